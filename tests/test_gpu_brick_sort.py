"""Bricks at the edges of the sort kernels: around the records copied ahead
(768) and the size that goes to a cluster of CTAs (8,192), few and many cells
per brick, on both sides of the plan size that skips the cluster kernel
(65,535), against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _bricks(seed, nb, box, sizes, n_bg):
    """Bricks holding the given numbers of particles, spread and clumped."""
    rng = np.random.default_rng(seed)
    h = box / nb
    parts = [rng.uniform(0.0, box, (n_bg, 3))] if n_bg else []
    for k, m in enumerate(sizes):
        c = np.array([k % nb, (k // nb) % nb, (nb - 1 - k) % nb])
        spread = rng.uniform(0.01, 0.99, (m - m // 3, 3))
        clump = rng.uniform(0.1, 0.9, 3) + rng.normal(scale=0.04, size=(m // 3, 3))
        p = np.clip(np.concatenate([spread, clump]), 1e-3, 1 - 1e-3)
        parts.append((c + p) * h)
    pos = np.concatenate(parts)
    pos = np.ascontiguousarray(pos[rng.permutation(len(pos))] % box, dtype=np.float32)
    pos[pos >= np.float32(box)] = 0.0
    return pos


# cells per brick side 1, 2, 4, 8, 16
@pytest.mark.parametrize("r", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("sizes,n_bg", [((767, 768, 769, 1025), 300), ((8191, 8192, 8193, 12000, 30000), 500),
                                        ((8193, 40000, 20000, 9000), 3000)])
def test_brick_sizes(cuda_lib, r, sizes, n_bg):
    import torch
    fof = cuda_lib
    nb, box = 4, 4.0
    pos = _bricks(10 * r + len(sizes), nb, box, sizes, n_bg)
    n = len(pos)
    l_x = 0.3 * box / (nb * 16)
    wid, wsz = oracle.groups(pos, box, l_x)
    opt = fof.fof_options()
    opt.cells_per_axis, opt.brick_cells = nb * r, r
    with fof.FoF(box, l_x, n, opt) as plan:
        dpos = torch.from_numpy(pos).cuda()
        for _ in range(2):                                    # the second call on a used workspace
            ids, sz, _, ng = plan.run(dpos)
            assert np.array_equal(ids.cpu().numpy(), wid)
            assert np.array_equal(sz.cpu().numpy(), wsz)
            assert ng == int((wsz > 0).sum())


def test_batch_of_uneven_bricks(cuda_lib):
    """Boxes of 1 to 16 cells per brick side in one plan: cell tables that start
    off a 16-byte boundary, skipped and listed bricks in turn."""
    import torch
    fof = cuda_lib
    rng = np.random.default_rng(11)
    ns = [1, 3, 7, 30, 500, 4000, 70000, 2, 12000, 90]
    boxes = [float(b) for b in rng.uniform(0.5, 3.0, len(ns))]
    poss, lxs = [], []
    for k, (m, L) in enumerate(zip(ns, boxes)):
        p = rng.uniform(0.0, L, (m, 3))
        if m > 1000:
            p[: m // 3] = L * (0.4 + 0.02 * rng.normal(size=(m // 3, 3)))
        p = np.float32(p % L)
        p[p >= np.float32(L)] = 0.0
        poss.append(p)
        lxs.append(0.2 * L / max(m, 8) ** (1 / 3))
    plan = fof.FoFBatch(boxes, lxs, ns)
    ids, sizes, _, ng, _ = plan.run(torch.from_numpy(np.concatenate(poss)).cuda())
    plan.close()
    ids, sizes = ids.cpu().numpy(), sizes.cpu().numpy()
    at = 0
    for k, m in enumerate(ns):
        wid, wsz = oracle.groups(poss[k], boxes[k], lxs[k])
        assert np.array_equal(ids[at:at + m], wid) and np.array_equal(sizes[at:at + m], wsz)
        assert ng[k] == int((wsz > 0).sum())
        at += m
