"""Team cells at the edges of the kernel's row blocks (32), of its two classes
(128) and of its range, sorted by z bin or not, with several groups per cell,
against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SIZES = [9, 10, 11, 24, 25, 26, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 160, 161, 224, 225, 254, 255]


def _cells(seed, nc, box, spread, layered):
    """Each cell holds a few strands through the whole cell and loose particles;
    layered: z takes few values, so bins are full and ties abound."""
    rng = np.random.default_rng(seed)
    h = box / nc
    parts = []
    for k, m in enumerate(SIZES):
        c = np.array([k % nc, (k // nc) % nc, (nc - 1 - k) % nc])
        n_strand = m // 2
        a, b = rng.uniform(0.0, 1.0, (2, 3))
        t = rng.uniform(0.0, 1.0, (n_strand, 1))
        strand = a + t * (b - a) + rng.normal(scale=spread, size=(n_strand, 3))
        p = np.concatenate([strand, rng.uniform(0.0, 1.0, (m - n_strand, 3))])
        if layered:
            p[:, 2] = rng.choice([0.001, 0.24, 0.26, 0.5, 0.75, 0.999], size=m)
        parts.append((c + np.clip(p, 1e-3, 1 - 1e-3)) * h)
    parts.append(rng.uniform(0.0, box, size=(500, 3)))
    pos = np.concatenate(parts)
    return np.ascontiguousarray(pos[rng.permutation(len(pos))] % box, dtype=np.float32)


# 2 cells per axis: every separation may wrap; 5 and 16: plain separations
@pytest.mark.parametrize("nc", [2, 5, 16])
@pytest.mark.parametrize("l_over_h", [0.12, 0.3, 0.6])
@pytest.mark.parametrize("layered", [False, True])
def test_team_cells(cuda_lib, nc, l_over_h, layered):
    import torch
    fof = cuda_lib
    box = 4.0
    l_x = l_over_h * box / nc
    pos = _cells(1000 * nc + int(100 * l_over_h), nc, box, 0.04, layered)
    pos[pos >= np.float32(box)] = 0.0
    wid, wsz = oracle.groups(pos, box, l_x)
    opt = fof.fof_options()
    opt.cells_per_axis = nc
    with fof.FoF(box, l_x, len(pos), opt) as plan:
        ids, sizes, _, ng = plan.run(torch.from_numpy(pos).cuda())
    assert np.array_equal(ids.cpu().numpy(), wid)
    assert np.array_equal(sizes.cpu().numpy(), wsz)
    assert ng == int((wsz > 0).sum())
