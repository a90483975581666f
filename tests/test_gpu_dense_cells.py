"""Dense cells at the edges of their size classes, with groups outside the
fullest sub-cell's, through both launch shapes (one launch with 1024 threads
per cell up to 3 * 2^20 particles, two size classes above), against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2003_11468_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [255, 256, 257, 700, 768, 769, 1500, 3071, 3072, 3073]


def _cells(seed, nc, box, l_x, sizes, n_bg):
    """Cells of the given sizes: a clump, a few small groups and loose particles
    spread over the whole cell (some beyond the clump's reach), on a sparse
    background, with dense cells side by side and at the periodic faces."""
    rng = np.random.default_rng(seed)
    h = box / nc
    parts = [rng.uniform(0.0, box, size=(n_bg, 3))]
    for k, m in enumerate(sizes):
        c = np.array([(3 * k) % nc, (nc - 1) if k % 3 == 0 else (k // 2) % nc, (5 * k) % nc])
        for side in range(2):                            # two dense neighbours along x
            cell = (c + [side, 0, 0]) % nc
            n_loose = max(8, m // 20)
            n_small = max(8, m // 10)
            centre = rng.uniform(0.2, 0.8, 3) * h
            clump = centre + rng.normal(scale=0.11 * h, size=(m - n_loose - n_small, 3))
            knots = rng.uniform(0.02, 0.98, size=(4, 3)) * h
            small = knots[rng.integers(0, 4, n_small)] + rng.uniform(-0.2, 0.2, size=(n_small, 3)) * l_x
            loose = rng.uniform(0.0, 1.0, size=(n_loose, 3)) * h
            inside = np.clip(np.concatenate([clump, small, loose]), 1e-4 * h, (1 - 1e-4) * h)
            parts.append(cell * h + inside)
    pos = np.concatenate(parts)
    return np.ascontiguousarray(pos[rng.permutation(len(pos))] % box, dtype=np.float32)


@pytest.mark.parametrize("l_over_h", [0.22, 0.30, 0.45])     # several sub-cells per cell axis
@pytest.mark.parametrize("large", [False, True])
def test_dense_cells(cuda_lib, l_over_h, large):
    import torch
    fof = cuda_lib
    nc, box = 16, 8.0
    l_x = l_over_h * box / nc
    pos = _cells(int(100 * l_over_h), nc, box, l_x, SIZES, 4000)
    pos[pos >= np.float32(box)] = 0.0
    n = len(pos)
    wid, wsz = oracle.groups(pos, box, l_x)
    assert fof.fof_box_geometry(box, l_x, n, _opt(fof, nc)).sub_cells > 1
    dpos = torch.from_numpy(pos).cuda()
    if large:                                                # a second, sparse box: past 3 * 2^20 particles
        m = (3 << 20) + 1
        filler = torch.from_numpy(synth.uniform_box(m, 50.0, seed=8)).cuda()
        plan = fof.FoFBatch([box, 50.0], [l_x, 0.005], [n, m], _opt(fof, nc))
        ids, sizes, _, ng, _ = plan.run(torch.cat([dpos, filler]))
        ng = ng[0]
    else:
        plan = fof.FoF(box, l_x, n, _opt(fof, nc))
        ids, sizes, _, ng = plan.run(dpos)
    plan.close()
    assert np.array_equal(ids[:n].cpu().numpy(), wid)
    assert np.array_equal(sizes[:n].cpu().numpy(), wsz)
    assert ng == int((wsz > 0).sum())


def _opt(fof, nc):
    o = fof.fof_options()
    o.cells_per_axis = nc
    return o
