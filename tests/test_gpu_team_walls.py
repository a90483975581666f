"""Team cells in boxes of two cells per axis, where every separation may wrap, at
the sizes of the kernel's row blocks, its two classes and its range: one listed
size per cell and nothing else in it, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# one box each: the eight cells hold these
SIZES = [(10, 11, 16, 17, 18, 31, 32, 33), (63, 64, 65, 95, 96, 97, 127, 128),
         (128, 129, 130, 159, 160, 161, 192, 193), (224, 225, 254, 255, 256, 256, 128, 12),
         (256, 129, 97, 33, 255, 160, 128, 65)]


def _cells(seed, sizes, nc, box, layered):
    """Strands through the whole cell, so that links run through the cell's faces
    and round the box, and loose particles; layered: few values of z."""
    rng = np.random.default_rng(seed)
    h = box / nc
    parts = []
    for k, m in enumerate(sizes):
        c = np.array([k % nc, (k // nc) % nc, (k // nc ** 2) % nc])
        a, b = rng.uniform(0.0, 1.0, (2, 3))
        t = rng.uniform(0.0, 1.0, (m // 2, 1))
        strand = a + t * (b - a) + rng.normal(scale=0.03, size=(m // 2, 3))
        p = np.concatenate([strand, rng.uniform(0.0, 1.0, (m - m // 2, 3))])
        if layered:
            p[:, 2] = rng.choice([0.001, 0.24, 0.26, 0.5, 0.75, 0.999], size=m)
        parts.append((c + np.clip(p, 1e-3, 1 - 1e-3)) * h)
    pos = np.concatenate(parts)
    return np.ascontiguousarray(pos[rng.permutation(len(pos))], dtype=np.float32)


# 2 cells per axis: the wrapped separations; 3: the plain ones, with every cell's
# neighbours on both sides the same
@pytest.mark.parametrize("nc", [2, 3])
@pytest.mark.parametrize("l_over_h", [0.08, 0.2, 0.5])
@pytest.mark.parametrize("layered", [False, True])
@pytest.mark.parametrize("sizes", SIZES)
def test_cells_of_listed_sizes(cuda_lib, nc, l_over_h, layered, sizes):
    import torch
    fof = cuda_lib
    box = 4.0
    l_x = l_over_h * box / nc
    pos = _cells(sum(sizes) + nc, sizes, nc, box, layered)
    held = np.unique(np.floor(pos / np.float32(box / nc)), axis=0, return_counts=True)[1]
    assert sorted(held.tolist()) == sorted(sizes)
    opt = fof.fof_options()
    opt.cells_per_axis, opt.dense_min = nc, 3000          # every cell a team cell
    wid, wsz = oracle.groups(pos, box, l_x)
    with fof.FoF(box, l_x, len(pos), opt) as plan:
        assert fof.fof_plan_info(plan.h)[0] == nc
        ids, sz, _, ng = plan.run(torch.from_numpy(pos).cuda())
    assert np.array_equal(ids.cpu().numpy(), wid) and np.array_equal(sz.cpu().numpy(), wsz)
    assert ng == int((wsz > 0).sum())
