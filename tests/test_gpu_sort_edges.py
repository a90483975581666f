"""Bricks at the edges of what the sort copies ahead into shared memory (512
records) and of its later rounds (512 more each), against the oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_brick_sort import _bricks

pytestmark = pytest.mark.gpu


# plans below and above 65,535 particles (there the full bricks' kernel runs before)
@pytest.mark.parametrize("n_bg", [0, 70_000])
@pytest.mark.parametrize("r", [1, 4, 16])
@pytest.mark.parametrize("sizes", [(511, 512, 513), (1023, 1024, 1025), (1535, 1536, 1537, 2047, 2048, 2049)])
def test_brick_sizes(cuda_lib, r, sizes, n_bg):
    import torch
    fof = cuda_lib
    nb, box = 16, 16.0
    pos = _bricks(r + len(sizes), nb, box, sizes, 0)
    h = box / nb
    if n_bg:                                  # outside the bricks under test
        rng = np.random.default_rng(n_bg)
        bg = rng.uniform(0.0, box, (n_bg, 3))
        inside = np.zeros(n_bg, dtype=bool)
        for k in range(len(sizes)):
            inside |= (np.floor(bg / h) == [k % nb, (k // nb) % nb, nb - 1 - k]).all(axis=1)
        pos = np.concatenate([pos, bg[~inside].astype(np.float32)])
    count = np.unique(np.floor(pos / np.float32(h)), axis=0, return_counts=True)[1]
    assert set(sizes) <= set(count.tolist())
    n = len(pos)
    l_x = 0.3 * h / 16
    opt = fof.fof_options()
    opt.cells_per_axis, opt.brick_cells = nb * r, r
    wid, wsz = oracle.groups(pos, box, l_x)
    with fof.FoF(box, l_x, n, opt) as plan:
        for _ in range(2):
            ids, sz, _, ng = plan.run(torch.from_numpy(pos).cuda())
            assert np.array_equal(ids.cpu().numpy(), wid) and np.array_equal(sz.cpu().numpy(), wsz)
            assert ng == int((wsz > 0).sum())
