"""Team cells in the largest boxes, where squared distances overflow float32 and
every pair takes the exact test: the places of a row block beyond the cell's
particles link to nothing there either."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


# sizes off the multiples of 8 and of 32 that the blocks are padded to; one warp
# per cell and, above 128, one CTA
@pytest.mark.parametrize("m", [10, 13, 31, 33, 41, 100, 127, 129, 161, 250])
@pytest.mark.parametrize("nc", [2, 3, 5])
@pytest.mark.parametrize("box", [1e30, 3e20])
def test_padding_links_nothing(cuda_lib, m, nc, box):
    import torch
    fof = cuda_lib
    rng = np.random.default_rng(m * nc)
    l_x = 0.18 * box / nc
    # the cell at the origin and the last one, so that padding that linked would
    # join other cells' particles
    corner = rng.uniform(0.0, 0.9, (m, 3)) * box / nc
    last = (nc - 1 + rng.uniform(0.1, 0.9, (m, 3))) * box / nc
    loose = rng.uniform(0.0, 1.0, (40, 3)) * box
    pos = np.concatenate([corner, last, loose]).astype(np.float32)
    pos[pos >= box] = 0.0
    pos = np.ascontiguousarray(pos[rng.permutation(len(pos))])
    wid, wsz = oracle.groups(pos, box, l_x)
    opt = fof.fof_options()
    opt.cells_per_axis = nc
    with fof.FoF(box, l_x, len(pos), opt) as plan:
        ids, sizes, _, ng = plan.run(torch.from_numpy(pos).cuda())
    assert np.array_equal(ids.cpu().numpy(), wid) and np.array_equal(sizes.cpu().numpy(), wsz)
    assert ng == int((wsz > 0).sum())
