"""Plans of very many small boxes: each box gives what it gives alone, and the
brick sort takes a time that follows the bricks, not the boxes before them."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _sort_ms(fof, plan, pos, n, nbox):
    import torch
    ids, sizes = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    best = np.inf
    fof.fof_set_timing(plan.h, True)
    for _ in range(4):
        fof.fof_reset_times(plan.h)
        fof.fof_link(plan.h, pos)
        fof.fof_groups(plan.h, ids, sizes, None, 0, 1, nbox)
        best = min(best, fof.fof_phase_times(plan.h)["brick_sort"][0])
    return best, ids, sizes


def test_a_million_boxes(cuda_lib):
    import torch
    fof = cuda_lib
    nbox, per, l_x = 1_000_000, 2, 0.2
    n = nbox * per
    g = torch.Generator("cuda").manual_seed(6)
    pos = torch.rand((n, 3), generator=g, device="cuda") * 0.999
    plan = fof.FoFBatch([1.0] * nbox, [l_x] * nbox, [per] * nbox)
    nc, r, nb = fof.fof_plan_info(plan.h, 0)
    many, ids, sizes = _sort_ms(fof, plan, pos, n, nbox)
    plan.close()
    host, ids, sizes = pos.cpu().numpy(), ids.cpu().numpy(), sizes.cpu().numpy()
    for b in [0, 1, 607, 608, nbox // 2, nbox - 1, *np.random.default_rng(1).integers(0, nbox, 200)]:
        at = slice(b * per, (b + 1) * per)
        wid, wsz = oracle.groups(host[at], 1.0, l_x)
        assert np.array_equal(ids[at], wid) and np.array_equal(sizes[at], wsz)
    # as many bricks in one box; a box's own table and its search are a few loads
    # more per brick, each about a tenth of what a brick takes
    opt = fof.fof_options()
    opt.cells_per_axis, opt.brick_cells = 100, 1
    with fof.FoF(1.0, 1e-3, n, opt) as one:
        assert 100 ** 3 == nbox * nb ** 3
        single, _, _ = _sort_ms(fof, one, pos, n, 1)
    assert many < 3 * single, (many, single, nc, r, nb)
