"""fof_relink where particles change cells inside their bricks (path 1): the sort
runs again on the kept brick order, with the kept list of full bricks."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _box(seed, nb, box, full):
    """`full` particles in each of two bricks, clumped and spread, and a thin
    background; every particle well inside its brick."""
    rng = np.random.default_rng(seed)
    h = box / nb
    parts = []
    for k in range(2):
        c = np.array([k + 1, nb - 1 - k, k])
        clump = rng.uniform(0.2, 0.8, (6, 3))[rng.integers(0, 6, full // 2)] + rng.normal(scale=0.02, size=(full // 2, 3))
        p = np.concatenate([clump, rng.uniform(0.0, 1.0, (full - full // 2, 3))])
        parts.append((c + np.clip(p, 0.05, 0.95)) * h)
    b = rng.integers(0, nb, (6_000, 3))
    parts.append((b + rng.uniform(0.05, 0.95, (6_000, 3))) * h)
    pos = np.concatenate(parts)
    pos = pos[rng.permutation(len(pos))]
    brick = np.floor(pos / h)
    return pos, brick, h


# with and without full bricks (above 8,192 particles in a plan above 65,535)
@pytest.mark.parametrize("full", [3_000, 8_193, 40_000])
@pytest.mark.parametrize("r", [4, 8])
def test_cells_change_inside_bricks(cuda_lib, full, r):
    import torch
    fof = cuda_lib
    nb, box = 5, 10.0
    pos, brick, h = _box(full + r, nb, box, full)
    rng = np.random.default_rng(9)
    l_x = 0.25 * h / 16
    n = len(pos)
    opt = fof.fof_options()
    opt.cells_per_axis, opt.brick_cells = nb * r, r
    ids, sizes = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    with fof.FoF(box, l_x, n, opt) as plan:
        assert fof.fof_plan_info(plan.h) == (nb * r, r, nb)
        fof.fof_link(plan.h, torch.from_numpy(pos.astype(np.float32)).cuda())
        fof.fof_groups(plan.h, ids, sizes, None, 0, 1)
        for step in range(3):
            # anywhere in the brick but for its faces: many particles change cells,
            # and cells change lists
            u = pos / h - brick
            u = 0.5 + (u - 0.5) * rng.uniform(0.7, 1.1) + rng.normal(scale=0.1, size=u.shape)
            pos = (brick + np.clip(u, 0.05, 0.95)) * h
            p32 = np.ascontiguousarray(pos.astype(np.float32))
            assert fof.fof_relink(plan.h, torch.from_numpy(p32).cuda()) == 1
            fof.fof_groups(plan.h, ids, sizes, None, 0, 1)
            wid, wsz = oracle.groups(p32, box, l_x)
            assert np.array_equal(ids.cpu().numpy(), wid), step
            assert np.array_equal(sizes.cpu().numpy(), wsz), step
