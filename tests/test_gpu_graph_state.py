"""A graph that was built and not launched has run nothing: the plan answers as
before the build, and as after a link once it has been launched."""
import numpy as np
import pytest

import oracle
from paper_2003_11468_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture
def case(cuda_lib):
    import torch
    n, box = 90_000, 20.0
    pos = synth.clustered_box(n, box, 60, seed=12)
    l_x = synth.linking_length(n, box)
    other = np.ascontiguousarray(pos[::-1])
    ids, sizes = (torch.full((n,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    want = [oracle.groups(p, box, l_x) for p in (pos, other)]
    dev = [torch.from_numpy(p).cuda() for p in (pos, other)]
    torch.cuda.synchronize()
    with cuda_lib.FoF(box, l_x, n) as plan:
        yield plan, dev, want, ids, sizes, torch.cuda.Stream()


def _same(ids, sizes, want):
    return np.array_equal(ids.cpu().numpy(), want[0]) and np.array_equal(sizes.cpu().numpy(), want[1])


def test_built_on_a_new_plan(cuda_lib, case):
    fof = cuda_lib
    plan, dev, want, ids, sizes, s = case
    fof.fof_graph_build(plan.h, dev[0], ids, sizes, None, 0, 2, s)
    with pytest.raises(fof.FoFError) as e:
        fof.fof_groups(plan.h, ids, sizes, None, 0, 2, 1, s)
    assert e.value.code == fof.FOF_ERR_STATE
    assert fof.fof_relink(plan.h, dev[1], s) == 2        # no binning to re-use
    fof.fof_groups(plan.h, ids, sizes, None, 0, 2, 1, s)
    assert _same(ids, sizes, want[1])


def test_launched_then_relinked(cuda_lib, case):
    import torch
    fof = cuda_lib
    plan, dev, want, ids, sizes, s = case
    fof.fof_graph_build(plan.h, dev[0], ids, sizes, None, 0, 2, s)
    fof.fof_graph_launch(plan.h, s)
    code, _, _ = fof.fof_result(plan.h, 1, s)
    assert code == 0 and _same(ids, sizes, want[0])
    assert fof.fof_relink(plan.h, dev[0], s) == 0
    ids.fill_(-7)
    torch.cuda.synchronize()
    fof.fof_groups(plan.h, ids, sizes, None, 0, 2, 1, s)
    assert _same(ids, sizes, want[0])


def test_built_between_link_and_groups(cuda_lib, case):
    fof = cuda_lib
    plan, dev, want, ids, sizes, s = case
    fof.fof_link(plan.h, dev[1], s)
    fof.fof_graph_build(plan.h, dev[0], ids, sizes, None, 0, 2, s)
    fof.fof_groups(plan.h, ids, sizes, None, 0, 2, 1, s)
    assert _same(ids, sizes, want[1])
    fof.fof_groups_async(plan.h, ids, sizes, None, 0, 2, s)
    fof.fof_graph_build(plan.h, dev[0], ids, sizes, None, 0, 2, s)
    code, ng, _ = fof.fof_result(plan.h, 1, s)           # of the call before the build
    assert code == 0 and ng[0] == int((want[1][1] > 0).sum())
