"""fof_groups more than once for one fof_link, and after graph replays: the
forest is flattened once, the outputs are written anew each time."""
import numpy as np
import pytest

import oracle
from paper_2003_11468_gb300 import synth

pytestmark = pytest.mark.gpu


def _buffers(n):
    import torch
    return (torch.full((n,), -7, dtype=torch.int32, device="cuda"),
            torch.full((n,), -7, dtype=torch.int32, device="cuda"),
            torch.full((n, 2), -7, dtype=torch.int32, device="cuda"))


def _expect(got, out, want, min_size):
    ids, sizes, cat = (t.cpu().numpy() for t in out)
    wid, wsz = want
    wcat = oracle.catalogue(wsz, min_size)
    code, ng, nk = got
    assert code == 0 and ng[0] == int((wsz > 0).sum()) and nk[0] == len(wcat)
    assert np.array_equal(ids, wid) and np.array_equal(sizes, wsz)
    assert np.array_equal(cat[:nk[0]], wcat)


def _box(n, seed):
    import torch
    box = 30.0
    pos = synth.clustered_box(n, box, max(1, n // 700), seed=seed)
    l_x = synth.linking_length(n, box)
    return box, l_x, torch.from_numpy(pos).cuda(), oracle.groups(pos, box, l_x)


# both size counts; one and several output tiles (4,096 inputs)
@pytest.mark.parametrize("size_count", [0, 1])
@pytest.mark.parametrize("n", [33, 4097, 150_001])
def test_again_after_one_link(cuda_lib, n, size_count):
    fof = cuda_lib
    box, l_x, pos, want = _box(n, n)
    opt = fof.fof_options()
    opt.size_count = size_count
    with fof.FoF(box, l_x, n, opt) as plan:
        for _ in range(2):
            fof.fof_link(plan.h, pos)
            for min_size in (2, 1, 20, 20):
                out = _buffers(n)
                _expect(fof.fof_groups(plan.h, *out, n, min_size), out, want, min_size)
        assert fof.fof_relink(plan.h, pos) == 0
        for min_size in (20, 2):
            out = _buffers(n)
            _expect(fof.fof_groups(plan.h, *out, n, min_size), out, want, min_size)


def test_again_above_the_direct_outputs(cuda_lib):
    """Outputs through buckets (above 2^24 inputs)."""
    import torch
    fof = cuda_lib
    n, box = (1 << 24) + 4097, 50.0
    pos = torch.rand((n, 3), generator=torch.Generator("cuda").manual_seed(5), device="cuda") * (box * 0.999)
    with fof.FoF(box, 0.5 * box / n ** (1 / 3), n) as plan:
        fof.fof_link(plan.h, pos)
        once = _buffers(n)
        want = fof.fof_groups(plan.h, *once, n, 2)
        for _ in range(2):
            out = _buffers(n)
            assert fof.fof_groups(plan.h, *out, n, 2) == want
            for a, b in zip(out, once):
                assert torch.equal(a, b)


def test_again_after_a_graph_launch(cuda_lib):
    import torch
    fof = cuda_lib
    n = 60_001
    box, l_x, pos, want = _box(n, 3)
    s = torch.cuda.Stream()
    with fof.FoF(box, l_x, n) as plan:
        out = _buffers(n)
        torch.cuda.synchronize()
        fof.fof_graph_build(plan.h, pos, *out, n, 20, s)
        for _ in range(2):
            fof.fof_graph_launch(plan.h, s)
            _expect(fof.fof_result(plan.h, 1, s), out, want, 20)
            for min_size in (2, 20):
                more = _buffers(n)
                torch.cuda.synchronize()
                _expect(fof.fof_groups(plan.h, *more, n, min_size, 1, s), more, want, min_size)


def test_captured_alone_and_replayed(cuda_lib):
    """The caller's own graphs: fof_groups_async alone, replayed several times, and
    fof_link with it, replayed between a link and a fof_groups outside."""
    import torch
    fof = cuda_lib
    n = 60_001
    box, l_x, pos, want = _box(n, 4)
    other = pos.flip(0).contiguous()
    s = torch.cuda.Stream()
    with fof.FoF(box, l_x, n) as plan:
        out = _buffers(n)
        fof.fof_link(plan.h, pos, s)
        alone, both = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(alone, stream=s):
            fof.fof_groups_async(plan.h, *out, n, 20, s)
        with torch.cuda.graph(both, stream=s):
            fof.fof_link(plan.h, other, s)
            fof.fof_groups_async(plan.h, *out, n, 20, s)

        def replay(graph):
            for t in out:
                t.fill_(-7)
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                graph.replay()
            s.synchronize()

        for _ in range(3):
            replay(alone)
            assert np.array_equal(out[0].cpu().numpy(), want[0]) and np.array_equal(out[1].cpu().numpy(), want[1])
        _expect(fof.fof_result(plan.h, 1, s), out, want, 20)
        fof.fof_link(plan.h, pos, s)
        replay(both)                          # the plan now holds the other order's groups
        flipped = oracle.groups(other.cpu().numpy(), box, l_x)
        assert np.array_equal(out[0].cpu().numpy(), flipped[0])
        assert np.array_equal(out[1].cpu().numpy(), flipped[1])
        more = _buffers(n)
        torch.cuda.synchronize()
        _expect(fof.fof_groups(plan.h, *more, n, 20, 1, s), more, flipped, 20)
