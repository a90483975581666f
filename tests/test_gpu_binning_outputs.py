"""Binning and outputs at the edges of their tiles and on both sides of the
sizes that choose a kernel, against the CPU oracle or against the other
kernel.  The partition is exact, so everything is compared bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2003_11468_gb300 import synth

pytestmark = pytest.mark.gpu


def _run(fof, h, pos, n, min_size, link=True, cap=None):
    import torch
    cap = n if cap is None else cap
    ids = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    sizes = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    cat = torch.full((max(cap, 1), 2), -7, dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream()
    if link:
        fof.fof_link(h, pos, s)
    code, ng, nk = fof.fof_groups(h, ids, sizes, cat, cap, min_size, 1, s, allow_capacity=True)
    return code, ids.cpu().numpy(), sizes.cpu().numpy(), cat.cpu().numpy()[:min(nk[0], cap)], ng[0], nk[0]


def _check(got, want, min_size):
    wid, wsz = want
    code, ids, sizes, cat, ng, nk = got
    wcat = oracle.catalogue(wsz, min_size)
    assert code == 0
    assert np.array_equal(ids, wid) and np.array_equal(sizes, wsz)
    assert nk == wcat.shape[0] and np.array_equal(cat, wcat)
    assert ng == int((wsz > 0).sum())


# edges of the warp, the binning tiles (1024, 4096, 8192) and the output tile
# (4096); 140,000 particles are 35 output tiles (the look-back's second round)
@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1025, 4095, 4096, 4097, 8191, 8193, 140_001])
def test_tile_edges(cuda_lib, n):
    import torch
    fof = cuda_lib
    box = 7.0
    pos = synth.clustered_box(n, box, max(1, n // 800), seed=700 + n)
    l_x = synth.linking_length(n, box) if n > 1 else 0.5
    want = oracle.groups(pos, box, l_x)
    with fof.FoF(box, l_x, n) as plan:
        dpos = torch.from_numpy(pos).cuda()
        for min_size in (1, 20):
            _check(_run(fof, plan.h, dpos, n, min_size), want, min_size)


# chunks of one to four tiles of 256 slots per CTA of the output scatter, with
# ragged last chunks: 152 SMs x 8 CTAs x 256 slots are 311,296
@pytest.mark.parametrize("n", [311_295, 622_593, 934_145, 1_245_183, 1_556_737])
def test_output_chunk_edges(cuda_lib, n):
    import torch
    fof = cuda_lib
    box = 40.0
    pos = synth.uniform_box(n, box, seed=900 + n)
    l_x = synth.linking_length(n, box)
    want = oracle.groups(pos, box, l_x)
    with fof.FoF(box, l_x, n) as plan:
        _check(_run(fof, plan.h, torch.from_numpy(pos).cuda(), n, 2), want, 2)


# bricks of one cell: counters a line apart and counted per tile in shared
# memory (up to 12,288), a sector apart (up to 131,072), side by side
@pytest.mark.parametrize("nc", [23, 24, 50, 51])
@pytest.mark.parametrize("shuffled", [False, True])
def test_brick_counters(cuda_lib, nc, shuffled):
    import torch
    fof = cuda_lib
    n, box = 60_000, 3.0
    pos = synth.clustered_box(n, box, 9, seed=77)
    if shuffled:
        pos = pos[np.random.default_rng(5).permutation(n)]
    l_x = synth.linking_length(n, box)
    opt = fof.fof_options()
    opt.cells_per_axis, opt.brick_cells = nc, 1
    want = oracle.groups(pos, box, l_x)
    with fof.FoF(box, l_x, n, opt) as plan:
        _check(_run(fof, plan.h, torch.from_numpy(pos).cuda(), n, 2), want, 2)


def test_direct_and_bucketed_outputs_agree(cuda_lib):
    """2^24 inputs store their pairs directly; with one more small box in the
    plan the same box goes through the buckets."""
    import torch
    fof = cuda_lib
    n, box = 1 << 24, 100.0
    l_x = synth.linking_length(n, box)
    g = torch.Generator(device="cuda").manual_seed(3)
    pos = torch.rand((n, 3), generator=g, device="cuda") * 99.9
    pos[: n // 4] = pos[: n // 4] * 0.3                    # a denser corner: larger groups
    pos = pos[torch.randperm(n, generator=g, device="cuda")].contiguous()
    with fof.FoF(box, l_x, n) as plan:
        one = plan.run(pos, min_size=3)
    small = torch.rand((5, 3), generator=g, device="cuda")
    with fof.FoF(1.0, 0.3, 5) as plan:
        tiny = plan.run(small, min_size=3)
    batch = fof.FoFBatch([box, 1.0], [l_x, 0.3], [n, 5])
    try:
        ids, sizes, cat, ng, nk = batch.run(torch.cat([pos, small]), min_size=3)
    finally:
        batch.close()
    assert torch.equal(ids[:n], one[0]) and torch.equal(sizes[:n], one[1])
    assert torch.equal(ids[n:], tiny[0]) and torch.equal(sizes[n:], tiny[1])
    assert torch.equal(cat, torch.cat([one[2], tiny[2]]))
    assert ng == [one[3], tiny[3]] and nk == [len(one[2]), len(tiny[2])]


def test_outputs_after_link_relink_and_graph(cuda_lib):
    """Each fof_groups starts from zero counts, whether it follows fof_link,
    fof_relink or a graph replay in between; a catalogue too small for its
    rows is cut."""
    import torch
    fof = cuda_lib
    n, box = 30_011, 5.0
    l_x = synth.linking_length(n, box)
    pos = synth.clustered_box(n, box, 30, seed=41)
    want = oracle.groups(pos, box, l_x)
    dpos = torch.from_numpy(pos).cuda()
    with fof.FoF(box, l_x, n) as plan:
        _check(_run(fof, plan.h, dpos, n, 20), want, 20)
        _check(_run(fof, plan.h, dpos, n, 2), want, 2)
        assert fof.fof_relink(plan.h, dpos) == 0
        _check(_run(fof, plan.h, dpos, n, 1, link=False), want, 1)
        s = torch.cuda.Stream()
        out = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        fof.fof_link(plan.h, dpos, s)
        fof.fof_graph_build(plan.h, dpos, out[0], out[1], None, 0, 2, s)
        fof.fof_graph_launch(plan.h, s)
        fof.fof_result(plan.h, 1, s)
        assert np.array_equal(out[0].cpu().numpy(), want[0]) and np.array_equal(out[1].cpu().numpy(), want[1])
        _check(_run(fof, plan.h, dpos, n, 5), want, 5)
        code, _, _, cat, _, nk = _run(fof, plan.h, dpos, n, 2, cap=7)
        wcat = oracle.catalogue(want[1], 2)
        assert code == fof.FOF_ERR_CAPACITY and nk == len(wcat) and np.array_equal(cat, wcat[:7])
