"""k_link's windows of 32 slots: several warps per window (small problems), one
warp with tickets of one or more windows (large ones), ragged ends of both,
against the oracle or between the two."""
import numpy as np
import pytest

import oracle
from paper_2003_11468_gb300 import synth

pytestmark = pytest.mark.gpu


# 8, 8, 8, 4, 2, 2 and 1 warps per window, one window each up to 389,120 particles, then tickets
@pytest.mark.parametrize("n", [33, 1_000, 9_727, 16_000, 32_000, 64_000, 100_000, 389_119, 389_153])
@pytest.mark.parametrize("b", [0.2, 0.5])
def test_small(cuda_lib, n, b):
    import torch
    fof = cuda_lib
    box = 5.0
    l_x = synth.linking_length(n, box, b)
    pos = synth.clustered_box(n, box, max(1, n // 1500), seed=n)
    wid, wsz = oracle.groups(pos, box, l_x)
    with fof.FoF(box, l_x, n) as plan:
        for _ in range(3):
            ids, sizes, _, ng = plan.run(torch.from_numpy(pos).cuda())
            assert np.array_equal(ids.cpu().numpy(), wid) and np.array_equal(sizes.cpu().numpy(), wsz)
            assert ng == int((wsz > 0).sum())


@pytest.mark.parametrize("n", [38_913, 320_001])
def test_batched_with_filler(cuda_lib, n):
    """The same box alone and in a plan of 40 million particles (tickets of
    several windows, other launch shapes in every kernel)."""
    import torch
    fof = cuda_lib
    box = 9.0
    l_x = synth.linking_length(n, box)
    pos = torch.from_numpy(synth.clustered_box(n, box, n // 900, seed=n)).cuda()
    with fof.FoF(box, l_x, n) as plan:
        alone = plan.run(pos)
    m = 40_000_001
    g = torch.Generator(device="cuda").manual_seed(9)
    filler = torch.rand((m, 3), generator=g, device="cuda") * 99.9
    l_f = synth.linking_length(m, 100.0)
    plan = fof.FoFBatch([100.0, box], [l_f, l_x], [m, n])
    ids, sizes, _, ng, _ = plan.run(torch.cat([filler, pos]))
    plan.close()
    assert torch.equal(ids[m:], alone[0]) and torch.equal(sizes[m:], alone[1]) and ng[1] == alone[3]
