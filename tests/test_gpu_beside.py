"""On both sides of the size up to which kernels run beside one another (2^26
particles): runs back to back, whose kernels may overlap, give the bits of a run
with timing events between its kernels, where none can."""
import pytest

from paper_2003_11468_gb300 import synth
from test_gpu_dependent_launches import _buffers, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1 << 26, (1 << 26) + 1])
def test_same_bits_with_and_without_overlap(cuda_lib, n):
    import torch
    fof = cuda_lib
    box = 50.0
    pos, = _inputs(n, box, 1, 77)
    s = torch.cuda.current_stream()
    with fof.FoF(box, synth.linking_length(n, box, 0.1), n) as plan:
        fof.fof_set_timing(plan.h, True)
        ids, sizes, _, ng = plan.run(pos, min_size=2)
        fof.fof_set_timing(plan.h, False)
        out = _buffers(n, 3)
        for i, z in out:
            fof.fof_link(plan.h, pos, s)
            fof.fof_groups_async(plan.h, i, z, None, 0, 2, s)
        code, got, _ = fof.fof_result(plan.h, 1, s)
        assert code == 0 and got[0] == ng
        for i, z in out:
            assert torch.equal(i, ids) and torch.equal(z, sizes)
