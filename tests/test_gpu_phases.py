"""What fof_phase_times counts under each phase, and the launches it reports."""
import pytest

pytestmark = pytest.mark.gpu


def _run(fof, n, relinks=0):
    import torch
    box = 20.0
    pos = torch.rand((n, 3), generator=torch.Generator("cuda").manual_seed(n), device="cuda") * (box * 0.999)
    ids, sizes = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    with fof.FoF(box, 0.3 * box / n ** (1 / 3), n) as plan:
        fof.fof_set_timing(plan.h, True)
        fof.fof_link(plan.h, pos)
        fof.fof_groups(plan.h, ids, sizes, None, 0, 2)
        phases = [fof.fof_phase_times(plan.h)]
        for _ in range(relinks):
            fof.fof_reset_times(plan.h)
            assert fof.fof_relink(plan.h, pos) == 0
            phases.append(fof.fof_phase_times(plan.h))
    return phases


# up to 2^24 inputs the write of ids and sizes leaves the catalogue behind too;
# above, a scan and the catalogue's own kernel follow
@pytest.mark.parametrize("n,catalogue", [(5_000, 0), ((1 << 24) + 1, 2)])
def test_outputs_hold_both_output_kernels(cuda_lib, n, catalogue):
    phases, = _run(cuda_lib, n)
    assert phases["outputs"][1] == 2
    assert phases["catalogue"][1] == catalogue


# with and without the second sort kernel (plans above 65,535 particles)
@pytest.mark.parametrize("n,sorts", [(65_535, 1), (65_536, 2)])
def test_relink_in_place_counts_one_launch(cuda_lib, n, sorts):
    first, again = _run(cuda_lib, n, relinks=1)
    assert first["brick_sort"][1] == sorts
    assert again["brick_sort"][1] == 1        # the forest alone is started anew
