"""Runs back to back, without a wait between them, on one and on several
streams, on both sides of the sizes that choose dependent launches (2^22) and
kernels beside each other (2^26): every run gives the same bits as a run alone."""
import threading

import numpy as np
import pytest

import oracle
from paper_2003_11468_gb300 import synth

pytestmark = pytest.mark.gpu


def _inputs(n, box, count, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for _ in range(count):                                # a third in a few clumps: heavy bricks, dense cells
        p = torch.rand((n, 3), generator=g, device="cuda") * (box * 0.999)
        k = n // 3
        c = torch.rand((12, 3), generator=g, device="cuda") * box * 0.9
        p[:k] = (c[torch.arange(k, device="cuda") % 12] + torch.randn((k, 3), generator=g, device="cuda") *
                 (box * 0.004)).remainder(box * 0.999)
        out.append(p[torch.randperm(n, generator=g, device="cuda")].contiguous())
    return out


def _buffers(n, count):
    import torch
    return [tuple(torch.full((n,), -5, dtype=torch.int32, device="cuda") for _ in range(2)) for _ in range(count)]


@pytest.mark.parametrize("n", [5_000, 300_000, 1 << 22, (1 << 22) + 1])
def test_back_to_back(cuda_lib, n):
    import torch
    fof = cuda_lib
    box = 10.0
    l_x = synth.linking_length(n, box)
    poss = _inputs(n, box, 3, n)
    with fof.FoF(box, l_x, n) as plan:
        alone = []
        for p in poss:
            torch.cuda.synchronize()
            ids, sizes, _, ng = plan.run(p, min_size=2)
            torch.cuda.synchronize()
            alone.append((ids, sizes, ng))
        if n <= 300_000:
            wid, wsz = oracle.groups(poss[0].cpu().numpy(), box, l_x)
            assert np.array_equal(alone[0][0].cpu().numpy(), wid) and np.array_equal(alone[0][1].cpu().numpy(), wsz)
        s = torch.cuda.current_stream()
        rounds = 6
        out = _buffers(n, 3 * rounds)
        for k in range(3 * rounds):                       # nothing waits until the end
            fof.fof_link(plan.h, poss[k % 3], s)
            fof.fof_groups_async(plan.h, out[k][0], out[k][1], None, 0, 2, s)
        code, ng, _ = fof.fof_result(plan.h, 1, s)
        assert code == 0 and ng[0] == alone[(3 * rounds - 1) % 3][2]
        for k, (ids, sizes) in enumerate(out):
            assert torch.equal(ids, alone[k % 3][0]) and torch.equal(sizes, alone[k % 3][1])


def test_threads_and_streams(cuda_lib):
    """Four threads, each with its own plan, stream and input, at the same time."""
    import torch
    fof = cuda_lib
    jobs = []
    for k, n in enumerate([4_001, 90_000, 700_000, 5_000_000]):
        box = 8.0
        l_x = synth.linking_length(n, box)
        pos = _inputs(n, box, 1, 50 + k)[0]
        plan = fof.FoF(box, l_x, n)
        want = plan.run(pos, min_size=2)
        jobs.append((plan, pos, want, torch.cuda.Stream(), _buffers(n, 12)))
    torch.cuda.synchronize()
    errors = []

    def work(plan, pos, want, stream, out):
        try:
            for ids, sizes in out:
                fof.fof_link(plan.h, pos, stream)
                fof.fof_groups_async(plan.h, ids, sizes, None, 0, 2, stream)
            code, ng, _ = fof.fof_result(plan.h, 1, stream)
            assert code == 0 and ng[0] == want[3]
        except BaseException as e:                        # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for plan, _, want, _, out in jobs:
        for ids, sizes in out:
            assert torch.equal(ids, want[0]) and torch.equal(sizes, want[1])
        plan.close()
