"""What a user of the group finder has it do, as timed cases.

Every case goes through the public entry points: a plan called on device
positions, the allocation-free call, host buffers (one snapshot, several
overlapped ones), a batch of uneven boxes replayed as one CUDA graph, time
steps re-linked on moved particles, and the server.  Positions follow the
repository's workloads (uniform boxes and Plummer-blob mixtures, the recipe of
synth.py), drawn on the GPU from the seed.  Sizes come from those workloads
(16^3..160^3 boxes of a batch, the 32^3 and 256^3 boxes, requests of 1e4
particles and more, and as much of the 1024^3 box as fits the card three
times over), with ragged sizes between them.

Outputs are whole numbers: group ids, group sizes, catalogue rows and counts.
How many rows a catalogue has depends on the input, so catalogues come back in
the caller's buffers, which hold zeros past the rows.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2003_11468_gb300 import fof
from paper_2003_11468_gb300.server import Server

EXACT_MAX = 40_000          # exact() compares every pair up to here
HOST_STEPS = 3              # snapshots of one overlapped host call


def _case(name, via, n, **kw):
    c = dict(name=name, via=via, n=n, boxes=1, box=100.0, b=0.2, kind="clustered", frac=0.5,
             order="generated", min_size=20, strict=False, move=0.0, n_top=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest box of a batch, on its own plan: latency of one small call
        _case("box_16", "box", 16 ** 3, box=50.0),
        # the small plain workload: 32^3 uniform particles in the unit box, pairs count
        _case("box_32_uniform", "box", 32 ** 3, box=1.0, kind="uniform", min_size=2),
        # inside a host application that owns all device memory: no allocation
        _case("noalloc_60k", "noalloc", 59_999, box=20.0),
        # one small job from pinned host buffers, results back on the host
        _case("host_300k", "host", 300_007, box=26.0),
        # a longer linking length, particles in no spatial order
        _case("box_2m_long", "box", 2_000_003, box=50.0, b=0.3, order="shuffled", min_size=32),
        # the middle plain workload: 256^3 particles, 20,000 blobs
        _case("box_256", "box", 256 ** 3),
        # the largest plain workload that fits three times over: 768^3 particles at the
        # 1024^3 box's blob density
        _case("box_768", "box", 768 ** 3),
        # many small boxes of uneven size in one graph replay: halo patches, zoom regions
        _case("batch_64_small", "batch", 16 ** 3, boxes=64, n_top=48 ** 3),
        # the batched workload: 512 boxes, 16^3..160^3 particles, one graph replay
        _case("batch_512", "batch", 16 ** 3, boxes=512, n_top=160 ** 3),
        # two time steps of a simulation that keeps its particles in cell order
        _case("relink_4m", "relink", 4_000_037, box=62.0, order="cells", move=0.01),
        # a run over snapshots in host memory, copies overlapped with the work
        _case("host_many_8m", "host_many", 8_000_009, box=78.0),
        # requests of very different sizes served together, host to host
        _case("served_16", "served", 10_000, boxes=16, n_top=10_000_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    via = rng.choice(["box", "box", "box", "noalloc", "host", "host_many", "batch", "batch", "relink", "served"])
    top = {"box": 512 ** 3, "noalloc": 400_000, "host": 2e7, "host_many": 1e7, "relink": 3e7}
    c = _case("", via, 0)
    del c["name"]
    c["min_size"] = rng.choice([1, 2, 20, 20, 32])
    if via in top:
        c["n"] = _log_int(rng, 16 ** 3, top[via])
        c["box"] = round(rng.uniform(0.5, 150.0), 3)
        c["b"] = round(rng.uniform(0.1, 0.3), 3)
        c["kind"] = rng.choice(["clustered", "clustered", "clustered", "uniform"])
        c["frac"] = round(rng.uniform(0.3, 0.7), 2)
        c["order"] = rng.choice(["generated", "shuffled", "cells"])
        c["strict"] = via != "noalloc" and rng.random() < 0.25
        if via == "relink":
            c["move"] = rng.choice([0.0, 0.001, 0.01, 0.1])
    else:                       # uneven boxes: sizes log-uniform on [n, n_top]
        c["n"] = 16 ** 3 if via == "batch" else 10_000
        c["boxes"] = _log_int(rng, 4, 256) if via == "batch" else rng.randint(4, 20)
        c["n_top"] = _log_int(rng, 32 ** 3, 160 ** 3) if via == "batch" else _log_int(rng, 1e5, 1e7)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _positions(gen, n, box, kind, frac, order):
    """n float32 positions in [0, box)^3 on the GPU: uniform, or frac of them in
    Plummer blobs (masses dN/dM ~ M^-1.9 on [1, 1e4], radii 0.05 mean separations
    times m^(1/3), cut at 10 radii), 20,000 blobs per 256^3 particles."""
    dev = torch.device("cuda")

    def rand(*shape):
        return torch.rand(*shape, generator=gen, device=dev)

    out = torch.empty((n, 3), device=dev)
    n_cl = int(round(frac * n)) if kind == "clustered" else 0
    if n_cl:
        blobs = max(1, round(20000 * n / 256 ** 3))
        mass = (1.0 + rand(blobs).double() * (1e4 ** -0.9 - 1.0)) ** (-1.0 / 0.9)
        counts = torch.floor(mass * (n_cl / mass.sum())).long()
        rest = n_cl - int(counts.sum())
        counts += rest // blobs
        counts[: rest % blobs] += 1
        centre = rand(blobs, 3) * box
        radius = 0.05 * box / n ** (1 / 3) * counts.float() ** (1 / 3)
        owner = torch.repeat_interleave(torch.arange(blobs, device=dev, dtype=torch.int32), counts)
        inside = 1000.0 / 101.0 ** 1.5                  # share of a Plummer sphere within 10 radii
        for lo in range(0, n_cl, 1 << 25):
            k = owner[lo:lo + (1 << 25)].long()
            u = (rand(len(k)) * inside).clamp_(min=1e-7)
            r = radius[k] / (u ** (-2 / 3) - 1.0).sqrt()
            cz = 2.0 * rand(len(k)) - 1.0
            phi = (2.0 * math.pi) * rand(len(k))
            st = (1.0 - cz * cz).clamp_(min=0.0).sqrt()
            d = torch.stack([st * phi.cos(), st * phi.sin(), cz], 1)
            out[lo:lo + len(k)] = centre[k] + r[:, None] * d
        del owner
    for lo in range(n_cl, n, 1 << 25):
        hi = min(n, lo + (1 << 25))
        out[lo:hi] = rand(hi - lo, 3) * box
    out.remainder_(box)
    out[out >= torch.tensor(box, device=dev)] = 0.0
    if order == "shuffled":
        out = out[torch.randperm(n, generator=gen, device=dev)]
    elif order == "cells":                              # cells of about 8 particles, row by row
        side = max(1, int((n / 8) ** (1 / 3)))
        c = (out * (side / box)).long().clamp_(max=side - 1)
        out = out[torch.argsort((c[:, 2] * side + c[:, 1]) * side + c[:, 0], stable=True)]
    return out.contiguous()


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _one(case, seed):
    return _positions(_generator(seed), case["n"], case["box"], case["kind"], case["frac"], case["order"])


def _l_x(n, box, b):
    return b * box / n ** (1 / 3)


def _many(case):
    """Sizes and sides of the uneven boxes: part of the case, not of the seed."""
    rng = random.Random(case["boxes"] * 1_000_003 + case["n_top"])
    ns = [_log_int(rng, case["n"], case["n_top"]) for _ in range(case["boxes"])]
    if case["via"] == "served":                         # one density for all requests
        return ns, [100.0 * (n / 256 ** 3) ** (1 / 3) for n in ns]
    return ns, [rng.uniform(50.0, 150.0) for _ in ns]


def _options(case):
    if not case["strict"]:
        return None
    o = fof.fof_options()
    o.tie_rule = fof.FOF_TIE_LT
    return o


class State:
    def __init__(self, case):
        self.case, self.n, self.min_size = case, case["n"], case["min_size"]
        self.box, self.l_x = case["box"], _l_x(case["n"], case["box"], case["b"])
        self.plan = self.server = None

    def __del__(self):
        if self.server is not None:
            self.server.close()
        if self.plan is not None:
            self.plan.close()


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def _to_host(x):
    h = _pinned(x.shape, x.dtype)
    h.copy_(x)
    return h


def prepare(case, seed):
    s = State(case)
    via, n, dev = case["via"], case["n"], torch.device("cuda")
    if via == "batch":
        ns, sides = _many(case)
        gen = _generator(seed)
        s.ns, total = ns, sum(ns)
        s.pos = torch.cat([_positions(gen, m, L, "clustered", 0.5, "generated") for m, L in zip(ns, sides)])
        s.plan = fof.FoFBatch(sides, [_l_x(m, L, case["b"]) for m, L in zip(ns, sides)], ns)
        s.ids, s.sizes = (torch.empty(total, dtype=torch.int32, device=dev) for _ in range(2))
        s.cat = torch.zeros((total, 2), dtype=torch.int32, device=dev)
        s.stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        fof.fof_graph_build(s.plan.h, s.pos, s.ids, s.sizes, s.cat, total, s.min_size, s.stream)
        return s
    if via == "served":
        ns, sides = _many(case)
        gen = _generator(seed)
        s.jobs = [(_to_host(_positions(gen, m, L, "clustered", 0.5, "generated")), L, _l_x(m, L, case["b"]))
                  for m, L in zip(ns, sides)]
        s.cat = [torch.zeros((m // max(s.min_size, 1) + 1, 2), dtype=torch.int32) for m in ns]
        s.server = Server()
        return s
    if via == "host_many":
        s.pos = [_to_host(_one(case, HOST_STEPS * seed + k)) for k in range(HOST_STEPS)]
        s.ids, s.sizes = ([_pinned(n, torch.int32) for _ in range(HOST_STEPS)] for _ in range(2))
        s.cat = [_pinned((n, 2), torch.int32).zero_() for _ in range(HOST_STEPS)]
        s.plan = fof.FoF(s.box, s.l_x, n, _options(case))
        return s
    s.pos = _one(case, seed)
    if via == "host":
        s.pos = _to_host(s.pos)
        s.ids, s.sizes = _pinned(n, torch.int32), _pinned(n, torch.int32)
        s.cat = _pinned((n, 2), torch.int32).zero_()
    else:
        k = 2 if via == "relink" else 1
        s.ids, s.sizes = ([torch.empty(n, dtype=torch.int32, device=dev) for _ in range(k)] for _ in range(2))
        s.cat = [torch.zeros((n, 2), dtype=torch.int32, device=dev) for _ in range(k)]
    if via != "noalloc":
        s.plan = fof.FoF(s.box, s.l_x, n, _options(case))
    if via == "relink":                                 # the step before: binned and linked
        step = torch.rand((n, 3), generator=_generator(seed + 1), device=dev) - 0.5
        moved = (s.pos + step * (2.0 * case["move"] * s.l_x)).remainder_(s.box)
        moved[moved >= torch.tensor(s.box, device=dev)] = 0.0
        s.steps = [moved.contiguous(), s.pos]
        fof.fof_link(s.plan.h, s.pos, torch.cuda.current_stream())
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    via, n, m = s.case["via"], s.n, s.min_size
    if via in ("box", "relink"):
        out, stream = [], torch.cuda.current_stream()
        for k, pos in enumerate(s.steps if via == "relink" else [s.pos]):
            if via == "relink":
                fof.fof_relink(s.plan.h, pos, stream)
            else:
                fof.fof_link(s.plan.h, pos, stream)
            _, ng, nk = fof.fof_groups(s.plan.h, s.ids[k], s.sizes[k], s.cat[k], n, m, 1, stream)
            out.append((s.ids[k], s.sizes[k], s.cat[k], ng[0], nk[0]))
        return out
    if via == "batch":
        fof.fof_graph_launch(s.plan.h, s.stream)
        _, ng, nk = fof.fof_result(s.plan.h, len(s.ns), s.stream)
        return s.ids, s.sizes, s.cat, torch.tensor(ng), torch.tensor(nk)
    if via == "noalloc":
        _, ng, nk = fof.fof_run_noalloc(s.box, s.l_x, n, s.pos, s.ids[0], s.sizes[0], s.cat[0], n, m,
                                        torch.cuda.current_stream())
        return s.ids[0], s.sizes[0], s.cat[0], ng, nk
    if via == "host":
        _, ng, nk = fof.fof_run_host(s.plan.h, s.pos, s.ids, s.sizes, s.cat, n, m, 1, torch.cuda.current_stream())
        return s.ids, s.sizes, s.cat, ng[0], nk[0]
    if via == "host_many":
        _, ng, nk = fof.fof_run_host_many(s.plan.h, s.pos, s.ids, s.sizes, s.cat, n, m, 1,
                                          torch.cuda.current_stream())
        return s.ids, s.sizes, s.cat, torch.tensor(ng), torch.tensor(nk)
    futures = [s.server.submit(pos, L, l_x, m) for pos, L, l_x in s.jobs]
    got = [f.result() for f in futures]
    for cat, r in zip(s.cat, got):
        cat[: len(r.catalogue)] = torch.from_numpy(r.catalogue)
    return [(r.ids, r.sizes, cat) for cat, r in zip(s.cat, got)], torch.tensor([r.n_groups for r in got])


def work(case):
    """Positions in (12 bytes a particle), ids and sizes out (8); at least one
    separation (8 operations) for each particle."""
    if case["via"] in ("batch", "served"):
        total = sum(_many(case)[0])
    else:
        total = case["n"] * {"relink": 2, "host_many": HOST_STEPS}.get(case["via"], 1)
    return {"bytes": 20.0 * total, "flops": 8.0 * total}


# ---------------------------------------------------------------------------
# the answer from every pair, in 64 bits
# ---------------------------------------------------------------------------

def _all_pairs(pos, box, l_x, strict, min_size):
    x, n, l2 = pos.double(), len(pos), l_x * l_x
    edges = []
    for lo in range(0, n, 512):
        s = 0.0
        for k in range(3):
            d = x[lo:lo + 512, k][:, None] - x[:, k][None, :]
            d = torch.where(d > box / 2, d - box, torch.where(d < -box / 2, d + box, d))
            s = s + d * d
        e = torch.nonzero(s < l2 if strict else s <= l2)
        e[:, 0] += lo
        edges.append(e[e[:, 0] != e[:, 1]])
    a, b = torch.cat(edges).T
    lab = torch.arange(n, device=pos.device)
    while True:                                         # smallest label over the links, then over the labels
        new = lab.scatter_reduce(0, a, lab[b], "amin")
        new = new[new]
        if torch.equal(new, lab):
            break
        lab = new
    count = torch.bincount(lab, minlength=n)
    rows = torch.nonzero(count >= max(min_size, 1))[:, 0]
    cat = torch.zeros((n, 2), dtype=torch.int32, device=pos.device)
    cat[: len(rows)] = torch.stack([rows, count[rows]], 1).int()
    return lab.int(), count.int(), cat, int((count > 0).sum()), len(rows)


def exact(case, seed):
    if case["n"] > EXACT_MAX or case["via"] not in ("box", "noalloc", "host"):
        return None
    out = _all_pairs(_one(case, seed), case["box"], _l_x(case["n"], case["box"], case["b"]), case["strict"],
                     case["min_size"])
    return [out] if case["via"] == "box" else out
