"""What the seed scan is timed on: cases of its use, each through the package's public entry points.

A case is one of five kinds of call:

* ``scan``     -- one turn partition of one event through ``scan.scan_partition`` (lattice, track
  recording, DCA and RSS, selection, classification): what every reconstruction program repeats.
* ``host``     -- whole events from pinned host buffers through ``scan.HostEventRunner`` with the
  pipelined driver: copies in, every turn partition in order, copies out.
* ``batch``    -- many uneven events at once through ``batch.BatchScanner.run``.
* ``refine``   -- one level of the iterative scan (top-M seeds, sparse references, finer lattices
  around them, their scan) through the binding's calls.
* ``jacobian`` -- the smoothed RSS of a few seeds, its gradient and the Gauss-Newton normal equations
  through ``experiments.GaussNewton.evaluate``.

Events are synthetic (``synth``): electrons of 100-105 MeV/c in 1 T, or a DIO-shaped spectrum in the
tabulated solenoid field.  ``exact`` restates the scan in plain torch in 64 bits from the same inputs.
"""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1911_09340_gb300 import batch as BT
from paper_1911_09340_gb300 import binding as B
from paper_1911_09340_gb300 import experiments, scan, synth

KAPPA = 299.792458
_DT = {"f32": torch.float32, "f64": torch.float64}
# buffers are sized once for any event of the chamber, as a program that takes event after event does
MAX_WIRES, MAX_HITS = 512, 1024

# ----------------------------------------------------------------------------------------------
# The cases
# ----------------------------------------------------------------------------------------------

_SCAN = dict(kind="scan", turns=3, part=1, n_z=16, n_phi=16, n_pz=32, n_pt=32, dtype="f32", stride=32,
             lam_mm=10.0, field="uniform", k=1, dca=False, backward=False)


def listed():
    return [
        # the smallest call: a first look at a partition on a few hundred seeds, all launches and latency
        dict(_SCAN, name="scan_f32_tiny", turns=1, part=0, n_z=4, n_phi=4, n_pz=4, n_pt=4),
        # the benchmark's partition: 2^18 seeds, every 32nd state recorded, hits of an earlier turn masked
        dict(_SCAN, name="scan_f32_2e18"),
        # odd node counts (no 2x4x4 lattice blocks), stride 16, the cutoff of the hit-classification
        # studies, and the ten best seeds of the partition instead of one
        dict(_SCAN, name="scan_f32_odd_top10", turns=4, part=0, n_z=9, n_phi=15, n_pz=21, n_pt=27, stride=16,
             lam_mm=0.8, k=10),
        # every RK4 state recorded, as the paper's Algorithm 1 does, in FP32
        dict(_SCAN, name="scan_f32_every_state", turns=2, part=0, n_z=8, n_phi=8, n_pz=16, n_pt=16, stride=1),
        # the DCA of every (wire, seed) kept, as an analysis of residuals wants it
        dict(_SCAN, name="scan_f32_dca_out", turns=2, part=1, n_z=8, n_phi=8, n_pz=16, n_pt=16, dca=True),
        # the paper's precision on the single-event configuration: 8^4 seeds, every state recorded
        dict(_SCAN, name="scan_f64_every_state", turns=2, part=0, n_z=8, n_phi=8, n_pz=8, n_pt=8, dtype="f64",
             stride=1),
        # FP64 on a larger lattice at stride 16
        dict(_SCAN, name="scan_f64_2e15", turns=3, part=2, n_z=8, n_phi=16, n_pz=16, n_pt=16, dtype="f64",
             stride=16),
        # the tabulated solenoid field with DIO-shaped momenta
        dict(_SCAN, name="scan_f32_table", turns=2, part=1, field="table"),
        # events end to end from host memory, back to back, as a reconstruction job feeds them
        dict(kind="host", name="host_f32_2e18", events=2, turns=3, n_z=16, n_phi=16, n_pz=32, n_pt=32,
             dtype="f32", stride=32, lam_mm=10.0),
        # uneven events (1-6 turns, 2^12-2^18 seeds per partition) in continuous batches
        dict(kind="batch", name="batch_f32_16", events=16, scale=0, dtype="f32", stride=32, lam_mm=10.0),
        # one level of the iterative scan: 2^14 coarse seeds in hand, 64 best, 16 lattices of 5^4 around them
        dict(kind="refine", name="refine_f32_16x625", turns=3, part=0, n_z=8, n_phi=8, n_pz=16, n_pt=16, fine=5,
             top=64, refs=16, dtype="f32", stride=16, lam_mm=10.0),
        # smoothed RSS, gradient and normal equations of the best 16 seeds
        dict(kind="jacobian", name="jacobian_f64_16", turns=3, part=0, seeds=16, stride=16, lam_mm=0.8,
             tau_mm=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice_counts(rng, most):
    """Four node counts, odd ones among them, whose product is log-uniform up to ``most``."""
    target = math.exp(rng.uniform(math.log(256), math.log(most)))
    while True:
        c = [rng.randint(2, 16), rng.randint(2, 16), rng.randint(2, 32), rng.randint(2, 32)]
        if rng.random() < 0.6:
            c = [max(2, c[0] // 2 * 2)] + [max(4, n // 4 * 4) for n in c[1:3]] + [c[3]]
        if 0.7 * target <= math.prod(c) <= min(most, 1.3 * target):
            return dict(n_z=c[0], n_phi=c[1], n_pz=c[2], n_pt=c[3])


def draw(rng):
    kind = rng.choices(["scan", "host", "batch", "refine", "jacobian"], [12, 2, 2, 2, 2])[0]
    turns = rng.randint(1, 5)
    if kind == "host":
        c = _lattice_counts(rng, 1 << 18)
        turns = rng.randint(2, 3)
        return dict(kind=kind, events=rng.randint(1, 2), turns=turns, dtype="f32",
                    stride=rng.choice([16, 24, 32]), lam_mm=10.0, **c)
    if kind == "batch":
        return dict(kind=kind, events=rng.randint(4, 16), scale=rng.randint(0, 2), dtype="f32",
                    stride=rng.choice([16, 32]), lam_mm=10.0)
    if kind == "refine":
        return dict(kind=kind, turns=turns, part=rng.randrange(turns), fine=rng.choice([3, 4, 5]),
                    top=rng.choice([32, 64]), refs=rng.randint(4, 16), dtype="f32",
                    stride=rng.choice([16, 32]), lam_mm=rng.choice([0.8, 10.0]), **_lattice_counts(rng, 1 << 15))
    if kind == "jacobian":
        return dict(kind=kind, turns=turns, part=rng.randrange(turns), seeds=_log_int(rng, 4, 64),
                    stride=rng.choice([1, 4, 16, 32]), lam_mm=rng.choice([0.8, 10.0]),
                    tau_mm=rng.choice([0.2, 1.0]))
    field = rng.choices(["uniform", "table", "table_planar"], [10, 2, 1])[0]
    dtype = rng.choices(["f32", "f64"], [7, 3])[0] if field == "uniform" else "f32"
    stride = rng.choice([1, 4, 8, 16, 24, 32]) if field == "uniform" else rng.choice([16, 32])
    # the recorded states of the largest listed cases of each type bound the drawn ones
    states = (1 << 18) * 70 if dtype == "f32" else (1 << 12) * 2240
    seeds = min(1 << 18, states * stride // 2240)
    if field != "uniform" or dtype == "f64":
        seeds = min(seeds, 1 << 16 if dtype == "f32" else 1 << 15)
    dca = field == "uniform" and rng.random() < 0.15
    if dca:
        seeds = min(seeds, 1 << 14 if dtype == "f32" and stride >= 16 else 1 << 11)
    return dict(kind="scan", turns=turns, part=rng.randrange(turns), dtype=dtype, stride=stride,
                lam_mm=rng.choice([0.8, 2.0, 10.0]), field=field, k=rng.choice([1, 1, 1, 10, 64]), dca=dca,
                backward=field == "uniform" and rng.random() < 0.15, **_lattice_counts(rng, seeds))


# ----------------------------------------------------------------------------------------------
# What a program keeps from call to call: the chamber, the field on the device, a context, drivers
# ----------------------------------------------------------------------------------------------


@functools.lru_cache(maxsize=None)
def _chamber():
    return synth.make_chamber()


@functools.lru_cache(maxsize=None)
def _host_field(name):
    return synth.uniform_field(1.0) if name == "uniform" else synth.table_field()


@functools.lru_cache(maxsize=None)
def _field(name):
    return B.DeviceField.from_synth(_host_field(name if name == "uniform" else "table"), interleaved=name == "table")


@functools.lru_cache(maxsize=None)
def _ctx():
    return B.Context(torch.cuda.current_device())


@functools.lru_cache(maxsize=1)
def _pipeline(S, n_rec, H, W, dtype):
    ctx = B.Context(torch.cuda.current_device())
    ps = scan.PipelinedScanner(ctx, _field("uniform"), S, n_rec, H, _DT[dtype])
    return scan.HostEventRunner(ctx, _field("uniform"), None, W, H, _DT[dtype], pipeline=ps)


@functools.lru_cache(maxsize=1)
def _batcher(slots, dtype, stride, lam_mm):
    # the configuration the batching study's tuner settles on: big partitions on lanes of their own
    return BT.BatchScanner(B.Context(torch.cuda.current_device()), _DT[dtype], stride, lam_mm * 1e-3, slots=slots,
                           max_total_seeds=1 << 20, max_wires=MAX_WIRES, max_hits=MAX_HITS, solo_min_seeds=1 << 16,
                           solo_lanes=4)


def _counts(c):
    return (c["n_z"], c["n_phi"], c["n_pz"], c["n_pt"])


def _event(c, seed, i=0):
    rng = np.random.default_rng([int(seed), i, 1911])
    turns = c["turns"]
    kw = dict(turns=(turns, turns), counts=_counts(c) if "n_z" in c else (8, 8, 16, 16), hits_window=(20, 400))
    if c.get("field", "uniform") == "uniform":
        return synth.make_event_random(_chamber(), rng, prescreen=True, **kw)
    return synth.make_event_random(_chamber(), rng, field=_host_field("table"), p_sampler=synth.dio_momentum_sampler, **kw)


def _batch_event(c, seed, i):
    """An event of the batching workload: 1-6 turns, seeds per partition by turn count."""
    rng = np.random.default_rng([int(seed), i, 340])
    turns = 1 + i % 6
    counts = list(synth.BATCH_COUNTS[turns])
    for _ in range(c["scale"]):
        counts[2], counts[3] = max(2, counts[2] // 2), max(2, counts[3] // 2)
    return synth.make_event_random(_chamber(), rng, turns=(turns, turns), counts=tuple(counts),
                                   hits_window=(20, 400), prescreen=True)


def _earlier_hits(ev, part):
    """The hit mask as earlier turn partitions leave it: the hits of earlier turns."""
    return ((ev.hit_turn >= 0) & (ev.hit_turn < part)).astype(np.uint8)


def _spec(ev, c):
    return synth.backward_partition(ev, c["part"]) if c.get("backward") else ev.partitions[c["part"]]


# ----------------------------------------------------------------------------------------------
# prepare and run
# ----------------------------------------------------------------------------------------------


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "scan":
        ev = _event(c, seed)
        dt = _DT[c["dtype"]]
        spec = _spec(ev, c)
        p = scan.params_for(spec, ev.n_steps[c["part"]], dt, c["stride"], c["lam_mm"] * 1e-3)
        dev = scan.DeviceEvent.from_event(ev, dt)
        ws = scan.Workspace(spec.n_seeds, p.n_rec, MAX_HITS, dt, k=c["k"])
        ws.hit_class.zero_()
        mask = torch.zeros(MAX_HITS, dtype=torch.uint8, device="cuda")
        mask[: ev.n_hits] = torch.as_tensor(_earlier_hits(ev, c["part"]), device="cuda")
        dev.mask = torch.zeros_like(mask)
        dca = torch.zeros((MAX_WIRES, spec.n_seeds), dtype=dt, device="cuda") if c["dca"] else None
        return dict(c=c, ev=ev, spec=spec, p=p, dev=dev, ws=ws, mask=mask, dca=dca, ctx=_ctx(), field=_field(c["field"]))
    if c["kind"] == "host":
        evs = [_event(c, seed, i) for i in range(c["events"])]
        n_rec = 2400 // c["stride"] + 1
        runner = _pipeline(math.prod(_counts(c)), n_rec, MAX_HITS, MAX_WIRES, c["dtype"])
        pinned = [runner.pin(ev, _DT[c["dtype"]]) for ev in evs]
        return dict(c=c, evs=evs, runner=runner, pinned=pinned, out=[runner.result_slots() for _ in evs])
    if c["kind"] == "batch":
        evs = [_batch_event(c, seed, i) for i in range(c["events"])]
        sc = _batcher(c["events"], c["dtype"], c["stride"], c["lam_mm"])
        return dict(c=c, evs=evs, sc=sc, pinned=sc.pin(evs))
    if c["kind"] == "refine":
        ev = _event(c, seed)
        dt = _DT[c["dtype"]]
        spec = ev.partitions[c["part"]]
        p = scan.params_for(spec, ev.n_steps[c["part"]], dt, c["stride"], c["lam_mm"] * 1e-3)
        dev = scan.DeviceEvent.from_event(ev, dt)
        dev.mask[: ev.n_hits] = torch.as_tensor(_earlier_hits(ev, c["part"]), device="cuda")
        ctx, field = _ctx(), _field("uniform")
        coarse = scan.Workspace(spec.n_seeds, p.n_rec, ev.n_hits, dt)
        scan.scan_partition(ctx, field, p, spec, dev, coarse, update_mask=False)
        half = tuple(0.75 * 2.0 * h / (n - 1) for h, n in zip(spec.half_width, spec.counts))
        shape = dataclasses.replace(spec, half_width=half, counts=(c["fine"],) * 4)
        ws = scan.Workspace(c["refs"] * shape.n_seeds, p.n_rec, ev.n_hits, dt, k=c["top"])
        return dict(c=c, ev=ev, spec=spec, shape=shape, half=half, p=p, dev=dev, ctx=ctx, field=field, ws=ws,
                    seeds=coarse.seeds, rss=coarse.rss,
                    top=torch.empty(c["top"], dtype=torch.int64, device="cuda"),
                    refs=torch.zeros((c["refs"], 4), dtype=torch.float64, device="cuda"),
                    n_refs=torch.zeros(1, dtype=torch.int32, device="cuda"))
    ev = _event(c, seed)
    g = experiments.GaussNewton(_ctx(), ev, c["part"], c["stride"], c["lam_mm"] * 1e-3, c["tau_mm"] * 1e-3, c["seeds"])
    spec = ev.partitions[c["part"]]
    # seeds about a coarse lattice step off the partition's centre, as a grid scan hands them over
    off = np.random.default_rng([int(seed), 7]).uniform(-0.15, 0.15, (c["seeds"], 4)) * np.array(spec.half_width)
    g.theta.copy_(torch.as_tensor(np.array(spec.centre) + off))
    g.dev.mask[: ev.n_hits] = torch.as_tensor(_earlier_hits(ev, c["part"]), device="cuda")
    return dict(c=c, ev=ev, g=g)


def run(s):
    kind = s["c"]["kind"]
    if kind == "scan":
        c, ws, dev, S = s["c"], s["ws"], s["dev"], s["spec"].n_seeds
        dev.mask.copy_(s["mask"])
        scan.scan_partition(s["ctx"], s["field"], s["p"], s["spec"], dev, ws, k=c["k"], want_dca=s["dca"])
        return dict(rss=ws.rss[:S], n_in=ws.n_in[:S], idx=ws.idx, best=ws.best, hit_class=ws.hit_class,
                    mask=dev.mask, dca=s["dca"])
    if kind == "host":
        c = s["c"]
        for ev, pinned, out in zip(s["evs"], s["pinned"], s["out"]):
            s["runner"].run(ev, pinned, c["stride"], c["lam_mm"] * 1e-3, out)
        return [dict(idx=o[0][: c["turns"]], best=o[1][: c["turns"]], mask=o[2]) for o in s["out"]]
    if kind == "batch":
        r = s["sc"].run(s["evs"], collect=True, pinned=s["pinned"])["results"]
        classes = [h for x in r for h in x.hit_class]
        hit_class = np.zeros((len(classes), MAX_HITS), np.uint8)
        for row, h in zip(hit_class, classes):
            row[: len(h)] = h
        return dict(idx=np.concatenate([x.best_idx for x in r]), best=np.concatenate([x.best_rss for x in r]),
                    hit_class=hit_class)
    if kind == "refine":
        c, ws, dev, p, ctx = s["c"], s["ws"], s["dev"], s["p"], s["ctx"]
        S = c["refs"] * s["shape"].n_seeds
        seeds, charge, pts, nv, rss, n_in = ws.views(S, p.n_rec)
        B.comet_scan_select(ctx, s["rss"], c["top"], s["top"])
        B.comet_scan_refine_refs(ctx, s["seeds"], s["top"], s["half"], c["refs"], s["refs"], s["n_refs"])
        B.comet_scan_lattice_refined(ctx, s["shape"], s["refs"], s["n_refs"], c["refs"], seeds, charge)
        B.comet_scan_propagate(ctx, s["field"], p, seeds, charge, pts, nv, bounds=ws.bounds)
        B.comet_scan_dca(ctx, s["field"], p, pts, nv, charge, dev.wires, dev.hit_offsets, dev.drift, dev.mask, rss,
                         n_in, n_wires=dev.W, bounds=ws.bounds)
        B.comet_scan_select(ctx, rss, c["top"], ws.idx, ws.best)
        return dict(refs=s["refs"], n_refs=s["n_refs"], seeds=seeds, rss=rss, n_in=n_in, idx=ws.idx, best=ws.best)
    g = s["g"]
    g.evaluate()
    return dict(srss=g.srss, grad=g.grad, jtj=g.jtj, jtr=g.jtr)


# ----------------------------------------------------------------------------------------------
# The work of a pass
# ----------------------------------------------------------------------------------------------


@functools.lru_cache(maxsize=256)
def _sizes(turns, field):
    """(wires, hits, steps per partition) of a typical event."""
    ev = _event(dict(turns=turns, field=field), 1)
    return ev.n_wires, ev.n_hits, int(np.mean(ev.n_steps))


def _scan_work(S, turns, stride, es, field="uniform", dca=False):
    """One partition: its wires and hits read, its RSS, counts and hit classes written; per recorded
    state one interval map (axial field) or per step four table lookups and an RK4 step; per (seed,
    wire) three virtual-plane evaluations, two refinement steps and the DCA, per (seed, hit) one residual."""
    W, H, steps = _sizes(turns, "uniform" if field == "uniform" else "table")
    rec = 18.0 * (steps // stride) if field == "uniform" else 438.0 * steps
    return dict(bytes=6 * W * es + 4 * (W + 1) + H * (es + 2) + S * (es + 4) + (W * S * es if dca else 0),
                flops=S * (rec + 201.0 * W + 8.0 * H))


def work(case):
    c = case
    es = 8 if c.get("dtype") == "f64" else 4
    if c["kind"] == "scan":
        return _scan_work(math.prod(_counts(c)), c["turns"], c["stride"], es, c["field"], c["dca"])
    if c["kind"] == "host":
        w = _scan_work(math.prod(_counts(c)), c["turns"], c["stride"], es)
        return {k: v * c["turns"] * c["events"] for k, v in w.items()}
    if c["kind"] == "batch":
        tot = dict(bytes=0.0, flops=0.0)
        for i in range(c["events"]):
            turns = 1 + i % 6
            S = math.prod(synth.BATCH_COUNTS[turns]) >> (2 * c["scale"])
            w = _scan_work(S, turns, c["stride"], es)
            for k in tot:
                tot[k] += turns * w[k]
        return tot
    if c["kind"] == "refine":
        w = _scan_work(c["refs"] * c["fine"] ** 4, c["turns"], c["stride"], es)
        return dict(bytes=w["bytes"] + 7 * es * math.prod(_counts(c)), flops=w["flops"])
    # per (seed, wire): the recorded states walked once (20 flops each), the refinement and its
    # derivatives in four parameters (about 800); per seed the sums
    W, H, steps = _sizes(c["turns"], "uniform")
    return dict(bytes=8.0 * (6 * W + 2 * H + c["seeds"] * 29),
                flops=c["seeds"] * W * (20.0 * (steps // c["stride"]) + 800.0))


# ----------------------------------------------------------------------------------------------
# The same results in 64 bits, in plain torch
# ----------------------------------------------------------------------------------------------


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _t(x):
    return torch.as_tensor(np.asarray(x, np.float64), device=_dev())


def _seen(x, dtype):
    """The values a path of that precision is given."""
    return x.to(torch.float32).to(torch.float64) if dtype == "f32" else x


def _grid(spec, centre=None):
    """Seeds [6, S] of a lattice in blocks of 2 x 4 x 4 x 1 nodes (fewer where a count does not divide)."""
    n = spec.counts
    b = [2 if n[0] % 2 == 0 else 1] + [4 if m % 4 == 0 else 2 if m % 2 == 0 else 1 for m in n[1:3]] + [1]
    ax = [_t([c if m == 1 else c + h * (2.0 * i / (m - 1) - 1.0) for i in range(m)])
          for m, c, h in zip(n, spec.centre if centre is None else centre, spec.half_width)]
    g = torch.meshgrid(*[torch.arange(m, device=_dev()) for m in n], indexing="ij")
    order = [x for m, k in zip(n, b) for x in (m // k, k)]
    g = [x.reshape(order).permute(0, 2, 4, 6, 1, 3, 5, 7).reshape(-1) for x in g]
    z, phi, pz, pt = (a[i] for a, i in zip(ax, g))
    one = torch.ones_like(z)
    return torch.stack([spec.vxy[0] * one, spec.vxy[1] * one, z, pt * torch.cos(phi), pt * torch.sin(phi), pz])


class _Axial:
    """RK4 in B = (0, 0, 1 T): one step of length h is P' = (1 + A) P, X' = X + N P with P = px + i py."""

    def __init__(self, P0, pz, q):
        self.P0, self.pz, self.w = P0, pz, KAPPA * q / P0

    def maps(self, h):
        t = h * self.w
        A = torch.complex(-t * t / 2 + t ** 4 / 24, -(t - t ** 3 / 6))
        N = torch.complex(h / self.P0 * (1 - t * t / 6), -h / self.P0 * (t / 2 - t ** 3 / 24))
        return A, N

    def after(self, X, P, z, h, k):
        """The states after k steps of length h."""
        A, N = self.maps(h)
        log_m = torch.complex(0.5 * torch.log1p(2 * A.real + A.real ** 2 + A.imag ** 2), torch.atan2(A.imag, 1 + A.real))
        mk = torch.exp(k * log_m)
        return X + N * (mk - 1) / A * P, P * mk, z + k * h * self.pz / self.P0

    def step(self, y, h):
        X, P = torch.complex(y[0], y[1]), torch.complex(y[3], y[4])
        A, N = self.maps(h)
        X, P = X + N * P, P + A * P
        return [X.real, X.imag, y[2] + h * self.pz / self.P0, P.real, P.imag, y[5]]


class _Table:
    """RK4 in a field interpolated trilinearly from its float32 table."""

    def __init__(self, f, P0, q):
        self.ip, self.c = 1.0 / P0, KAPPA * q / P0
        t = torch.as_tensor(f.table, device=_dev())
        self.n = torch.tensor(t.shape[:0:-1], device=_dev(), dtype=torch.float64)[:, None]
        self.tab = t.permute(1, 2, 3, 0).reshape(-1, 3).contiguous()
        self.o, self.sp = _t(f.origin)[:, None], f.spacing
        nx, ny = t.shape[3], t.shape[2]
        self.stride = torch.tensor([1, nx, nx * ny], device=_dev())[:, None]
        self.off = torch.tensor([dx + nx * dy + nx * ny * dz for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)],
                                device=_dev())[:, None]

    def at(self, x):
        sh = x.shape[1:]
        g = (x.reshape(3, -1) - self.o) / self.sp
        g = torch.minimum(g.clamp(min=0.0), self.n - 1)
        i = torch.minimum(g.floor(), self.n - 2)
        t = (g - i)[:, :, None]
        v = self.tab[(i.long() * self.stride).sum(0) + self.off].double()
        v = v[0::2] + t[0] * (v[1::2] - v[0::2])
        v = v[0::2] + t[1] * (v[1::2] - v[0::2])
        return (v[0] + t[2] * (v[1] - v[0])).T.reshape((3,) + sh)

    def _deriv(self, y):
        return torch.cat([y[3:] * self.ip, self.c * torch.linalg.cross(y[3:], self.at(y[:3]), dim=0)])

    def step(self, y, h):
        y = torch.stack(list(y))
        k1 = self._deriv(y)
        k2 = self._deriv(y + 0.5 * h * k1)
        k3 = self._deriv(y + 0.5 * h * k2)
        k4 = self._deriv(y + h * k3)
        return list(y + h / 6 * (k1 + 2 * (k2 + k3) + k4))


def _tracks(seeds, q, p, field):
    """Recorded states [n_rec, 6, S], how many are valid, and the stepper."""
    P0 = seeds[3:].norm(dim=0)
    if field == "uniform":
        st = _Axial(P0, seeds[5], q)
        k = torch.arange(p.n_rec, device=_dev(), dtype=torch.float64)[:, None] * p.stride
        X, P, z = st.after(torch.complex(seeds[0], seeds[1]), torch.complex(seeds[3], seeds[4]), seeds[2], p.h, k)
        pts = torch.stack([X.real, X.imag, z, P.real, P.imag, seeds[5].expand_as(z)], 1)
    else:
        st = _Table(_host_field("table"), P0, q)
        y, rec = list(seeds), [seeds]
        for i in range(1, (p.n_rec - 1) * p.stride + 1):
            y = st.step(y, p.h)
            if i % p.stride == 0:
                rec.append(torch.stack(y))
        pts = torch.stack(rec)
    out = (pts[:, 2] < p.zmin) | (pts[:, 2] > p.zmax) | (pts[:, 0] ** 2 + pts[:, 1] ** 2 > p.rmax ** 2)
    # valid: every state up to and with the first one outside
    valid = torch.cat([torch.zeros_like(out[:1]), out[:-1]]).cumsum(0) == 0
    return pts, valid, st


def _perp(v, u):
    t = v[0] * u[0] + v[1] * u[1] + v[2] * u[2]
    return [v[i] - t * u[i] for i in range(3)]


def _closest(pts, valid, wire):
    """Index of the recorded state closest to the wire, per seed (the first of equals)."""
    e = _perp([pts[:, i] - wire[i] for i in range(3)], wire[3:])
    return torch.where(valid, e[0] ** 2 + e[1] ** 2 + e[2] ** 2, math.inf).argmin(0)


def _refined(y, wire, st, p):
    """DCA by the virtual plane from state y, moving at most one recording interval, and the steps taken."""
    h_rec = p.h * p.stride
    sigma, steps = torch.zeros_like(y[0]), []
    for _ in range(min(p.max_iter, 8)):
        pn = (y[3] ** 2 + y[4] ** 2 + y[5] ** 2).sqrt()
        n = _perp([y[3] / pn, y[4] / pn, y[5] / pn], wire[3:])
        nn = (n[0] ** 2 + n[1] ** 2 + n[2] ** 2).sqrt()
        d = ((y[0] - wire[0]) * n[0] + (y[1] - wire[1]) * n[1] + (y[2] - wire[2]) * n[2]) / nn
        to = (sigma - d / nn).clamp(-h_rec, h_rec)
        y = st.step(y, to - sigma)
        steps.append(to - sigma)
        sigma = to
    e = _perp([y[i] - wire[i] for i in range(3)], wire[3:])
    return (e[0] ** 2 + e[1] ** 2 + e[2] ** 2).sqrt(), steps


def _dcas(seeds, q, p, field, wires):
    """DCA [W, S] of every seed's track to every wire."""
    out = []
    per = max(1, int(6e7 // (p.n_rec * 6)))
    for s0 in range(0, seeds.shape[1], per):
        sd = seeds[:, s0:s0 + per]
        pts, valid, st = _tracks(sd, q, p, field)
        at = torch.arange(sd.shape[1], device=_dev())
        D = []
        for i in range(wires.shape[1]):
            k = _closest(pts, valid, wires[:, i])
            D.append(_refined(list(pts[k, :, at].T), wires[:, i], st, p)[0])
        out.append(torch.stack(D) if D else torch.zeros((0, sd.shape[1]), device=_dev(), dtype=torch.float64))
    return torch.cat(out, 1)


def _hits(ev, mask, drift):
    """Per wire: its unmasked drifts."""
    return [drift[a:b][mask[a:b] == 0] for a, b in zip(ev.hit_offsets[:-1], ev.hit_offsets[1:])]


def _residuals(D, hits):
    """Smallest |D - r| of each wire with an unmasked hit, [n, S]."""
    e = [(D[i][None] - r[:, None]).abs().amin(0) for i, r in enumerate(hits) if len(r)]
    return torch.stack(e) if e else D[:0]


def _inputs(ev, dtype):
    return _seen(_t(ev.wires), dtype), _seen(_t(ev.drift), dtype)


def _rss(D, hits, lam):
    return _residuals(D, hits).clamp(max=lam).square().sum(0)


def _exact_partition(ev, spec, p, dtype, field, mask):
    wires, drift = _inputs(ev, dtype)
    D = _dcas(_seen(_grid(spec), dtype), spec.charge, p, field, wires)
    return D, _rss(D, _hits(ev, mask, drift), p.lam)


def _exact_event(ev, c):
    """Lowest RSS of each turn partition, each classifying its best seed's hits out of the next."""
    mask, best = np.zeros(ev.n_hits, np.uint8), []
    for p, spec in zip(scan.event_params(ev, _DT[c["dtype"]], c["stride"], c["lam_mm"] * 1e-3), ev.partitions):
        D, rss = _exact_partition(ev, spec, p, c["dtype"], "uniform", mask)
        s = int(rss.argmin())
        best.append(float(rss[s]))
        d = D[:, s].cpu().numpy()
        for i, (a, b) in enumerate(zip(ev.hit_offsets[:-1], ev.hit_offsets[1:])):
            e = np.where(mask[a:b] == 0, np.abs(d[i] - ev.drift[a:b]), np.inf)
            if len(e) and e.min() < p.lam:
                mask[a + int(e.argmin())] = 1
    return best


def _exact_jacobian(s):
    """Smoothed RSS and its derivatives: D differentiated at the fixed arc length of the closest approach."""
    c, ev, g = s["c"], s["ev"], s["g"]
    p, spec, lam, tau = g.params, g.spec, c["lam_mm"] * 1e-3, c["tau_mm"] * 1e-3
    th = g.theta.detach().to(_dev()).clone().requires_grad_(True)
    wires, drift = _inputs(ev, "f64")
    hits = _hits(ev, _earlier_hits(ev, c["part"]), drift)

    def seed_of(t):
        one = torch.ones_like(t[:, 0])
        return torch.stack([spec.vxy[0] * one, spec.vxy[1] * one, t[:, 0], t[:, 3] * t[:, 1].cos(),
                            t[:, 3] * t[:, 1].sin(), t[:, 2]])

    sd = seed_of(th)
    with torch.no_grad():
        pts, valid, st0 = _tracks(sd, spec.charge, p, "uniform")
    st = _Axial((sd[3] ** 2 + sd[4] ** 2 + sd[5] ** 2).sqrt(), sd[5], spec.charge)
    at = torch.arange(c["seeds"], device=_dev())
    srss = torch.zeros(c["seeds"], dtype=torch.float64, device=_dev())
    jtj, jtr = torch.zeros((c["seeds"], 16), device=_dev()).double(), torch.zeros((c["seeds"], 4), device=_dev()).double()
    for i, r in enumerate(hits):
        if not len(r):
            continue
        with torch.no_grad():
            k = _closest(pts, valid, wires[:, i])
            steps = _refined(list(pts[k, :, at].T), wires[:, i], st0, p)[1]
        X, P, z = st.after(torch.complex(sd[0], sd[1]), torch.complex(sd[3], sd[4]), sd[2], p.h, k.double() * p.stride)
        y = [X.real, X.imag, z, P.real, P.imag, sd[5]]
        for ds in steps:
            y = st.step(y, ds)
        e = _perp([y[j] - wires[j, i] for j in range(3)], wires[3:, i])
        D = (e[0] ** 2 + e[1] ** 2 + e[2] ** 2).sqrt()
        J = torch.autograd.grad(D.sum(), th, retain_graph=True)[0]
        j = (D[None] - r[:, None]).abs().argmin(0)
        rho = D - r[j]
        w = torch.sigmoid((lam - rho.abs()) / tau)
        srss = srss + w * rho ** 2 + (1 - w) * lam ** 2
        wd = w.detach()[:, None]
        jtj += (wd[:, :, None] * J[:, :, None] * J[:, None, :]).reshape(-1, 16)
        jtr += wd * J * rho.detach()[:, None]
    grad = torch.autograd.grad(srss.sum(), th)[0]
    return dict(srss=srss.detach(), grad=grad, jtj=jtj, jtr=jtr)


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "scan":
        ev = _event(c, seed)
        spec, lam = _spec(ev, c), c["lam_mm"] * 1e-3
        p = scan.params_for(spec, ev.n_steps[c["part"]], _DT[c["dtype"]], c["stride"], lam)
        D, rss = _exact_partition(ev, spec, p, c["dtype"], c["field"], _earlier_hits(ev, c["part"]))
        return dict(rss=rss, n_in=None, idx=None, best=rss.sort()[0][: c["k"]], hit_class=None, mask=None,
                    dca=torch.nn.functional.pad(D, (0, 0, 0, MAX_WIRES - len(D))) if c["dca"] else None)
    if c["kind"] == "host":
        return [dict(idx=None, best=_t(_exact_event(_event(c, seed, i), c)), mask=None) for i in range(c["events"])]
    if c["kind"] == "batch":
        evs = [_batch_event(c, seed, i) for i in range(c["events"])]
        if sum(ev.n_wires * sp.n_seeds for ev in evs for sp in ev.partitions) > 4e8:
            return None   # over 20 seconds
        return dict(idx=None, best=_t(sum((_exact_event(ev, c) for ev in evs), [])), hit_class=None)
    s = prepare(c, seed)
    if c["kind"] == "jacobian":
        return _exact_jacobian(s)
    # the references: the coarse scan's best seeds in order, none within two half-widths of another
    ev, p, half = s["ev"], s["p"], s["half"]
    coarse = s["seeds"].double().cpu().numpy()
    refs = []
    for i in torch.sort(s["rss"], stable=True)[1][: c["top"]].cpu().numpy():
        x, y, z, px, py, pz = coarse[:, i]
        v = np.array([z, math.atan2(py, px), pz, math.hypot(px, py)])
        d = [np.abs([math.remainder(a, 2 * math.pi) if n == 1 else a for n, a in enumerate(v - r)]) for r in refs]
        if len(refs) < c["refs"] and not any((e < 2 * np.array(half)).all() for e in d):
            refs.append(v)
    seeds = torch.cat([_grid(s["shape"], refs[i] if i < len(refs) else refs[0]) for i in range(c["refs"])], 1)
    wires, drift = _inputs(ev, c["dtype"])
    D = _dcas(_seen(seeds, c["dtype"]), s["shape"].charge, p, "uniform", wires)
    rss = _rss(D, _hits(ev, _earlier_hits(ev, c["part"]), drift), p.lam)
    out = np.zeros((c["refs"], 4))
    out[: len(refs)] = refs
    return dict(refs=_t(out), n_refs=None, seeds=seeds, rss=rss, n_in=None, idx=None, best=rss.sort()[0][: c["top"]])
