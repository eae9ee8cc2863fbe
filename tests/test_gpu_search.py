"""The closest-state search and the refinement where they can go wrong: tracks that are not finite or too far
away to square, runs of candidate states that a track's valley leaves, and the refinement's precision."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1911_09340_gb300 import binding as B
from paper_1911_09340_gb300 import scan, synth

from gpu_util import FP32_DCA_TOL, gpu_dca, gpu_propagate, per_wire_residual, rss_bound, seen
from test_batch import _events, _reference

pytestmark = pytest.mark.gpu
UNIFORM = synth.uniform_field(1.0)
KAPPA = 299.792458


def test_fp64_refinement_step_is_full_precision(ctx):
    """One Newton step of up to half a metre from the recorded state (max_iter = 1, RK4 step 1 m), against
    the same step in extended precision from the device's own states.  The step is not stationary in its
    length there, so a relative error of the reciprocal root shows in the DCA with up to half its size in
    metres.  Coordinates stay below 8 m and some thirty roundings of 2^-53 reach the result: 32 x 8 x 1.1e-16."""
    rng = np.random.default_rng(5)
    S, n = 64, 60
    mom = rng.normal(size=(S, 3)) * [60.0, 60.0, 30.0] + [40.0, 0.0, 0.0]
    seeds = np.concatenate([rng.uniform(-0.2, 0.2, (S, 3)), mom], axis=1)
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    wires = np.concatenate([rng.uniform(-1.5, 1.5, (n, 3)), u], axis=1).T
    bz = 0.05
    bp = B.ScanParams(h=1.0, n_steps=3, stride=1, zmin=-90.0, zmax=90.0, rmax=90.0, tol=1e-12, max_iter=1)
    out = gpu_dca(ctx, B.DeviceField.from_synth(synth.uniform_field(bz)), bp, seeds, -1, wires, np.arange(n + 1),
                  np.full(n, 1e-3), np.zeros(n, np.uint8), torch.float64, use_bounds=False)
    L = np.longdouble
    P = out["pts"].cpu().numpy().astype(L)                       # [6][n_rec][S]
    A, U = wires[:3].astype(L), wires[3:].astype(L)
    d = P[:3, :, :, None] - A[:, None, None, :]
    e = d - (d * U[:, None, None, :]).sum(0) * U[:, None, None, :]
    d2 = (e * e).sum(0)                                          # [n_rec][S][n]
    k = d2.argmin(0)
    two = np.sort(d2, axis=0)
    clear = two[1] - two[0] > 1e-9
    y = np.take_along_axis(P[:, :, :, None], k[None, None], axis=1)[:, 0]   # [6][S][n]
    p0 = np.sqrt((P[3:, 0] ** 2).sum(0))[:, None]
    t = y[3:] / p0
    nv = t - (t * U[:, None, :]).sum(0) * U[:, None, :]
    nn = np.sqrt((nv * nv).sum(0))
    ds = np.clip(-((y[:3] - A[:, None, :]) * nv).sum(0) / nn / nn, -1, 1)
    # one RK4 step of length ds in a uniform axial field: P' = m P, X' = X + N P
    th, hp = ds * (L(KAPPA) * -1 * L(bz) / p0), ds / p0
    m = 1 - th * th * (L(1) / 2 - th * th / 24) - 1j * (th * (1 - th * th / 6))
    N = hp * (1 - th * th / 6) - 1j * (hp * th * (L(1) / 2 - th * th / 24))
    X = y[0] + 1j * y[1] + N * (y[3] + 1j * y[4])
    assert m.dtype == np.clongdouble
    r = np.stack([X.real, X.imag, y[2] + ds * y[5] / p0]) - A[:, None, :]
    er = r - (r * U[:, None, :]).sum(0) * U[:, None, :]
    D = np.sqrt((er * er).sum(0))
    usable = clear & (np.abs(ds) < 0.999) & (nn > 0.1)
    assert usable.mean() > 0.3 and np.abs(ds)[usable].max() > 0.4
    assert np.abs(out["dca"] - D.astype(np.float64))[usable].max() <= 32 * 8 * 2.0 ** -53


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("use_bounds", [False, True])
@pytest.mark.parametrize("stride,bad", [(1, 0), (4, 33), (16, 5), (32, 31)])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 0.0])
def test_sums_beside_a_track_that_is_not_finite(ctx, dtype, use_bounds, stride, bad, value):
    """A seed that is not finite (or has no momentum, so that its states are not) leaves the sums of the other
    seeds of its group as they are: against the oracle's, within the DCA bars' bound."""
    ev = synth.multi_turn_event(1, counts=(4, 4, 4, 2))
    spec = ev.partitions[0]
    seeds = seen(O.lattice(spec)[:70], dtype).copy()
    others = np.arange(70) != bad
    drift, wires, lam = seen(ev.drift, dtype), seen(ev.wires, dtype), 1e-2
    mask = np.zeros(ev.n_hits, np.uint8)
    op, bp = (c(n_steps=ev.n_steps[0], stride=stride, lam=lam) for c in (O.Params, B.ScanParams))
    ref = O.scan(UNIFORM, op, seeds[others], spec.charge, O.wires_aos(wires), ev.hit_offsets, drift, mask, want_dca=True)
    seeds[bad, 3:] = value
    got = gpu_dca(ctx, B.DeviceField.from_synth(UNIFORM), bp, seeds, spec.charge, wires, ev.hit_offsets, drift, mask, dtype,
                  want_dca=False, use_bounds=use_bounds)
    delta = FP32_DCA_TOL if dtype == torch.float32 else 1e-9
    e = per_wire_residual(ref["dca"], ev.hit_offsets, drift, mask)
    assert (np.abs(got["rss"][others] - ref["rss"]) <= rss_bound(e, lam, delta, dtype == torch.float32) + 1e-15).all()
    edge = (np.abs(e - lam) <= delta).sum(1)
    assert (np.abs(got["n_in"][others] - ref["n_in"]) <= edge).all() and (ref["n_in"] > 0).any()


@pytest.mark.parametrize("dtype,far", [(torch.float32, 1e25), (torch.float64, 1e200)])
@pytest.mark.parametrize("use_bounds", [False, True])
@pytest.mark.parametrize("n_seeds,not_finite", [(1, None), (70, None), (70, 3), (70, 69)])
def test_every_dca_of_a_track_without_distances(ctx, dtype, far, use_bounds, n_seeds, not_finite):
    """A track whose squared distances overflow has its DCAs written when every DCA is wanted: infinite, as the
    distance of its state is, and counted as not converged.  Where there is no distance at all they are NaN."""
    ev = synth.multi_turn_event(1, counts=(4, 4, 4, 2))
    spec = ev.partitions[0]
    seeds = O.lattice(spec)[:n_seeds].copy()
    seeds[0, :2] = far
    if not_finite is not None:
        seeds[not_finite, 3] = np.nan
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=16, lam=1e-2)
    field = B.DeviceField.from_synth(UNIFORM)
    out = gpu_dca(ctx, field, bp, seeds, spec.charge, ev.wires, ev.hit_offsets, ev.drift, np.zeros(ev.n_hits, np.uint8),
                  dtype, use_bounds=use_bounds)
    assert out["n_unconv"] >= ev.n_wires and out["n_in"][0] == 0
    dca = torch.full((ev.n_wires, n_seeds), -1.0, dtype=dtype, device="cuda")
    again = torch.empty(n_seeds, dtype=dtype, device="cuda"), torch.empty(n_seeds, dtype=torch.int32, device="cuda")
    B.comet_scan_dca(ctx, field, bp, out["pts"], out["nv"], out["charge"], out["w"], out["o"], out["d"], out["m"], *again,
                     dca_out=dca, n_wires=ev.n_wires, bounds=out["bounds"])
    dca = dca.double().cpu().numpy().T
    assert np.array_equal(dca, out["dca"], equal_nan=True)
    finite = np.arange(n_seeds) > 0
    assert np.isposinf(dca[0]).all()
    if not_finite is not None:
        assert np.isnan(dca[not_finite]).all()
        finite[not_finite] = False
    assert (np.isfinite(dca[finite]) & (dca[finite] >= 0)).all()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("stride,n_rec", [(1, 201), (1, 401), (2, 201)])
def test_walk_into_another_run(ctx, dtype, stride, n_rec):
    """Two bundles of nearly straight tracks cross at a wide angle beside a few wires.  The group's spheres
    reach the wires before and after the crossing but not at it, so there are two runs of candidate
    states, and each track's closest state lies in one of them: a search of the other run must not keep it
    without its neighbours.  The sums are those of the scan of every state, bit for bit (each closest state
    lies well inside its run)."""
    rng = np.random.default_rng(n_rec)
    h = 4e-3 / stride
    S, ang = 32, np.deg2rad(65.0)
    half = (n_rec - 1) * 4e-3 / 2
    seeds = np.zeros((S, 6))
    for s in range(S):
        a = (ang if s % 2 else -ang) + (rng.normal() * 5e-4)
        seeds[s] = [-half * np.cos(a), -half * np.sin(a), rng.normal() * 1e-3, 100 * np.cos(a), 100 * np.sin(a), 8.0]
    hw = np.array([0.055, 0.058, 0.060, 0.062, 0.065])
    wires = np.stack([np.zeros(5), -hw, np.zeros(5), np.zeros(5), np.zeros(5), np.ones(5)])
    drift = hw * np.cos(ang)
    bp = B.ScanParams(h=h, n_steps=(n_rec - 1) * stride, stride=stride, lam=4e-3, rmax=9.0, zmin=-9.0, zmax=9.0)
    field = B.DeviceField.from_synth(synth.uniform_field(0.001))
    run = lambda all_: gpu_dca(ctx, field, bp, seeds, -1, wires, np.arange(6), drift, np.zeros(5, np.uint8), dtype,
                               want_dca=all_, use_bounds=not all_)
    full, kept = run(True), run(False)
    assert (full["n_in"] > 0).all()
    for name in ("rss", "n_in"):
        assert np.array_equal(full[name], kept[name])
    with_spheres = gpu_dca(ctx, field, bp, seeds, -1, wires, np.arange(6), drift, np.zeros(5, np.uint8), dtype)
    for name in ("dca", "rss", "n_in"):
        assert np.array_equal(full[name], with_spheres[name])


@pytest.mark.parametrize("stride,cut", [(1, 40), (4, 40), (12, 33), (16, 64)])
def test_byte_offsets_of_64_bits_equal_those_of_32(ctx, stride, cut):
    """FP64 and every DCA wanted over a track array above 4 GiB (64-bit byte offsets) against its first seeds
    alone (32-bit): the same states, sums and DCAs."""
    ev = synth.multi_turn_event(1, counts=(16, 16, 32, 32))
    spec = ev.partitions[0]
    n_rec = ev.n_steps[0] // stride + 1
    S = ((1 << 32) // (48 * n_rec) + 64) // 32 * 32
    base = O.lattice(spec)
    seeds = np.concatenate([base[:cut], np.resize(base[::97], (S - cut, 6))])
    W = min(ev.n_wires, 12)
    wires, offs = ev.wires[:, :W], ev.hit_offsets[: W + 1]
    drift, mask = ev.drift[: offs[-1]], np.zeros(offs[-1], np.uint8)
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=stride, lam=1e-2)
    field = B.DeviceField.from_synth(UNIFORM)
    ctx.set_record_blocks(0)
    ctx.set_dca_chunk_wires(32)     # the sums' order depends on the number of seeds otherwise
    try:
        for want in (False, True):
            big = gpu_dca(ctx, field, bp, seeds, spec.charge, wires, offs, drift, mask, torch.float64, want_dca=want)
            n32 = cut // 32 * 32
            small = gpu_dca(ctx, field, bp, seeds[:n32], spec.charge, wires, offs, drift, mask, torch.float64, want_dca=want)
            assert 48 * n_rec * S >= 1 << 32
            for name in ("rss", "n_in") + (("dca",) if want else ()):
                assert np.array_equal(big[name][:n32], small[name])
            assert torch.equal(big["pts"][:, :, :n32], small["pts"])
            del big, small
    finally:
        ctx.set_record_blocks(1)
        ctx.set_dca_chunk_wires(0)


@pytest.mark.parametrize("dtype_name", ["float32", "float64"])
@pytest.mark.parametrize("stride", [1, 4])
def test_batch_of_long_recordings_equals_per_event_scan(ctx, dtype_name, stride):
    """More than 192 recorded states (level-1 segments of several states): the batched launches scan the runs
    of candidate states that the single-event launches walk, with the same bits."""
    from paper_1911_09340_gb300 import batch
    dtype = getattr(torch, dtype_name)
    events = _events(5)
    ctx.set_record_blocks(0)
    try:
        ref = _reference(ctx, events, dtype, stride)
        bs = batch.BatchScanner(ctx, dtype, stride=stride, lam=1e-2, slots=3, max_seeds=4096, max_total_seeds=1 << 13,
                                max_wires=512, max_hits=1024)
        r = bs.run(events, collect=True)
    finally:
        ctx.set_record_blocks(1)
    for rr, res in zip(ref, r["results"]):
        for p, part in enumerate(rr):
            assert res.best_idx[p] == part["idx"] and res.best_rss[p] == part["rss"]
            assert np.array_equal(res.hit_class[p], part["hit_class"])


@pytest.mark.parametrize("fault,step", [("k0", 3), ("k65", 3), ("k_above_S", 3), ("no_idx", 3), ("no_rss", 2), ("no_class", 4),
                                        ("no_points", 1)])
def test_partition_call_refuses_what_its_steps_refuse(ctx, fault, step):
    """comet_scan_partition ends at the step that refuses its arguments, with that step's status; the results
    of the later steps stay as they were, and the context serves the next call."""
    ev = synth.multi_turn_event(1, counts=(2, 3, 2, 2))
    spec = ev.partitions[0]
    S = spec.n_seeds
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=16, lam=1e-2)
    dev = scan.DeviceEvent.from_event(ev)
    field = B.DeviceField.from_synth(UNIFORM)

    def call(k=2, **kw):
        ws = scan.Workspace(S, bp.n_rec, ev.n_hits, k=64)
        ws.idx.fill_(-7), ws.hit_class.fill_(9), ws.rss.fill_(-3.0)
        a = dict(seeds=ws.seeds, charge=ws.charge, points=ws.points, n_valid=ws.n_valid, bounds=ws.bounds, wires=dev.wires,
                 hit_offsets=dev.hit_offsets, drift=dev.drift, hit_mask=dev.mask, rss=ws.rss, n_in=ws.n_in, idx=ws.idx,
                 best=ws.best, hit_class=ws.hit_class, n_wires=dev.W)
        a.update(kw)
        try:
            B.comet_scan_partition(ctx, field, bp, spec, k, **a)
            failed = False
        except B.CometError as e:
            failed = True
            assert e.status == 1
        torch.cuda.synchronize()
        return failed, ws
    kw = {"k0": dict(k=0), "k65": dict(k=65), "k_above_S": dict(k=S + 1), "no_idx": dict(idx=None), "no_rss": dict(rss=None),
          "no_class": dict(hit_class=None),
          "no_points": dict(points=None)}[fault]
    failed, ws = call(**kw)
    assert failed and bool((ws.hit_class == 9).all())
    if step <= 3:
        assert bool((ws.idx == -7).all())
    if step <= 2:
        assert bool((ws.rss == -3.0).all())
    (ok_a, a), (ok_b, b) = call(), call()
    assert not ok_a and not ok_b and torch.equal(a.idx, b.idx) and torch.equal(a.rss[:S], b.rss[:S])
    assert a.idx[:2].tolist() == np.argsort(a.rss[:S].cpu().numpy(), kind="stable")[:2].tolist()


@pytest.mark.parametrize("counts,stride", [((3, 5, 7, 9), 16), ((3, 5, 7, 9), 12), ((4, 4, 8, 3), 32)])
def test_fp32_sums_over_tiles_of_wires(ctx, counts, stride):
    """More wires than one tile holds, FP32 with one-state segments: each seed's counts are those of its wires
    taken in three calls that fit one tile, and its RSS is their sum to the rounding of four FP32 results."""
    ev = synth.multi_turn_event(1, counts=counts)
    spec = ev.partitions[0]
    wires, drift = [], []
    for i in range(12):
        other = synth.multi_turn_event(i, counts=counts)
        wires.append(other.wires)
        drift.append(other.drift[other.hit_offsets[:-1]])
    wires, drift = np.concatenate(wires, 1)[:, :1100], np.concatenate(drift)[:1100]
    assert wires.shape[1] == 1100
    seeds = O.lattice(spec)
    mask = (np.random.default_rng(2).random(1100) < 0.1).astype(np.uint8)
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=stride, lam=1e-2, tol=1e-6)
    field = B.DeviceField.from_synth(UNIFORM)
    run = lambda a, b: gpu_dca(ctx, field, bp, seeds, spec.charge, wires[:, a:b], np.arange(b - a + 1), drift[a:b],
                               mask[a:b], torch.float32, want_dca=False)
    whole = run(0, 1100)
    parts = [run(0, 500), run(500, 1000), run(1000, 1100)]
    assert np.array_equal(whole["n_in"], sum(p["n_in"] for p in parts)) and (whole["n_in"] > 0).any()
    assert whole["n_unconv"] == sum(p["n_unconv"] for p in parts)
    assert np.allclose(whole["rss"], sum(p["rss"] for p in parts), rtol=4 * 2.0 ** -24, atol=0)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("above,stride,n_wires", [(-0.3, 16, 40), (1e-3, 16, 40), (2e-3, 16, 40), (1e-4, 1, 40), (1e-3, 16, 1030)])
def test_every_dca_of_short_tracks(ctx, dtype, above, stride, n_wires):
    """Tracks that leave the region after one to some tens of states: groups whose tracks all have a few states
    are scanned, the others searched by their spheres, in either kernel, with the bits of the scan without spheres."""
    ev = synth.multi_turn_event(1, counts=(7, 4, 8, 9))
    spec = ev.partitions[0]
    zmax = spec.centre[0] + above      # the fourth of the seven values of z0
    seeds = O.lattice(spec)[576:1311]
    wires = np.resize(np.arange(ev.n_wires), n_wires)
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=stride, lam=1e-2, zmax=float(zmax))
    drift = np.random.default_rng(1).uniform(0.0, 8e-3, n_wires)
    full, kept = (gpu_dca(ctx, B.DeviceField.from_synth(UNIFORM), bp, seeds, spec.charge, ev.wires[:, wires],
                          np.arange(n_wires + 1), drift, np.zeros(n_wires, np.uint8), dtype, use_bounds=b) for b in (False, True))
    most = np.array([max(full["nv"].cpu().numpy()[i:i + 32]) for i in range(0, len(seeds), 32)])
    assert (most < 8).any() and (above < 0 or ((most >= 8).any() and (most[most < 8] > 1).any()))
    for name in ("dca", "rss", "n_in"):
        assert np.array_equal(full[name], kept[name])


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("S", [4, 5, 2047, 2048, 2049, 3 * 2048 + 2])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_top_k_by_rounds_or_lists(ctx, dtype, S, k):
    """The smallest k by rounds of an argmin, larger ones by lists, against the oracle's order: one chunk, a last
    chunk shorter than k, signed zeros (equal, so by index), infinities and NaN, ascending and descending input."""
    rng = np.random.default_rng(S + k)
    special = rng.choice(np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1.5, -2.0]), size=S)
    few = np.full(S, np.nan)
    few[rng.integers(S, size=2)] = 7.0
    for v in (special, few, np.full(S, np.inf), np.arange(S, 0, -1.0), np.arange(S) * 1.0):
        v = v.astype(np.float32 if dtype == torch.float32 else np.float64)
        idx = torch.full((k,), -7, dtype=torch.int64, device="cuda")
        val = torch.zeros(k, dtype=dtype, device="cuda")
        B.comet_scan_select(ctx, torch.as_tensor(v, device="cuda"), k, idx, val)
        order = np.lexsort((np.arange(S), np.where(np.isnan(v), 0.0, v), np.isnan(v)))[:k]
        assert np.array_equal(idx.cpu().numpy(), order)
        assert np.array_equal(val.cpu().numpy(), v[order], equal_nan=True)
        only = torch.full((k,), -7, dtype=torch.int64, device="cuda")
        B.comet_scan_select(ctx, torch.as_tensor(v, device="cuda"), k, only, None)
        assert torch.equal(only, idx)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n_seeds,stride,leaving", [(20001, 64, 0), (20001, 64, 3), (20031, 200, 1), (20000, 64, 0), (19999, 5000, 0)])
def test_recording_side_by_side_equals_the_one_with_spheres(ctx, dtype, n_seeds, stride, leaving):
    """Without spheres the warps of a block record side by side when the number of seeds is no multiple of 32: the
    states and counts of the recording with spheres, in full blocks, in the last one (which has fewer warps), in
    blocks with a track that leaves the region, and with a single recorded state."""
    ev = synth.multi_turn_event(1, counts=(4, 4, 8, 4))
    spec = ev.partitions[0]
    seeds = np.resize(O.lattice(spec), (n_seeds, 6))
    for s in np.linspace(40, n_seeds - 1, leaving).astype(int):
        seeds[s, 3:] = [5.0, 0.0, 100.0]
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=stride, zmin=-0.8, zmax=0.8)
    field = B.DeviceField.from_synth(UNIFORM)
    ctx.set_record_blocks(0)
    try:
        bounds = torch.empty(B.bounds_shape(n_seeds), dtype=torch.float32, device="cuda")
        with_spheres = gpu_propagate(ctx, field, bp, seeds, spec.charge, dtype, bounds=bounds)
        alone = gpu_propagate(ctx, field, bp, seeds, spec.charge, dtype)
    finally:
        ctx.set_record_blocks(1)
    assert torch.equal(alone[3], with_spheres[3])
    assert int((alone[3] < bp.n_rec).sum()) == (leaving if bp.n_rec > 1 else 0)
    assert torch.equal(torch.nan_to_num(alone[2], nan=-1e3), torch.nan_to_num(with_spheres[2], nan=-1e3))


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n_seeds,stride", [(1, 1), (33, 16), (70, 7), (5000, 32), (20001, 64)])
def test_recording_in_a_uniform_field_of_any_direction(ctx, dtype, n_seeds, stride):
    """Recorded without spheres (few seeds: a loop of its own) and with them: the same counts, and states that
    agree to two ulp of the largest coordinate and momentum, also for tracks that leave the region."""
    ev = synth.multi_turn_event(1, counts=(4, 4, 8, 4))
    spec = ev.partitions[0]
    seeds = np.resize(O.lattice(spec), (n_seeds, 6))
    bp = B.ScanParams(n_steps=1600, stride=stride, zmin=-0.8, zmax=0.1, rmax=0.65)
    field = B.DeviceField(0, b=(0.05, -0.1, 1.0))
    bounds = torch.empty(B.bounds_shape(n_seeds), dtype=torch.float32, device="cuda")
    a = gpu_propagate(ctx, field, bp, seeds, spec.charge, dtype, bounds=bounds)
    b = gpu_propagate(ctx, field, bp, seeds, spec.charge, dtype)
    assert torch.equal(a[3], b[3])
    if n_seeds > 32:
        assert int(a[3].min()) < bp.n_rec and int(a[3].max()) > 1
    assert torch.equal(torch.isnan(a[2]), torch.isnan(b[2]))
    diff = torch.nan_to_num(a[2] - b[2]).abs().amax((1, 2))
    eps = torch.finfo(dtype).eps
    assert float(diff[:3].max()) <= 2 * eps and float(diff[3:].max()) <= 2 * 128 * eps


@pytest.mark.parametrize("interleaved", [False, True])
def test_fp32_cells_of_many_seeds(ctx, interleaved):
    """More than two warps per scheduler take their cells by another lookup than a few seeds: the same track
    points to 1 um of FP64, for tracks that leave the grid, enter it and run along its edge."""
    half, n = 0.25, 11
    g = np.linspace(-half, half, n)
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    table = np.stack([0.03 * z + 0.02 * y, 0.05 * x * z, 1.0 + 0.1 * x - 0.05 * y * z]).astype(np.float32)
    field = B.DeviceField(1, table=table, origin=(-half,) * 3, spacing=2 * half / (n - 1), interleaved=interleaved)
    start = [(0.0, 0.0, 0.0), (half, 0.0, 0.0), (-half, half, -half), (0.0, -half, half), (half + 0.01, 0.02, 0.0),
             (g[n // 2], g[0], g[n // 2]), (-0.05, 0.04, -half - 0.02), (-3e6, 2e6, 3e6)]
    few = np.array([[*p, 90.0 * np.cos(a), 90.0 * np.sin(a), 20.0] for p in start for a in (0.0, 1.3, 2.9, 4.4, 5.6)])
    few = few.astype(np.float32).astype(np.float64)
    bp = B.ScanParams(n_steps=400, stride=8, zmin=-9e9, zmax=9e9, rmax=9e9)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many = np.resize(few, (256 * sms + 64, 6))
    _, _, p32, n32 = gpu_propagate(ctx, field, bp, many, -1, torch.float32)
    _, _, p64, n64 = gpu_propagate(ctx, field, bp, few, -1, torch.float64)
    m = len(few)
    assert torch.equal(n32[:m], n64) and torch.equal(n32[m:2 * m], n64)
    near = torch.as_tensor(np.abs(few[:, 0]) < 1.0, device="cuda")
    for c in (p32[:, :, :m], p32[:, :, m:2 * m]):
        assert float((c[:3].double() - p64[:3])[:, :, near].abs().max()) < 1e-6
        assert torch.equal(c[:3].isfinite(), p64[:3].isfinite())


@pytest.mark.parametrize("use_bounds", [False, True])
@pytest.mark.parametrize("counts,stride", [((4, 4, 4, 2), 16), ((3, 5, 3, 7), 16), ((3, 5, 3, 7), 8), ((1, 1, 1, 1), 32)])
def test_fp32_sums_in_a_uniform_field_of_any_direction(ctx, use_bounds, counts, stride):
    """Segments of one state (short and long runs) and of several against the oracle, within the DCA bars' bound."""
    ev = synth.multi_turn_event(1, counts=counts)
    spec = ev.partitions[0]
    f32 = torch.float32
    seeds, wires, drift, lam = seen(O.lattice(spec), f32), seen(ev.wires, f32), seen(ev.drift, f32), 1e-2
    mask = np.zeros(ev.n_hits, np.uint8)
    b = tuple(seen((0.05, -0.1, 1.0), f32))
    op, bp = (c(n_steps=ev.n_steps[0], stride=stride, lam=lam) for c in (O.Params, B.ScanParams))
    ref = O.scan(synth.Field(kind=0, b=b), op, seeds, spec.charge, O.wires_aos(wires), ev.hit_offsets, drift, mask, want_dca=True)
    got = gpu_dca(ctx, B.DeviceField(0, b=b), bp, seeds, spec.charge, wires, ev.hit_offsets, drift, mask, f32, want_dca=False,
                  use_bounds=use_bounds)
    e = per_wire_residual(ref["dca"], ev.hit_offsets, drift, mask)
    assert (np.abs(got["rss"] - ref["rss"]) <= rss_bound(e, lam, FP32_DCA_TOL)).all()
    assert (np.abs(got["n_in"] - ref["n_in"]) <= (np.abs(e - lam) <= FP32_DCA_TOL).sum(1)).all() and (ref["n_in"] > 0).all()
