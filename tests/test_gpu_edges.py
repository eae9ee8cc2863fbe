"""Edges of the kernels' own branches: warps with fewer than 32 seeds, tile and list sizes, and the paths
a launch takes by size, each against the general path or the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from paper_1911_09340_gb300 import binding as B
from paper_1911_09340_gb300 import scan, synth

from gpu_util import gpu_dca, gpu_propagate

pytestmark = pytest.mark.gpu
UNIFORM = synth.uniform_field(1.0)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("stride,n_seeds", [(1, 33), (5, 64), (16, 1), (16, 31), (24, 97), (32, 4100)])
def test_recording_inside_the_region_equals_the_tested_one(ctx, dtype, stride, n_seeds):
    """A warp whose tracks provably stay inside the target region records without the per-state test.
    With the region's radius 20 um above the largest recorded one the proof's margin (0.1 mm) fails but
    no track leaves, so the same seeds take the general loop: points, counts and spheres are the same
    bits, also in a last warp with fewer than 32 seeds."""
    ev = synth.multi_turn_event(1, counts=(8, 8, 16, 8))
    spec = ev.partitions[0]
    seeds = O.lattice(spec)[:n_seeds]
    field = B.DeviceField.from_synth(UNIFORM)
    bp = B.ScanParams(n_steps=ev.n_steps[0] // stride * stride, stride=stride, zmin=-9.0, zmax=9.0, rmax=9.0)
    ctx.set_record_blocks(0)
    try:
        def record(p):
            bounds = torch.full(B.bounds_shape(n_seeds), -7.0, dtype=torch.float32, device="cuda")
            _, _, pts, nv = gpu_propagate(ctx, field, p, seeds, spec.charge, dtype, bounds=bounds)
            return pts, nv, bounds
        free = record(bp)
        rho = float(torch.hypot(free[0][0], free[0][1]).max())
        edge = record(dataclasses.replace(bp, rmax=rho + 2e-5))
    finally:
        ctx.set_record_blocks(1)
    for a, b in zip(free, edge):
        assert torch.equal(a, b)
    assert bool((free[1] == bp.n_rec).all())


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("S", [64, 65, 127, 2048 + 63, 2 * 2048 + 1, 40 * 2048 + 5])
@pytest.mark.parametrize("k", [2, 32, 33, 64])
def test_top_k_lists(ctx, dtype, S, k):
    """The warps' sorted lists of 64 against the oracle's selection: a last chunk shorter than k, list
    halves, signed zeros (equal, so by index), infinities and NaN, descending input (every key enters)."""
    rng = np.random.default_rng(S + k)
    special = rng.choice(np.array([0.0, -0.0, np.inf, np.nan, 1.5, -2.0, 3.0]), size=S)
    for v in (special, np.arange(S, 0, -1, dtype=np.float64)):
        v = v.astype(np.float32 if dtype == torch.float32 else np.float64)
        rss = torch.as_tensor(v, device="cuda")
        idx = torch.full((k,), -7, dtype=torch.int64, device="cuda")
        val = torch.zeros(k, dtype=dtype, device="cuda")
        B.comet_scan_select(ctx, rss, k, idx, val)
        order = np.lexsort((np.arange(S), np.where(np.isnan(v), 0.0, v), np.isnan(v)))[:k]
        assert np.array_equal(idx.cpu().numpy(), order)
        assert np.array_equal(val.cpu().numpy(), v[order], equal_nan=True)
        assert np.array_equal(np.signbit(val.cpu().numpy()), np.signbit(v[order]))


@pytest.mark.parametrize("M", [1, 127, 128, 129, 700])
@pytest.mark.parametrize("half_width", [(0.03125, 0.5, 2.0, 3.0), (0.015625, 1.6, 1.5, 5.0), (0.0, 0.0, 0.0, 0.0)])
def test_reference_walk_over_tiles(ctx, M, half_width):
    """References from more candidates than one tile, with unused slots and with z0 and pz on a lattice
    (differences that equal the width exactly) and phi across the +-pi seam, against the oracle."""
    rng = np.random.default_rng(M)
    n = 900
    z, phi = rng.integers(-8, 9, n) / 64.0, rng.uniform(-np.pi, np.pi, n)
    pz, pt = np.round(rng.uniform(10, 20, n)), rng.uniform(95, 105, n)
    seeds = np.stack([0 * z, 0 * z, z, pt * np.cos(phi), pt * np.sin(phi), pz], axis=1)
    idx = rng.integers(-2, n + 2, size=M)
    idx[0] = 5
    K = 32
    refs = torch.zeros((K, 4), dtype=torch.float64, device="cuda")
    nref = torch.zeros(1, dtype=torch.int32, device="cuda")
    dev = torch.as_tensor(np.ascontiguousarray(seeds.T), device="cuda")
    B.comet_scan_refine_refs(ctx, dev, torch.as_tensor(idx, device="cuda"), half_width, K, refs, nref)
    got = refs[: int(nref)].cpu().numpy()
    want = O.refine_refs(seeds, idx, half_width, K)
    assert got.shape == want.shape
    assert np.allclose(got, want, rtol=1e-14, atol=1e-14)


@pytest.mark.parametrize("n_seeds,n_wires,stride", [(1, 1, 16), (5, 2, 1), (7, 3, 16), (3, 16, 4), (2, 33, 16), (65, 5, 32)])
def test_jacobian_lane_groups(ctx, n_seeds, n_wires, stride):
    """Few wires share a warp between seeds (2^n lanes each), more than 32 take several warps: the DCAs are
    the oracle's to 1e-9 m where the refinement converges, and the sums are those of the per-wire
    values in ascending wire order."""
    ev = synth.single_event_fp64()
    spec = ev.partitions[0]
    rng = np.random.default_rng(n_seeds)
    theta = np.array(spec.centre) + rng.uniform(-0.2, 0.2, (n_seeds, 4)) * np.array(spec.half_width)
    near = np.nonzero([np.any(ev.hit_turn[a:b] == 0) for a, b in zip(ev.hit_offsets[:-1], ev.hit_offsets[1:])])[0]
    wires = ev.wires[:, near[:n_wires]]
    W = wires.shape[1]
    assert W == n_wires
    drift = rng.uniform(0.0, 8e-3, W)
    lam, tau = 1e-2, 1e-3
    p = B.ScanParams(n_steps=ev.n_steps[0], stride=stride, lam=lam)
    f64 = dict(dtype=torch.float64, device="cuda")
    t = lambda x, d=torch.float64: torch.as_tensor(np.ascontiguousarray(x), dtype=d, device="cuda")
    work, D, J = torch.empty(n_seeds * W * 11, **f64), torch.empty((n_seeds, W), **f64), torch.empty((n_seeds, W, 4), **f64)
    srss, grad, jtj, jtr = (torch.empty(s, **f64) for s in (n_seeds, (n_seeds, 4), (n_seeds, 16), (n_seeds, 4)))
    B.comet_scan_jacobian(ctx, B.DeviceField.from_synth(UNIFORM), p, t(theta), *spec.vxy, spec.charge, t(wires),
                          t(np.arange(W + 1), torch.int32), t(drift), t(np.zeros(W), torch.uint8), tau, work, srss,
                          grad, jtj, jtr, dca_out=D, jac_out=J)
    seeds = np.stack([np.full(n_seeds, spec.vxy[0]), np.full(n_seeds, spec.vxy[1]), theta[:, 0],
                      theta[:, 3] * np.cos(theta[:, 1]), theta[:, 3] * np.sin(theta[:, 1]), theta[:, 2]], axis=1)
    ref = O.scan(UNIFORM, O.Params(n_steps=ev.n_steps[0], stride=stride, lam=lam), seeds, spec.charge,
                 O.wires_aos(wires), np.arange(W + 1, dtype=np.int32), drift, np.zeros(W, np.uint8), want_dca=True)
    D, J = D.cpu().numpy(), J.cpu().numpy()
    assert np.abs(D - ref["dca"]).max() <= 1e-9
    rho = D - drift
    e = np.abs(rho)
    w = 1.0 / (1.0 + np.exp(-(lam - e) / tau))
    assert np.allclose(srss.cpu(), (w * e * e + (1 - w) * lam * lam).sum(1), rtol=1e-12)
    assert np.allclose(jtr.cpu(), ((w * rho)[..., None] * J).sum(1), rtol=1e-10, atol=1e-12)
    assert np.allclose(jtj.cpu().numpy().reshape(-1, 4, 4), np.einsum("sw,swi,swj->sij", w, J, J), rtol=1e-10, atol=1e-12)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("stride,n_seeds,zmax", [(1, 64, 9.0), (2, 33, 9.0), (8, 97, 9.0), (11, 64, 9.0), (12, 40, 9.0),
                                                 (16, 1, 9.0), (32, 64, 9.0), (32, 97, -0.3), (1, 40, -0.3)])
def test_closest_state_without_scanning_equals_the_scan(ctx, dtype, stride, n_seeds, zmax):
    """The walk down a track's valley and the spheres' bounds against the scan of every recorded state
    (DCAs wanted, no spheres given): the same DCAs, sums and counts, bit for bit.  Level-1 segments of one
    state (more than 192 states have several each), runs across super-segments, tracks that leave the
    region, chamber wires, wires of any direction (along the tracks too, where the valley is not
    convex and is scanned) and wires around the helix axis, which every state is equally far from."""
    ev = synth.multi_turn_event(1, counts=(8, 8, 16, 8))
    spec = ev.partitions[0]
    seeds = O.lattice(spec)[:n_seeds]
    rng = np.random.default_rng(stride)
    path, _ = O.propagate(UNIFORM, O.Params(n_steps=ev.n_steps[0], stride=1), seeds[:1], spec.charge)
    n = 60
    at = path[0, rng.integers(0, path.shape[1], n), :3] + rng.normal(scale=6e-3, size=(n, 3))
    u = rng.normal(size=(n, 3)) * [1.0, 1.0, 2.0]
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    centre = path[0, :, :3].mean(0)
    wires = np.concatenate([ev.wires, np.concatenate([at, u], 1).T,
                            np.array([[*centre, 0.0, 0.0, 1.0], [*path[0, 0, :3], 0.0, 0.0, 1.0]]).T], axis=1)
    W = wires.shape[1]
    offs = np.arange(W + 1, dtype=np.int32)
    drift = rng.uniform(0.0, 8e-3, W)
    mask = (rng.random(W) < 0.1).astype(np.uint8)
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=stride, zmax=zmax, lam=1e-2)

    def run(p, want_dca, use_bounds):
        return gpu_dca(ctx, B.DeviceField.from_synth(UNIFORM), p, seeds, spec.charge, wires, offs, drift, mask, dtype,
                       want_dca=want_dca, use_bounds=use_bounds)
    full, kept = run(bp, True, False), run(bp, True, True)
    for name in ("dca", "rss", "n_in"):
        assert np.array_equal(full[name], kept[name])


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("stride,bad", [(1, 0), (16, 5), (16, 31), (32, 33)])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_every_dca_beside_a_track_that_is_not_finite(ctx, dtype, stride, bad, value):
    """A seed that is not finite spoils its group's spheres; when every DCA is wanted the other seeds of
    the group still get theirs, as without spheres."""
    ev = synth.multi_turn_event(1, counts=(4, 4, 4, 2))
    spec = ev.partitions[0]
    seeds = O.lattice(spec)[:70].copy()
    seeds[bad, 3] = value
    W = ev.n_wires
    bp = B.ScanParams(n_steps=ev.n_steps[0], stride=stride, lam=1e-2)
    full, kept = (gpu_dca(ctx, B.DeviceField.from_synth(UNIFORM), bp, seeds, spec.charge, ev.wires, ev.hit_offsets,
                          ev.drift, np.zeros(ev.n_hits, np.uint8), dtype, want_dca=True, use_bounds=b) for b in (False, True))
    others = np.arange(70) != bad
    assert full["dca"].shape == (70, W) and np.isfinite(full["dca"][others]).all()
    for name in ("dca", "rss", "n_in"):
        assert np.array_equal(full[name], kept[name], equal_nan=True)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("k,counts,want_dca", [(1, (2, 3, 4, 5), False), (1, (1, 1, 1, 1), True), (10, (3, 4, 5, 6), True),
                                               (64, (4, 4, 4, 4), False)])
def test_partition_in_one_call_equals_the_five(ctx, dtype, k, counts, want_dca):
    """scan_partition without a timer is one native call, with one it is five: the same results, in a
    workspace larger than the partition, with and without the optional outputs."""
    ev = synth.multi_turn_event(1, counts=counts)
    spec = ev.partitions[0]
    bp = scan.event_params(ev, dtype, 16)[0]
    out = []
    for timer in (None, scan.KernelTimer()):
        dev = scan.DeviceEvent.from_event(ev, dtype)
        ws = scan.Workspace(spec.n_seeds + 40, bp.n_rec + 3, ev.n_hits + 5, dtype, k=k)
        ws.hit_class.fill_(7)
        dca = torch.full((dev.W, spec.n_seeds), -1.0, dtype=dtype, device="cuda") if want_dca else None
        wire = torch.full((dev.W,), -1.0, dtype=dtype, device="cuda") if want_dca else None
        best = torch.full((1,), -5, dtype=torch.int64, device="cuda") if k == 1 and want_dca else None
        scan.scan_partition(ctx, B.DeviceField.from_synth(UNIFORM), bp, spec, dev, ws, k=k, want_dca=dca, dca_wire=wire,
                            best_idx=best, timer=timer)
        n = spec.n_seeds
        out.append([ws.rss[:n], ws.n_in[:n], ws.idx if best is None else best, ws.best[:k], ws.hit_class, dev.mask,
                    ws.n_unconv] + ([dca, wire] if want_dca else []))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    small = scan.Workspace(max(spec.n_seeds - 1, 1), bp.n_rec - 1, ev.n_hits, dtype, k=k)
    with pytest.raises(RuntimeError):
        scan.scan_partition(ctx, B.DeviceField.from_synth(UNIFORM), bp, spec, dev, small, k=k)


@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("half,n", [(0.9, 37), (0.25, 11), (0.0625, 2), (0.5, 3)])
def test_fp32_field_cells_and_the_grid_edge(ctx, half, n, interleaved):
    """FP32 recording in a table that the track leaves, enters and runs along (seeds on nodes, on the edge
    and outside, where coordinates are clamped; a grid of one cell) against the FP64 kernel, whose cells
    come from the general lookup: within 1 um, the bar of the FP32 points."""
    g = np.linspace(-half, half, n)
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    table = np.stack([0.03 * z + 0.02 * y, 0.05 * x * z, 1.0 + 0.1 * x - 0.05 * y * z]).astype(np.float32)
    field = B.DeviceField(1, table=table, origin=(-half,) * 3, spacing=2 * half / (n - 1), interleaved=interleaved)
    start = [(0.0, 0.0, 0.0), (half, 0.0, 0.0), (-half, half, -half), (0.0, -half, half), (half + 0.01, 0.02, 0.0),
             (g[n // 2], g[0], g[n // 2]), (-0.05, 0.04, -half - 0.02)]
    seeds = np.array([[*p, 90.0 * np.cos(a), 90.0 * np.sin(a), 20.0] for p in start for a in (0.0, 1.3, 2.9, 4.4, 5.6)])
    bp = B.ScanParams(n_steps=1600, stride=8, zmin=-9.0, zmax=9.0, rmax=9.0)
    seeds = seeds.astype(np.float32).astype(np.float64)
    _, _, p32, n32 = gpu_propagate(ctx, field, bp, seeds, -1, torch.float32)
    _, _, p64, n64 = gpu_propagate(ctx, field, bp, seeds, -1, torch.float64)
    assert torch.equal(n32, n64)
    assert float((p32[:3].double() - p64[:3]).abs().max()) < 1e-6
