"""Edges of the kernels' own branches: warps with fewer than 32 seeds, tile and list sizes, and the paths
a launch takes by size, each against the general path or the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from paper_1911_09340_gb300 import binding as B
from paper_1911_09340_gb300 import synth

from gpu_util import gpu_propagate

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
