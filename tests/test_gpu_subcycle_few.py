"""Tiled sub-cycling of few FP32 packets: levels pushed as order-free slices of the
sorted arrays (default CTA width) against levels pushed in bins' tiles (16 warps asked
for).  Packets must agree bit for bit; the densities to twice the FP32 bar of 1e-5
relative L2 that each keeps to the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2111_14704_gb300 as rs
import rsol_inputs as ri
from tests.gpu_helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n,grid", [(2, 1, (16, 16, 16)), (2, 4099, (32, 24, 20)), (1, 30011, (32, 32, 32)),
                                          (2, 117953, (29, 109, 18))])
def test_slices_match_tiles(shape, n, grid):
    import torch
    parts = ri.make_particles(n, grid, 41)
    modes = ri.alfven_modes(8, 41, L=tuple(map(float, grid)), kmax=4, dB_rms=0.2)
    planes = ri.field_grid(grid, modes=modes, vA=0.01, u_gas=(0.0, 0.01, 0.0))
    out = []
    for warps in (0, 16):
        ctx = rs.Context(rs.Params(*grid, shape=shape, precision=32, c_tilde=0.1, warps=warps))
        F = rs.fields_to_device(planes, 32)
        P, Q, fb = rs.Particles.from_numpy(parts, 32), rs.Particles.empty(n, 32), ctx.grid_tensor()
        counts = ctx.sort_push_subcycled(P, Q, F, 10.0, 0.2, fb)
        torch.cuda.synchronize()
        ctx.check()
        out.append((Q, rs.grid_to_planes(fb), np.asarray(counts)))
    (A, a, ca), (B, b, cb) = out
    assert np.array_equal(ca, cb)
    for x, y in zip(A.tensors(), B.tensors()):
        assert torch.equal(x, y)
    for q in range(8):
        assert rel_l2(a[q], b[q]) <= 2e-5, q
