"""Deterministic FP32 deposits do not depend on the CTA width: 8 and 16 warps give the same
bits in one box (bins of one and of several chunks of 1232 packets, 776 in bins of 4 cells),
and a batch of dense bins at either width equals one push per box."""
from __future__ import annotations

import pytest

import paper_2111_14704_gb300 as rs
import rsol_inputs as ri
from tests.test_gpu_batch import _batch, _det_batch_equals_per_box

pytestmark = pytest.mark.gpu

GRID = (32, 32, 32)


@pytest.mark.parametrize("shape,bin_,n", [(2, 8, 1232), (2, 8, 1233), (2, 8, 2000), (1, 8, 2000), (2, 8, 3001),
                                          (2, 8, 9000), (2, 4, 1000), (2, 4, 1553), (2, 4, 2100)])
def test_widths_give_the_same_bits(shape, bin_, n):
    import torch
    parts = ri.make_particles(n, GRID, 71)
    for a in range(3):
        parts["cell"][a] = 9 + parts["cell"][a] % 2
    modes = ri.alfven_modes(8, 71, L=(32.0,) * 3, kmax=4, dB_rms=0.2)
    planes = ri.field_grid(GRID, modes=modes, vA=0.01, u_gas=(0.0, 0.01, 0.0))
    out = []
    for warps in (8, 16, 0):
        ctx = rs.Context(rs.Params(*GRID, shape=shape, precision=32, c_tilde=0.1, deterministic=1, bin=bin_,
                                   warps=warps))
        A, P = rs.Particles.from_numpy(parts, 32), rs.Particles.empty(n, 32)
        ctx.sort(A, P)
        fb = ctx.grid_tensor()
        ctx.push_gather(P, rs.fields_to_device(planes, 32), 2.0, fb)
        ctx.check()
        out.append(fb)
    assert torch.equal(out[0], out[1]) and torch.equal(out[1], out[2])


@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("warps", [8, 16])
def test_dense_batch_of_either_width_equals_per_box(shape, warps):
    _det_batch_equals_per_box(_batch(6, 13, 32, shape=shape, det=1, n_lo=8, n_hi=20, p_lo=2 ** 11, p_hi=2 ** 15),
                              shape, warps)
