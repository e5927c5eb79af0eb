"""The FP64 totals of FP32 packets (summed in pairs of floats) against numpy in
FP64: a few packets, a ragged count over all blocks, values outside the pairs'
range (which the kernel sums in FP64) and a feedback grid that is not 16-byte
aligned.  gamma and beta are rounded to FP32 per packet, so totals agree to
2^-23 relative to the sum of magnitudes; a total of weights and momenta, whose
terms are exact, to 2^-44."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2111_14704_gb300 as rs
import rsol_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,wscale,uscale", [(1, 1.0, 1.0), (1000003, 1.0, 1.0), (5000, 1e-30, 1.0),
                                             (5000, 1e30, 1e-20), (5000, 1.0, 0.0)])
def test_totals_against_numpy(n, wscale, uscale):
    import torch
    grid = (12, 10, 8)
    parts = ri.make_particles(n, grid, 5)
    rng = np.random.default_rng(3)
    parts["w"] = (rng.random(n) * wscale).astype(np.float32).astype(np.float64)
    parts["u"] = (parts["u"] * uscale).astype(np.float32).astype(np.float64)
    ctx = rs.Context(rs.Params(*grid, precision=32, c=2.0, c_tilde=0.5, q=3.0, q_over_m=1.5, dx=0.5))
    P = rs.Particles.from_numpy(parts, 32)
    flat = torch.randn(12 * 10 * 8 * 8 + 1, device="cuda")
    fb = flat[1:]  # 4-byte aligned
    got = ctx.moments(P, fb)
    m, c, q = 2.0, 2.0, 3.0
    N, u = parts["w"], parts["u"]
    g = np.sqrt(1.0 + (u * u).sum(0))
    terms = np.stack([N, *(N * m * c * u), N * g * m * c * c, *(N * q * c * u / g)])
    want, mag = terms.sum(1), np.abs(terms).sum(1)
    tol = np.array([2.0 ** -44] * 4 + [2.0 ** -22] * 4)
    assert np.all(np.abs(got[:8] - want) <= tol * mag)
    G = fb.double().cpu().numpy().reshape(-1, 8) * 0.125
    assert np.all(np.abs(got[8:] - G.sum(0)) <= 2.0 ** -44 * np.abs(G).sum(0))
    assert np.array_equal(got, ctx.moments(P, fb))
