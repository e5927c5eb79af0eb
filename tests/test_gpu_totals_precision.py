"""Totals of FP32 packets carry at least the 53 bits of FP64, whatever the path.

The packets of `test_no_bits_lost` repeat 64 weights and momenta so that every thread of
the first level sums the same 64 products: rounding errors of its sums add up instead of
averaging out.  The exact total is the sum of those 64 (products of two FP32 numbers are
exact in FP64, math.fsum rounds once), times 2^18.  Bar: 48 roundings of FP64, those of
the additions over warps (7) and blocks (37) and of the factors."""
from __future__ import annotations

import math

import numpy as np
import pytest

import paper_2111_14704_gb300 as rs

pytestmark = pytest.mark.gpu


def totals(w, u, fb=None):
    import torch
    n = w.numel()
    ctx = rs.Context(rs.Params(8, 8, 8, precision=32, c_tilde=0.1))
    z = torch.zeros(n, device="cuda")
    P = rs.Particles(torch.zeros(n, dtype=torch.int32, device="cuda"), [z, z.clone(), z.clone()], u, w)
    got = ctx.moments(P, fb)
    assert np.array_equal(got, ctx.moments(P, fb))
    return got


@pytest.mark.parametrize("scale", [1.0, 2.0**-60, 2.0**70])
def test_no_bits_lost(scale):
    import torch
    g = np.random.default_rng(39)
    w = (np.exp(g.uniform(-3, 3, 64)).astype(np.float32) * np.float32(scale)).astype(np.float32)
    u = [np.exp(g.uniform(0, 4, 64)).astype(np.float32) for _ in range(3)]
    n = 1 << 24  # 1024 blocks of 16384, 64 packets a thread, one per 256
    spread = lambda p: torch.from_numpy(p).cuda().repeat_interleave(256).repeat(n // 16384)
    got = totals(spread(w), [spread(x) for x in u])
    for q, f in enumerate([np.ones(64, np.float32), *u]):
        terms = w.astype(np.float64) * f
        want = math.fsum(terms) * (n // 64)
        assert abs(got[q] - want) <= 48 * 2.0**-53 * want, (q, (got[q] - want) / want * 2.0**53)


def test_feedback_sums_lose_no_bits():
    import torch
    g = np.random.default_rng(40)
    ctx_nodes = 512
    fb = torch.from_numpy(np.exp(g.uniform(-8, 8, (ctx_nodes, 8))).astype(np.float32)).cuda()
    one = torch.ones(1, device="cuda")
    got = totals(one, [one.clone() for _ in range(3)], fb)
    v = fb.double().cpu().numpy()
    for q in range(8):
        want = math.fsum(v[:, q])
        assert abs(got[8 + q] - want) <= 48 * 2.0**-53 * want, q


@pytest.mark.parametrize("n,late", [(20000, False), (3000001, False), (200001, True), (3000001, True)])
@pytest.mark.parametrize("wlo,whi,ulo,uhi", [(0.9 * 2.0**60, 2.0**60, 0.9 * 2.0**60, 2.0**60), (1e-14, 1e-13, 1.0, 10.0),
                                             (1e-30, 1e30, 1e-3, 1e3), (1e37, 1e38, 1e-12, 1e-9)])
def test_values_at_and_past_the_range(n, late, wlo, whi, ulo, uhi):
    """Large enough for FP32 sums to overflow, small weights, weights too far apart for one
    scale, momenta too small; in every block from its first packets on, or from its second
    thousand (late).  Terms of weights and momenta are exact: 2^-44 of the magnitudes."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    logu = lambda lo, hi: torch.exp(math.log(lo) + (math.log(hi) - math.log(lo)) *
                                    torch.rand(n, dtype=torch.float64, device="cuda", generator=g)).float()
    w, u = logu(wlo, whi), [logu(ulo, uhi) for _ in range(3)]
    if late:
        blocks = min(1024, n // 1024 + 1)
        first = torch.arange(n, device="cuda") % -(-n // blocks) < 1024
        w = torch.where(first, torch.ones_like(w), w)
        u = [torch.where(first, torch.ones_like(x), x) for x in u]
    got = totals(w, u)
    N, U = w.double(), [x.double() for x in u]
    gam = torch.sqrt(1 + U[0] ** 2 + U[1] ** 2 + U[2] ** 2)
    want = [float(x.sum()) for x in [N, *(N * x for x in U), N * gam, *(N * x / gam for x in U)]]
    for q in range(8):
        assert abs(got[q] - want[q]) <= (2.0**-44 if q < 4 else 2.0**-22) * want[q], q
