"""State moments of FP32 packets in a sort order, at the sizes where the staged
deposit turns: bins too sparse for a tile (160 packets, CIC 384), chunks of 2136
packets, two of them ordered at a time; packets of one bin spread over its cells or
crowded into one, and on bins of 4 cells.  Tolerance per node: 200 rounded FP32
additions (at most that many meet on a node outside a tile) of the node's sum of
magnitudes, plus one fixed-point unit (2^-31 of the tile's bound) per packet."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2111_14704_gb300 as rs
import rsol_inputs as ri

pytestmark = pytest.mark.gpu

GRID = (32, 32, 32)


@pytest.mark.parametrize("shape,n,crowded", [(2, 1, False), (2, 160, False), (2, 161, False),
                                             (1, 384, False), (1, 385, True), (2, 2136, False),
                                             (2, 2137, True), (2, 4272, False), (2, 4273, False),
                                             (1, 4273, False), (2, 9001, True), (2, 30011, False)])
def test_moments_of_one_bin_against_oracle(shape, n, crowded):
    parts = ri.make_particles(n, GRID, 37)
    for a in range(3):
        parts["cell"][a] = 11 if crowded else 9 + parts["cell"][a] % 6
    A, P = rs.Particles.from_numpy(parts, 32), rs.Particles.empty(n, 32)
    ctx = rs.Context(rs.Params(*GRID, shape=shape, precision=32, c_tilde=0.1, warps=16))
    ctx.sort(A, P)
    M = ctx.grid_tensor()
    ctx.deposit(P, M)
    ctx.check()
    got = rs.grid_to_planes(M).astype(np.float64)
    host = P.to_numpy()
    op = oracle.params(GRID, shape=shape, dt=1.0, c_tilde=0.1)
    ref = oracle.state_moments(op, oracle.Particles(host))
    # magnitudes: every component of every packet positive (the weights are)
    pos = dict(host, u=np.abs(host["u"]))
    mag = oracle.state_moments(op, oracle.Particles(pos))
    one = dict(host, w=np.ones(n))
    crowd = max(1.0, float(oracle.state_moments(op, oracle.Particles(one))[0].max()))
    w = float(host["w"].max())
    u = np.sqrt((host["u"] ** 2).sum(axis=0)).max()
    bound = [w, w * u, w * u, w * u, w * np.sqrt(1 + u * u), w, w, w]
    for q in range(8):
        tol = 200 * 2.0**-24 * mag[q] + n * 2.0**-31 * 2.01 * crowd * bound[q]
        err = np.abs(got[q] - ref[q])
        assert (err <= tol).all(), (q, float((err - tol).max()))
