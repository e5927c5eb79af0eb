"""State moments of a sorted FP32 set over the range of FP32: very large and very small
weights, and a packet with a value that is not finite, or whose |u|^2 is not, in a bin
summed through its tile and in one too sparse for it.  Such a packet changes only its
own nodes, as it does in a set that was never sorted.  Tolerance per node: the rounding
of the FP32 additions that can meet there (200 in a tile's set, as in an ordinary one; one
per packet where a whole bin goes to the grid packet by packet) of the node's sum of
magnitudes, plus one fixed-point unit (2^-31 of the tile's bound) per packet."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2111_14704_gb300 as rs
import rsol_inputs as ri

pytestmark = pytest.mark.gpu

GRID = (32, 32, 32)


def one_bin(n, seed):
    parts = ri.make_particles(n, GRID, seed)
    for a in range(3):
        parts["cell"][a] = 9 + parts["cell"][a] % 6
    return parts


def moments(parts, shape, sort):
    n = parts["w"].size
    ctx = rs.Context(rs.Params(*GRID, shape=shape, precision=32, c_tilde=0.1))
    P = rs.Particles.from_numpy(parts, 32)
    if sort:
        Q = rs.Particles.empty(n, 32)
        ctx.sort(P, Q)
        P = Q
    M = ctx.grid_tensor()
    ctx.deposit(P, M)
    return rs.grid_to_planes(M).astype(np.float64)


def reference(parts, shape, adds):
    """The oracle's moments and the tolerance per component."""
    n = parts["w"].size
    op = oracle.params(GRID, shape=shape, dt=1.0, c_tilde=0.1)
    run = lambda p: oracle.state_moments(op, oracle.Particles(p))
    ref, mag = run(parts), run(dict(parts, u=np.abs(parts["u"])))
    crowd = max(1.0, float(run(dict(parts, w=np.ones(n)))[0].max()))
    w, u = float(parts["w"].max()), np.sqrt((parts["u"] ** 2).sum(axis=0)).max()
    bound = [w, w * u, w * u, w * u, w * np.sqrt(1 + u * u), w, w, w]
    return ref, [adds * 2.0**-24 * mag[q] + n * 2.0**-31 * 2.01 * crowd * bound[q] for q in range(8)]


@pytest.mark.parametrize("shape,n", [(2, 100), (2, 3000), (1, 3000), (2, 5000)])
@pytest.mark.parametrize("scale", [1e-25, 1e-12, 1e20, 1e25, 1e30])
def test_weights_over_the_range_of_fp32(shape, n, scale):
    parts = one_bin(n, 43)
    parts["w"] = (parts["w"] * scale).astype(np.float32).astype(np.float64)
    got = moments(parts, shape, True)
    ref, tol = reference(parts, shape, 200)
    for q in range(8):
        err = np.abs(got[q] - ref[q])
        assert (err <= tol[q]).all(), (q, float((err / np.maximum(tol[q], 1e-300)).max()))


@pytest.mark.parametrize("n", [100, 3000, 5000])
@pytest.mark.parametrize("what,value", [("u", np.nan), ("u", np.inf), ("u", 1e20), ("w", np.nan), ("w", np.inf),
                                        ("off", np.nan)])
def test_a_packet_out_of_range_changes_only_its_own_nodes(n, what, value):
    parts = one_bin(n, 47)
    bad = {k: v.copy() for k, v in parts.items()}
    j = n // 3
    if what == "w":
        bad["w"][j] = value
    else:
        bad[what][0][j] = value
    got, plain = moments(bad, 2, True), moments(bad, 2, False)
    others = {k: np.delete(v, j, axis=-1) for k, v in parts.items()}
    ref, tol = reference(others, 2, n)
    # nodes within two cells of the packet's (its stencil's, whatever the offset)
    idx = [np.arange(g) for g in GRID]
    near = [np.abs(idx[a] - parts["cell"][a][j]) <= 2 for a in range(3)]
    mine = near[2][:, None, None] & near[1][None, :, None] & near[0][None, None, :]
    for q in range(8):
        g = got[q].reshape(mine.shape)
        assert (np.abs(g - ref[q].reshape(mine.shape)) <= np.reshape(tol[q], mine.shape))[~mine].all(), q
        p = plain[q].reshape(mine.shape)
        assert np.array_equal(np.isfinite(g), np.isfinite(p)), q
