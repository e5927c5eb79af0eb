"""FP32 pushes of boxes with few bins, default CTA width: sparse bins dealt to several
CTAs (8 bins: 16 slices, 64 bins: 2), at the packet counts where a bin turns to its tile
(160 TSC or 384 CIC packets a slice, at most 768), and dense bins, whose sums must keep
the tile's accuracy however few the bins.

Sums of K positive FP32 values that grow evenly round by 2^-24 / sqrt(12) sqrt(K / 3) of
the total in the root mean square; the bar for rho is twice that, K the additions of
tiles to the grid that meet on a node (eight bins, one per two chunks of 2176 packets);
as global sums of one value per packet the same boxes miss it by a factor of 3 or more."""
from __future__ import annotations

import math

import numpy as np
import pytest

import oracle
import paper_2111_14704_gb300 as rs
import rsol_inputs as ri
from tests.gpu_helpers import rel_l2

pytestmark = pytest.mark.gpu


def fields(grid):
    modes = ri.alfven_modes(8, 53, L=tuple(map(float, grid)), kmax=4, dB_rms=0.2)
    return ri.field_grid(grid, modes=modes, vA=0.01, u_gas=(0.0, 0.01, 0.0)).astype(np.float32).astype(np.float64)


def bar(k):
    return 2 * 2.0**-24 / math.sqrt(12) * math.sqrt(k / 3)


@pytest.mark.parametrize("deterministic", [0, 1])
@pytest.mark.parametrize("edge,shape,n", [(16, 2, 1), (16, 2, 15), (16, 2, 161), (16, 2, 768), (16, 2, 769),
                                          (16, 1, 768), (16, 1, 769), (32, 2, 320), (32, 2, 321), (32, 1, 768)])
def test_slices_of_a_sparse_bin(edge, shape, n, deterministic):
    import torch
    grid = (edge,) * 3
    parts = ri.make_particles(n, grid, 59)
    for a in range(3):
        parts["cell"][a] = 9 + parts["cell"][a] % 6
    planes = fields(grid)
    params = rs.Params(*grid, shape=shape, precision=32, c_tilde=0.1, deterministic=deterministic)
    ctx, other = rs.Context(params), rs.Context(params)
    A, P, R = rs.Particles.from_numpy(parts, 32), rs.Particles.empty(n, 32), rs.Particles.empty(n, 32)
    ctx.sort(A, P)
    for x, y in zip(R.tensors(), P.tensors()):
        x.copy_(y)
    op = oracle.params(grid, shape=shape, dt=2.0, c_tilde=0.1)
    OP = oracle.Particles(P.to_numpy())
    F = rs.fields_to_device(planes, 32)
    for _ in range(2):
        fb, free = ctx.grid_tensor(), ctx.grid_tensor()
        ctx.push_gather(P, F, 2.0, fb)
        other.push_gather(R, F, 2.0, free)
        G, got = oracle.step(op, planes, OP), rs.grid_to_planes(fb)
        for q in range(8):
            assert rel_l2(got[q], G[q]) <= 1e-5, q
    ctx.check()
    for x, y in zip(P.tensors(), R.tensors()):
        assert torch.equal(x, y)


@pytest.mark.parametrize("edge,shape,n,crowded", [(16, 2, 1 << 20, False), (24, 1, 1 << 20, False),
                                                  (16, 2, 20001, True)])
def test_dense_bins_keep_the_accuracy_of_tiles(edge, shape, n, crowded):
    grid = (edge,) * 3
    parts = ri.make_particles(n, grid, 61)
    if crowded:
        parts["cell"][:] = 11
    planes = fields(grid)
    ctx = rs.Context(rs.Params(*grid, shape=shape, precision=32, c_tilde=0.1))
    A, P = rs.Particles.from_numpy(parts, 32), rs.Particles.empty(n, 32)
    ctx.sort(A, P)
    G = oracle.step(oracle.params(grid, shape=shape, dt=2.0, c_tilde=0.1), planes, oracle.Particles(P.to_numpy()))
    fb = ctx.grid_tensor()
    ctx.push_gather(P, rs.fields_to_device(planes, 32), 2.0, fb)
    ctx.check()
    got = rs.grid_to_planes(fb)
    bins = 1 if crowded else math.ceil(edge / 8) ** 3
    assert rel_l2(got[0], G[0]) <= bar(8 * math.ceil(n / bins / 4352))
    for q in range(1, 8):
        assert rel_l2(got[q], G[q]) <= 1e-5, q


def test_a_crowded_bin_of_a_sub_cycled_level_keeps_the_accuracy_of_tiles():
    """About 20000 packets in one cell of 64^3, few for the box: a level of more than 768
    of them takes the tiles, so rho is as near the oracle's as with the tiles asked for (16
    warps), up to the order of the additions.  Tiles make 28 additions on a node, global
    sums 111,000, whose rms rounding is sqrt(111000 / 28) = 63 times as large; the bar is the
    geometric middle, 8.  (The sub-steps add nearly equal values, whose roundings are not
    independent: no bar from their number alone.  Packets whose limits lie within 1e-3 of a
    level's edge are left out.)"""
    grid, dt = (64, 64, 64), 10.0
    parts = ri.make_particles(20400, grid, 67)
    parts["cell"][:] = 11
    planes = fields(grid)
    op = oracle.params(grid, shape=2, dt=dt, c_tilde=0.1)
    r = np.log2(dt / oracle.dt_limits(op, planes, oracle.Particles(parts), 0.2))
    keep = np.abs(r - np.round(r)) > 1e-3
    parts = {k: np.ascontiguousarray(v[..., keep]) for k, v in parts.items()}
    G, levels = oracle.step_subcycled(op, planes, oracle.Particles(parts), 0.2)
    err = []
    for warps in (0, 16):
        ctx = rs.Context(rs.Params(*grid, shape=2, precision=32, c_tilde=0.1, warps=warps))
        P, fb = rs.Particles.from_numpy(parts, 32), ctx.grid_tensor()
        counts = ctx.sort_push_subcycled(P, rs.Particles.empty(P.n, 32), rs.fields_to_device(planes, 32), dt, 0.2,
                                         fb)
        ctx.check()
        assert np.array_equal(counts, np.bincount(levels, minlength=len(counts)))
        err.append([rel_l2(x, y) for x, y in zip(rs.grid_to_planes(fb), G)])
    assert err[0][0] <= 8 * err[1][0]
    assert max(err[0]) <= 1e-5
