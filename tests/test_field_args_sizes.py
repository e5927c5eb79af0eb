"""Too few directions of travel or gas velocity components are an error, not one value
spread over the rest; more than needed are cut."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2111_14704_gb300 as rs
import rsol_inputs as ri


def modes_with(sigma):
    m = ri.alfven_modes(4, 3, L=(16.0,) * 3, kmax=4, dB_rms=0.1)
    return dict(m, sigma=np.asarray(sigma, dtype=np.float64))


@pytest.mark.parametrize("sigma", [[-1.0], [], [1.0, -1.0, 1.0]])
def test_too_few_directions(sigma):
    with pytest.raises(ValueError):
        rs._field_args(modes_with(sigma), (0.0, 0.0, 0.0))


@pytest.mark.parametrize("u_gas", [0.5, [0.5], [0.5, 0.1], []])
def test_too_few_velocity_components(u_gas):
    for m in (None, modes_with([1.0, -1.0, 1.0, 1.0])):
        with pytest.raises(ValueError):
            rs._field_args(m, u_gas)


def test_longer_arrays_are_cut():
    buf, _, nm = rs._field_args(modes_with([1.0, -1.0, 1.0, 1.0, 5.0]), (1.0, 2.0, 3.0, 4.0))
    assert nm == 4 and list(buf[32:]) == [1.0, -1.0, 1.0, 1.0, 1.0, 2.0, 3.0]
