"""The one-buffer packing of a field-source call against the separate records."""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest

import paper_2111_14704_gb300 as rs
import rsol_inputs as ri


@pytest.mark.parametrize("nm", [0, 1, 17])
def test_field_args_match_mode_records(nm):
    modes = ri.alfven_modes(nm, 3, L=(16.0,) * 3, kmax=4, dB_rms=0.1) if nm else None
    if nm:
        modes["sigma"].flags.writeable = False
    buf, at, n = rs._field_args(modes, (1, 2.0, 3.5))
    assert n == nm and buf.ctypes.data == at
    got = np.array((C.c_double * (9 * nm + 3)).from_address(at))
    if nm:
        rec, sig, _ = rs._mode_records(modes)
        assert np.array_equal(got[:8 * nm], rec.ravel()) and np.array_equal(got[8 * nm:9 * nm], sig)
    assert list(got[9 * nm:]) == [1.0, 2.0, 3.5]
