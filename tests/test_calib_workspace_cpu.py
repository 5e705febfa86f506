"""The calibration workspace's size is part of the C interface: callers keep it."""
import ctypes as C

import pytest

from paper_2609_38169_gb300 import _lib, api as A


@pytest.mark.parametrize("gate", [A.GATE_SCALAR, A.GATE_CHANNEL])
@pytest.mark.parametrize("layers,hv,n", [(1, 1, 1), (4, 32, 8), (40, 16, 1), (3, 7, 5)])
def test_workspace_size(gate, layers, hv, n):
    cfg = A.Config(n_layers=layers, n_key_heads=hv, n_value_heads=hv, gate_kind=gate)
    heads, units, k1 = layers * hv, A.stepq_num_units(cfg), len(cfg.candidates) + 1
    parts = [heads * 128 * 8, units * 8, units * k1 * 8, heads * 128 * 4, units,
             4 * n, n * hv * 128 * 128 * 4, n * hv * 128 * 4]
    c = cfg.c()
    assert _lib.lib().stepq_calib_workspace_bytes(C.byref(c), n) == sum((p + 255) // 256 * 256 for p in parts)
