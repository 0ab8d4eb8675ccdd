"""gwc_workspace_bytes: a function of the sizes and options alone, the same on a machine without a GPU."""
import ctypes
import math

import numpy as np
import pytest


def _bytes(prec, n_aux, n_states, n_occ, batch):
    from paper_2412_17132_gb300 import gwc

    core = np.zeros(1, dtype=np.int32)
    eps = np.linspace(-10, 5, n_states)
    s = gwc.System(n_states, n_occ, n_aux, 1, core.ctypes.data_as(ctypes.POINTER(ctypes.c_int)), eps.ctypes.data, 1, 1, None,
                   math.nan, 1)
    o = gwc.default_options()
    o.prec, o.batch = gwc.PREC[prec], batch
    b = ctypes.c_size_t()
    assert gwc.lib().gwc_workspace_bytes(ctypes.byref(s), ctypes.byref(o), 400, ctypes.byref(b)) == 0
    return b.value


@pytest.mark.parametrize("n_aux,n_states,n_occ", [(64, 40, 6), (300, 120, 20), (63, 40, 6)])
@pytest.mark.parametrize("batch", [1, 16])
def test_the_fp64_mode_counts_its_digit_planes(n_aux, n_states, n_occ, batch):
    n_ov = n_occ * (n_states - n_occ)
    pad, opad, ldm = -(-n_aux // 128) * 128, -(-n_ov // 64) * 64, -(-n_aux // 4) * 4
    planes = 22 * pad * opad
    row = 22 * opad + 4  # the scaled operand's planes and the row's exponent
    work = max(128 * row, min(2 * batch * pad * row + 1024, 1 << 30))
    # what the FP64 mode holds in place of the split mode: wider matrices and right-hand sides, no BF16 and FP32 copies of O
    wider = batch * (n_aux * ldm + ldm) * 8 + n_states * ldm * 4 - pad * opad * 8
    got = _bytes("fp64", n_aux, n_states, n_occ, batch) - _bytes("bf16x3", n_aux, n_states, n_occ, batch) - wider
    want = planes + work if n_aux >= 64 else 0
    assert abs(got - want) <= 2048, (got, want)
