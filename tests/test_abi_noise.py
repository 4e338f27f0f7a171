"""Status and wait controls of a noise handle refuse a NULL handle before any device work (no GPU needed)."""
import ctypes

import pytest


def test_null_noise_handles_are_refused():
    from paper_2603_19600_gb300 import build
    try:
        lib = ctypes.CDLL(build.build())
    except RuntimeError as e:  # no nvcc on this machine
        pytest.skip(str(e))
    lib.furax_last_error.restype = ctypes.c_char_p
    assert lib.furax_noise_status(None, None) == -1
    assert b"noise handle" in lib.furax_last_error()
    assert lib.furax_noise_set_wait_budget(None, ctypes.c_int64(1 << 20), None) == -1
    assert lib.furax_debug_hold_noise(None, 1, None) == -1
