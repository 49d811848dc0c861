"""The hardware logarithm on the arguments the tensor-core epilogues of orders
2 and 3 take it of: class counts times the power of two of the sample count."""
import ctypes

import numpy as np
import pytest


def test_bad_arguments():
    import paper_2201_03331_gb300 as fc
    from paper_2201_03331_gb300 import build
    build.build()
    lib = fc.library()
    assert lib.fc_log2_approx_scaled(None, 4, 3, None) == fc.FC_EINVAL
    n, out = (ctypes.c_uint32 * 1)(1), (ctypes.c_float * 1)()
    for shift in (-1, 32):
        assert lib.fc_log2_approx_scaled(n, 1, shift, out) == fc.FC_EINVAL
    assert lib.fc_log2_approx_scaled(None, 0, 3, None) == fc.FC_OK


def test_shifts_of_the_sample_counts():
    """fc::triples_scale(M) is 2^-s, s = max(floor(log2 M) - 2, 0): at most 2^-14
    for two classes of 65,535, and the samples come to less than 8."""
    from paper_2201_03331_gb300 import build
    scale = ctypes.CDLL(build.build())._ZN2fc13triples_scaleEl
    scale.argtypes, scale.restype = [ctypes.c_int64], ctypes.c_float
    for M in range(2, 131071):
        q = scale(M)
        assert q == 2.0 ** -max(M.bit_length() - 3, 0) and q >= 2.0 ** -14 and M * q < 8


@pytest.mark.gpu
@pytest.mark.parametrize("shift", range(15))
def test_error_within_the_assumed_bound(shift):
    import paper_2201_03331_gb300 as fc
    from paper_2201_03331_gb300 import build
    build.build()
    n = np.arange(0, 2 ** 17 + 1, dtype=np.uint32)
    lg = fc.fc_log2_approx_scaled(n, shift).astype(np.float64)
    assert np.isfinite(lg).all()   # (a count of 0 has a finite one, which 0 then multiplies)
    exact = np.log2(n[1:].astype(np.float64)) - shift
    err = np.abs(lg[1:] - exact) / np.maximum(1.0, np.abs(exact))
    assert err.max() <= 2.0 ** -22, (err.max() * 2 ** 22, n[1 + err.argmax()])
