"""The reciprocal square root of the Cholesky pivots and the square root made from it against CUDA's, over all exponents."""
import ctypes
import os

import numpy as np
import pytest

from paper_2407_19930_gb300 import build

pytestmark = pytest.mark.gpu


def test_against_cuda():
    rng = np.random.default_rng(3)
    m = 1.0 + rng.random(200_000)
    d = np.concatenate([
        np.ldexp(m, rng.integers(-1022, 1023, m.size)),                        # even and odd exponents
        1.0 + np.arange(4096) * 2.0 ** -52, 4.0 - np.arange(1, 4096) * 2.0 ** -51, 2.0 - np.arange(1, 4096) * 2.0 ** -52,
        np.ldexp(1.0, np.arange(-1074, 1024)),                                 # powers of two, subnormal ones among them
        np.ldexp(m[:1000], -1060), [np.finfo(float).tiny, np.finfo(float).max]])
    lib = ctypes.CDLL(os.path.join(build.BUILD, "libpeaks.so"))
    out = np.empty((4, d.size))
    P = ctypes.POINTER(ctypes.c_double)
    assert lib.librpa_probe_rsqrt(d.size, d.ctypes.data_as(P), out.ctypes.data_as(P)) == 0
    r, s, r0, s0 = out
    # ours: a half unit in the last place of the product d r0 and the final rounding, 1.5 x 2^-53; CUDA's rsqrt: one unit
    # (2^-52 relative at most)
    assert np.abs(r / r0 - 1.0).max() <= 2.0 ** -51
    # the Newton step leaves its own rounding, 2^-53, and CUDA's sqrt is correctly rounded, 2^-53 (subnormal results: none)
    n = d >= np.finfo(float).tiny
    assert np.abs(s[n] / s0[n] - 1.0).max() <= 1.1 * 2.0 ** -52
