"""Rounding of the operator's transforms, every line length in the three arithmetics, against numpy's
FP64 transforms of the library's own kernel table (which takes the table's own error out).

A transform of P points rounds log2(P) times; independent roundings of unit u leave a relative error
of about u sqrt(log2 P), forward and inverse u sqrt(2 log2 P) on a vector of random entries (flat
spectrum, so the symbol weights error and value alike).  Bound: twice that, with u = 2^-24 (FP32), 2^-45
(float-float: two FP32 numbers carry 48 bits, a product or a deferred renormalisation loses up to
three), 2^-53 (FP64, once for each side).
"""

import math

import numpy as np
import pytest

from paper_1408_4495_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n", [(2, 16), (2, 24), (2, 32), (2, 48), (2, 64), (2, 128), (2, 256), (2, 512), (2, 1024), (2, 2048),
                                 (3, 8), (3, 24)])
def test_apply_rounding(d, n):
    from paper_1408_4495_gb300 import build, ls
    build.build()
    omega, L = 2 * np.pi * n / 8, 2 * n
    m = W.enforce_buffer(W.bumps(n, d, [-0.2], [0.12], [(0.5,) * d]), 2)
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n,) * d) + 1j * rng.standard_normal((n,) * d)
    with ls.Solver(m, omega, mixed=True) as s:
        kt = s.kernel_table()
        y = {u: s.apply(x[None], prec=p)[0]
             for u, p in ((2.0**-24, ls.LS_PREC_MIXED), (2.0**-45, ls.LS_PREC_FF), (2.0**-53, ls.LS_PREC_FP64))}
    t = np.minimum(np.arange(L), L - np.arange(L))
    k = kt[np.ix_(*[t] * d)]
    for a in range(d):
        k[(slice(None),) * a + (n,)] = 0.0
    v = np.fft.ifftn(np.fft.fftn(omega**2 * m * x, s=(L,) * d, axes=range(d)) * np.fft.fftn(k))[(slice(0, n),) * d]
    grow = math.sqrt(2 * d * math.log2(L))
    for u, yu in y.items():
        # the FP32 operator rounds x, the added vector, to FP32 as well
        bound = 2 * grow * (u + 2.0**-53) * np.linalg.norm(v) + (2 * u * np.linalg.norm(x) if u == 2.0**-24 else 2.0**-52 * np.linalg.norm(x))
        assert np.linalg.norm(yu - (x + v)) < bound, u
