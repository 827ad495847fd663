"""The longest line transforms (L = 4096, 2D n = 2048) through the C-ABI in the three arithmetics,
with the bounds of the shorter ones (test_gpu_parity.py), and the FP64 plane-wave right-hand sides
from their per-axis phase tables at an odd batch."""

import numpy as np
import pytest

import oracle as O
from paper_1408_4495_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def LS():
    from paper_1408_4495_gb300 import build, ls
    build.build()
    return ls


def test_operator_apply_longest_lines(LS):
    n, omega = 2048, 2 * np.pi * 256
    m = W.enforce_buffer(W.bumps(n, 2, [-0.2, 0.15], [0.1, 0.08], [(0.4, 0.5), (0.6, 0.55)]), 2)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((1, n, n)) + 1j * rng.standard_normal((1, n, n))
    ref = O.apply_operator(O.kernel_table(n, 2, omega), omega, m, x[0])
    with LS.Solver(m, omega, mixed=True) as s:
        for prec, bound in ((LS.LS_PREC_MIXED, 2e-5), (LS.LS_PREC_FF, 1e-11), (LS.LS_PREC_FP64, 1e-11)):
            y = s.apply(x, prec=prec)[0]
            assert np.linalg.norm(y - ref) < bound * np.linalg.norm(ref)


@pytest.mark.parametrize("d,n", [(2, 48), (3, 24)])
def test_fp64_rhs_odd_batch(LS, d, n):
    omega = 2 * np.pi * n / 8
    m = W.enforce_buffer(W.bumps(n, d, [-0.2], [0.1], [(0.5,) * d]), 2)
    dirs = W.directions_circle(5) if d == 2 else W.directions_sphere(5, 3)
    kt = O.kernel_table(n, d, omega)
    with LS.Solver(m, omega, mixed=False) as s:
        g = s.rhs_plane_wave(dirs)
    for j in range(5):
        ref = O.rhs(kt, omega, m, dirs[j])
        assert np.max(np.abs(g[j] - ref)) < 1e-11 * np.max(np.abs(ref))
