"""One-CTA-per-front solve levels at the edges of their range: one to four groups of 16 right-hand
sides, the last one partly empty, fronts of 3 to 64 rows, more than one column chunk, few and many
fronts a level."""

import numpy as np
import pytest

from paper_1408_4495_gb300 import workloads as W

pytestmark = pytest.mark.gpu

OFF = 1 << 30


@pytest.mark.parametrize("d,n,nrhs", [(2, 16, 5), (2, 24, 17), (2, 48, 33), (2, 128, 16), (2, 128, 64),
                                      (3, 8, 16), (3, 16, 49)])
def test_small_levels_against_general_sweep(d, n, nrhs):
    """Both sum the same FP32 products in another order, so their errors against the FP64
    preconditioner are alike: within a factor of 5 of the general sweep's."""
    from paper_1408_4495_gb300 import build, ls
    build.build()
    m = W.enforce_buffer(W.bumps(n, d, [-0.2], [0.1], [(0.5,) * d]), d)
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((nrhs,) + (n,) * d) + 1j * rng.standard_normal((nrhs,) + (n,) * d)
    omega = 2 * np.pi * n / 8
    with ls.Solver(m, omega, mixed=False) as s:
        s.factor()
        ref = s.precond(x)
    err = {}
    with ls.Solver(m, omega, mixed=True) as s:
        s.factor()
        for k in (256, 0):
            s.set_tune({"tcs_min_rows": OFF, "tcs_bwd_min_rows": OFF, "small_max_k": k})
            z = s.precond(x)
            err[k] = max(np.linalg.norm(z[j] - ref[j]) / np.linalg.norm(ref[j]) for j in range(nrhs))
    assert err[256] <= 5 * err[0]
