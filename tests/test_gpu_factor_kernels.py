"""The kernels of the factorization at the edges of their ranges, through matrices of the caller's own.

ls_general_setup with every point on the boundary of the domain makes the preconditioner's matrix M
and the stencil matrix [A;B] the same: the matrix of the given rows.  precond(x) is then x to the
rounding of the factorization, at any size and without a reference solution.

Rows with a small diagonal and a large entry next to it (pairs of points that ask for each other's
row) make every panel and elimination exchange rows.  Front sizes: 2D leaves of 16 own rows with 64
(n = 32, one CTA a front) to 4096 fronts (n = 256, one warp a front), levels of 4, 8 and 16 rows on both sides of 256
fronts at every width that kernel is built for (n = 128, 256, 512), panels of 8 to 32 columns (n = 24, 3D n = 24), of 64, 96, 128 rows (four threads a row) and above.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2, 16), (2, 24), (2, 32), (2, 48), (2, 64), (2, 128), (2, 256), (2, 512), (3, 8), (3, 16), (3, 24)]


@pytest.fixture(scope="module")
def LS():
    from paper_1408_4495_gb300 import build, ls
    build.build()
    return ls


def rows(d, n, seed):
    """Random rows (n^d x 3^d): unit diagonal, small couplings, and 30 % of the pairs of neighbours
    along the last axis with diagonal 0.1 and mutual entries 1."""
    rng = np.random.default_rng(seed)
    N, P3 = n**d, 3**d
    c = (P3 - 1) // 2
    amp = 0.3 if d == 2 else 0.15
    a = amp * (rng.uniform(-1, 1, (N, P3)) + 1j * rng.uniform(-1, 1, (N, P3)))
    a[:, c] = 1.0
    first = np.flatnonzero((np.arange(N) % n % 2 == 0) & (rng.uniform(size=N) < 0.3))
    a[first, c] = a[first + 1, c] = 0.1
    a[first, c + 1] = a[first + 1, c - 1] = 1.0
    return a


def solver(LS, d, n, alpha, mixed):
    s = LS.Solver(np.zeros((n,) * d), 2 * np.pi * n / 8, mixed=mixed)
    s.general_setup(np.ones((n,) * d, dtype=np.uint8), alpha, np.ones(n**d, dtype=np.int32))
    s.factor()
    return s


@pytest.mark.parametrize("d,n", SIZES)
def test_factorization_inverts_the_rows(LS, d, n):
    """FP64: 1e-10 (rounding times a condition number of at most 1e5).  FP32: the same elimination with
    unit roundoff 2^-24 instead of 2^-53 and products at 2^-22 (3xTF32), with a factor of 4 for the
    scatter between two orders of summation: 16 * 2^29 times the FP64 error."""
    nrhs = 3
    rng = np.random.default_rng(n)
    x = rng.standard_normal((nrhs,) + (n,) * d) + 1j * rng.standard_normal((nrhs,) + (n,) * d)
    alpha = rows(d, n, n + d)
    err = {}
    for mixed in (False, True):
        with solver(LS, d, n, alpha, mixed) as s:
            s.precond_refine(0)
            err[mixed] = np.linalg.norm(s.precond(x) - x) / np.linalg.norm(x)
    assert err[False] < 1e-10
    assert err[True] < 16 * 2.0**29 * max(err[False], 2.0**-53)


# a pair of neighbours of one front: its 2 x 2 block of ones is exactly singular, every other row is
# a unit row.  The leaf at the origin; the root separator (middle plane of axis 0)
@pytest.mark.parametrize("mixed", [True, False])
@pytest.mark.parametrize("d,n,where", [(2, 16, "leaf"), (2, 64, "leaf"), (2, 256, "leaf"), (3, 8, "leaf"), (2, 24, "root"),
                                       (2, 64, "root"), (2, 128, "root"), (2, 256, "root"), (3, 24, "root")])
def test_singular_front_is_reported(LS, d, n, where, mixed):
    N, P3 = n**d, 3**d
    c = (P3 - 1) // 2
    alpha = np.zeros((N, P3), dtype=complex)
    alpha[:, c] = 1.0
    p = 0 if where == "leaf" else n // 2 * n ** (d - 1) + 2
    x = np.ones((1,) + (n,) * d, dtype=complex)
    with solver(LS, d, n, alpha, mixed) as s:  # unit rows alone: exact
        assert np.array_equal(s.precond(x), x)
    alpha[p, c + 1] = alpha[p + 1, c - 1] = 1.0
    with solver(LS, d, n, alpha, mixed) as s:
        with pytest.raises(LS.LsError) as e:
            s.precond(x)
        assert e.value.status == LS.LS_EINVAL
