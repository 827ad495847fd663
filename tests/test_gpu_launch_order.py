"""Launches that start ahead of the end of the one before them give the bits of a run in which every
launch is timed by itself (events between the launches keep them apart)."""

import numpy as np
import pytest

from paper_1408_4495_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,nrhs,mixed", [(2, 16, 1, True), (2, 32, 5, False), (2, 64, 3, True),
                                            (2, 128, 7, True), (3, 8, 2, True), (3, 16, 5, False)])
def test_overlapped_launches_same_bits(d, n, nrhs, mixed):
    from paper_1408_4495_gb300 import build, ls
    build.build()
    m = W.enforce_buffer(W.bumps(n, d, [-0.2], [0.1], [(0.5,) * d]), d)
    rng = np.random.default_rng(n)
    dirs = rng.standard_normal((nrhs, d))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    with ls.Solver(m, 2 * np.pi * n / 8, mixed=mixed) as s:
        s.factor()
        g = s.rhs_plane_wave(dirs)

        def run():
            return [np.array(s.apply(g)), np.array(s.solve(g, tol=1e-6)[0])]

        ls.profile_start("**")
        ref = run()
        assert ls.profile_stop()["ms_by_class"]
        for _ in range(5):
            for a, b in zip(run(), ref):
                assert np.array_equal(a, b)
