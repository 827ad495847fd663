"""Device arrays that the kernels read and write in place: the same results as through host arrays
for aligned and misaligned arrays, for in == out and for arrays that overlap."""

import numpy as np
import pytest

from paper_1408_4495_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1408_4495_gb300 import build, ls
    build.build()
    n = 32
    m = W.enforce_buffer(W.bumps(n, 2, [-0.2], [0.1], [(0.5, 0.5)]), 2)
    with ls.Solver(m, 2 * np.pi * 4, mixed=True) as s:
        s.factor()
        yield ls, s, n


def _at(torch, total, offset):
    """total complex doubles on the device, `offset` doubles past a 16-byte boundary."""
    raw = torch.zeros(2 * total + 4, dtype=torch.float64, device="cuda")
    return raw, raw[offset:offset + 2 * total]


@pytest.mark.parametrize("op", ["mixed", "ff", "fp64", "stencil", "precond"])
@pytest.mark.parametrize("where", ["aligned", "misaligned", "same", "shifted"])
def test_arrays_in_place(ctx, op, where):
    import torch
    ls, s, n = ctx
    nrhs, N = 3, n * n
    rng = np.random.default_rng(4)
    x = rng.standard_normal((nrhs, n, n)) + 1j * rng.standard_normal((nrhs, n, n))
    fn = {"mixed": lambda a, b: s.lib.ls_apply(s.h, nrhs, a, b, ls.LS_PREC_MIXED),
          "ff": lambda a, b: s.lib.ls_apply(s.h, nrhs, a, b, ls.LS_PREC_FF),
          "fp64": lambda a, b: s.lib.ls_apply(s.h, nrhs, a, b, ls.LS_PREC_FP64),
          "stencil": lambda a, b: s.lib.ls_stencil_apply(s.h, nrhs, a, b, ls.LS_PREC_MIXED),
          "precond": lambda a, b: s.lib.ls_precond(s.h, nrhs, a, b)}[op]
    ref = np.empty_like(x)
    assert fn(ls._ptr(x), ls._ptr(ref)) == ls.LS_OK
    off = 1 if where == "misaligned" else 0
    extra = N // 2 if where == "shifted" else 0  # out starts half a vector behind in
    raw, flat = _at(torch, nrhs * N + extra, off)
    a = flat[:2 * nrhs * N]
    a.copy_(torch.from_numpy(x.view(np.float64).reshape(-1)))
    if where == "same":
        b = a
    elif where == "shifted":
        b = flat[2 * extra:]
    else:
        _, b = _at(torch, nrhs * N, off)
    torch.cuda.synchronize()
    assert fn(a.data_ptr(), b.data_ptr()) == ls.LS_OK
    got = b.cpu().numpy().view(np.complex128).reshape(x.shape)
    assert np.array_equal(got, ref)


def test_rhs_and_far_field_in_place(ctx):
    import torch
    ls, s, n = ctx
    dirs, obs = W.directions_circle(3), W.directions_circle(5)
    g = s.rhs_plane_wave(dirs)
    pts = np.array([[3, 4], [20, 9]], dtype=np.int32)
    ps = s.rhs_point_source(pts)
    rng = np.random.default_rng(2)
    us = rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n))
    F = s.far_field(dirs, us, obs)
    for off in (0, 1):
        raw, out = _at(torch, 3 * n * n, off)
        _, u = _at(torch, 3 * n * n, off)
        d = torch.tensor(dirs, device="cuda")
        torch.cuda.synchronize()
        assert s.lib.ls_rhs_plane_wave(s.h, 3, d.data_ptr(), out.data_ptr()) == ls.LS_OK
        assert np.array_equal(out.cpu().numpy().view(np.complex128).reshape(g.shape), g)
        assert s.lib.ls_rhs_point_source(s.h, 2, ls._ptr(pts), None, out.data_ptr()) == ls.LS_OK
        assert np.array_equal(out[:4 * n * n].cpu().numpy().view(np.complex128).reshape(ps.shape), ps)
        u.copy_(torch.from_numpy(us.view(np.float64).reshape(-1)))
        torch.cuda.synchronize()
        o = torch.tensor(obs, device="cuda")
        # the result over the start of the fields
        assert s.lib.ls_far_field(s.h, 3, d.data_ptr(), u.data_ptr(), 5, o.data_ptr(), u.data_ptr()) == ls.LS_OK
        assert np.array_equal(u[:30].cpu().numpy().view(np.complex128).reshape(F.shape), F)
