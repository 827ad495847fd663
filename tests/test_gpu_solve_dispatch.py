"""Which solve levels the automatic rule sends to the tensor cores: a preconditioner application with
the automatic choice is bit for bit the one with none where the rule names none (the sweeps are
deterministic)."""

import numpy as np
import pytest

from paper_1408_4495_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NONE = 1 << 30


@pytest.fixture(scope="module")
def LS():
    from paper_1408_4495_gb300 import build, ls
    build.build()
    return ls


@pytest.mark.parametrize("n,nrhs", [(1024, 5), (1024, 16), (512, 17), (512, 32)])
def test_levels_stay_on_the_cuda_cores(LS, n, nrhs):
    """One group of right-hand sides in 2D, where levels exceed the rule's number of terms: FP32 at
    every level.  Two groups at n = 512: every level has 0.25 to 1.25 times 2^25 terms."""
    import torch
    m = W.enforce_buffer(W.bumps(n, 2, [-0.2], [0.1], [(0.5, 0.5)]), 2)
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((nrhs, n, n), dtype=torch.complex128, device="cuda", generator=gen)
    with LS.Solver(torch.tensor(m, device="cuda"), 2 * np.pi * n / 8, dim=2, mixed=True,
                   stream=torch.cuda.current_stream()) as s:
        s.factor()
        s.precond_refine(0)
        z = s.precond(x)
        s.set_tune({"tcs_min_rows": NONE, "tcs_bwd_min_rows": NONE})
        assert torch.equal(torch.view_as_real(s.precond(x)), torch.view_as_real(z))
