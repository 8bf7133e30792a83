"""A solve that ends on a device error returns an iterate and a residual that
belong together."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2509_08109_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def _indefinite(n, seed):
    """A diagonal lowered at random until the operator is indefinite: the
    setup still goes through, and CG finds p.Ap <= 0 in every other iteration
    (the even ones, whose step waits for the next, succeed)."""
    rng = np.random.default_rng(seed)
    kappa = np.exp(rng.normal(0, rng.uniform(0, 2), (n - 1, n - 1)))
    A = oracle.assemble(inputs.coords_identity(n, 2), kappa)
    A[1:-1, 1:-1, 4] -= rng.uniform(0, 1, (n - 2, n - 2)) * 10 ** rng.uniform(-3, 0.3) * kappa[:-1, :-1]
    b = np.zeros((n, n))
    b[1:-1, 1:-1] = np.random.default_rng(seed).uniform(-1, 1, (n - 2, n - 2))
    return A, b


def _relres(A, x, b):
    r = b - oracle.apply(A, x)
    return np.linalg.norm(r[1:-1, 1:-1]) / np.linalg.norm(b[1:-1, 1:-1])


# Both residuals are FP64 sums of ten terms of the size of |A| |x| (below
# 1e3 |b| here): equal to 1e-12, and the residual is larger than |b|.
@pytest.mark.parametrize("maxit", [13, 14, 500])
@pytest.mark.parametrize("n,seed,way", [(17, 134, "single"), (17, 134, "concurrent"), (65, 210, "single"),
                                        (65, 210, "concurrent"), (65, 210, "batch")])
def test_residual_after_an_indefinite_operator(n, seed, way, maxit):
    A, b = _indefinite(n, seed)
    lib = binding.load()
    s = binding.Solver(2, n, precision="fp32", outer="refine")
    s.set_stencil(torch.as_tensor(A)).setup()
    f = torch.as_tensor(b, device="cuda")
    x = torch.zeros_like(f)
    info = binding._Info()
    one = ctypes.c_void_p * 1
    rest = (1, one(f.data_ptr()), one(x.data_ptr()), 1e-10, maxit, ctypes.byref(info))
    if way == "single":
        code = lib.bmg_solve(s._h, 1, f.data_ptr(), x.data_ptr(), 1e-10, maxit, ctypes.byref(info))
    elif way == "concurrent":
        code = lib.bmg_solve_many(one(s._h.value), 1, *rest)
    else:
        batch = binding.Batch([s])
        code = lib.bmg_batch_solve(batch._h, *rest)
    torch.cuda.synchronize()
    assert code == 7 and info.status == 7       # not SPD
    assert info.iterations == 13                # the first run
    res = _relres(A, x.cpu().numpy(), b)
    assert res > 1.0                            # steps have been taken
    assert abs(info.true_relres - res) <= 1e-9 * res
