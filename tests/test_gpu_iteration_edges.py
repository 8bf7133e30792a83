"""The iteration kernels where they can go wrong: counts that end on either
parity (the refinement mode leaves an even iteration's step to the next one),
and grids below, at and above the tiles of the products, half sweeps and
tails."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_08109_gb300 import binding, inputs
from tests.gpu_util import relerr, solver_for

pytestmark = pytest.mark.gpu


def _problem(dim, n):
    coords = inputs.coords_bump(n, 0.11, -0.13) if dim == 2 else inputs.coords_identity(n, 3)
    rng = np.random.default_rng(100 * dim + n)
    kappa = np.exp(rng.normal(0.0, 0.5, size=(n - 1,) * dim))
    rhs = inputs.rhs_uniform(rng, (n,) * dim)
    return coords, kappa, rhs


def _relres(A, x, b):
    r = b - oracle.apply(A, x)
    inner = (slice(1, -1),) * b.ndim
    return np.linalg.norm(r[inner]) / np.linalg.norm(b[inner])


# The reported residual is that of the returned iterate: a step that is left
# out or added twice changes it by its own size.  Both residuals are FP64 sums
# of 3^d + 1 terms of the size of |A| |x|; their rounding is below 1e-12 |b| at
# these sizes, so relative to residuals above 1e-5 |b| they agree to 1e-6.
@pytest.mark.parametrize("precision,outer", [("fp32", "refine"), ("fp64", "cg"), ("fp32", "flexible")])
@pytest.mark.parametrize("dim,n", [(2, 5), (2, 33), (2, 65), (2, 129), (3, 5), (3, 9), (3, 17), (3, 65)])
def test_reported_residual_is_that_of_the_iterate(dim, n, precision, outer):
    coords, kappa, rhs = _problem(dim, n)
    A = oracle.assemble(coords, kappa)
    s = binding.Solver(dim, n, precision=precision, outer=outer)
    s.assemble(torch.as_tensor(coords), torch.as_tensor(kappa)).setup()
    b = torch.as_tensor(rhs, device="cuda")
    seen = []
    for maxit in (1, 2, 3):
        x, info = s.solve(b, tol=1e-14, maxit=maxit, raise_on_nonconv=False)
        if info.iterations < maxit:
            break            # the smallest grids are solved to rounding by then
        res = _relres(A, x.cpu().numpy(), rhs)
        if res < 1e-5:
            break
        assert abs(info.true_relres - res) <= 1e-6 * res, (maxit, info.true_relres, res)
        seen.append(res)
    if n >= 17:
        assert len(seen) >= 2


@pytest.mark.parametrize("maxit", [1, 2, 3])
def test_batch_counts_of_either_parity(maxit):
    sizes = (65, 129, 257)
    probs = [_problem(2, n) for n in sizes]
    solvers = []
    for n, (coords, kappa, _) in zip(sizes, probs):
        s = binding.Solver(2, n, precision="fp32", outer="refine")
        solvers.append(s.assemble(torch.as_tensor(coords), torch.as_tensor(kappa)).setup())
    bs = [[torch.as_tensor(f.copy(), device="cuda") for f in (rhs, 2.0 * rhs[::-1])] for _, _, rhs in probs]
    xs = [[torch.zeros_like(f) for f in b] for b in bs]
    infos = binding.Batch(solvers).solve(bs, xs, tol=1e-14, maxit=maxit, raise_on_nonconv=False)
    for (coords, kappa, _), b, x, inf in zip(probs, bs, xs, infos):
        A = oracle.assemble(coords, kappa)
        for f, u, info in zip(b, x, inf):
            res = _relres(A, u.cpu().numpy(), f.cpu().numpy())
            assert info.iterations == maxit
            assert abs(info.true_relres - res) <= 1e-6 * res


# Flexible CG (beta from r.z - r.z_old) with an FP64 V-cycle against the
# oracle's: the same iterates, so after a fixed count they agree as closely as
# the plain iteration is required to.
@pytest.mark.parametrize("n,iters", [(5, 2), (17, 4), (33, 5), (129, 6), (257, 5)])
def test_flexible_cg_fixed_iterations(n, iters):
    coords, kappa, rhs = _problem(2, n)
    H = oracle.Hierarchy(oracle.assemble(coords, kappa))
    s = binding.Solver(2, n, precision="fp64", outer="flexible")
    s.assemble(torch.as_tensor(coords), torch.as_tensor(kappa)).setup()
    x, info = s.solve(torch.as_tensor(rhs, device="cuda"), tol=0.0, maxit=iters, raise_on_nonconv=False)
    xo = H.pcg(rhs, tol=0.0, maxit=iters, flexible=True)[0]
    assert info.iterations == iters
    assert relerr(x.cpu().numpy(), xo) <= 1e-9
