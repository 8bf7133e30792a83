"""Run lengths of the refinement mode: how far a run goes sets how exact the
returned solution is at a given tolerance."""
import math

import numpy as np
import pytest
import torch

from paper_2509_08109_gb300 import binding, inputs
from tests.gpu_util import relerr

pytestmark = pytest.mark.gpu

# what a first run that aims at a reduction takes at least: the count for the
# guessed contraction 0.3, ceil(ln(reduction) / ln 0.3) + 1
FIRST = math.ceil(math.log(1e-6) / math.log(0.3)) + 1


def _box(n, seed=0):
    rng = np.random.default_rng(1000 + n + seed)
    kappa = np.exp(rng.normal(0.0, 0.5, size=(n - 1,) * 3))
    return inputs.coords_identity(n, 3), kappa, inputs.rhs_uniform(rng, (n,) * 3)


def _solver(n, seed=0, precision="fp32", outer="refine"):
    coords, kappa, rhs = _box(n, seed)
    s = binding.Solver(3, n, precision=precision, outer=outer)
    s.assemble(torch.as_tensor(coords), torch.as_tensor(kappa)).setup()
    return s, torch.as_tensor(rhs, device="cuda")


def _solve_each_way(n, tol):
    """The same solve alone and beside another one: (solution, info) twice."""
    s, f = _solver(n)
    x, info = s.solve(f, tol=tol)
    t, g = _solver(n, 1)
    y, z = torch.zeros_like(f), torch.zeros_like(g)
    infos = binding.solve_many([s, t], [[f], [g]], [[y], [z]], tol=tol)
    return (x, info), (y, infos[0][0])


# On the box the cycle contracts by far more than 0.3, so the first run meets
# a tolerance of 1e-6 with the count it starts with and is the only one.
@pytest.mark.parametrize("n", [17, 33, 65])
def test_first_run_takes_the_predicted_count(n):
    for x, info in _solve_each_way(n, 1e-6):
        assert info.true_relres <= 1e-6
        assert info.iterations == FIRST and info.refinements == 1


# At 1e-10 the second run aims at the remaining 1e-4 or less with the rate of
# the first, which its FP32 residual limits to about 1e-7 in 13 iterations
# (0.29 each); the cycle contracts by 0.2 or less, so the run of at least
# ceil(ln 1e-4 / ln 0.29) + 1 = 9 goes 0.2^9 = 5e-7 beyond the first one's
# 1e-6: the FP64 iterate ends below 1e-12 of the solution, whose own rounding
# (an FP64 solve to 1e-13) is smaller.
@pytest.mark.parametrize("n", [33, 65])
def test_solution_is_more_exact_than_the_tolerance(n):
    s, f = _solver(n, precision="fp64", outer="cg")
    ref, _ = s.solve(f, tol=1e-13)
    for x, info in _solve_each_way(n, 1e-10):
        assert info.true_relres <= 1e-10
        assert relerr(x.cpu().numpy(), ref.cpu().numpy()) <= 1e-12
