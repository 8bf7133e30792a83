"""Inner runs that start on an odd iteration: the run before ended on an even
one, whose step was added at the end, and must not be added again by the odd
iteration that follows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_08109_gb300 import binding, inputs

pytestmark = pytest.mark.gpu


def _problem(dim, n):
    rng = np.random.default_rng(10 * n + dim)
    kappa = np.exp(rng.normal(0.0, 0.3, size=(n - 1,) * dim))
    s = binding.Solver(dim, n, precision="fp32", outer="refine")
    coords = inputs.coords_identity(n, dim)
    s.assemble(torch.as_tensor(coords), torch.as_tensor(kappa)).setup()
    return s, oracle.assemble(coords, kappa), inputs.rhs_uniform(rng, (n,) * dim)


def _relres(A, x, b):
    inner = (slice(1, -1),) * b.ndim
    return np.linalg.norm((b - oracle.apply(A, x))[inner]) / np.linalg.norm(b[inner])


# The first run takes 13 iterations or an odd number more and reduces the
# residual by 1e-6 or so, the second the rest.  The last step of the first run,
# a part of the iterate of the size of its residual or so, added twice would
# leave the second run with a residual above the tolerance and a third would
# follow.  The library's residual and this one's are FP64 sums: 1e-13 apart.
@pytest.mark.parametrize("concurrent", [False, True])
@pytest.mark.parametrize("dim,n", [(2, 65), (2, 257), (3, 17), (3, 65)])
def test_a_run_that_starts_on_odd_parity(dim, n, concurrent):
    s, A, rhs = _problem(dim, n)
    f = torch.as_tensor(rhs, device="cuda")
    _, one = s.solve(f, tol=1e-10, maxit=13, raise_on_nonconv=False)
    assert one.iterations == 13 and one.refinements == 1
    if concurrent:
        x = torch.zeros_like(f)
        info = binding.solve_many([s], [[f]], [[x]], tol=1e-10)[0][0]
    else:
        x, info = s.solve(f, tol=1e-10)
    assert info.refinements == 2 and info.iterations > 13
    assert info.true_relres <= 1e-10
    assert abs(info.true_relres - _relres(A, x.cpu().numpy(), rhs)) <= 1e-13


# Systems of one batch that stop at different counts: the right-hand side of a
# nearly known solution converges at once from it as a guess, others later.
def test_batch_systems_that_stop_at_different_counts():
    probs = [_problem(2, n) for n in (65, 129)]
    bs, xs = [], []
    for s, A, rhs in probs:
        f = [torch.as_tensor(v, device="cuda") for v in (rhs, rhs[::-1].copy(), rhs.T.copy())]
        exact, _ = s.solve(f[1], tol=1e-12)
        bs.append(f)
        xs.append([torch.zeros_like(f[0]), exact * (1 + 1e-7), torch.zeros_like(f[0])])
    infos = binding.Batch([s for s, _, _ in probs]).solve(bs, xs, tol=1e-10)
    for (s, A, rhs), f, x, inf in zip(probs, bs, xs, infos):
        assert inf[1].iterations < inf[0].iterations
        for b, u, i in zip(f, x, inf):
            assert i.true_relres <= 1e-10 and i.refinements <= 3
            assert abs(i.true_relres - _relres(A, u.cpu().numpy(), b.cpu().numpy())) <= 1e-13
