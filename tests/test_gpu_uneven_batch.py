"""Batches of very uneven sizes: every problem's rows are worked on, and only
those, and the scratch of a batch is that of its problems."""
import numpy as np
import pytest
import torch

from paper_2509_08109_gb300 import binding, inputs
from tests.gpu_util import relerr

pytestmark = pytest.mark.gpu


def _problem(n, seed):
    rng = np.random.default_rng(seed)
    coords = inputs.coords_bump(n, 0.1, 0.05)
    kappa = np.exp(rng.normal(0.0, 0.5, size=(n - 1, n - 1)))
    s = binding.Solver(2, n, precision="fp32", outer="refine")
    s.assemble(torch.as_tensor(coords), torch.as_tensor(kappa)).setup()
    return s, torch.as_tensor(inputs.rhs_uniform(rng, (n, n)), device="cuda")


# Every array of a batch's workspace belongs to one problem or holds an entry
# per problem, tile or row, so joining two batches costs no more than both:
# 256 bytes of alignment for each array at most (ten per class, eight per
# problem, twelve of the batch).
def test_workspace_is_the_sum_of_the_problems():
    big = _problem(1025, 0)[0]
    small = [_problem(65, 0)[0] for _ in range(64)]
    both, one, many = (binding.Batch(s).workspace_bytes for s in ([big] + small, [big], small))
    assert both <= one + many + 256 * (10 * 6 + 8 * 65 + 12)


# A problem beside others gives what it gives in a batch of its own: to the
# tolerance, since its tiles, and with them the order of its dot products, may
# be others there.
@pytest.mark.parametrize("sizes", [(513, 65, 65, 129), (65, 257, 65), (129, 65)])
def test_a_problem_is_the_same_beside_others(sizes):
    probs = [_problem(n, k) for k, n in enumerate(sizes)]
    bs = [[f, 0.5 * f.flip(0)] for _, f in probs]
    bs = [[f.contiguous() for f in b] for b in bs]
    xs = [[torch.zeros_like(f) for f in b] for b in bs]
    infos = binding.Batch([s for s, _ in probs]).solve(bs, xs, tol=1e-10)
    for (s, _), b, x, inf in zip(probs, bs, xs, infos):
        ys = [torch.zeros_like(f) for f in b]
        alone = binding.Batch([s]).solve([b], [ys], tol=1e-10)[0]
        for u, y, i, a in zip(x, ys, inf, alone):
            assert i.true_relres <= 1e-10
            assert abs(i.iterations - a.iterations) <= 1
            assert relerr(u.cpu().numpy(), y.cpu().numpy()) <= 1e-7
