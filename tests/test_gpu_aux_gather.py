"""Products of the auxiliary-space cycle on either side of the row count where
their gathers change form, and with rows left over, against plain FP64
products with the exported operators."""
import functools

import numpy as np
import pytest
import scipy.sparse as sp
import torch

from oracle import aux
from paper_2509_08109_gb300 import binding, inputs
from tests.gpu_util import relerr

pytestmark = pytest.mark.gpu

OMEGA = 2.0 / 3.0
N = 65

# (304 x 512) interior vertices are the most that take the deep form; 305 x 512
# and 307 x 521 (no multiple of a slice or a block) the other one
SIZES = [(306, 514), (307, 514), (309, 523)]


@functools.lru_cache(maxsize=None)
def _mesh(nr, nt):
    return inputs.annulus_mesh(nr, nt)


class _Plain:
    def __init__(self, a, m, s, mass_steps):
        self.iv = np.flatnonzero(~m.dirichlet)
        nv = len(self.iv)

        def get(w, shape):
            rp, col, val = a.export(w)
            return sp.csr_matrix((val, col, rp), shape=shape)
        self.A, self.M, self.C = get("A", (nv, nv)), get("M", (nv, nv)), get("C", (nv, N * N))
        self.d = self.A.diagonal()
        p = m.xy[m.tri]
        e, f = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
        area = 0.5 * np.abs(e[:, 0] * f[:, 1] - e[:, 1] * f[:, 0])
        lump = np.bincount(m.tri.reshape(-1), np.repeat(area / 3, 3), len(m.xy))[self.iv]
        self.minv = (lambda r: r / lump) if mass_steps == 0 else (lambda r: aux.cg_steps(self.M, r, mass_steps))
        self.s = s

    def cycle(self, f, u):
        u = u + OMEGA * (f - self.A @ u) / self.d
        rc = (self.C.T @ self.minv(f - self.A @ u)).reshape(N, N)
        ec = self.s.vcycle(torch.as_tensor(rc, device="cuda")).cpu().numpy().reshape(-1)
        u = u + self.minv(self.C @ ec)
        return u + OMEGA * (f - self.A @ u) / self.d


def _setup(nr, nt, precision, mass_steps, krylov):
    m = _mesh(nr, nt)
    s = binding.Solver(2, N, precision=precision)
    s.assemble(torch.as_tensor(inputs.coords_quarter_annulus(N)), torch.ones((N - 1, N - 1), dtype=torch.float64))
    s.setup()
    a = binding.AuxSolver(s, m, mass_steps=mass_steps, krylov=krylov)
    return m, a, _Plain(a, m, s, mass_steps)


# FP64 sums of at most some forty terms on both sides, in other orders, through
# two cycles: as the cycles at a fixed count against the oracle, 1e-11.
@pytest.mark.parametrize("mass_steps", [0, 2])
@pytest.mark.parametrize("nr,nt", SIZES)
def test_cycles(nr, nt, mass_steps):
    m, a, p = _setup(nr, nt, "fp64", mass_steps, False)
    f = m.f[p.iv]
    u = p.cycle(f, p.cycle(f, np.zeros_like(f)))
    got, info = a.solve(torch.as_tensor(m.f, device="cuda"), tol=0.0, maxit=2, raise_on_nonconv=False)
    assert info.iterations == 2
    got = got.cpu().numpy()[p.iv]
    assert relerr(got, u) <= 1e-11
    res = np.linalg.norm(f - p.A @ got) / np.linalg.norm(f)
    assert abs(info.true_relres - res) <= 1e-10 * res


# One step of flexible CG is alpha z with z = B f, alpha = f.z / z.Az.  FP64: as
# above.  FP32: z carries the roundings of sums of some forty FP32 terms at each
# of the cycle's five stages, 200 u = 1.2e-5 of the stages' values, which add to z.
@pytest.mark.parametrize("precision,bound", [("fp64", 1e-11), ("fp32", 1.2e-5)])
@pytest.mark.parametrize("nr,nt", SIZES)
def test_first_step_of_flexible_cg(nr, nt, precision, bound):
    m, a, p = _setup(nr, nt, precision, 0, True)
    f = m.f[p.iv]
    z = p.cycle(f, np.zeros_like(f))
    u = (f @ z) / (z @ (p.A @ z)) * z
    got, info = a.solve(torch.as_tensor(m.f, device="cuda"), tol=1e-10, maxit=1, raise_on_nonconv=False)
    assert info.iterations == 1
    got = got.cpu().numpy()[p.iv]
    assert relerr(got, u) <= bound
    res = np.linalg.norm(f - p.A @ got) / np.linalg.norm(f)
    assert abs(info.true_relres - res) <= 1e-10 * res
