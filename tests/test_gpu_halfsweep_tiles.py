"""The half-sweep smoother's tile shapes on the GPU: column tiles with a
three-column halo (levels above 129^3: 257^3 is the smallest) and FP64 levels,
against the per-colour kernels on the same operator, which have no tiles."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_08109_gb300 import binding, inputs
from tests.gpu_util import U32, relerr

pytestmark = pytest.mark.gpu


def _box(n):
    """Identity map and log-normal kappa: well conditioned on every level."""
    gen = torch.Generator(device="cuda").manual_seed(n)
    kappa = torch.randn((n - 1,) * 3, dtype=torch.float64, device="cuda", generator=gen).mul_(0.5).exp_()
    r = torch.randn((n,) * 3, dtype=torch.float64, device="cuda", generator=gen)
    return torch.as_tensor(inputs.coords_identity(n, 3)), kappa, r


def _vcycle(n, precision, unfused):
    coords, kappa, r = _box(n)
    s = binding.Solver(3, n, precision=precision, unfused=unfused)
    return s.assemble(coords, kappa).setup().vcycle(r)


# Both smoothers sum a point's 26 products in the same order, and the other
# kernels are the same, so in FP32 the cycles differ by at most a few roundings
# of the result's largest value (bound 4 u, as at 33^3 to 129^3).  In FP64 one
# multiplies by the stored reciprocal diagonal where the other divides, 2 u a
# point and colour, over 8 levels x 16 colours: 256 u = 3e-14, held to 1e-12 as
# the cycle is against the oracle.
@pytest.mark.parametrize("n", [33, 65, 129, 257])
@pytest.mark.parametrize("precision,bound", [("fp32", 4 * U32), ("fp64", 1e-12)])
def test_half_sweeps_match_the_colour_sweeps(n, precision, bound):
    z = _vcycle(n, precision, False)
    ref = _vcycle(n, precision, True)
    scale = ref.abs().max()
    assert bool((z[1:-1, 1:-1, 1:-1] != 0).all())
    assert float((z - ref).abs().max() / scale) <= bound


@pytest.mark.parametrize("n", [33, 65])
def test_fp64_colour_sweeps_match_oracle(n):
    coords, kappa, r = _box(n)
    z = _vcycle(n, "fp64", True).cpu().numpy()
    H = oracle.Hierarchy(oracle.assemble(coords.numpy(), kappa.cpu().numpy()))
    assert relerr(z, H.vcycle(r.cpu().numpy())) <= 1e-12
