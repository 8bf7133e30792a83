"""Finest-grid assembly at the edges of the kernels' tiles (2-D strips of 63
node columns and bands of rows, 3-D columns of 15 x 15 nodes and bands of
planes): one node more and less than a tile, the smallest grids and odd sizes,
against the oracle.  The bound is the oracle's own rounding: it sums
coordinates of order one to Jacobian entries of order 1/n, which loses a few
n eps; 20 n eps of the row's diagonal covers it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_08109_gb300 import binding, inputs
from tests.gpu_util import rel_to_diag

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, n) for n in (3, 4, 62, 63, 64, 65, 126, 127, 128, 190)]
                         + [(3, n) for n in (3, 4, 14, 15, 16, 17, 30, 31, 32)])
def test_assembly_at_tile_edges(dim, n):
    if dim == 2:
        coords = inputs.coords_bump(n, 0.11, -0.13)
    else:
        coords = inputs.coords_identity(n, 3)
        bump = np.prod(np.sin(np.pi * coords), axis=0)
        coords = coords + np.array([0.1, -0.08, 0.06])[:, None, None, None] * bump
    kappa = np.exp(np.random.default_rng(n).normal(0.0, 0.5, size=(n - 1,) * dim))
    ref = oracle.assemble(coords, kappa)
    out = torch.full((n,) * dim + (3 ** dim,), float("nan"), dtype=torch.float64, device="cuda")
    binding.assemble_noalloc(dim, n, torch.as_tensor(coords, device="cuda"), torch.as_tensor(kappa, device="cuda"), out)
    got = out.cpu().numpy()
    assert np.isfinite(got).all()
    inner = (slice(1, -1),) * dim
    assert rel_to_diag(got[inner], ref[inner]) <= 20 * n * np.finfo(float).eps
    edge = np.ones((n,) * dim, bool)
    edge[inner] = False
    assert not got[edge].any()
