"""CPU check of the tiles that the 3-D half-sweep kernels run (no GPU): the
model of test_halfsweep_schedule with the rows and columns a CTA really
computes.  Its region is the owned rows and one row on each side; a row parity
at a time, first the one that the direction starts with, on all of the
region's rows, then the other one on the owned rows alone (the halo row of the
second parity is left out).  Columns: the whole row without a halo (levels up
to 129^3), or the owned columns and three on each side."""
import numpy as np
import pytest

from tests.test_halfsweep_schedule import _operator, _plain_sweep, _update


def _half(a, f, xin, xz, xout, parity, forward, ti, tj, drop=None):
    """One half sweep of all planes of one parity in tiles of tj rows (even)
    and ti columns (None: the whole row).  drop: a row parity whose halo row is
    left out as well ("first")."""
    n = xin.shape[0]
    m = n - 2
    first = 0 if forward else 1
    for k in range(2 - parity, n - 1, 2):
        for j0 in range(1, 1 + m, tj):
            for i0 in range(1, 1 + m, ti or m):
                plane = xin[k].copy()
                lo, hi = (1, m + 1) if ti is None else (i0 - 3, i0 + ti + 3)
                for jpar in (first, 1 - first):
                    rows = [j for j in range(j0 - 1, j0 + tj + 1) if (j - (j0 - 1)) % 2 == jpar]
                    if jpar != first or drop == "first":
                        rows = [j for j in rows if j0 <= j < j0 + tj]
                    for ipar in ((0, 1) if forward else (1, 0)):
                        for j in rows:
                            for i in range(lo, hi):
                                if (i & 1) == ipar and 1 <= i <= m and 1 <= j <= m:
                                    plane[j, i] = _update(a, f, None, i, j, k,
                                                          lambda dz: plane if dz == 0 else xz[k + dz])
                j1 = min(j0 + tj, m + 1)
                i1 = m + 1 if ti is None else min(i0 + ti, m + 1)
                xout[k, j0:j1, i0:i1] = plane[j0:j1, i0:i1]


def _both(n, ti, tj, drop=None):
    """(down, up) by half sweeps and by plain 8-colour sweeps."""
    a = _operator(n, n)
    rng = np.random.default_rng(n + 1)
    inner = (slice(1, -1),) * 3
    f = np.zeros((n, n, n))
    f[inner] = rng.uniform(-1, 1, (n - 2,) * 3)
    zero = np.zeros((n, n, n))
    ref, x = zero.copy(), zero.copy()
    _plain_sweep(a, f, ref, range(8))
    _half(a, f, zero, zero, x, 0, True, ti, tj, drop)
    _half(a, f, zero, x, x, 1, True, ti, tj, drop)
    x0 = zero.copy()
    x0[inner] = rng.uniform(-1, 1, (n - 2,) * 3)
    up, y = x0.copy(), x0.copy()
    _plain_sweep(a, f, up, range(7, -1, -1))
    _half(a, f, x0, x0, y, 1, False, ti, tj, drop)
    _half(a, f, x0, y, y, 0, False, ti, tj, drop)
    return (x, ref), (y, up)


@pytest.mark.parametrize("n,ti,tj", [(9, None, 4), (17, None, 4), (17, None, 8), (17, 6, 4), (17, 10, 2), (11, 4, 6)])
def test_tiles_give_the_eight_colour_sweep(n, ti, tj):
    for got, ref in _both(n, ti, tj):
        assert np.array_equal(got, ref)


def test_the_first_parity_needs_its_halo_row():
    for got, ref in _both(17, None, 4, drop="first"):
        assert not np.array_equal(got, ref)
