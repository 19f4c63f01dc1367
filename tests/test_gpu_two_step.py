"""The two-step passes (csrc/xrow.cuh, csrc/colpass.cuh) on every axis length they take, against
the FP64 oracle: one axis runs over all lengths that split into two radices while the others are
short and odd, so that tiles, lanes and boxes have remainders in every shape.  Tolerance: three
complex64 iterations carry about 1e-6 each (six short transforms of length <= 1024 and a dozen
complex products), so 2e-5 of the field in relative L2, as for the other parity cases."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import cbs_oracle as co
from paper_2506_15411_gb300 import inputs

pytestmark = pytest.mark.gpu

LAM = 1.064e-6
K = 3


def _lengths(lo, hi):
    def ok(m):
        for p in (2, 3, 5, 7, 11, 13):
            while m % p == 0:
                m //= p
        return m == 1
    return [n for n in range(lo, hi + 1) if ok(n)]


def _check(nx, ny, nz):
    import torch

    from paper_2506_15411_gb300 import CBSPlan, PlaneWave
    pads = tuple(min(2, n // 5) for n in (nx, ny, nz))
    g = co.Grid(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads)
    eps = inputs.random_eps(nx, ny, nz, seed=nx + 3 * ny + 7 * nz)
    pol = (1.0, 0.25j, 0.5)
    ref = co.forward(g, eps, co.plane_wave_source(g, pol=pol), tol=0.0, max_iter=K)
    with CBSPlan(nx, ny, nz, g.pitch, LAM, 1.0, pads, pads, tol=0.0, max_iter=K, check_every=K) as plan:
        plan.set_permittivity(torch.from_numpy(eps).cuda())
        E, st = plan.forward(PlaneWave(pol=pol))
        E = E.cpu().numpy()
    assert st.iters == K
    err = np.linalg.norm(E - ref.E) / np.linalg.norm(ref.E)
    assert err <= 2e-5, (nx, ny, nz, err)
    r = ref.history[-1] / ref.history[0]
    assert abs(st.rel_resid - r) <= 1e-4 * r, (nx, ny, nz)


# every length: the rows' remainders (21 rows, 35 rows), partial tiles of 8 and 16 columns
@pytest.mark.parametrize("lo,hi", [(4, 128), (129, 400), (401, 1024)])
def test_every_x_length(lo, hi):
    for n in _lengths(lo, hi):
        _check(n, 7, 3 if n % 2 else 5)


@pytest.mark.parametrize("lo,hi", [(4, 128), (129, 400), (401, 1024)])
def test_every_y_length(lo, hi):
    for n in _lengths(lo, hi):
        if n % 2 and n > 853:
            continue    # refused: two tiles of 16 columns, the only width for odd y, do not fit
        _check(18 if n % 2 else 9, n, 3)


@pytest.mark.parametrize("lo,hi", [(4, 128), (129, 432)])
def test_every_z_length(lo, hi):
    for n in _lengths(lo, hi):
        _check(9 if n % 2 else 18, 3, n)


@pytest.mark.parametrize("grid", [(40, 132, 64), (45, 56, 130), (96, 270, 63)])
def test_several_tiles_of_each_kind_per_block(grid):
    """Enough tiles that every block runs its ring of tiles more than once round."""
    _check(*grid)
