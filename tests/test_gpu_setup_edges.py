"""The set-up kernels where their FP32 filter is at its edge: permittivities so small that the squares of
their deviations underflow in FP32, and odd rows with tails in the absorbing layers.  The splitting is the
oracle's in FP64 (the same sums in the same precision: 1e-12)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import cbs_oracle as co
from paper_2506_15411_gb300 import inputs

pytestmark = pytest.mark.gpu

LAM = 1.064e-6


def _check(grid, lo, hi, eps, corner="sum"):
    import torch

    from paper_2506_15411_gb300 import CBSPlan
    nx, ny, nz = grid
    g = co.Grid(nx, ny, nz, LAM / 8, LAM, 1.0, lo, hi, corner=corner)
    sp = co.splitting(co.k_squared(g, eps))
    with CBSPlan(nx, ny, nz, g.pitch, LAM, 1.0, lo, hi, tol=0.0, max_iter=1, check_every=1,
                 layer_corner_max=corner == "max") as plan:
        plan.set_permittivity(torch.from_numpy(eps).cuda())
        k0, shift = plan.splitting()
    assert abs(k0 - sp.k0sq) <= 1e-12 * max(abs(sp.k0sq), sp.epsilon)
    assert abs(shift - sp.epsilon) <= 1e-12 * sp.epsilon


@pytest.mark.parametrize("scale", [1e-14, 1e-19, 1e-22, 1e-30])
@pytest.mark.parametrize("kind", ["random", "voxel"])
def test_permittivities_whose_squares_underflow(kind, scale):
    nx, ny, nz = 40, 12, 9
    if kind == "random":
        eps = inputs.random_eps(nx, ny, nz, lo=0.5, hi=3.0, seed=11)
    else:
        eps = np.ones((nz, ny, nx), np.float32)
        eps[4, 5, 37] = 3.0
    _check((nx, ny, nz), (0, 0, 0), (0, 0, 0), (eps * np.float32(scale)).astype(np.float32))


@pytest.mark.parametrize("corner", ["sum", "max"])
@pytest.mark.parametrize("grid,lo,hi", [((135, 7, 9), (16, 1, 0), (16, 1, 0)), ((273, 9, 8), (40, 2, 0), (11, 1, 3)),
                                        ((325, 5, 4), (1, 0, 0), (30, 1, 1)), ((65, 6, 5), (30, 1, 1), (30, 1, 1))])
def test_odd_rows_with_their_tails_in_the_layers(grid, lo, hi, corner):
    _check(grid, lo, hi, inputs.random_eps(*grid, lo=0.5, hi=3.0, seed=grid[0]), corner)
