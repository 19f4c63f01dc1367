"""The set-up kernels: the splitting they find against the oracle's in FP64 (the same sums in the
same precision, so all but the last digits: 1e-12), on permittivities whose voxels repeat, differ
everywhere or hide their one extreme voxel, with layers on and off, both corner rules, odd and
short axes; and a refused permittivity leaves the plan as it was."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import cbs_oracle as co
from paper_2506_15411_gb300 import inputs

pytestmark = pytest.mark.gpu

LAM = 1.064e-6


def _eps(kind, g, seed):
    nx, ny, nz = g.nx, g.ny, g.nz
    if kind == "random":
        return inputs.random_eps(nx, ny, nz, lo=0.5, hi=3.0, seed=seed)
    e = np.ones((nz, ny, nx), np.float32)
    if kind == "slab":
        e[nz // 3: nz // 2] = 2.25
        e[nz // 2, :, ::2] = 1.7
    else:   # one voxel decides: the lowest, in the interior; the rest alike
        e[:] = 2.0
        e[nz // 2, ny // 2, nx // 2] = -0.75
    return e


@pytest.mark.parametrize("kind", ["random", "slab", "voxel"])
@pytest.mark.parametrize("grid,pads", [((40, 36, 44), (4, 5, 6)), ((131, 7, 9), (16, 1, 0)), ((33, 21, 5), (0, 0, 0)),
                                       ((300, 20, 12), (40, 3, 2))])
@pytest.mark.parametrize("corner", ["sum", "max"])
def test_splitting_matches_the_oracle(kind, grid, pads, corner):
    import torch

    from paper_2506_15411_gb300 import CBSPlan
    nx, ny, nz = (n if n != 131 else 132 for n in grid)
    g = co.Grid(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads, corner=corner)
    eps = _eps(kind, g, seed=nx + ny)
    sp = co.splitting(co.k_squared(g, eps))
    with CBSPlan(nx, ny, nz, g.pitch, LAM, 1.0, pads, pads, tol=0.0, max_iter=1, check_every=1,
                 layer_corner_max=corner == "max") as plan:
        plan.set_permittivity(torch.from_numpy(eps).cuda())
        k0, shift = plan.splitting()
    assert abs(k0 - sp.k0sq) <= 1e-12 * max(abs(sp.k0sq), sp.epsilon)
    assert abs(shift - sp.epsilon) <= 1e-12 * sp.epsilon


def test_a_refused_permittivity_leaves_the_plan_as_it_was():
    import torch

    from paper_2506_15411_gb300 import CBSPlan, PlaneWave
    from paper_2506_15411_gb300._lib import CBSError
    nx, ny, nz = 24, 20, 16
    eps = torch.from_numpy(inputs.random_eps(nx, ny, nz, seed=3)).cuda()
    bad = eps.clone()
    bad[5, 6, 7] = float("inf")
    flat = torch.ones_like(eps)
    with CBSPlan(nx, ny, nz, LAM / 8, LAM, 1.0, (0, 0, 0), (0, 0, 0), tol=0.0, max_iter=6, check_every=3) as plan:
        plan.set_permittivity(eps)
        want, sp = plan.forward(PlaneWave(z_plane=4))[0].clone(), plan.splitting()
        for e in (bad, flat):   # a non-finite voxel; no layers and no contrast: epsilon = 0
            with pytest.raises(CBSError):
                plan.set_permittivity(e)
            assert plan.splitting() == sp
            assert torch.equal(plan.forward(PlaneWave(z_plane=4))[0], want)
        plan.set_permittivity(eps)
        assert torch.equal(plan.forward(PlaneWave(z_plane=4))[0], want)
