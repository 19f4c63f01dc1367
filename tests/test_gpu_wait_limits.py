"""GPU: tile waits that run out.  With a limit of no polls every wait of the tile kernels gives up at once,
while copies are under way; with a few polls some do.  Each kernel then has to end by itself with its error
recorded, and the plan's next solve has to be what it was.  Grids: both kinds of the x, y and z kernels,
tiles stored by the copying warp and by the groups, one and many tiles a block."""
from __future__ import annotations

import pytest

from paper_2506_15411_gb300 import inputs

pytestmark = pytest.mark.gpu

LAM = 1.064e-6


@pytest.mark.parametrize("grid", [(40, 36, 44), (128, 56, 130), (64, 512, 48), (343, 36, 44), (36, 343, 3), (343, 343, 169)])
def test_waits_that_run_out_end_the_solve_and_leave_the_plan_usable(grid):
    import torch

    from paper_2506_15411_gb300 import CBSPlan, PlaneWave
    from paper_2506_15411_gb300 import _lib as L
    nx, ny, nz = grid
    pads = tuple(min(3, n // 5) for n in grid)
    with CBSPlan(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads, tol=0.0, max_iter=6, check_every=3) as plan:
        plan.set_permittivity(torch.from_numpy(inputs.random_eps(nx, ny, nz, seed=2)).cuda())
        want = plan.forward(PlaneWave())[0].clone()
        for polls in (0, 1, 3, 0):
            L.check(plan.lib.cbs_selftest_wait_limit(plan.handle, polls))
            try:
                E = plan.forward(PlaneWave())[0]
                assert polls > 0 and torch.equal(E, want)   # (no wait ran out)
            except L.CBSError as e:
                assert e.code == L.CBS_ERR_CUDA and "timed out" in str(e)
        L.check(plan.lib.cbs_selftest_wait_limit(plan.handle, -1))
        E, st = plan.forward(PlaneWave())
        assert st.iters == 6 and torch.equal(E, want)
