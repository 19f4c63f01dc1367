"""The rings of the two-step passes and of the residual partials, gone round more than twice, against the
FP64 oracle: every block has more than twice as many tiles as its ring has sets (checked against the axis
plans), on y tiles stored by the groups and by the copying warp, with and without sets to spare; and blocks
of iterations longer than the ring of residual partials.  Fields to 2e-5 of their norm, residuals to 1e-4, as
in the parity tests."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import cbs_oracle as co
from paper_2506_15411_gb300 import inputs
from test_two_step_host import _plan, ts   # noqa: F401  (ts is a fixture)

pytestmark = pytest.mark.gpu

LAM = 1.064e-6


def _ring_turns(ts, nx, ny, nz, sms):   # noqa: F811
    """Tiles of the busiest block over sets of its ring, of the x, y and z passes."""
    _, _, _, rpb, sx, _ = _plan(ts, nx, 0, ny * nz)[:6]
    _, ty, _, _, sy = _plan(ts, ny, 1)[:5]
    _, tz, _, _, sz = _plan(ts, nz, 2)[:5]
    tiles = -(-ny * nz // rpb), -(-nx // ty) * nz * 3, -(-nx // tz) * ny
    return [t / min(t, sms) / s for t, s in zip(tiles, (sx, sy, sz))]


# y of 56 and 128: tiles the groups store; 256: a copying warp with sets to spare; 512: without
@pytest.mark.parametrize("grid", [(128, 56, 224), (96, 128, 192), (128, 256, 98), (192, 512, 50)])
def test_rings_of_tiles_go_round_more_than_twice(ts, grid):   # noqa: F811
    import torch

    from paper_2506_15411_gb300 import CBSPlan, PlaneWave
    nx, ny, nz = grid
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    turns = _ring_turns(ts, nx, ny, nz, sms)
    assert turns[1] > 2.0, turns
    pads = (2, 2, 2)
    K = 2
    g = co.Grid(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads)
    eps = inputs.random_eps(nx, ny, nz, seed=ny)
    ref = co.forward(g, eps, co.plane_wave_source(g), tol=0.0, max_iter=K)
    with CBSPlan(nx, ny, nz, g.pitch, LAM, 1.0, pads, pads, tol=0.0, max_iter=K, check_every=K) as plan:
        plan.set_permittivity(torch.from_numpy(eps).cuda())
        E, st = plan.forward(PlaneWave())
        E = E.cpu().numpy()
    assert np.linalg.norm(E - ref.E) <= 2e-5 * np.linalg.norm(ref.E)
    r = ref.history[-1] / ref.history[0]
    assert abs(st.rel_resid - r) <= 1e-4 * r


def test_x_and_z_rings_go_round_more_than_twice(ts):   # noqa: F811
    import torch

    from paper_2506_15411_gb300 import CBSPlan, PlaneWave
    grid = nx, ny, nz = 64, 336, 130
    turns = _ring_turns(ts, nx, ny, nz, torch.cuda.get_device_properties(0).multi_processor_count)
    assert min(turns[0], turns[2]) > 2.0, turns
    pads = (2, 2, 2)
    g = co.Grid(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads)
    eps = inputs.random_eps(*grid, seed=4)
    ref = co.forward(g, eps, co.plane_wave_source(g), tol=0.0, max_iter=2)
    with CBSPlan(nx, ny, nz, g.pitch, LAM, 1.0, pads, pads, tol=0.0, max_iter=2, check_every=2) as plan:
        plan.set_permittivity(torch.from_numpy(eps).cuda())
        E = plan.forward(PlaneWave())[0].cpu().numpy()
    assert np.linalg.norm(E - ref.E) <= 2e-5 * np.linalg.norm(ref.E)


def test_blocks_longer_than_the_ring_of_residuals():
    """140 iterations in one block (two turns of the ring and a part) and in blocks of 7 and 70 give one
    field and one residual, the oracle's; so does a served request."""
    import torch

    from paper_2506_15411_gb300 import CBSPlan, PlaneWave
    from paper_2506_15411_gb300.serve import GridSpec, Server
    nx, ny, nz = 40, 36, 44
    pads = (5, 5, 5)
    K = 140
    g = co.Grid(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads)
    eps = inputs.random_eps(nx, ny, nz, seed=9)
    ref = co.forward(g, eps, co.plane_wave_source(g), tol=0.0, max_iter=K)
    dev = torch.from_numpy(eps).cuda()
    out = []
    for check in (140, 70, 7):
        with CBSPlan(nx, ny, nz, g.pitch, LAM, 1.0, pads, pads, tol=0.0, max_iter=K, check_every=check) as plan:
            plan.set_permittivity(dev)
            E, st = plan.forward(PlaneWave())
            out.append((E.clone(), st.rel_resid))
    with Server(max_active=3, tol=0.0, max_iter=K, check_every=140) as srv:
        spec = GridSpec(nx, ny, nz, g.pitch, LAM, 1.0, pads, pads)
        for t in range(2):
            srv.submit(spec, dev, PlaneWave(), (nx // 2, ny // 2, nz // 2), adjoint=False, want_field=True, tag=t)
        out += [(r.E, r.fwd.rel_resid) for r in srv.wait(2)]
    for E, rel in out[1:]:
        assert torch.equal(E, out[0][0]) and rel == out[0][1]
    r = ref.history[-1] / ref.history[0]
    assert abs(out[0][1] - r) <= 1e-4 * r
    assert np.linalg.norm(out[0][0].cpu().numpy() - ref.E) <= 2e-5 * np.linalg.norm(ref.E)


def test_a_served_adjoint_starts_its_twiddle_tables_anew():
    """Blocks of 12 iterations: the forward series ends at the fifth of eight tables, and the adjoint begins
    at the first, as it does through a plan."""
    import torch

    from paper_2506_15411_gb300 import CBSPlan, PlaneWave
    from paper_2506_15411_gb300.serve import GridSpec, Server
    nx, ny, nz = 40, 36, 44
    pads = (5, 5, 5)
    r0 = (nx // 2, ny // 2, nz // 2)
    dev = torch.from_numpy(inputs.random_eps(nx, ny, nz, seed=10)).cuda()
    with CBSPlan(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads, tol=0.0, max_iter=20, check_every=12) as plan:
        plan.set_permittivity(dev)
        E, _ = plan.forward(PlaneWave())
        Ea, _ = plan.adjoint(r0, E)
        grad, _ = plan.gradient(E, Ea, r0)
    with Server(max_active=2, tol=0.0, max_iter=20, check_every=12) as srv:
        spec = GridSpec(nx, ny, nz, LAM / 8, LAM, 1.0, pads, pads)
        for t in range(2):
            srv.submit(spec, dev, PlaneWave(), r0, adjoint=True, want_field=True, want_grad=True, tag=t)
        for r in srv.wait(2):
            assert torch.equal(r.E, E) and torch.equal(r.grad, grad)
