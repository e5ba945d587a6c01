"""The tile kernel that steps small lattices against the strip kernel: the same operations
in the same order, so the whole stored state has to be equal to the last bit."""
import math

import pytest

from paper_1903_01168_gb300 import lbm as L
from paper_1903_01168_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FLOWS = {
    "periodic": dict(),
    "walls": dict(bc_y=L.LBM_BC_WALL, gx=5e-6, gy=-2e-6),
    "slip": dict(bc_y=L.LBM_BC_WALL, gx=5e-6, wall_slip=1, contact_angle=math.radians(60.0)),
    "angle": dict(bc_y=L.LBM_BC_WALL, contact_angle=math.radians(110.0)),
}
MODELS = {
    "bgk": dict(),
    "bgk_hermite": dict(equilibrium=L.LBM_EQ_HERMITE),
    "mrt": dict(collision=L.LBM_MRT),
    "mrt_hermite": dict(collision=L.LBM_MRT, equilibrium=L.LBM_EQ_HERMITE),
}


def _state(nx, ny, steps, plan, stop=-1, **kw):
    with L.Simulation(nx, ny, gamma=10.0, tau_r=0.7, tau_b=1.0, sigma=0.01, beta=0.7, plan=plan, **kw) as s:
        s.init_fields(*W.random_fields(nx, ny, seed=nx * 1000 + ny, gamma=10.0, u_amp=0.02,
                                       walls_y=kw.get("bc_y", 0) == L.LBM_BC_WALL))
        if stop >= 0:
            s.set_stop(stop)
        s.step(steps)
        return s.save_state()


@pytest.mark.parametrize("storage", [L.LBM_F32, L.LBM_F16DEV, L.LBM_BF16DEV])
@pytest.mark.parametrize("nx,ny", [(8, 4), (9, 5), (62, 7), (63, 8), (64, 9), (65, 16), (66, 17), (127, 33), (129, 6), (200, 140)])
def test_tiles_equal_strips(nx, ny, storage):
    for flow in FLOWS.values():
        for model in MODELS.values():
            kw = dict(flow, **model, storage=storage)
            # 7 direct launches, then a graph of 32 steps and 4 more
            for steps in (7, 36):
                assert _state(nx, ny, steps, L.LBM_PLAN_AUTO, **kw) == _state(nx, ny, steps, L.LBM_PLAN_SPLIT, **kw)


def test_tiles_stop():
    kw = dict(storage=L.LBM_F32)
    assert _state(64, 64, 40, L.LBM_PLAN_AUTO, stop=35, **kw) == _state(64, 64, 35, L.LBM_PLAN_SPLIT, stop=35, **kw)
