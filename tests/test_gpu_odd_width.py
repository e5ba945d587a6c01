"""Strips of odd widths, whose side columns are stored in the pass after their row's: against tiles to
the last bit, with last strips of 1 to 9 columns (the strip before then has some of the side columns)
and in a batch with even widths.  The start state is noise in every node."""
import math

import numpy as np
import pytest

from paper_1903_01168_gb300 import lbm as L

pytestmark = pytest.mark.gpu

FLOWS = {
    "periodic": dict(),
    "walls": dict(bc_y=L.LBM_BC_WALL, gx=5e-6, gy=-2e-6),
    "slip": dict(bc_y=L.LBM_BC_WALL, wall_slip=1, contact_angle=math.radians(60.0)),
}
MODELS = {"bgk": dict(), "mrt_hermite": dict(collision=L.LBM_MRT, equilibrium=L.LBM_EQ_HERMITE)}
STORAGE = [L.LBM_F32, L.LBM_F16DEV, L.LBM_BF16DEV]


def start(nx, ny, **kw):
    rng = np.random.default_rng(nx * 10007 + ny)
    red = rng.uniform(0.0, 1.0, (ny, nx))
    flow = 0.01 * rng.uniform(-1.0, 1.0, (2, ny, nx))
    s = L.Simulation(nx, ny, gamma=2.0, tau_r=0.9, tau_b=1.0, sigma=0.002, beta=0.7, **kw)
    s.init_fields(2.0 * red, 1.0 - red, flow[0], flow[1])
    return s


def state(nx, ny, steps, **kw):
    with start(nx, ny, **kw) as s:
        s.step(steps)
        return s.save_state()


@pytest.mark.parametrize("storage", STORAGE)
@pytest.mark.parametrize("nx,ny", [(9, 4), (11, 30), (15, 19), (17, 8), (127, 21), (129, 40), (131, 17), (135, 33), (137, 6),
                                   (255, 50), (385, 35)])
def test_strips_equal_tiles(nx, ny, storage):
    for flow in FLOWS.values():
        for model in MODELS.values():
            kw = dict(flow, **model, storage=storage)
            tiles = state(nx, ny, 3, **kw)
            for rows in (1, 16):      # pieces of a row, of more rows than are kept
                assert state(nx, ny, 3, plan=L.LBM_PLAN_SPLIT, plan_rows=rows, **kw) == tiles


@pytest.mark.parametrize("storage", STORAGE)
def test_odd_and_even_widths_in_one_batch(storage):
    sizes = [(64, 20), (129, 33), (255, 16), (256, 9), (9, 50)]
    sims = [start(nx, ny, storage=storage) for nx, ny in sizes]
    for plan in (L.LBM_PLAN_SPLIT, L.LBM_PLAN_BALANCED):
        b = L.Batch(sims, plan=plan)
        b.step(5)
        b.close()
    got = [s.save_state() for s in sims]
    for s in sims:
        s.close()
    assert got == [state(nx, ny, 10, storage=storage) for nx, ny in sizes]
