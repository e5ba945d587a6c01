"""Tiles against strips where the tile kernel can go wrong: a lone column right of the last full
tile, and every launch shape at ragged sizes.  The start state is noise in every node, so that no
node's colour field is saturated and any difference in the order of a sum shows; the stored
states have to be equal to the last bit."""
import math

import numpy as np
import pytest

from paper_1903_01168_gb300 import lbm as L

pytestmark = pytest.mark.gpu

FLOWS = {
    "periodic": dict(),
    "walls": dict(bc_y=L.LBM_BC_WALL, gx=5e-6, gy=-2e-6),
    "slip": dict(bc_y=L.LBM_BC_WALL, gx=5e-6, wall_slip=1, contact_angle=math.radians(60.0)),
}
MODELS = {
    "bgk": dict(),
    "mrt_hermite": dict(collision=L.LBM_MRT, equilibrium=L.LBM_EQ_HERMITE),
}


def noise(nx, ny):
    rng = np.random.default_rng(nx * 10007 + ny)
    red = rng.uniform(0.0, 1.0, (ny, nx))
    flow = 0.01 * rng.uniform(-1.0, 1.0, (2, ny, nx))
    return 2.0 * red, 1.0 - red, flow[0], flow[1]


def states(nx, ny, plan, steps, **kw):
    """Stored states after each number of steps, stepped on from one to the next."""
    out = []
    with L.Simulation(nx, ny, gamma=2.0, tau_r=0.9, tau_b=1.0, sigma=0.002, beta=0.7, plan=plan, **kw) as s:
        s.init_fields(*noise(nx, ny))
        for n in steps:
            s.step(n)
            assert s.diagnostics()["nonfinite"] == 0
            out.append(s.save_state())
    return out


@pytest.mark.parametrize("storage", [L.LBM_F32, L.LBM_F16DEV, L.LBM_BF16DEV])
@pytest.mark.parametrize("nx,ny", [(65, 4), (65, 23), (193, 24), (321, 6)])
@pytest.mark.parametrize("flow", ["walls", "slip"])
def test_lone_column_beside_the_last_tile(flow, nx, ny, storage):
    """nx = 65 mod 128 between walls: the strip that ends with the lone column forms the column
    beyond it link by link, and so has the tile left of it."""
    for model in MODELS.values():
        kw = dict(FLOWS[flow], **model, storage=storage)
        assert states(nx, ny, L.LBM_PLAN_AUTO, (1, 1, 3), **kw) == states(nx, ny, L.LBM_PLAN_SPLIT, (1, 1, 3), **kw)


def launch_shape(nx, ny):
    """Rows and warps of a tile's block by the library's rule: the first shape whose tiles are all
    resident (None: strips)."""
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for rows, warps, per_sm in ((2, 5, 3), (4, 7, 2), (4, 4, 4)):
        if -(-nx // 64) * -(-ny // rows) <= per_sm * sms:
            return rows, warps
    return None


@pytest.mark.parametrize("storage", [L.LBM_F32, L.LBM_F16DEV, L.LBM_BF16DEV])
@pytest.mark.parametrize("nx,ny,shape", [(201, 139, (2, 5)), (300, 203, (4, 7)), (193, 301, (4, 7)), (509, 254, (4, 4)),
                                         (449, 301, (4, 4)), (1025, 131, (4, 4)), (450, 313, None)])
def test_every_launch_shape(nx, ny, shape, storage):
    """Ragged sizes of every shape: last columns odd, a last row of tiles of one to three rows; five
    direct launches and a graph of 32 with one more."""
    assert launch_shape(nx, ny) == shape
    for flow in FLOWS.values():
        for model in MODELS.values():
            kw = dict(flow, **model, storage=storage)
            assert states(nx, ny, L.LBM_PLAN_AUTO, (5, 33), **kw) == states(nx, ny, L.LBM_PLAN_SPLIT, (5, 33), **kw)
