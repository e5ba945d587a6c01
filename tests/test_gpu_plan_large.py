"""The plan of large FP32 lattices: wholly periodic BGK ones of even widths whose pieces come out even
are cut for 4 blocks per SM, the others for 5; 16-bit storage and MRT with the Hermite source for all
6.  (Cut for 5, some of both were slower than with the kernel before.)"""
import numpy as np
import pytest

from paper_1903_01168_gb300 import lbm as L

pytestmark = pytest.mark.gpu

WALLS = dict(bc_y=L.LBM_BC_WALL, gx=1e-6)
SLIP = dict(bc_y=L.LBM_BC_WALL, wall_slip=1)
MRT_HERMITE = dict(collision=L.LBM_MRT, equilibrium=L.LBM_EQ_HERMITE)


@pytest.mark.parametrize("nx,ny,per_sm,kw", [
    (256, 8192, 4, dict()), (2048, 2048, 4, dict()), (2048, 2048, 4, dict(equilibrium=L.LBM_EQ_HERMITE)),
    (4096, 2048, 4, WALLS), (2048, 1280, 5, WALLS), (2048, 2048, 6, MRT_HERMITE), (2048, 2048, 5, dict(collision=L.LBM_MRT)), (4096, 2048, 5, SLIP),
    (2000, 2000, 4, dict()), (2047, 2048, 5, dict()), (2496, 820, 5, dict()), (8192, 256, 5, dict()), (1024, 1792, 5, dict()), (2048, 2048, 6, dict(storage=L.LBM_F16DEV))])
def test_blocks_of_a_large_lattice(nx, ny, per_sm, kw):
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with L.Simulation(nx, ny, gamma=2.0, **kw) as s:
        b = L.Batch([s])
        assert -(-b.items // sms) == per_sm       # one piece per block
        b.close()


def test_states_do_not_depend_on_it():
    nx, ny = 256, 8200
    rng = np.random.default_rng(5)
    red = rng.uniform(0.0, 1.0, (ny, nx))
    flow = 0.01 * rng.uniform(-1.0, 1.0, (2, ny, nx))

    def state(**plan):
        with L.Simulation(nx, ny, gamma=2.0, tau_r=0.9, tau_b=1.0, sigma=0.002, beta=0.7, **plan) as s:
            s.init_fields(2.0 * red, 1.0 - red, flow[0], flow[1])
            s.step(3)
            s.step(34)
            return s.save_state()

    assert state() == state(plan=L.LBM_PLAN_BALANCED, plan_rows=100)
