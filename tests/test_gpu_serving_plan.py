"""The plan that the server gives its batches is not slower than the library's own for an uneven set
of open channels (a tenth allowed, above what timings of one plan differ by)."""
import numpy as np
import pytest

from paper_1903_01168_gb300 import autotune as A
from paper_1903_01168_gb300 import lbm as L
from paper_1903_01168_gb300.serving import Server

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [L.LBM_F32, L.LBM_F16DEV])
def test_server_plan_against_the_default(storage):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(4)
    server = Server()
    with torch.cuda.stream(torch.cuda.Stream()):
        sims = []
        for _ in range(8):
            nx, ny = 32 * int(rng.integers(16, 257)), 32 * int(rng.integers(2, 9))
            s = L.Simulation(nx, ny, torch_memory=True, gamma=5.0, tau_r=0.8, tau_b=0.8, sigma=1e-3, bc_x=L.LBM_BC_INOUT,
                             bc_y=L.LBM_BC_WALL, u_in_r=0.0125, u_in_b=0.025, p_out=0.48, inlet_period_r=40,
                             inlet_period_b=20, storage=storage)
            s.init_fields(np.full((ny, nx), 5.0), *[np.zeros((ny, nx))] * 3)
            sims.append(s)

        def ms(**plan):
            b = L.Batch(sims, **plan)
            try:
                return A._event_ms(b.step, 32)
            finally:
                b.close()

        got, default = (min(v) for v in zip(*((ms(plan=server.plan, row_overhead=server.row_overhead), ms())
                                              for _ in range(3))))
        print(f"storage {storage}: server's plan {1e3 * got:.1f} us a step, the library's {1e3 * default:.1f}")
        for s in sims:
            s.close()
    assert got <= 1.1 * default
