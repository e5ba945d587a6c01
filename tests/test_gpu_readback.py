"""Read-backs wait for their own simulation only.  A simulation's first read-backs must not allocate
or free memory in a way that waits for the rest of the device."""
import pytest

from paper_1903_01168_gb300 import lbm as L
from paper_1903_01168_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [L.LBM_F32, L.LBM_BF16DEV])
@pytest.mark.parametrize("nx,ny", [(8, 4), (333, 31)])
def test_first_readbacks_do_not_wait_for_other_streams(nx, ny, storage):
    torch = pytest.importorskip("torch")
    kw = dict(gamma=10.0, sigma=0.005, beta=0.7, bc_y=L.LBM_BC_WALL, storage=storage)
    fields = W.bubble_fields(nx, ny, nx / 2, ny / 2, ny / 4, 10.0)

    def start():
        s = L.Simulation(nx, ny, **kw)
        s.init_fields(*fields)
        s.step(5)
        s.synchronize()
        return s

    def read(s):
        d = s.diagnostics()
        geometry, gas = s.slug_geometry()
        return d, geometry, gas.tolist()

    busy = torch.cuda.Stream()
    with start() as s, start() as other:
        want = read(other)          # loads the kernels
        done = torch.cuda.Event()
        with torch.cuda.stream(busy):
            torch.cuda._sleep(1_500_000_000)      # under a second, on one SM
            done.record()
        got = read(s)
        waited = done.query()
        torch.cuda.synchronize()
        assert got == want
        assert not waited, "the read-backs returned only after another stream's work"
