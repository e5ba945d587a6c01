"""Steps of a plan with more than half and at most two thirds of the resident blocks are not launched
early: such a batch is not slower (a tenth allowed) than with a tiny lattice of another storage type
beside it, whose launches keep the others from being early."""
import pytest

from paper_1903_01168_gb300 import autotune as A
from paper_1903_01168_gb300 import lbm as L
from paper_1903_01168_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,other", [(L.LBM_F32, L.LBM_F16DEV), (L.LBM_F16DEV, L.LBM_F32)])
def test_between_half_and_two_thirds_of_the_blocks(storage, other):
    torch = pytest.importorskip("torch")
    with torch.cuda.stream(torch.cuda.Stream()):
        fields = W.bubble_fields(64, 64, 32, 32, 16, 10.0)
        members = 55 * 6 * torch.cuda.get_device_properties(0).multi_processor_count // 90   # one block each
        sims = []
        for _ in range(members):
            s = L.Simulation(64, 64, torch_memory=True, gamma=10.0, sigma=0.005, beta=0.7, storage=storage)
            s.init_fields(*fields)
            sims.append(s)
        tiny = L.Simulation(8, 4, torch_memory=True, gamma=10.0, storage=other)
        tiny.init_fields(*W.bubble_fields(8, 4, 4, 2, 1, 10.0))

        def ms(which):
            b = L.Batch(which)
            try:
                return A._event_ms(b.step, 32)
            finally:
                b.close()

        alone, beside = (min(v) for v in zip(*((ms(sims), ms(sims + [tiny])) for _ in range(3))))
        for s in sims + [tiny]:
            s.close()
    print(f"storage {storage}: {1e3 * alone:.1f} us a step alone, {1e3 * beside:.1f} beside the other group")
    assert alone <= 1.1 * beside
