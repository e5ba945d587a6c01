"""What the tuner picks for one lattice is not slower than the library's default (a quarter allowed,
well above what timings of one choice differ by)."""
import pytest

from paper_1903_01168_gb300 import autotune as A

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 64), (200, 200), (2048, 128)])
def test_tuned_single_lattice_against_the_default(nx, ny):
    t = A.Autotuner(steps=60)
    t.tune_single(nx, ny, gamma=10.0)
    tuned = t.params_for(nx, ny, False, gamma=10.0)

    def ms(params):
        s = A._start(nx, ny, params, {})
        try:
            return A._event_ms(s.step, 200)
        finally:
            s.close()

    got, default = (min(v) for v in zip(*((ms(tuned), ms(dict(gamma=10.0))) for _ in range(4))))
    print(f"{nx}x{ny}: tuned {tuned} {1e3 * got:.2f} us a step, default {1e3 * default:.2f}")
    assert got <= 1.25 * default
