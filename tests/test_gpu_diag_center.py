"""Pressure jump around a bubble centre outside the box: nodes within rounding of the inner or outer
radius count by their FP64 distance, whatever the sign of the wrapped coordinate difference."""
import numpy as np
import pytest

from paper_1903_01168_gb300 import lbm as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("which,factor,add", [("p_out", 1.0, 8.0), ("p_in", 0.5, 0.0)])
def test_nodes_on_the_radius_of_a_centre_outside_the_box(which, factor, add, axis):
    n = 100
    rng = np.random.default_rng(2)
    blue = np.zeros((n, n))
    blue[30:70, 20:60] = 1.0
    red = (1.0 - blue) * rng.uniform(0.5, 1.5, (n, n))
    y, x = np.mgrid[0:n, 0:n]
    with L.Simulation(n, n, gamma=1.0) as s:
        def start(cx, cy):
            s.init_bubble(cx, cy, 20.0)       # sets the centre
            s.init_fields(red, blue, 0 * red, 0 * red)
            return s.diagnostics()

        r = start(50.0, 50.0)["r_eff"] * factor + add
        p = s.fields()["p"]
        for node in range(10, 90, 8):
            for side in (1e-10, -1e-10):      # the node (x, y) = (node, 40) lies just out of or inside the radius
                c = [node - n - r * (1.0 + side), 40.0]
                got = start(*(c if axis == 0 else c[::-1]))[which]
                d = [np.abs(q - v) for q, v in zip((x, y), c if axis == 0 else c[::-1])]
                dist = np.sqrt(sum(np.minimum(q, n - q) ** 2 for q in d))
                want = p[dist > r if which == "p_out" else dist < r].mean()
                assert abs(got - want) <= 1e-12 * want, (node, side)
