"""The strip kernel of lattices periodic in x against the FP64 oracle.  Small lattices are stepped in
tiles by default, so these set a plan: pieces of at least 16 rows, longer than the row ring.  The
bars are the ones of the parity, wetting and precision tests."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_1903_01168_gb300 import lbm as L
from paper_1903_01168_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PLAN = dict(plan=L.LBM_PLAN_SPLIT, plan_rows=16)
MRT_HERMITE = dict(collision=L.LBM_MRT, equilibrium=L.LBM_EQ_HERMITE)
U_S = {L.LBM_F16DEV: 2.0 ** -11, L.LBM_BF16DEV: 2.0 ** -8}

CASES = {
    # name: (nx, ny, params); flow speed 0.02
    "periodic_bgk": (200, 67, dict(gamma=10.0, tau_r=0.6, tau_b=1.1, sigma=0.01, beta=0.7, gx=2e-6, gy=-1e-6)),
    "periodic_mrt_hermite": (200, 67, dict(gamma=10.0, tau_r=0.6, tau_b=1.1, sigma=0.01, beta=0.7, gx=2e-6, gy=-1e-6,
                                           **MRT_HERMITE)),
    "walls_bgk": (137, 50, dict(gamma=5.0, tau_r=0.7, tau_b=0.9, sigma=0.005, beta=0.99, bc_y=L.LBM_BC_WALL, gx=1e-5)),
    "walls_mrt_hermite": (96, 65, dict(gamma=10.0, tau_r=0.55, tau_b=1.0, sigma=0.01, beta=0.7, bc_y=L.LBM_BC_WALL, gx=5e-6,
                                       **MRT_HERMITE)),
    "slip_angle": (150, 41, dict(gamma=2.0, tau_r=0.8, tau_b=1.0, sigma=0.01, beta=0.7, gx=2e-6, bc_y=L.LBM_BC_WALL,
                                 wall_slip=1, contact_angle=math.radians(60.0))),
    "angle_mrt_hermite": (150, 41, dict(gamma=2.0, tau_r=0.8, tau_b=1.0, sigma=0.01, beta=0.7, gx=2e-6, bc_y=L.LBM_BC_WALL,
                                        contact_angle=math.radians(120.0), **MRT_HERMITE)),
}


def fields_of(nx, ny, kw):
    if kw.get("contact_angle"):      # a drop on the wall
        rb = np.zeros((ny, nx))
        rb[:12, nx // 2 - 20:nx // 2 + 20] = 1.0
        ux = 0.01 * np.random.default_rng(3).standard_normal((ny, nx))
        return 1.0 - rb, rb, ux, np.zeros((ny, nx))
    return W.random_fields(nx, ny, seed=nx + ny, gamma=kw["gamma"], u_amp=0.02, walls_y=kw.get("bc_y", 0) == L.LBM_BC_WALL)


def oracle_after(nx, ny, kw, fields, library=None):
    o = O.Oracle(O.OracleParams(nx=nx, ny=ny, **kw), library)
    o.init_fields(*fields)
    o.step(100)
    return o.fields()


def errors(fo, f):
    ro = fo["rho_r"] + fo["rho_b"]
    umax = max(np.abs(fo["ux"]).max(), np.abs(fo["uy"]).max(), 0.02)
    return (np.max(np.abs(f["rho_r"] + f["rho_b"] - ro) / ro),
            max(np.abs(f["ux"] - fo["ux"]).max(), np.abs(f["uy"] - fo["uy"]).max()) / umax,
            np.max(np.abs(f["rho_r"] - fo["rho_r"]) / ro))


@pytest.fixture(scope="module")
def fp32_oracle(tmp_path_factory):
    return O.fp32_library(str(tmp_path_factory.mktemp("oracle_fp32")))


def stepped(nx, ny, kw, fields):
    with L.Simulation(nx, ny, **PLAN, **kw) as s:
        s.init_fields(*fields)
        s.step(100)
        return s.fields()


@pytest.mark.parametrize("name", sorted(CASES))
def test_strips_100_steps(name, fp32_oracle):
    nx, ny, kw = CASES[name]
    f = fields_of(nx, ny, kw)
    fo = oracle_after(nx, ny, kw, f)
    got, floor = errors(fo, stepped(nx, ny, kw, f)), errors(fo, oracle_after(nx, ny, kw, f, fp32_oracle))
    print(name, " ".join(f"{what} {e:.2e} (floor {F:.2e})" for what, e, F in zip(("rho", "u", "colour"), got, floor)))
    for e, F in zip(got, floor):
        assert e <= max(1e-5, 2.0 * F)


@pytest.mark.parametrize("storage", sorted(U_S))
def test_strips_16_bit(storage):
    nx, ny, kw = CASES["periodic_mrt_hermite"]
    f = fields_of(nx, ny, kw)
    e_rho, e_u, _ = errors(oracle_after(nx, ny, kw, f), stepped(nx, ny, dict(kw, storage=storage), f))
    print(f"storage {storage}: rho {e_rho:.2e} u {e_u:.2e}")
    assert e_rho <= 2 * U_S[storage] and e_u <= 20 * U_S[storage]
