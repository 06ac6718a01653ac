"""The product-form collision (unforced or a uniform force along x, unit higher-order rates) against the
oracle, in every storage, with the one-cell and the two-cell kernels, on both lattices.

One step from the same state at the bounds of test_gpu_parity.py (derived there), on planes of 2048
cells and more (below, a force along x keeps the transforms), and with a force large enough
(1e-2 of rho c_s) that the terms of second order in it would show.
"""
import pytest

import helpers as H
from test_gpu_parity import ONE_STEP_ATOL, ONE_STEP_RTOL, _inputs, _pair, cm  # noqa: F401

pytestmark = pytest.mark.gpu

WALL = [[[0, 0, 0], [0, 0, 0]], [[0.02, 0, 0.0], [-0.03, 0.0, 0.0]], [[0, 0, 0], [0, 0, 0]]]
CASES = {
    "d2q9_unforced": dict(lattice="D2Q9", shape=(1, 47, 61), kw=dict(tau=0.55)),
    "d2q9_channel": dict(lattice="D2Q9", shape=(1, 32, 64), force=6e-3,
                         kw=dict(tau=0.8, omega_bulk=1.2, bc=("periodic", "bounceback", "periodic"), wall_velocity=WALL)),
    "d3q27_unforced_les": dict(lattice="D3Q27", shape=(3, 33, 65), kw=dict(tau=0.52, smagorinsky_cs=0.15)),
    "d3q27_forced": dict(lattice="D3Q27", shape=(4, 16, 128), force=6e-3, kw=dict(tau=0.6, omega_bulk=1.0)),
    "d3q27_forced_walls_les": dict(lattice="D3Q27", shape=(3, 33, 63), force=-6e-3,
                                   kw=dict(tau=0.53, smagorinsky_cs=0.15, van_driest=(26.0, 8.0), wall_velocity=WALL,
                                           bc=("bounceback", "bounceback", "periodic"))),
}


@pytest.mark.parametrize("kernel", ["auto", "direct"])
@pytest.mark.parametrize("storage", ["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("name", list(CASES))
def test_one_step_elementwise(cm, name, storage, kernel):  # noqa: F811
    case = CASES[name]
    rho, u, _ = _inputs(dict(case, flow="tgv_unforced"))
    s, o = _pair(cm, case["lattice"], case["shape"], storage, rho, u, uniform=(case.get("force", 0.0), 0.0, 0.0),
                 kernel=kernel, **case["kw"])
    o.set_state(H.decode(s.get_state(), case["lattice"]))
    s.step(1)
    o.step(1)
    w = H.lattice(case["lattice"]).w.view(-1, 1, 1, 1)
    got, ref = H.decode(s.get_state(), case["lattice"]) / w - 1, o.s / w - 1
    err = (got - ref).abs()
    assert bool((err <= ONE_STEP_ATOL[storage] + ONE_STEP_RTOL[storage] * ref.abs()).all()), f"{err.max().item():.3e}"
    s.close()


@pytest.mark.parametrize("nx,ny", [(33, 70), (57, 41), (130, 19), (129, 16), (1, 70)])
@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q27"])
def test_fp64_rows_of_any_length(cm, lattice, nx, ny):  # noqa: F811
    """The FP64 one-cell step lays rows that do not fill their blocks end to end over the plane."""
    nz = 1 if lattice == "D2Q9" else 3
    case = dict(lattice=lattice, shape=(nz, ny, nx), flow="tgv")
    rho, u, F = _inputs(case)
    s, o = _pair(cm, lattice, case["shape"], "f64", rho, u, F, tau=0.7, bc=("periodic", "bounceback", "periodic"))
    o.set_state(H.decode(s.get_state(), lattice))
    s.step(1)
    o.step(1)
    w = H.lattice(lattice).w.view(-1, 1, 1, 1)
    err = (H.decode(s.get_state(), lattice) / w - o.s / w).abs().max().item()
    assert err <= ONE_STEP_ATOL["f64"], f"{err:.3e}"
    s.close()
