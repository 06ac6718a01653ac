"""A uniform force along x on small grids: the one-cell step takes the product form there too.

One step against the oracle at the bounds of test_gpu_parity.py (derived there), and against the same
force given as a field, whose step goes through the transforms: both are within the bound of the oracle,
so within twice the bound of each other.
"""
import numpy as np
import pytest

import helpers as H
from test_gpu_parity import ONE_STEP_ATOL, ONE_STEP_RTOL, _inputs, _pair, cm  # noqa: F401

pytestmark = pytest.mark.gpu

WALL = [[[0, 0.01, 0], [0, 0, 0.02]], [[0.02, 0, 0.0], [-0.03, 0.0, 0.0]], [[0, 0, 0], [0, 0, 0]]]
CASES = {
    "d2q9_channel": dict(lattice="D2Q9", shape=(1, 12, 31), kw=dict(tau=0.8, bc=("periodic", "bounceback", "periodic"), wall_velocity=WALL)),
    "d2q9_one_row": dict(lattice="D2Q9", shape=(1, 1, 5), kw=dict(tau=0.7)),
    "d2q9_one_column": dict(lattice="D2Q9", shape=(1, 33, 1), kw=dict(tau=0.6, omega_bulk=1.1)),
    "d2q9_below_2048": dict(lattice="D2Q9", shape=(1, 31, 66), kw=dict(tau=0.55, smagorinsky_cs=0.15)),
    "d3q27_tiny": dict(lattice="D3Q27", shape=(2, 3, 4), kw=dict(tau=0.6)),
    "d3q27_walls_les": dict(lattice="D3Q27", shape=(5, 9, 33), kw=dict(tau=0.53, smagorinsky_cs=0.15, van_driest=(26.0, 8.0), wall_velocity=WALL,
                                                                       bc=("bounceback", "bounceback", "periodic"))),
    # above 65,536 cells: blocks of several rows, of which the plane's last are partly empty
    "d2q9_rows_of_94": dict(lattice="D2Q9", shape=(1, 702, 94), kw=dict(tau=0.6)),
    "d3q27_rows_of_94_walls": dict(lattice="D3Q27", shape=(38, 19, 94), kw=dict(tau=0.56, bc=("periodic", "bounceback", "periodic"), wall_velocity=WALL)),
    "d3q27_rows_of_7": dict(lattice="D3Q27", shape=(4, 40, 7), kw=dict(tau=0.56, omega_bulk=1.0)),
}


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("name", list(CASES))
def test_one_step_elementwise(cm, name, storage):  # noqa: F811
    case = CASES[name]
    rho, u, _ = _inputs(dict(case, flow="tgv_unforced"))
    force = (5e-3, 0.0, 0.0)
    s, o = _pair(cm, case["lattice"], case["shape"], storage, rho, u, uniform=force, **case["kw"])
    field = np.zeros((3,) + case["shape"])
    field[0] = force[0]
    f, _ = _pair(cm, case["lattice"], case["shape"], storage, rho, u, field, **case["kw"])
    f.set_state(s.get_state())
    o.set_state(H.decode(s.get_state(), case["lattice"]))
    s.step(1)
    f.step(1)
    o.step(1)
    w = H.lattice(case["lattice"]).w.view(-1, 1, 1, 1)
    got, other, ref = (x / w - 1 for x in (H.decode(s.get_state(), case["lattice"]), H.decode(f.get_state(), case["lattice"]), o.s))
    bound = ONE_STEP_ATOL[storage] + ONE_STEP_RTOL[storage] * ref.abs()
    assert bool(((got - ref).abs() <= bound).all()), f"{(got - ref).abs().max().item():.3e}"
    assert bool(((got - other).abs() <= 2 * bound).all()), f"{(got - other).abs().max().item():.3e}"
    s.close()
    f.close()
