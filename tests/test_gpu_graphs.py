"""Steps replayed as graphs of sixteen and of two chained steps against steps launched one by one.

The kernels and their order are the same either way, so the states must agree bit for bit: for a call
with every graph length and a single step in it, from both state buffers, and across a force change.
"""
import pytest
import torch

from test_gpu_parity import _inputs, _pair, cm  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = {
    "d2q9_f64_channel": dict(lattice="D2Q9", shape=(1, 32, 64), storage="f64",
                             kw=dict(tau=0.8, bc=("periodic", "bounceback", "periodic"))),
    "one_cell_f32": dict(lattice="D3Q27", shape=(5, 6, 40), storage="f32", kw=dict(tau=0.6)),
    "pair_bf16_field": dict(lattice="D3Q27", shape=(8, 12, 64), storage="bf16", kw=dict(tau=0.6)),
    "ragged_f32_walls": dict(lattice="D3Q27", shape=(6, 34, 62), storage="f32", kw=dict(tau=0.6, bc=("bounceback",) * 3)),
    "many_blocks_f32": dict(lattice="D3Q27", shape=(40, 64, 128), storage="f32", kw=dict(tau=0.6)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_long_runs_equal_single_steps_bitwise(cm, name):  # noqa: F811
    case = CASES[name]
    rho, u, F = _inputs(dict(case, flow="tgv"))
    a, _ = _pair(cm, case["lattice"], case["shape"], case["storage"], rho, u, F, **case["kw"])
    b, _ = _pair(cm, case["lattice"], case["shape"], case["storage"], rho, u, F, **case["kw"])
    la, lb = a.launch_count, b.launch_count
    for n in (39, 34):                 # 2 x 16 + 3 x 2 + 1 from one buffer, 2 x 16 + 2 from the other
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert torch.equal(a.get_state().view(torch.uint8), b.get_state().view(torch.uint8))
    for s in (a, b):
        s.set_force((3e-5, 0.0, 0.0 if case["lattice"] == "D2Q9" else -1e-5))
    a.step(33)
    for _ in range(33):
        b.step(1)
    assert torch.equal(a.get_state().view(torch.uint8), b.get_state().view(torch.uint8))
    assert a.launch_count - la == b.launch_count - lb
    a.close()
    b.close()


def test_two_steps_per_pass_with_a_force_along_x(cm):  # noqa: F811
    """The plane-ring schedule takes the collision variants of single steps: the same bits."""
    rho, u, _ = _inputs(dict(lattice="D3Q27", shape=(18, 6, 64), flow="tgv_unforced"))
    a, _ = _pair(cm, "D3Q27", (18, 6, 64), "f32", rho, u, uniform=(3e-4, 0.0, 0.0), kernel="pair_two_steps", tau=0.6)
    b, _ = _pair(cm, "D3Q27", (18, 6, 64), "f32", rho, u, uniform=(3e-4, 0.0, 0.0), kernel="pair", tau=0.6)
    a.step(5)
    b.step(5)
    assert torch.equal(a.get_state(), b.get_state())
    a.close()
    b.close()
