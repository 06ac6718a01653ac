"""Chained steps (one call of many steps) of the kernels that large and long-row grids run, against
steps launched one by one: the same kernels in the same order, so the same bits.

The staged 16-bit step is taken where every resident warp has 8 tiles of 64 cells or more (60 with a
force field); the grids here have a quarter more than that on this device's multiprocessors. States of
up to 256 MiB run graphs of sixteen steps, larger ones graphs of two.
"""
import pytest
import torch

from test_gpu_parity import cm  # noqa: F401

pytestmark = pytest.mark.gpu

CHANNEL = dict(bc=("periodic", "bounceback", "periodic"), smagorinsky_cs=0.1, van_driest=(26.0, 0.3))
# rows (nx, ny), tiles per resident warp and resident warps per multiprocessor behind the planes
CASES = {
    "staged_unforced": dict(row=(128, 128), tiles=8 * 20, kw=dict(omega_bulk=1.0)),
    "staged_unforced_walls_graphs_of_two": dict(row=(192, 133), tiles=24 * 20,
                                                kw=dict(bc=("periodic", "bounceback", "bounceback"), smagorinsky_cs=0.1)),
    "staged_channel": dict(row=(192, 61), tiles=8 * 16, force="x", kw=CHANNEL),
    "staged_channel_graphs_of_two": dict(row=(256, 101), tiles=30 * 16, force="x", kw=CHANNEL),
    "staged_field": dict(row=(256, 256), tiles=60 * 16, force="field", kw=dict(smagorinsky_cs=0.1, omega_bulk=1.0)),
    "two_cells_x_force": dict(shape=(9, 20, 128), force="x", kw=dict(omega_bulk=1.0)),
    "ragged_x_force": dict(shape=(5, 33, 66), force="x", kw=dict(bc=("bounceback", "bounceback", "periodic"))),
}
PLAIN = {
    "fp64_rows_end_to_end": dict(lattice="D3Q27", shape=(6, 41, 57), storage="f64", force="x", kw=dict(tau=0.6)),
    "fp64_plane_end_to_end": dict(lattice="D2Q9", shape=(1, 70, 130), storage="f64", force="x", kw=dict(tau=0.7)),
    "f32_one_cell_x_force": dict(lattice="D2Q9", shape=(1, 41, 97), storage="f32", force="x", kw=dict(tau=0.6)),
}


def _shape(case, margin=1.25):
    if "shape" in case:
        return case["shape"]
    nx, ny = case["row"]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return (int(margin * case["tiles"] * sms / (nx // 64 * ny)) + 1, ny, nx)


def _compare(cm, lattice, shape, storage, name, case):  # noqa: F811
    nz, ny, nx = shape
    if "row" in case:
        assert (27 * 2 * nx * ny * nz > 256 << 20) == ("graphs_of_two" in name or "field" in name)
    g = torch.Generator(device="cuda").manual_seed(11)
    kw = dict(dict(tau=0.53), **case["kw"])
    a, b = (cm.Solver(lattice=lattice, nx=nx, ny=ny, nz=nz, storage=storage, **kw) for _ in range(2))
    field = None
    if case.get("force") == "field":
        field = 1e-4 * torch.randn((3,) + shape, generator=g, device="cuda", dtype=torch.float64)
    uniform = (2e-5, 0.0, 0.0) if case.get("force") == "x" else (0.0, 0.0, 0.0)
    u = 0.03 * torch.randn((3,) + shape, generator=g, device="cuda", dtype=torch.float64)
    if lattice == "D2Q9":
        u[2] = 0.0
    for s in (a, b):
        s.set_force(uniform, field)
        s.init(None, u)
    for n in (35, 34):                   # from either state buffer
        a.step(n)
        for _ in range(n):
            b.step(1)
        got, ref = a.get_state(), b.get_state()
        assert torch.isfinite(got.float() if got.dtype != torch.float64 else got).all()
        assert torch.equal(got.view(torch.uint8), ref.view(torch.uint8))
    a.close()
    b.close()


@pytest.mark.parametrize("storage", ["bf16", "f16"])
@pytest.mark.parametrize("name", list(CASES))
def test_chained_16_bit_steps_equal_single_steps_bitwise(cm, name, storage):  # noqa: F811
    _compare(cm, "D3Q27", _shape(CASES[name]), storage, name, CASES[name])


@pytest.mark.parametrize("name", list(PLAIN))
def test_chained_steps_equal_single_steps_bitwise(cm, name):  # noqa: F811
    case = PLAIN[name]
    _compare(cm, case["lattice"], case["shape"], case["storage"], name, case)
