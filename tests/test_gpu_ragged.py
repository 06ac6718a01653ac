"""GPU parity of the two-cells-per-thread step on rows of any length and with walls across x.

On planes of at least 2048 cells the automatic choice updates two cells per thread whatever the row
length: even rows pair adjacent cells, odd rows cells half a row apart with the last thread's second
cell left out, and the rows of a plane are laid end to end over the blocks. One step is held to the
bounds of test_gpu_parity.py (derived there) at row lengths around the edges of a warp's 64 cells,
and against the one-cell kernel.
"""
import pytest
import torch

import helpers as H
from paper_1202_6074_gb300 import slab as SL
from test_gpu_parity import ONE_STEP_ATOL, ONE_STEP_RTOL, _inputs, _pair, cm  # noqa: F401

pytestmark = pytest.mark.gpu

MOVING = [[[0, 0.01, 0], [0, 0, 0.02]], [[0.03, 0, 0], [0, 0, -0.01]], [[0.01, 0.01, 0], [-0.02, 0, 0]]]
CASES = {
    "periodic_62": dict(shape=(3, 34, 62), flow="tgv_unforced", kw=dict(tau=0.6, omega_bulk=1.0)),
    "periodic_65": dict(shape=(3, 33, 65), flow="tgv_unforced", kw=dict(tau=0.6, omega_bulk=1.0)),
    "field_66_les": dict(shape=(3, 32, 66), flow="tgv", kw=dict(tau=0.52, smagorinsky_cs=0.15)),
    "field_63_rates": dict(shape=(3, 33, 63), flow="tgv", kw=dict(tau=0.62, omega_3=1.2, omega_4=0.9)),
    "short_rows": dict(shape=(3, 230, 9), flow="tgv", kw=dict(tau=0.6)),
    "channel_190_vd": dict(shape=(4, 12, 190), flow="channel",
                           kw=dict(tau=0.52, smagorinsky_cs=0.15, van_driest=(26.0, 8.0), wall_velocity=MOVING,
                                   bc=("periodic", "bounceback", "periodic"))),
    "cavity_130": dict(shape=(4, 16, 130), flow="tgv_unforced",
                       kw=dict(tau=0.6, omega_bulk=1.0, bc=("bounceback",) * 3, wall_velocity=MOVING)),
    "cavity_47_field": dict(shape=(4, 45, 47), flow="tgv",
                            kw=dict(tau=0.6, bc=("bounceback",) * 3, wall_velocity=MOVING)),
    "x_walls_128": dict(shape=(3, 16, 128), flow="tgv",
                        kw=dict(tau=0.6, bc=("bounceback", "periodic", "periodic"), wall_velocity=MOVING)),
    "factorized_50": dict(shape=(3, 42, 50), flow="tgv", kw=dict(tau=0.58, attractor="factorized")),
    "reduced_51_z_walls": dict(shape=(3, 42, 51), flow="tgv_unforced",
                               kw=dict(tau=0.6, reduced_compressibility=True, rho0=1.02,
                                       bc=("bounceback", "periodic", "bounceback"))),
}


def _one_step(cm, case, storage, uniform=(0.0, 0.0, 0.0), **kw):  # noqa: F811
    rho, u, F = _inputs(dict(case, lattice="D3Q27"))
    s, o = _pair(cm, "D3Q27", case["shape"], storage, rho, u, F, uniform=uniform, **case["kw"], **kw)
    o.set_state(H.decode(s.get_state(), "D3Q27"))
    s.step(1)
    o.step(1)
    w = H.lattice("D3Q27").w.view(-1, 1, 1, 1)
    got, ref = H.decode(s.get_state(), "D3Q27") / w - 1, o.s / w - 1
    s.close()
    return got, ref


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("name", list(CASES))
def test_one_step_elementwise(cm, name, storage):  # noqa: F811
    got, ref = _one_step(cm, CASES[name], storage)
    err = (got - ref).abs()
    assert bool((err <= ONE_STEP_ATOL[storage] + ONE_STEP_RTOL[storage] * ref.abs()).all()), f"{err.max().item():.3e}"
    # the one-cell kernel on the same state: both are within the one-step bound of the oracle
    one, _ = _one_step(cm, CASES[name], storage, kernel="direct")
    assert bool(((got - one).abs() <= 2 * (ONE_STEP_ATOL[storage] + ONE_STEP_RTOL[storage] * ref.abs())).all())


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("nx", [62, 63, 126])
def test_uniform_force_along_x(cm, nx, storage):  # noqa: F811
    case = dict(shape=(3, 34, nx), flow="tgv_unforced", kw=dict(tau=0.53, omega_bulk=1.0, smagorinsky_cs=0.12,
                                                                bc=("bounceback", "periodic", "periodic")))
    got, ref = _one_step(cm, case, storage, uniform=(3e-5, 0.0, 0.0))
    err = (got - ref).abs()
    assert bool((err <= ONE_STEP_ATOL[storage] + ONE_STEP_RTOL[storage] * ref.abs()).all()), f"{err.max().item():.3e}"


@pytest.mark.parametrize("storage,nx", [("f32", 66), ("f32", 67), ("bf16", 66)])
def test_slabs_equal_the_whole_grid_bitwise(cm, storage, nx):  # noqa: F811
    ny, nz = 32, 9
    rho, u, _ = _inputs(dict(shape=(nz, ny, nx), lattice="D3Q27", flow="tgv_unforced"))
    kw = dict(lattice="D3Q27", nx=nx, ny=ny, storage=storage, tau=0.53, omega_bulk=1.0)
    ref = cm.Solver(nz=nz, **kw)
    ref.init(torch.tensor(rho, device="cuda"), torch.tensor(u, device="cuda"))
    slabs = []
    for r in range(2):
        s, z0 = SL.cuda_slab(cm, nz, r, 2, **kw)
        sl = slice(z0, z0 + s.shape[0])
        s.init(torch.tensor(rho[sl], device="cuda"), torch.tensor(u[:, sl], device="cuda"))
        slabs.append(s)
    SL.SlabRun(slabs, SL.LocalExchange(slabs)).step(4)
    ref.step(4)
    own = torch.cat([s.get_state()[:, 1:-1] for s in slabs], dim=1)
    assert torch.equal(own.view(torch.uint8), ref.get_state().view(torch.uint8))
    for s in slabs + [ref]:
        s.close()
