"""The 16-bit step with its pull staged in shared memory against the two-cell kernel.

Large grids at 16-bit storage take the staged step where the source buffer is aligned to 16 bytes, and the
two-cell kernel otherwise (buffers offset by two entries here). Both run the same lane arithmetic on
the same populations: the bits must agree, for every collision variant the staged step has, with
walls (rows next to one are pulled directly), on slabs and with force fields, on grids just above
the line where a warp gets a partial last run of tiles.
"""
import pytest
import torch

from test_gpu_parity import cm  # noqa: F401

pytestmark = pytest.mark.gpu

CHANNEL = dict(bc=("periodic", "bounceback", "periodic"), smagorinsky_cs=0.1, van_driest=(26.0, 0.3))
LID = [[[0, 0, 0], [0, 0, 0]], [[0.03, 0, 0], [0, 0, -0.01]], [[0.01, 0.01, 0], [-0.02, 0, 0]]]
CASES = {
    "unforced": dict(shape=(103, 128, 128), kw=dict(omega_bulk=1.0)),
    "unforced_one_tile_rows": dict(shape=(131, 199, 64), kw=dict(omega_bulk=1.0)),
    "unforced_walls_les": dict(shape=(67, 133, 192), kw=dict(bc=("periodic", "bounceback", "bounceback"), wall_velocity=LID,
                                                            smagorinsky_cs=0.1)),
    "channel": dict(shape=(97, 101, 192), force="x", kw=CHANNEL),
    "uniform_x_periodic": dict(shape=(103, 128, 128), force="x", kw=dict(omega_bulk=1.0)),
    "field_les": dict(shape=(148, 256, 256), force="field", kw=dict(smagorinsky_cs=0.1, omega_bulk=1.0)),
    "field_walls": dict(shape=(193, 253, 192), force="field", kw=dict(bc=("periodic", "bounceback", "periodic"))),
    "slab": dict(shape=(103, 128, 128), kw=dict(bc=("periodic", "periodic", "halo"))),
}


@pytest.mark.parametrize("storage", ["bf16", "f16"])
@pytest.mark.parametrize("name", list(CASES))
def test_staged_step_equals_the_two_cell_kernel_bitwise(cm, name, storage):  # noqa: F811
    case = CASES[name]
    nz, ny, nx = case["shape"]
    g = torch.Generator(device="cuda").manual_seed(7)
    s = cm.Solver(lattice="D3Q27", nx=nx, ny=ny, nz=nz, storage=storage, tau=0.53, **case["kw"])
    if case.get("force") == "x":
        s.set_force((2e-5, 0.0, 0.0))
    elif case.get("force") == "field":
        s.set_force((0.0, 0.0, 0.0), 1e-4 * torch.randn((3, nz, ny, nx), generator=g, device="cuda", dtype=torch.float64))
    n = s.new_state().numel()
    s0 = (0.05 * torch.randn(n, generator=g, device="cuda")).to(s.state_dtype)
    outs = []
    for off in (0, 2):
        a = torch.zeros(n + 2, dtype=s0.dtype, device="cuda")
        b = torch.zeros_like(a)
        a[off:off + n].copy_(s0)
        s.step_buffers(a[off:off + n], b[off:off + n])
        outs.append(b[off:off + n].reshape(s.state_shape)[:, 1:-1] if s.slab else b[off:off + n])
    assert torch.isfinite(outs[0].float()).all()
    assert torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))
    s.close()
