"""Ragged rows of even length pair adjacent cells, or (x, x + nx/2) where a buffer is not aligned to two
entries: every cell goes through the same lane arithmetic either way, so the bits must agree."""
import pytest
import torch

from test_gpu_parity import cm  # noqa: F401

pytestmark = pytest.mark.gpu

MOVING = [[[0, 0.01, 0], [0, 0, 0.02]], [[0.03, 0, 0], [0, 0, -0.01]], [[0.01, 0.01, 0], [-0.02, 0, 0]]]
CASES = {
    "periodic": dict(shape=(3, 34, 62), kw=dict()),
    "periodic_66_les": dict(shape=(3, 32, 66), kw=dict(smagorinsky_cs=0.1)),
    "short_rows": dict(shape=(3, 260, 8), kw=dict()),
    "cavity": dict(shape=(4, 16, 130), kw=dict(bc=("bounceback",) * 3, wall_velocity=MOVING)),
    "x_walls_128": dict(shape=(3, 16, 128), kw=dict(bc=("bounceback", "periodic", "periodic"), wall_velocity=MOVING)),
    "factorized": dict(shape=(3, 42, 50), kw=dict(attractor="factorized")),
    "reduced": dict(shape=(3, 42, 50), kw=dict(reduced_compressibility=True, rho0=1.02)),
    "x_force": dict(shape=(3, 34, 62), force=(2e-5, 0.0, 0.0), kw=dict()),
    "force_rates": dict(shape=(3, 34, 62), force=(2e-5, 1e-5, -1e-5), kw=dict(omega_3=1.2)),
    "slab": dict(shape=(3, 34, 62), kw=dict(bc=("periodic", "periodic", "halo"))),
}


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("name", list(CASES))
def test_pairings_agree_bitwise(cm, name, storage):  # noqa: F811
    case = CASES[name]
    nz, ny, nx = case["shape"]
    s = cm.Solver(lattice="D3Q27", nx=nx, ny=ny, nz=nz, storage=storage, tau=0.55, **case["kw"])
    s.set_force(case.get("force", (0.0, 0.0, 0.0)))
    g = torch.Generator(device="cuda").manual_seed(5)
    n = s.new_state().numel()
    s0 = (0.05 * torch.randn(n, generator=g, device="cuda")).to(s.state_dtype)
    outs = []
    for off in (0, 1):
        a = torch.zeros(n + 1, dtype=s0.dtype, device="cuda")
        b = torch.zeros_like(a)
        a[off:off + n].copy_(s0)
        s.step_buffers(a[off:off + n], b[off:off + n])
        out = b[off:off + n].reshape(s.state_shape)
        outs.append((out[:, 1:-1] if s.slab else out).contiguous())
    assert torch.isfinite(outs[0].float()).all()
    assert torch.equal(outs[0].view(torch.uint8), outs[1].view(torch.uint8))
    s.close()
