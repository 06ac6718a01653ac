"""Ragged rows of even length pair adjacent cells, or (x, x + nx/2) where a buffer is not aligned to two
entries: every cell goes through the same lane arithmetic either way, so the bits must agree."""
import pytest
import torch

from paper_1202_6074_gb300 import slab as SL
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


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("nx", [66, 67])
def test_block_sizes_agree_bitwise(cm, nx, storage):  # noqa: F811
    """A grid whose blocks of 128 threads fill the multiprocessors more than once, against four slabs
    of it, which run blocks of one warp."""
    ny, sms = 32, torch.cuda.get_device_properties(0).multi_processor_count
    planes = (nx + 1) // 2 * ny // 128 + 1
    nz = 7 * sms // planes + 2                 # up to six blocks a multiprocessor are one wave
    g = torch.Generator(device="cuda").manual_seed(6)
    u = 0.03 * torch.randn((3, nz, ny, nx), generator=g, device="cuda", dtype=torch.float64)
    kw = dict(lattice="D3Q27", nx=nx, ny=ny, storage=storage, tau=0.53)
    whole = cm.Solver(nz=nz, **kw)
    whole.init(None, u)
    parts = 4
    slabs = []
    for r in range(parts):
        s, z0 = SL.cuda_slab(cm, nz, r, parts, **kw)
        s.init(None, u[:, z0:z0 + s.shape[0]].contiguous())
        slabs.append(s)
    SL.SlabRun(slabs, SL.LocalExchange(slabs)).step(3)
    whole.step(3)
    assert whole.step_path == slabs[0].step_path == "ragged"
    own = torch.cat([s.get_state()[:, 1:-1] for s in slabs], dim=1)
    assert torch.equal(own.view(torch.uint8), whole.get_state().view(torch.uint8))
    for s in slabs + [whole]:
        s.close()
