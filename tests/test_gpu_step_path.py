"""Which kernel a step runs (cmlbm_step_path): the automatic choice on both sides of its lines, for single
steps, captured graphs, buffers passed in, and split steps. The staged step's lines go with the device's
multiprocessors; the grids have a quarter more, or a quarter less, than the tiles they ask for.
"""
import pytest
import torch

from test_gpu_parity import cm  # noqa: F401

pytestmark = pytest.mark.gpu

WALLS = ("bounceback", "bounceback", "bounceback")
CASES = [
    # lattice, (nz, ny, nx), storage, kw, force, path
    ("D2Q9", (1, 40, 64), "f32", {}, None, "one_cell"),
    ("D3Q27", (4, 40, 64), "f64", {}, None, "one_cell"),
    ("D3Q27", (4, 40, 64), "f32", {}, None, "two_cells"),
    ("D3Q27", (4, 40, 64), "bf16", {}, "x", "two_cells"),
    ("D3Q27", (4, 2, 64), "f16", dict(omega_3=1.2), "field", "two_cells"),
    ("D3Q27", (4, 40, 64), "f32", dict(kernel="direct"), None, "one_cell"),
    ("D3Q27", (4, 33, 62), "f32", {}, None, "one_cell"),              # 2046 cells a plane
    ("D3Q27", (4, 64, 32), "f32", {}, None, "ragged"),                # 2048
    ("D3Q27", (4, 33, 63), "bf16", {}, "field", "ragged"),
    ("D3Q27", (4, 32, 64), "f16", dict(bc=WALLS), None, "ragged"),    # walls across x
    ("D3Q27", (4, 31, 64), "f16", dict(bc=WALLS), None, "one_cell"),
    ("D3Q27", (4, 300, 7), "f32", {}, None, "one_cell"),              # rows below 8
    ("D3Q27", (4, 260, 8), "f32", dict(attractor="factorized"), None, "ragged"),
    ("D3Q27", (4, 33, 63), "f32", dict(kernel="direct"), None, "one_cell"),
    ("D3Q27", (16, 4, 64), "f32", dict(kernel="pair_two_steps"), None, "two_steps"),
    ("D3Q27", (4, 4, 128), "f32", dict(kernel="tma"), None, "tma"),
]


def _solver(cm, lattice, shape, storage, kw, force):  # noqa: F811
    nz, ny, nx = shape
    s = cm.Solver(lattice=lattice, nx=nx, ny=ny, nz=nz, storage=storage, tau=0.6, **kw)
    field = torch.full((3,) + shape, 1e-6, device="cuda", dtype=torch.float64) if force == "field" else None
    s.set_force((1e-6, 0.0, 0.0) if force == "x" else (0.0, 0.0, 0.0), field)
    s.init()
    return s


@pytest.mark.parametrize("case", CASES)
def test_path_of_small_grids(cm, case):  # noqa: F811
    s = _solver(cm, *case[:5])
    assert s.step_path is None
    s.step(2 if case[5] == "two_steps" else 1)
    assert s.step_path == case[5]
    s.step(40)
    assert s.step_path == case[5]
    s.close()


@pytest.mark.parametrize("force,tiles,kw", [
    (None, 8 * 20, dict(omega_bulk=1.0)),
    (None, 8 * 20, dict(bc=("periodic", "bounceback", "bounceback"), smagorinsky_cs=0.1)),
    ("x", 7 * 16, dict(bc=("periodic", "bounceback", "periodic"))),
    ("field", 60 * 16, dict(smagorinsky_cs=0.1)),
])
@pytest.mark.parametrize("storage", ["bf16", "f16"])
def test_path_of_the_staged_step(cm, storage, force, tiles, kw):  # noqa: F811
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for margin, path in ((1.25, "staged"), (0.75, "two_cells")):
        s = _solver(cm, "D3Q27", (int(margin * tiles * sms / (2 * 128)) + 1, 128, 128), storage, kw, force)
        s.step(3)                                    # a graph of two and a single step
        assert s.step_path == path
        a = torch.zeros(s.new_state().numel() + 2, dtype=s.state_dtype, device="cuda")
        b = torch.zeros_like(a)
        s.step_buffers(a[:-2], b[:-2])
        assert s.step_path == path
        s.step_buffers(a[2:], b[2:])                 # not aligned to the staged copies
        assert s.step_path == "two_cells"
        s.step_split()
        assert s.step_path in (path, "two_cells")    # by the planes of its last part
        s.close()


def test_null_handle(cm):  # noqa: F811
    assert cm.load().cmlbm_step_path(None) == cm.ERR_INVALID
