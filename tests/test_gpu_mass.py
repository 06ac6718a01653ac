"""FP32 runs conserve mass up to unbiased rounding.

A step rounds the 27 (9) populations of a cell, of size up to 0.1, so a cell's mass is off by about
s = 1.5e-9 (ulp(0.1) / sqrt(12) = 2.2e-9 a population, weighted). Over N cells of which 16 at a time
repeat each other by symmetry and T steps, the mean density then walks by s sqrt(16 T / N). Six times
that is the bound; a bias of 1e-11 a cell and step, which grows with T, is beyond it on these grids.
"""
import math

import pytest
import torch

import helpers as H
from test_gpu_parity import cm  # noqa: F401

pytestmark = pytest.mark.gpu

S = 1.5e-9


def _mean_density(s, lattice):
    w = H.lattice(lattice).w.double().cuda()
    return float((s.get_state().double().flatten(1).mean(1) * w).sum())


def _flow(name, shape):
    nz, ny, nx = shape
    z, y, x = (2 * math.pi * torch.arange(n, dtype=torch.float64, device="cuda") / n for n in shape)
    z, y, x = z[:, None, None], y[None, :, None], x[None, None, :]
    u = torch.zeros((3,) + shape, dtype=torch.float64, device="cuda")
    rho = 1 + 1e-3 * torch.cos(x) * torch.sin(2 * y) + 0 * z
    if name == "taylor_green":
        u[0] = 0.04 * torch.sin(x) * torch.cos(y) * torch.cos(z)
        u[1] = -0.04 * torch.cos(x) * torch.sin(y) * torch.cos(z)
    else:                    # a strong shear along one axis beside a weak flow along the others
        strong, weak = 0.04 * torch.sin(y) + 0 * x + 0 * z, 2e-5 * torch.sin(2 * x + y) + 0 * z
        axis = {"shear_x": 0, "shear_z": 2}[name]
        u[:] = weak
        u[axis] = strong
        if nz == 1:
            u[2] = 0.0
    return rho, u


@pytest.mark.parametrize("lattice,shape,flow,steps,force", [
    ("D3Q27", (128, 128, 128), "taylor_green", 60, 0.0),
    ("D3Q27", (128, 128, 128), "taylor_green", 60, 1e-5),
    ("D3Q27", (96, 111, 130), "shear_x", 200, 0.0),
    ("D3Q27", (96, 128, 128), "shear_z", 200, 1e-6),
    ("D2Q9", (1, 1024, 1024), "shear_x", 2000, 0.0),
    ("D2Q9", (1, 1024, 1024), "shear_x", 2000, 1e-7),
])
def test_mass_of_an_fp32_run(cm, lattice, shape, flow, steps, force):  # noqa: F811
    nz, ny, nx = shape
    rho, u = _flow(flow, shape)
    s = cm.Solver(lattice=lattice, nx=nx, ny=ny, nz=nz, storage="f32", tau=0.505)
    s.set_force((force, 0.0, 0.0))
    s.init(rho, u)
    before = _mean_density(s, lattice)
    s.step(steps)
    drift = _mean_density(s, lattice) - before
    s.close()
    assert abs(drift) <= 6 * S * math.sqrt(16 * steps / (nx * ny * nz)), f"{drift:.2e}"
