"""Plan creation: kernel generation over several tiles and runs of layers, and
spectra built in FP32 pairs, at cell sizes far from one metre.  Bars: a
kernel value is a sum of eight corner terms that largely cancel, so it is good
to a few roundings of the terms, not of itself: eight units of 2^-53 of their
magnitudes for the terms and the sum, twice that for the difference of two such
values, 2e-15; FP32 fields 2e-5 and FP64 fields 1e-10 relative L2 per component
as in the parity tests."""
import numpy as np
import pytest
import torch

from paper_2005_10160_gb300 import capi
from paper_2005_10160_gb300.plan import Plan, kernel_values

pytestmark = pytest.mark.gpu

NINE = [0x7F, 0x3F | capi.GRAV_GX | capi.GRAV_GY]


def corner_magnitudes(mesh, u, v, n):
    """Sum over the eight corners of |F_c| (gravitational constant included) per
    component gz, gxx, gxy, gxz, gyy, gyz, gzz, gx, gy: what the kernel value
    is the cancelling sum of."""
    dx, dy, dz, h = mesh[3:]
    x = (0.5 - u - np.arange(2)[:, None, None]) * dx
    y = (0.5 - v - np.arange(2)[None, :, None]) * dy
    z = -h - (n + np.arange(2)[None, None, :]) * dz
    r = np.sqrt(x * x + y * y + z * z)
    ax, ay, az = np.arcsinh(x / np.hypot(y, z)), np.arcsinh(y / np.hypot(x, z)), np.arcsinh(z / np.hypot(x, y))
    tx, ty, tz = np.arctan(y * z / (x * r)), np.arctan(x * z / (y * r)), np.arctan(x * y / (z * r))
    F = [abs(x * ay) + abs(y * ax) + abs(z * tz), tx, az, ay, ty, ax, tz, abs(y * az) + abs(z * ay) + abs(x * tx),
         abs(z * ax) + abs(x * az) + abs(y * ty)]
    return np.array([6.672e-11 * np.abs(f).sum() for f in F])


@pytest.mark.parametrize("mesh", [(33, 17, 16, 10.0, 25.0, 20.0, 2.0), (66, 3, 40, 1e-3, 4e-3, 2e-3, 1e-3),
                                  (2, 49, 9, 5e4, 1e3, 2e2, 30.0)])
def test_kernel_values_across_tiles_and_runs(gravlib, orc, mesh):
    nx, ny, nz, dx, dy, dz, h = mesh
    rng = np.random.default_rng(nx)
    for comps in NINE:
        lst = capi.comp_list(comps)
        K = kernel_values(mesh, comps).cpu().numpy()
        edges = [(u, v, n) for u in (-nx + 1, 0, min(nx - 1, 32)) for v in (-ny + 1, 0, min(ny - 1, 16)) for n in (0, nz - 1)]
        some = [(int(rng.integers(-nx + 1, nx)), int(rng.integers(-ny + 1, ny)), int(rng.integers(0, nz))) for _ in range(150)]
        for u, v, n in edges + some:
            box = ((u - 0.5) * dx, (u + 0.5) * dx, (v - 0.5) * dy, (v + 0.5) * dy, n * dz, (n + 1) * dz)
            ref = orc.prism((0.0, 0.0, -h), box)[lst]
            got = K[:, n, v + ny - 1, u + nx - 1]
            bar = 2e-15 * corner_magnitudes(mesh, u, v, n)[lst]
            assert np.all(np.abs(got - ref) <= bar), (u, v, n, got, ref, bar)


@pytest.mark.parametrize("cell", [(1e-3, 2e-3, 1e-3, 1e-3), (5e4, 1e4, 2e4, 1e3), (1.0, 300.0, 20.0, 0.5)])
@pytest.mark.parametrize("comps", NINE)
def test_spectra_at_any_cell_size(gravlib, orc, cell, comps):
    mesh = (19, 12, 7, *cell)
    rng = np.random.default_rng(5)
    rho = rng.uniform(-500, 500, (7, 12, 19)).astype(np.float32)
    ref = orc.forward(mesh, comps, rho.astype(np.float64)).reshape(len(capi.comp_list(comps)), -1)
    norm = np.linalg.norm(ref, axis=1)
    for fp64, tol in ((False, 2e-5), (True, 1e-10)):
        with Plan(mesh, comps, fp64=fp64) as plan:
            d = plan.forward(torch.as_tensor(rho, dtype=plan.dtype, device="cuda")).cpu().double().numpy()
        err = np.linalg.norm(d.reshape(ref.shape) - ref, axis=1)
        assert np.all(err <= tol * norm), (fp64, err / norm)
