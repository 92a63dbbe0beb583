"""The lane-group FP32 kernels (rows of 128 .. 2048 points, columns of 128 ..
512 points) at the sizes where their tiles, rounds and layer groups end:
forward and adjoint against the FP64 path over the whole field, batches bit
for bit against single calls.  Bar 2e-5 relative L2, the FP32 bar of the
other parity tests (about fifty rounding stages of 6e-8 add up to 4e-7)."""
import numpy as np
import pytest
import torch

from paper_2005_10160_gb300 import capi
from paper_2005_10160_gb300.batch import BatchRunner
from paper_2005_10160_gb300.plan import Plan, Plan3D

pytestmark = pytest.mark.gpu

TOL32 = 2e-5
MESHES = [
    # nx, ny, nz: row classes 64 .. 1024 with ragged ends, column classes 64 .. 256, layers around the rounds of 8
    (33, 33, 1), (64, 64, 8), (63, 47, 9), (65, 65, 7), (128, 128, 33), (127, 100, 16), (129, 129, 5), (256, 256, 17),
    (255, 193, 64), (257, 34, 24), (511, 66, 3), (512, 130, 65), (513, 35, 2), (777, 129, 11), (1023, 65, 4),
    (40, 257, 3), (600, 300, 5), (70, 700, 6),
]
MASKS = [capi.GRAV_GZ, capi.GRAV_GZ | capi.GRAV_GXY, 0x7F & ~capi.GRAV_GZ, 0x7F, 0x3F | capi.GRAV_GX | capi.GRAV_GY]


def worst(got, ref):
    """Largest relative L2 error over the components, with a floor of 1e-3 of the largest norm of the same kind."""
    got, ref = got.double(), ref.double()
    d = (got - ref).flatten(1).norm(dim=1)
    n = ref.flatten(1).norm(dim=1)
    return d, n


@pytest.mark.parametrize("i,size", list(enumerate(MESHES)))
def test_lane_group_kernels_match_the_fp64_path(gravlib, i, size):
    nx, ny, nz = size
    mesh = (nx, ny, nz, 20.0, 25.0, 15.0, 8.0)
    comps = MASKS[i % len(MASKS)]
    lst = capi.comp_list(comps)
    first = torch.tensor([c in (0, 7, 8) for c in lst])
    gen = torch.Generator(device="cuda").manual_seed(i)
    rho = torch.empty((3, nz, ny, nx), device="cuda").uniform_(-500, 500, generator=gen)
    # residuals of equal weight in the product: scaled by the kernels' sizes
    scale = torch.where(first, 1.0, 20.0).to("cuda")[:, None, None]
    r = torch.empty((3, len(lst), ny, nx), device="cuda").normal_(generator=gen) * scale
    with Plan(mesh, comps) as plan, Plan(mesh, comps, fp64=True) as plan64:
        d, g = plan.forward(rho[0]), plan.adjoint(r[0])
        d64, g64 = plan64.forward(rho[0].double()), plan64.adjoint(r[0].double())
        diff, norm = worst(d, d64)
        for kind in (True, False):
            sel = (first == kind).to("cuda")
            if sel.any():
                floor = 1e-3 * norm[sel].max()
                assert bool((diff[sel] <= TOL32 * torch.maximum(norm[sel], floor)).all()), (diff, norm)
        assert float((g.double() - g64).norm()) <= TOL32 * float(g64.norm())
        runner = BatchRunner(plan, 3)
        db, gb = runner.forward(rho), runner.adjoint(r)
        for k in range(3):
            assert torch.equal(db[k], plan.forward(rho[k]))
            assert torch.equal(gb[k], plan.adjoint(r[k]))


MESHES3D = [
    # Pz = 64 and 128 with the least and most layers, Py = 128 .. 1024 and 2048 (untiled inverse)
    (20, 33, 17), (33, 64, 32), (40, 100, 33), (17, 257, 64), (65, 300, 40), (24, 40, 20), (30, 700, 18), (130, 129, 63),
]


@pytest.mark.parametrize("i,size", list(enumerate(MESHES3D)))
def test_equal_dim_lane_groups_match_the_fp64_path(gravlib, i, size):
    nx, ny, nz = size
    mesh = (nx, ny, nz, 20.0, 25.0, 15.0)
    comps = MASKS[i % len(MASKS)]
    lst = capi.comp_list(comps)
    first = torch.tensor([c in (0, 7, 8) for c in lst])
    gen = torch.Generator(device="cuda").manual_seed(100 + i)
    rho = torch.empty((nz, ny, nx), device="cuda").uniform_(-500, 500, generator=gen)
    scale = torch.where(first, 1.0, 20.0).to("cuda")[:, None, None, None]
    r = torch.empty((len(lst), nz, ny, nx), device="cuda").normal_(generator=gen) * scale
    with Plan3D(mesh, comps) as plan, Plan3D(mesh, comps, fp64=True) as plan64:
        d, g = plan.forward(rho), plan.adjoint(r)
        d64, g64 = plan64.forward(rho.double()), plan64.adjoint(r.double())
    diff, norm = worst(d, d64)
    for kind in (True, False):
        sel = (first == kind).to("cuda")
        if sel.any():
            floor = 1e-3 * norm[sel].max()
            assert bool((diff[sel] <= TOL32 * torch.maximum(norm[sel], floor)).all()), (diff, norm)
    assert float((g.double() - g64).norm()) <= TOL32 * float(g64.norm())
