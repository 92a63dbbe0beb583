"""The layer sums of the FP32 forward columns at the edges of their blocks.

1024-point columns (513 <= ny <= 1024) keep the compensated sums of blocks of 32
layers in tensor memory, 16 columns a component (eight components use all of
it): one block and less, the edges, and several blocks, with one, six, seven
and eight components.  64-point columns (33 <= ny <= 64) give eight layers a
round to each of up to eight layer groups of a CTA: idle groups, a second and a
third round, and the sum over the groups with the corrections in registers and in
shared memory.

Forward against the FP64 path over the whole field, 2e-5 relative L2 as in the
other parity tests; batches bit for bit against single calls."""
import pytest
import torch

from paper_2005_10160_gb300 import capi
from paper_2005_10160_gb300.batch import BatchRunner
from paper_2005_10160_gb300.plan import Plan

pytestmark = pytest.mark.gpu

TOL32 = 2e-5
MASKS = [capi.GRAV_GZ, 0x3F, 0x7F, 0x7F | capi.GRAV_GX]
SIZES = [(3, 600, nz) for nz in (31, 32, 33, 64, 65, 97)] + [(33, 33, 33), (40, 50, 64), (35, 64, 65), (34, 40, 130)]


@pytest.mark.parametrize("comps", MASKS)
@pytest.mark.parametrize("size", SIZES)
def test_layer_sums_match_the_fp64_path(gravlib, size, comps):
    nx, ny, nz = size
    mesh = (nx, ny, nz, 20.0, 25.0, 15.0, 8.0)
    gen = torch.Generator(device="cuda").manual_seed(nz)
    rho = torch.empty((2, nz, ny, nx), device="cuda").uniform_(-500, 500, generator=gen)
    with Plan(mesh, comps) as plan, Plan(mesh, comps, fp64=True) as plan64:
        d = torch.stack([plan.forward(rho[0]), plan.forward(rho[1])])
        assert torch.equal(BatchRunner(plan, 2).forward(rho), d)
        for k in range(2):
            ref = plan64.forward(rho[k].double()).flatten(1)
            err = (d[k].double().flatten(1) - ref).norm(dim=1)
            assert bool((err <= TOL32 * ref.norm(dim=1)).all()), err / ref.norm(dim=1)
