"""The inversion loop enqueued by the library against the same loop operation
by operation (a plan subclass takes that path): FP64 on planes whose size is
and is not a multiple of the vector width, more layers than block rows, full
and per-component weights, kept models, no steps, and a vanished gradient.
Bar 1e-10, that of the host test of the same recurrence: the two differ only
in rounding order, which CG amplifies to about 1e-12 within eight steps."""
import pytest
import torch

from paper_2005_10160_gb300 import capi
from paper_2005_10160_gb300.inversion import cgls
from paper_2005_10160_gb300.plan import Plan

pytestmark = pytest.mark.gpu


class StepwisePlan(Plan):
    """Takes the loop's own operations instead of the library's."""


@pytest.mark.parametrize("size,full,keep,iters", [((12, 10, 3), False, True, 4), ((7, 5, 4), True, True, 3),
                                                  ((1, 1, 1), False, False, 2), ((33, 2, 1300), False, False, 2),
                                                  ((64, 64, 5), True, False, 0), ((65, 31, 2), False, True, 4)])
def test_enqueued_loop_matches_the_stepwise_loop(gravlib, size, full, keep, iters):
    mesh = (*size, 20.0, 25.0, 15.0, 8.0)
    comps = capi.GRAV_GZ | capi.GRAV_GZZ
    gen = torch.Generator(device="cuda").manual_seed(sum(size))
    shape = (2, size[1], size[0])
    sigma = torch.tensor([1e-6, 1e-9], dtype=torch.float64, device="cuda")[:, None, None]
    d = torch.empty(shape, dtype=torch.float64, device="cuda").normal_(generator=gen) * sigma * 50
    w = 1.0 / sigma
    if full:
        w = w * torch.empty(shape, dtype=torch.float64, device="cuda").uniform_(0.5, 2.0, generator=gen)
    with Plan(mesh, comps, fp64=True) as a, StepwisePlan(mesh, comps, fp64=True) as b:
        lam = 1.0
        got, ref = cgls(a, d, w, lam, iters=iters, keep_models=keep), cgls(b, d, w, lam, iters=iters, keep_models=keep)
        assert len(got.objectives) == len(ref.objectives) == iters + 1
        assert all(abs(x - y) <= 1e-10 * abs(y) for x, y in zip(got.objectives, ref.objectives))
        assert float((got.m - ref.m).norm()) <= 1e-10 * float(ref.m.norm())
        assert len(got.models) == len(ref.models) == (iters if keep else 0)
        for x, y in zip(got.models, ref.models):
            assert x.shape == y.shape and float((x - y).norm()) <= 1e-10 * float(y.norm())
        zero = cgls(a, torch.zeros_like(d), w, lam, iters=2)
        assert zero.objectives == [0.0, 0.0, 0.0] and not bool(zero.m.any())
