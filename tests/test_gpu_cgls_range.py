"""The inversion loop enqueued by the library, against the loop operation by
operation (a plan subclass takes that path): FP32 sums of squares, steps that
have no length, kept models, workspace.

Bar 1e-3: the two differ in the rounding of FP32 vector updates, 2^-24, which CG
amplifies about 1e4 times within eight steps (the FP64 loops differ by 1e-12)."""
import pytest
import torch

from paper_2005_10160_gb300 import capi
from paper_2005_10160_gb300.inversion import cgls
from paper_2005_10160_gb300.plan import Plan

pytestmark = pytest.mark.gpu

BAR = 1e-3


class StepwisePlan(Plan):
    """Takes the loop's own operations instead of the library's."""


def assert_same(got, ref):
    assert len(got.objectives) == len(ref.objectives)
    assert all(abs(x - y) <= BAR * abs(y) for x, y in zip(got.objectives, ref.objectives)), (got.objectives, ref.objectives)
    diff, norm = float((got.m.double() - ref.m.double()).norm()), float(ref.m.double().norm())
    assert 0 < norm < float("inf") and diff <= BAR * norm, (diff, norm)


def test_sums_past_the_fp32_range(gravlib):
    """Every square is finite in FP32, a thread's sum of four is not.  Stations far above an 8 x 8 x 1 mesh: the kernel
    is nearly the same everywhere, so with w = 1 / (sum of a row) every vector of the loop is about 1.5e19."""
    mesh = (8, 8, 1, 20.0, 25.0, 15.0, 2000.0)
    with Plan(mesh, capi.GRAV_GZ) as a, StepwisePlan(mesh, capi.GRAV_GZ) as b:
        row = float(a.forward(torch.ones(1, 8, 8, device="cuda")).mean())
        w = torch.full((1, 1, 1), 1.0 / row, device="cuda")
        d = torch.full((1, 8, 8), 1.5e19 * row, device="cuda")
        assert_same(cgls(a, d, w, 1.0, iters=1), cgls(b, d, w, 1.0, iters=1))


# planes of both vector widths; several values a thread over more layers than block rows (33 x 2 x 1300) and within
# a plane too (131 x 97 x 1217)
@pytest.mark.parametrize("size", [(12, 10, 3), (7, 5, 4), (33, 2, 1300), (131, 97, 1217)])
def test_fp32_loop_matches_the_stepwise_loop(gravlib, size):
    mesh = (*size, 20.0, 25.0, 15.0, 8.0)
    comps = capi.GRAV_GZ | capi.GRAV_GZZ
    gen = torch.Generator(device="cuda").manual_seed(sum(size))
    sigma = torch.tensor([1e-6, 1e-9], device="cuda")[:, None, None]
    d = torch.empty((2, size[1], size[0]), device="cuda").normal_(generator=gen) * sigma * 50
    with Plan(mesh, comps) as a, StepwisePlan(mesh, comps) as b:
        assert_same(cgls(a, d, 1.0 / sigma, 1.0, iters=3), cgls(b, d, 1.0 / sigma, 1.0, iters=3))


# (q, q) below FP32's range with data in SI units and no weights; a product of scale 1e-20, whose step is 1e40
@pytest.mark.parametrize("scale,data,error", [(None, 1e-9, ZeroDivisionError), (1e-20, 1e19, RuntimeError)])
def test_a_step_without_a_length_is_an_error(gravlib, scale, data, error):
    mesh = (8, 8, 1, 20.0, 25.0, 15.0, 2000.0 if scale else 8.0)
    comps = capi.GRAV_GZ if scale else capi.GRAV_GZZ
    for cls in (Plan, StepwisePlan):
        with cls(mesh, comps) as plan:
            w = scale / float(plan.forward(torch.ones(1, 8, 8, device="cuda")).mean()) if scale else 1.0
            weights = torch.full((1, 1, 1), w, device="cuda")
            with pytest.raises(error):
                cgls(plan, torch.full((1, 8, 8), data / w, device="cuda"), weights, 0.0, iters=2)


def test_kept_models_have_memory_of_their_own(gravlib):
    """Keeping one model must not keep the others alive."""
    mesh = (12, 10, 3, 20.0, 25.0, 15.0, 8.0)
    gen = torch.Generator(device="cuda").manual_seed(1)
    d = torch.empty((1, 10, 12), device="cuda").normal_(generator=gen) * 5e-5
    with Plan(mesh, capi.GRAV_GZ) as plan:
        res = cgls(plan, d, torch.full((1, 1, 1), 1e6, device="cuda"), 1.0, iters=3, keep_models=True)
    stores = [m.untyped_storage() for m in (*res.models, res.m)]
    assert len({s.data_ptr() for s in stores}) == 4
    assert all(s.nbytes() == m.numel() * m.element_size() for s, m in zip(stores, (*res.models, res.m)))
    assert torch.equal(res.models[-1], res.m)


def test_workspace_of_a_long_loop(gravlib):
    """A step adds three dot products of 16 bytes to the workspace."""
    with Plan((12, 10, 3, 20.0, 25.0, 15.0, 8.0), capi.GRAV_GZ) as plan:
        assert capi.grav_cgls_work_bytes(plan.handle, 1001) - capi.grav_cgls_work_bytes(plan.handle, 1) == 1000 * 48
