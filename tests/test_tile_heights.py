"""Stencil tiles, whole-realization tiles and row groups over the grid sizes: the
true residual of batched solves, and a lone solve against the batch bit for bit."""
import pytest
import torch

from paper_1903_12227_gb300 import rve, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [rve.FP64, rve.MIXED])
@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("n,count", [(32, 300), (64, 300), (128, 40), (256, 9), (512, 3), (1024, 2)])
def test_lone_and_batched_solves(n, count, scheme, precision):
    ds = workloads.batch(n // 8, 8, 10.0, 4, count)
    tol = 1e-10
    opts = rve.make_opts(scheme=scheme, precision=precision, tol=tol)
    mask = rve.gen_field(ds)
    u, info = rve.solve(ds, mask=mask, opts=opts)
    assert all(i["status"] == rve.RVE_OK for i in rve.info_to_dicts(info, count))
    f = rve.rhs(ds, mask=mask)
    r = (f - rve.apply_stiffness(ds, u, mask=mask, scheme=scheme)).view(count, n * n, 2)
    # the solver's own residual met tol; this one differs by FP64 rounding of
    # A u (8 eps |A| |u| per node, |A| <= 16 a_max) and, mixed, of the final u
    floor = 64 * 2.0 ** -53 * 160.0 * u.view(count, -1, 2).abs().amax(1) * n
    assert bool((r.norm(dim=1) <= tol * f.view(count, n * n, 2).norm(dim=1) + floor).all())
    words = n * n // 32
    for k in (0, count - 1):
        m = mask[k * words:(k + 1) * words]
        v, _ = rve.solve(ds[k:k + 1], mask=m, opts=opts)
        assert torch.equal(v, u[k * n * n:(k + 1) * n * n])


@pytest.mark.parametrize("precision", [rve.FP64, rve.MIXED])
@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("n", [512, 1024, 2048])
def test_explicit_cells_equal_mask(n, scheme, precision):
    """The stencil passes (one launch, and two from 1024 on) on explicit cells and on the mask."""
    ds = workloads.batch(n // 8, 8, 10.0, 6, 1)
    opts = rve.make_opts(scheme=scheme, precision=precision, tol=1e-10)
    mask = rve.gen_field(ds)
    coef = rve.coef_from_mask(ds, mask)
    u, info = rve.solve(ds, mask=mask, opts=opts)
    v, info2 = rve.solve(ds, coef=coef, opts=opts)
    assert all(i["status"] == rve.RVE_OK for t in (info, info2) for i in rve.info_to_dicts(t, 1))
    if precision == rve.MIXED:   # the same arithmetic on the same values
        assert torch.equal(u, v)
    A = rve.a_hom(ds, u, mask=mask, scheme=scheme)
    B = rve.a_hom(ds, v, coef=coef, scheme=scheme)
    # two answers to one tolerance: the energies differ by its square times the
    # condition number, far below 1e-10 of them
    assert float((A - B).abs().max()) <= 1e-10 * float(A.abs().max())
