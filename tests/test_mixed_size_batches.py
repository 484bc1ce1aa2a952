"""A realization's results are the same bits alone and in a batch of other sizes:
every sum is cut into tiles by the grid's own size."""
import pytest
import torch

from paper_1903_12227_gb300 import rve, workloads

pytestmark = pytest.mark.gpu

SIZES = (64, 2048, 32, 512, 1024, 128, 256, 32)


def _batch(sizes, contrast=10.0):
    ds = [workloads.realization(n // 8, 8, contrast, 9, k) for k, n in enumerate(sizes)]
    mask = rve.gen_field(ds)
    node = [0]
    for n in sizes:
        node.append(node[-1] + n * n)
    return ds, mask, node


@pytest.mark.parametrize("path", [rve.PATH_FUSED, rve.PATH_PERSISTENT])
@pytest.mark.parametrize("precision", [rve.FP64, rve.MIXED])
@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
def test_solve(scheme, precision, path):
    ds, mask, node = _batch(SIZES)
    opts = rve.make_opts(scheme=scheme, precision=precision, path=path, tol=1e-9)
    u, info = rve.solve(ds, mask=mask, opts=opts)
    infos = rve.info_to_dicts(info, len(ds))
    for k in range(len(ds)):
        v, one = rve.solve(ds[k:k + 1], mask=mask[node[k] // 32:node[k + 1] // 32], opts=opts)
        assert rve.info_to_dicts(one, 1)[0] == infos[k]
        assert infos[k]["status"] == rve.RVE_OK
        assert torch.equal(v, u[node[k]:node[k + 1]]), SIZES[k]


@pytest.mark.parametrize("precision", [rve.FP64, rve.MIXED])
def test_captured_plan(precision):
    ds, _, _ = _batch(SIZES)
    opts = rve.make_opts(precision=precision, path=rve.PATH_FUSED, tol=1e-9)
    A, info = rve.Plan(ds, opts).execute()
    infos = rve.info_to_dicts(info, len(ds))
    for k in range(len(ds)):
        B, one = rve.Plan(ds[k:k + 1], opts).execute()
        assert rve.info_to_dicts(one, 1)[0] == infos[k]
        if precision == rve.MIXED:
            assert torch.equal(A[k:k + 1], B), SIZES[k]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("delta", [0.0, 0.2])
def test_preconditioner(delta, dtype):
    ds, _, node = _batch(SIZES)
    x = torch.randn(node[-1], 2, dtype=dtype, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    y = rve.apply_precond(ds, x, delta=delta)
    for k in range(len(ds)):
        assert torch.equal(rve.apply_precond(ds[k:k + 1], x[node[k]:node[k + 1]], delta=delta), y[node[k]:node[k + 1]])


@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("want_flux", [False, True])
@pytest.mark.parametrize("sizes", [SIZES, (32,) * 700, (128,) * 40, (256, 512, 256)])
def test_a_hom(sizes, want_flux, scheme):
    ds, mask, node = _batch(sizes)
    u = 0.01 * torch.randn(node[-1], 2, dtype=torch.float64, device="cuda",
                           generator=torch.Generator(device="cuda").manual_seed(4))
    kw = {"scheme": scheme, "want_lo": True, "want_flux": want_flux}
    whole = rve.a_hom(ds, u, mask=mask, **kw)
    for k in sorted({0, 1, len(ds) // 2, len(ds) - 1} | set(range(min(8, len(ds))))):
        lone = rve.a_hom(ds[k:k + 1], u[node[k]:node[k + 1]], mask=mask[node[k] // 32:node[k + 1] // 32], **kw)
        for a, b in zip(lone, whole):
            assert torch.equal(a, b[k:k + 1]), (k, sizes[k])


@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("sizes", [(64, 256, 32, 128, 512, 256, 64), (256, 256, 32), (32,) * 97 + (256, 64, 256)])
def test_chebyshev_moments(sizes, scheme):
    ds, mask, node = _batch(sizes, contrast=5.0)
    K, hi = 33, 16 * 5.0
    v = torch.randn(node[-1], 2, dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(5))
    mu = rve.cheb_moments(ds, v, K, 0.0, hi, mask=mask, scheme=scheme)
    for k in sorted({0, 1, len(ds) // 2, len(ds) - 1} | set(range(max(0, len(ds) - 7), len(ds)))):
        one = rve.cheb_moments(ds[k:k + 1], v[node[k]:node[k + 1]], K, 0.0, hi,
                               mask=mask[node[k] // 32:node[k + 1] // 32], scheme=scheme)
        assert torch.equal(one, mu[k:k + 1]), (k, sizes[k])
