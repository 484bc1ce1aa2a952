"""The FP64 stiffness application up to the largest doubles, and on cell values
that are zero, tiny or not finite."""
import numpy as np
import pytest
import torch

from paper_1903_12227_gb300 import rve, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("explicit", [False, True])
@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("n", [32, 256])
def test_large_vectors(n, scheme, explicit):
    """2^e x gives 2^e (A x) exactly as long as that is a double."""
    ds = workloads.batch(n // 8, 8, 3.0, 2, 2)
    mask = rve.gen_field(ds)
    kw = {"coef": rve.coef_from_mask(ds, mask)} if explicit else {"mask": mask}
    x = torch.rand(2 * n * n, 2, dtype=torch.float64, device="cuda",
                   generator=torch.Generator(device="cuda").manual_seed(n)) + 1.0   # in [1, 2)
    y = rve.apply_stiffness(ds, x, scheme=scheme, **kw)
    # the weights' centre times x stays below (8/3) 3 2^1020 2 = 2^1024; the
    # other terms have the opposite sign
    z = rve.apply_stiffness(ds, x * 2.0 ** 1020, scheme=scheme, **kw)
    assert torch.equal(z, y * 2.0 ** 1020)


@pytest.mark.parametrize("explicit", [False, True])
@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
def test_large_cells(scheme, explicit):
    """2^1020 A gives 2^1020 (A x) exactly as long as that is a double."""
    n, e = 64, 1020
    x = torch.randn(n * n, 2, dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(2)) * 2.0 ** -20
    ds = [workloads.realization(8, 8, 3.0, 2, 0, a_matrix=s) for s in (1.0, 2.0 ** e)]
    mask = rve.gen_field(ds[:1])
    y, z = (rve.apply_stiffness([d], x, scheme=scheme, **({"coef": rve.coef_from_mask([d], mask)} if explicit else {"mask": mask}))
            for d in ds)
    assert torch.equal(z, y * 2.0 ** e)


def test_unusual_cells():
    ds = workloads.batch(8, 8, 3.0, 2, 1)
    n = 64
    a = torch.ones(n * n, dtype=torch.float64, device="cuda")
    bad = {(5, 7): 0.0, (20, 40): 2.0 ** -1021, (30, 10): 2.0 ** -1040, (40, 33): np.inf, (50, 50): np.nan}
    for (i, j), v in bad.items():
        a[i * n + j] = v
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(n * n, 2, dtype=torch.float64, device="cuda", generator=g)
    y = rve.apply_stiffness(ds, x, coef=a).view(n, n, 2).cpu().numpy()
    ok = np.ones((n, n), dtype=bool)
    for (i, j), v in bad.items():
        if not np.isfinite(v):
            ok[i:i + 2, j:j + 2] = False   # the cell's nodes
    assert np.isfinite(y[ok]).all() and not np.isfinite(y[~ok]).any()
    for v in (0.0, 2.0 ** -1021, 2.0 ** -1040):   # such cells add less than a unit of the others
        b = torch.ones_like(a)
        b[5 * n + 7] = v
        c = torch.ones_like(a)
        c[5 * n + 7] = 0.0
        u, w = (rve.apply_stiffness(ds, x, coef=t) for t in (b, c))
        assert torch.equal(u, w)
