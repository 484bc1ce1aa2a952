"""Stiffness application and Chebyshev moments over every grid size and form of
their kernels (column pairs and single columns, row groups, masks and explicit
cells, 8-byte aligned vectors; clusters and the per-step form), against plain
torch in double."""
import numpy as np
import pytest
import torch

from paper_1903_12227_gb300 import rve, workloads

pytestmark = pytest.mark.gpu


def _cells(ds, mask):
    n = ds[0]["L"] * ds[0]["m0"]
    return rve.coef_from_mask(ds, mask).view(len(ds), n, n)


def _apply(a, x, scheme):
    """A x element by element; a [B, n, n], x [B, n, n, 2] float64."""
    w0, w1 = (1 / 3, 1 / 6) if scheme == rve.CONSISTENT else (0.5, 0.0)
    at = lambda v, i, j: torch.roll(v, (-i, -j), (1, 2))  # noqa: E731
    bits = [(0, 0), (0, 1), (1, 0), (1, 1)]
    y = torch.zeros_like(x)
    for p in bits:
        t = torch.zeros_like(x)
        for q in bits:
            d1, d2 = p[0] != q[0], p[1] != q[1]
            k = -2 * w1 if d1 and d2 else (w1 - w0) if d1 or d2 else 2 * w0
            t += k * at(x, *q)
        y += torch.roll(a[..., None] * t, p, (1, 2))
    return y


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("n,count", [(32, 1), (32, 700), (64, 3), (128, 100), (256, 1), (512, 2), (1024, 3), (2048, 1)])
def test_stiffness(n, count, scheme, dtype):
    ds = workloads.batch(n // 4, 4, 7.3, 2, count)
    mask = rve.gen_field(ds)
    a = _cells(ds, mask)
    g = torch.Generator(device="cuda").manual_seed(n)
    base = torch.randn(count * n * n * 2 + 2, dtype=dtype, device="cuda", generator=g)
    eps = 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24
    for off in ((0,) if dtype == torch.float64 else (0, 2)):   # float32: 16- and 8-byte aligned
        x = base[off:off + count * n * n * 2].view(-1, 2)
        ref = _apply(a, x.double().view(count, n, n, 2), scheme).view(-1, 2)
        for kw in ({"mask": mask}, {"coef": a.reshape(-1)}):
            y = rve.apply_stiffness(ds, x, scheme=scheme, **kw).double()
            # nine products and their sum, weights of up to four roundings:
            # 16 eps of sum |w| |x| <= 16 a_max / 3 max |x|
            assert float((y - ref).abs().max()) <= 16 * eps * 16 * 7.3 / 3 * float(x.abs().max())


@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("explicit", [False, True])
@pytest.mark.parametrize("n,count,K", [(32, 3, 2), (32, 1, 129), (64, 100, 40), (128, 2, 65), (256, 2, 24)])
def test_chebyshev_moments(n, count, K, explicit, scheme):
    ds = workloads.batch(n // 8, 8, 5.0, 3, count)
    mask = rve.gen_field(ds)
    a = _cells(ds, mask)
    g = torch.Generator(device="cuda").manual_seed(n + K)
    v = torch.randn(count * n * n * 2 + 1, dtype=torch.float64, device="cuda", generator=g)[1:].view(-1, 2)
    if n > 128:
        v = v.clone()
    lo, hi = -0.5, 16 * 5.0 * (1 / 3 if scheme == rve.CONSISTENT else 0.5)
    mu = rve.cheb_moments(ds, v, K, lo, hi, scheme=scheme, **({"coef": a.reshape(-1)} if explicit else {"mask": mask}))
    w = v.view(count, n, n, 2)
    tilde = lambda x: (2 * _apply(a, x, scheme) - (hi + lo) * x) / (hi - lo)  # noqa: E731
    prev, cur, ref = w, tilde(w), [(w * w).sum((1, 2))]
    for k in range(1, K):
        ref.append((w * cur).sum((1, 2)))
        prev, cur = cur, 2 * tilde(cur) - prev
    ref = torch.stack(ref, -1)
    # every step adds a few roundings of |w| and the recurrence carries them on linearly
    bound = 8 * K * K * 2.0 ** -53 * float(ref[..., 0].max())
    assert float((mu - ref).abs().max()) <= bound
