"""FP64 A_hom in double-double arithmetic: the energy form is the same bits with
and without the flux form, and A + A_lo against exact rational arithmetic."""
from fractions import Fraction

import pytest
import torch

from paper_1903_12227_gb300 import rve, workloads

pytestmark = pytest.mark.gpu


def _u(nodes, seed, size=0.1):
    return size * torch.randn(nodes, 2, dtype=torch.float64, device="cuda",
                              generator=torch.Generator(device="cuda").manual_seed(seed))


@pytest.mark.parametrize("explicit", [False, True])
@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("n,count", [(32, 40), (64, 3), (128, 9), (256, 5), (512, 2), (1024, 1), (2048, 1)])
def test_with_and_without_flux(n, count, scheme, explicit):
    ds = workloads.batch(n // 8, 8, 7.3, 1, count)
    mask = rve.gen_field(ds)
    kw = {"coef": rve.coef_from_mask(ds, mask)} if explicit else {"mask": mask}
    u = _u(count * n * n, n)
    A, lo = rve.a_hom(ds, u, scheme=scheme, want_lo=True, **kw)
    B, lo2, _ = rve.a_hom(ds, u, scheme=scheme, want_lo=True, want_flux=True, **kw)
    assert torch.equal(A, B)
    assert torch.equal(lo, lo2)


@pytest.mark.parametrize("scheme", [rve.CONSISTENT, rve.LUMPED])
@pytest.mark.parametrize("L,m0,contrast", [(4, 8, 10.0), (8, 4, 7.3), (4, 16, 100.0)])
def test_against_rationals(L, m0, contrast, scheme):
    n = L * m0
    ds = workloads.batch(L, m0, contrast, 3, 1)
    mask = rve.gen_field(ds)
    a = rve.coef_from_mask(ds, mask).cpu().tolist()
    u = _u(n * n, L, 0.5 / m0)
    A, lo, F = (t[0].cpu().tolist() for t in rve.a_hom(ds, u, mask=mask, scheme=scheme, want_lo=True, want_flux=True))
    v = [[Fraction(x) for x in row] for row in u.cpu().tolist()]
    diag = 2 if scheme == rve.CONSISTENT else 0
    K = 6 if scheme == rve.CONSISTENT else 2
    pairs = [((0, 0), (0, 1), 1), ((1, 0), (1, 1), 1), ((0, 0), (1, 0), 1), ((0, 1), (1, 1), 1),
             ((0, 0), (1, 1), diag), ((0, 1), (1, 0), diag)]
    h = Fraction(1, m0)
    E = [[Fraction(0)] * 2 for _ in range(2)]
    P = [[Fraction(0)] * 2 for _ in range(2)]   # P[j][i]
    for i in range(n):
        for j in range(n):
            at = lambda p: v[((i + p[0]) % n) * n + (j + p[1]) % n]  # noqa: E731
            c = Fraction(a[i * n + j])
            for p, q, w in pairs:
                if w == 0:
                    continue
                du = [x - y for x, y in zip(at(q), at(p))]
                xi = [h * (q[0] - p[0]), h * (q[1] - p[1])]
                dv = [du[0] + xi[0], du[1] + xi[1]]
                for r in range(2):
                    for s in range(2):
                        E[r][s] += c * w * dv[r] * dv[s]
                        P[r][s] += c * w * xi[r] * du[s]
    mean = sum(Fraction(x) for x in a) / (n * n)
    scale = float(max(E[0][0], E[1][1])) / (K * L * L)
    for r in range(2):
        for s in range(2):
            # under 40 operations of relative error 3 2^-106 to a cell's energies
            # and their products with the cell value, under 40 sums above them
            err = abs(Fraction(A[r][s]) + Fraction(lo[r][s]) - E[r][s] / (K * L * L))
            assert float(err) <= 240 * 2.0 ** -106 * scale
            flux = (mean if r == s else 0) + P[s][r] / (K * L * L)
            assert abs(float(Fraction(F[r][s]) - flux)) <= 2.0 ** -52 * max(abs(float(flux)), scale)
