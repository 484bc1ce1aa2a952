"""Rows at the ends of the exponent range: the fixed-point transforms of double
pairs take no row whose result could leave the doubles, so that an overflow
shows as an infinity or a NaN and never as a wrong finite number."""
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1903_12227_gb300 import build, rve, rve3, workloads

HERE = os.path.dirname(os.path.abspath(__file__))


def test_rows_taken_on_the_host(tmp_path):
    exe = str(tmp_path / "fixed_rows_range")
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "-w", "-I", build.CSRC,
                    os.path.join(HERE, "fixed_rows_range_host.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout[-1000:]


def _rows(g, shape):
    """Rows with a mean (their DC terms are the first to overflow) and some noise."""
    return 0.75 + 0.25 * g.standard_normal(shape).clip(-0.9, 0.9)


def _finite_values_are_right(y, ref):
    """y against s B^-1 x formed at an ordinary magnitude."""
    ok = np.isfinite(y)
    assert np.abs(y[ok] - ref[ok]).max(initial=0.0) <= 1e-12 * np.abs(ref).max()
    return ok.all()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 128, 512, 2048])
def test_preconditioner_large_rows(n):
    ds = [workloads.realization(n // 8, 8, 10.0, 0, 0)]
    x = _rows(np.random.default_rng(n), (n * n, 2))
    one = rve.apply_precond(ds, torch.tensor(x, device="cuda"), delta=0.5).cpu().numpy()
    whole = []
    for e in (1000, 1006, 1010, 1012, 1014, 1016, 1018, 1019, 1020, 1021, 1022, 1023):
        y = rve.apply_precond(ds, torch.tensor(np.ldexp(x, e), device="cuda"), delta=0.5).cpu().numpy()
        # the reference stays a double: |B^-1| = 1 / delta = 2, |x| < 1
        whole.append(_finite_values_are_right(np.ldexp(y, -e), one))
    assert whole[0] and whole[1]   # 2048 2^1006 is far below the largest double


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 64])
def test_preconditioner_large_rows_3d(n):
    ds = [workloads.realization3(n // 8, 8, 10.0, 0, 0)]
    x = _rows(np.random.default_rng(n), (n ** 3, 3))
    one = rve3.apply_precond(ds, torch.tensor(x, device="cuda"), delta=0.5).cpu().numpy()
    whole = []
    for e in (1000, 1006, 1010, 1012, 1014, 1016, 1018, 1019, 1020, 1021, 1022, 1023):
        y = rve3.apply_precond(ds, torch.tensor(np.ldexp(x, e), device="cuda"), delta=0.5).cpu().numpy()
        whole.append(_finite_values_are_right(np.ldexp(y, -e), one))
    assert whole[0] and whole[1]


def test_rows_of_zeros_on_the_host(tmp_path):
    exe = str(tmp_path / "fixed_rows_zero")
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "-w", "-I", build.CSRC,
                    os.path.join(HERE, "fixed_rows_zero_host.cu"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 64, 256, 1024])
def test_preconditioner_zero_and_subnormal_rows(n):
    """Sparse fields, and subnormals beside rows of zeros (their results keep every bit that FP64 keeps)."""
    ds = [workloads.realization(n // 8, 8, 10.0, 0, 0)]
    x = np.zeros((n, n, 2))
    x[n // 2, 3], x[n // 2 + 5, n - 1] = (1.0, -2.0), (0.5, 0.0)
    lam = 4 * np.sin(np.pi * np.arange(n) / n) ** 2
    ref = np.fft.ifft2(np.fft.fft2(x, axes=(0, 1)) / (5.5 * (lam[:, None] + lam) + 0.5)[..., None], axes=(0, 1)).real
    apply = lambda v: rve.apply_precond(ds, torch.tensor(v.reshape(-1, 2), device="cuda"), delta=0.5).cpu().numpy()  # noqa: E731
    y = apply(x).reshape(x.shape)
    assert np.linalg.norm(y - ref) <= 1e-12 * np.linalg.norm(ref)
    assert not apply(np.zeros_like(x)).any()
    small = apply(np.ldexp(x, -1060)).reshape(x.shape)
    # one unit of the subnormals per pass and mode: 4 n of them at most
    assert np.abs(np.ldexp(small, 1060) - ref).max() <= 4 * n * 2.0 ** (1060 - 1074)
