"""The fixed-point row transforms of double pairs (csrc/rve_fixed.cuh): their
bounds and their error on the host, and the preconditioner that runs them on
the GPU over every grid size and the rows that leave the fixed-point path."""
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1903_12227_gb300 import build, rve, workloads

HERE = os.path.dirname(os.path.abspath(__file__))


def test_bounds_and_error_on_the_host(tmp_path):
    exe = str(tmp_path / "fixed_rows")
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "-w", "-I", build.CSRC,
                    os.path.join(HERE, "fixed_rows_host.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout[-300:]
    rows = [line.split() for line in out.stdout.splitlines()]
    assert len(rows) == 7 * 9
    for p, kind, fixed, double in rows:
        # no less exact than the stages in double (one rounding of the result
        # where both are exact to it, 2^-54 of the norm)
        assert float(fixed) <= max(1.1 * float(double), 2.0 ** -54), (p, kind, fixed, double)


def _precond(x, c0, delta):
    """B^-1 x for [batch, n, n, 2] by numpy's FFT."""
    n = x.shape[1]
    lam = 4 * np.sin(np.pi * np.arange(n) / n) ** 2
    sym = c0 * (lam[:, None] + lam[None, :]) + delta
    inv = np.where(sym > 0, 1.0 / np.where(sym > 0, sym, 1.0), 0.0)
    return np.fft.ifft2(np.fft.fft2(x, axes=(1, 2)) * inv[None, :, :, None], axes=(1, 2)).real


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 64, 128, 256, 512, 1024, 2048])
def test_preconditioner_rows(n):
    ds = [workloads.realization(n // 8, 8, 10.0, 0, k) for k in range(3)]
    g = np.random.default_rng(n)
    x = g.standard_normal((3, n, n, 2))
    x[0, ::3] = 0.0                                  # whole rows of zeros
    x[1, 1] *= 1e-290                                # a row too small for the fixed-point path
    x[2] = 0.0
    x[2, n // 3, [1, n - 2], :] = [[1.0, 0.0], [-1.0, 3.0]]   # spikes
    x[2] *= 2.0 ** -300
    y = rve.apply_precond(ds, torch.tensor(x.reshape(-1, 2), device="cuda"), delta=0.5)
    y = y.cpu().numpy().reshape(x.shape)
    ref = _precond(x, 5.5, 0.5)
    for k in range(3):   # delta = 0.5: |B^-1| |B| < 100, so 1e-12 is above 100 n eps
        assert np.linalg.norm(y[k] - ref[k]) <= 1e-12 * np.linalg.norm(ref[k])


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 256, 512])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_preconditioner_not_finite(n, bad):
    """An infinity or NaN leaves no finite value in its row and does not reach other realizations."""
    ds = [workloads.realization(n // 8, 8, 10.0, 0, k) for k in range(2)]
    x = np.random.default_rng(1).standard_normal((2, n, n, 2))
    ref = rve.apply_precond(ds, torch.tensor(x.reshape(-1, 2), device="cuda"), delta=0.5)
    x[0, n // 2, 3, 1] = bad
    y = rve.apply_precond(ds, torch.tensor(x.reshape(-1, 2), device="cuda"), delta=0.5)
    y, ref = (t.cpu().numpy().reshape(x.shape) for t in (y, ref))
    assert not np.isfinite(y[0, n // 2]).any()
    np.testing.assert_array_equal(y[1], ref[1])


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 64, 128])
def test_preconditioner_lines_3d(n):
    """Lines of the 3D transforms: zeros, spikes and magnitudes that leave the fixed-point path."""
    from paper_1903_12227_gb300 import rve3
    ds = [workloads.realization3(n // 8, 8, 10.0, 0, k) for k in range(2)]
    g = np.random.default_rng(n)
    x = g.standard_normal((2, n, n, n, 3))
    x[0, ::3] = 0.0
    x[0, 1, 1] *= 1e-290
    x[1] = 0.0
    x[1, n // 3, 2, [1, n - 2], :] = [[1.0, 0.0, 2.0], [-1.0, 3.0, 0.0]]
    y = rve3.apply_precond(ds, torch.tensor(x.reshape(-1, 3), device="cuda"), delta=0.5)
    y = y.cpu().numpy().reshape(x.shape)
    lam = 4 * np.sin(np.pi * np.arange(n) / n) ** 2
    sym = 5.5 * (lam[:, None, None] + lam[:, None] + lam) + 0.5
    for k in range(2):   # as in 2D: |B^-1| |B| < 200
        ref = np.fft.ifftn(np.fft.fftn(x[k], axes=(0, 1, 2)) / sym[..., None], axes=(0, 1, 2)).real
        assert np.linalg.norm(y[k] - ref) <= 1e-12 * np.linalg.norm(ref)
