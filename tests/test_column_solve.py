"""The preconditioner over every grid size, precision and shift: the segment
lengths and carries of the column pass, its singular column, and blocks of few
columns, against numpy's FFT."""
import numpy as np
import pytest
import torch

from paper_1903_12227_gb300 import rve, workloads
from test_fixed_rows import _precond

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("delta", [0.0, 0.03])
@pytest.mark.parametrize("n", [32, 64, 128, 256, 512, 1024, 2048])
def test_preconditioner(n, delta, precision):
    ds = [workloads.realization(n // 8, 8, 10.0, 0, k) for k in range(2)]
    x = np.random.default_rng(n).standard_normal((2, n, n, 2))
    if precision == "fp32":
        x = x.astype(np.float32)
    y = rve.apply_precond(ds, torch.tensor(x.reshape(-1, 2), device="cuda"), delta=delta)
    y = y.cpu().numpy().reshape(x.shape).astype(np.float64)
    ref = _precond(x.astype(np.float64), 5.5, delta)
    # noise is dominated by the lowest modes, whose filters have a memory of up
    # to n rows (delta = 0: n / 2 pi of them): n eps per row transform and
    # filter, 20 of them in all
    eps = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    bound = 20 * n * eps
    for k in range(2):
        assert np.linalg.norm(y[k] - ref[k]) <= bound * np.linalg.norm(ref[k])
