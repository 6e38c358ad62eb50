"""Shells, forces and pressure through the forward-only plane passes (compile-time
and 256^3) against the tiled transforms of the same plan type."""
import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import plan_for_cell
from workloads.cells import random_cell


# Both sides transform the same density with FP32 (FP64) butterflies grouped
# differently: sums over shells or all G of terms with 1e-7 (1e-16) errors.
@pytest.mark.gpu
@pytest.mark.parametrize("precision,n,alpha", [("fp64", 24, 0.5), ("fp32", 24, 5 / 6), ("fp64", 45, 5 / 6), ("fp32", 75, 0.5),
                                               ("fp32", 96, 0.5), ("fp64", 128, 0.5), ("fp32", 160, 0.5), ("fp32", 256, 0.5)])
def test_analysis_matches_the_tiled_transforms(monkeypatch, precision, n, alpha):
    cell = random_cell(5, 12, 1.0, 2.0, 0.8, n)
    dt = torch.float32 if precision == "fp32" else torch.float64
    x = np.arange(n) * (2 * np.pi / n)
    rho = 1.0 + 0.3 * np.cos(x)[:, None, None] * np.cos(2 * x)[None, :, None] + 0.2 * np.sin(x)[None, None, :]
    rho = torch.tensor(rho * cell.n_electrons / cell.volume, dtype=dt, device="cuda").reshape(-1)
    got = []
    for env in ({}, {"OFDFT_PLANE": "0", "OFDFT_Z256": "0"}):
        for k, v in env.items():
            monkeypatch.setenv(k, v)
        plan = plan_for_cell(cell, precision, alpha=alpha)
        got.append((plan.sei_shells(rho, 40)[1], plan.forces(rho), plan.pressure(rho)))
        plan.close()
    tol = 3e-6 if precision == "fp32" else 1e-12
    (s1, f1, p1), (s0, f0, p0) = got
    assert np.max(np.abs(s1 - s0)) <= tol * np.max(np.abs(s0))
    assert np.max(np.abs(f1 - f0)) <= tol * np.max(np.abs(f0))
    size = max(abs(v) for v in p0.values())
    for k in p0:
        assert abs(p1[k] - p0[k]) <= tol * size, k
