"""The compile-time passes (csrc/cpass.cuh) against the generic ones of the same
plane path on every grid that has them: one evaluation with two and three
transformed fields, the preconditioning pass inside a short minimisation, and a
density that is aligned to single values only."""
import os

import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import plan_for_cell
from workloads.cells import random_cell

GRIDS = [24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128, 135,
         144, 150, 160]


def density(cell, dtype):
    n = cell.n
    rng = np.random.default_rng(n)
    x = np.arange(n) * (2 * np.pi / n)
    X, Y, Z = np.meshgrid(x, x, x, indexing="ij")
    p = np.ones((n, n, n))
    for _ in range(5):
        m = rng.integers(-3, 4, size=3)
        p += 0.12 * np.cos(m[0] * X + m[1] * Y + m[2] * Z + rng.uniform(0, 2 * np.pi))
    p *= cell.n_electrons / cell.volume / p.mean()
    return torch.tensor(p, dtype=dtype, device="cuda").reshape(-1)


def both(monkeypatch, cell, precision, go, **kw):
    out = []
    for v in ("1", "0"):
        monkeypatch.setenv("OFDFT_CPASS", v)
        plan = plan_for_cell(cell, precision, **kw)
        out.append(go(plan))
        plan.close()
    return out


# The transforms have the generic passes' radices, twiddles and order, so the
# potentials differ at most where the compiler contracts a product differently:
# a few roundings of the psi transform, amplified by G^2 of these fine grids to
# 2e-5 (FP32, the error of such a potential against FP64) and 1e-12 (FP64) of
# max|v|; the energies by the order of their sums.
@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol_v,tol_e", [("fp32", 2e-5, 1e-6), ("fp64", 1e-12, 1e-13)])
@pytest.mark.parametrize("alpha", [0.5, 5.0 / 6.0])
@pytest.mark.parametrize("n", GRIDS)
def test_evaluation_matches_the_generic_passes(monkeypatch, n, alpha, precision, tol_v, tol_e):
    cell = random_cell(7, 8, 1.0, 2.0, 0.8, n)
    rho = density(cell, torch.float32 if precision == "fp32" else torch.float64)

    def go(plan):
        v = torch.empty_like(rho)
        e = plan.energy_potential(rho, v)
        plan.profile_enable(False)
        plan.energy_potential(rho, v)
        return v, e, set(plan.profile_read())

    (v1, e1, k1), (v0, e0, k0) = both(monkeypatch, cell, precision, go, alpha=alpha)
    assert "k_plane_c" in k1 and "k_zinv_c" in k1 and "k_plane_c" not in k0
    assert float((v1 - v0).abs().max()) <= tol_v * float(v0.abs().max())
    scale = max(abs(e0[k]) for k in ("F_TF", "E_loc", "E_xc", "E_H", "E_ion"))
    for k in e0:
        assert abs(e1[k] - e0[k]) <= tol_e * max(scale, abs(e0[k])), k


# FP32 above 160: planes over clusters, where the generic passes are the tiled ones
# with another order of the stages along x and y.  Both round the psi transform,
# amplified by G^2; against the FP64 plan the error must not be larger (a factor
# 1.5 for two independent roundings).
@pytest.mark.gpu
@pytest.mark.parametrize("n", [162, 180, 192, 200, 216, 225, 240, 243, 250])
def test_large_grids_are_as_exact_as_the_tiled_passes(monkeypatch, n):
    cell = random_cell(7, 8, 1.0, 2.0, 0.8, n)
    cell.L *= 2.5
    cell.pos *= 2.5
    rho = density(cell, torch.float32)

    def go(plan):
        r = rho.to(plan.dtype)
        v = torch.empty_like(r)
        e = plan.energy_potential(r, v)
        return v.double(), e

    v64, e64 = both(monkeypatch, cell, "fp64", go)[1]
    (v1, e1), (v0, e0) = both(monkeypatch, cell, "fp32", go)
    err = [float((v - v64).norm() / v64.norm()) for v in (v1, v0)]
    assert err[0] <= 1.5 * err[1]
    size = max(abs(x) for x in e64.values())
    for k in e64:
        assert abs(e1[k] - e64[k]) <= max(1.5 * abs(e0[k] - e64[k]), 1e-6 * size), k


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol", [("fp32", 2e-6), ("fp64", 1e-12)])
@pytest.mark.parametrize("n", [24, 45, 64, 75, 128])
def test_minimisation_matches_the_generic_passes(monkeypatch, n, precision, tol):
    cell = random_cell(7, 8, 1.0, 2.0, 0.8, n)
    dt = torch.float32 if precision == "fp32" else torch.float64

    def go(plan):
        rho = torch.empty(n ** 3, dtype=dt, device="cuda")
        plan.minimize(rho, max_iter=5)
        return rho

    r1, r0 = both(monkeypatch, cell, precision, go)
    assert float((r1 - r0).norm() / r0.norm()) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 75])
def test_density_aligned_to_single_values(n):
    cell = random_cell(7, 8, 1.0, 2.0, 0.8, n)
    rho = density(cell, torch.float64)
    off = torch.empty(n ** 3 + 1, dtype=torch.float64, device="cuda")[1:]
    off.copy_(rho)
    plan = plan_for_cell(cell, "fp64")
    a, b = torch.empty_like(rho), torch.empty_like(rho)
    plan.energy_potential(rho, a)
    plan.energy_potential(off, b)
    plan.close()
    assert float((a - b).abs().max()) <= 1e-12 * float(a.abs().max())


# FP64 passes whose rows per block are none of a tile schedule's usual counts: the
# plan's own schedule, one it does not have a compile-time pass for, and the
# autotuner's choice give the same potential (bound as above).
@pytest.mark.gpu
@pytest.mark.parametrize("n", [45, 54, 100])
def test_tile_schedules_beside_the_compile_time_rows(n):
    cell = random_cell(11, 8, 1.0, 2.0, 0.8, n)
    rho = density(cell, torch.float64)
    plan = plan_for_cell(cell, "fp64")

    def go():
        v = torch.empty_like(rho)
        plan.profile_enable(False)
        plan.energy_potential(rho, v)
        return v, set(plan.profile_read())

    v0, k0 = go()
    plan.set_tiles((16, 16, 16))
    v1, k1 = go()
    tiles, _ = plan.autotune()
    v2, _ = go()
    plan.close()
    assert "k_zinv_c" in k0 and "k_zinv_epi" in k1
    assert all(8 <= t <= 64 for t in tiles)
    for v in (v1, v2):
        assert float((v - v0).abs().max()) <= 1e-12 * float(v0.abs().max())
