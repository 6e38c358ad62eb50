"""Positions many cells away: the minimum image's cell count beyond the whole numbers a float holds
(2^24), from host and device memory."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import Plan


# Against the same positions wrapped exactly.  A separation x near k cells is rounded to
# 1e-16 k L as x - k L is formed: forces of some hartree/bohr times that, with the
# factor of 100 of test_gpu_ions.py.
@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("k", [16777219, 40000003, -123456789])
def test_positions_many_cells_away(k, precision):
    L, n, n_ion = 9.0, 36, 6
    pos = np.random.default_rng(3).uniform(0.0, L, (n_ion, 3))
    far = pos.copy()
    far[::2, 0] += k * L
    far[1::3, 2] -= k * L
    near = np.array([[float(Fraction(float(x)) % Fraction(L)) for x in p] for p in far])
    rho = torch.full((n ** 3,), n_ion / L ** 3, dtype=torch.float32 if precision == "fp32" else torch.float64, device="cuda")
    got = []
    for p in (near, far, torch.tensor(far, device="cuda")):
        plan = Plan(L, n, np.ones(n_ion), 0.4, precision=precision)
        plan.structure_factor(p)
        got.append((plan.energy_potential(rho)["E_ion"], plan.forces(rho)))
        plan.close()
    tol = (1e-11 if precision == "fp64" else 1e-6) + 1e-14 * abs(k) * L * 100
    for e, f in got[1:]:
        assert abs(e - got[0][0]) <= tol
        assert np.max(np.abs(f - got[0][1])) <= tol
