"""Structure factor of FP32 plans on the largest grids, whose k_struct tiles take more
shared memory than a kernel has without raising its limit, with the full S(G) and
with the rows of the local potential only."""
import math

import numpy as np
import pytest
import torch

from oracle.cell import ewald_energy
from paper_2601_23002_gb300 import Plan


# S: phases and products rounded to 6e-8, sums of n_ion unit vectors (as in
# test_gpu_ions.py); E_ion: FP32 S and the reciprocal cut at 1e-9.
@pytest.mark.gpu
@pytest.mark.parametrize("n", [324, 360, 375, 500])
def test_fp32_structure_factor_of_large_grids(n):
    L, n_ion = 0.2 * n, 5
    rng = np.random.default_rng(n)
    Z, pos = np.full(n_ion, 3.0), rng.uniform(0.0, L, (n_ion, 3))
    plan = Plan(L, n, Z, 0.3, precision="fp32")
    plan.structure_factor(pos)
    rho = torch.full((n ** 3,), 3.0 * n_ion / L ** 3, dtype=torch.float32, device="cuda")
    e = [plan.energy_potential(rho)]
    S = torch.empty(n, n, n // 2 + 1, dtype=torch.complex64, device="cuda")
    plan.structure_factor(pos, S)
    e.append(plan.energy_potential(rho))
    plan.close()
    m = np.rint(np.fft.fftfreq(n) * n)
    ph = [torch.tensor(np.exp(-2j * math.pi * np.outer(pos[:, d] / L, m)), device="cuda") for d in range(3)]
    worst = 0.0
    for a in range(0, n, 60):
        ref = torch.einsum("ia,ib->abi", ph[0][:, a:a + 60], ph[1]).reshape(-1, n_ion) @ ph[2][:, :n // 2 + 1]
        got = S[a:a + 60].reshape(-1, n // 2 + 1).to(torch.complex128)
        worst = max(worst, float((got - ref).abs().max()))
    assert worst <= 2e-6 * math.sqrt(n_ion) * 4
    ref = ewald_energy(Z, pos, L)
    for x in e:
        assert abs(x["E_ion"] - ref) <= 1e-6 * float(np.sum(Z * Z))
