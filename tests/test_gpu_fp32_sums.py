"""Sums that FP32 plans form in FP64: the Ewald energy's reciprocal part, the pressure's
local and nonlocal parts."""
import math

import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import Plan


def _m2(n):
    m = torch.tensor(np.rint(np.fft.fftfreq(n) * n), device="cuda")
    return m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :n // 2 + 1] ** 2


def _weights(n):
    w = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1.0
    if n % 2 == 0:
        w[-1] = 1.0
    return w


# An FP32 plan's S(G) is rounded to FP32, and nothing after it is: the energies of the
# FP32 and the FP64 plan differ by the weighted sum of the differences of |S_Z|^2.  The
# grids' Nyquist |G| (below 9.1) bounds the reciprocal range of both plans alike.
# 1e-12: FP64 sums of some thousand positive terms.
@pytest.mark.gpu
@pytest.mark.parametrize("Z", [1.0, 3.0])
@pytest.mark.parametrize("n,L,n_ion", [(24, 10.0, 30), (45, 20.0, 17)])
def test_ewald_sum_of_the_fp32_structure_factor(n, L, n_ion, Z):
    pos = np.random.default_rng(n).uniform(0.0, L, (n_ion, 3))
    rho = torch.full((n ** 3,), Z * n_ion / L ** 3, dtype=torch.float64, device="cuda")
    E, A2 = [], []
    for precision, ct in (("fp32", torch.complex64), ("fp64", torch.complex128)):
        S = torch.empty(n, n, n // 2 + 1, dtype=ct, device="cuda")
        plan = Plan(L, n, np.full(n_ion, Z), 0.3, precision=precision)
        plan.structure_factor(pos, S)
        E.append(plan.energy_potential(rho.to(plan.dtype))["E_ion"])
        plan.close()
        s = Z * torch.view_as_real(S)                     # (rounded to the plan's type, as S_Z)
        A2.append((s.double() ** 2).sum(dim=-1))
    G2 = (2.0 * math.pi / L) ** 2 * _m2(n)
    G2[0, 0, 0] = 1.0
    eta2 = (math.pi * n / L) ** 2 / (4.0 * 39.0)
    f = 2.0 * math.pi / L ** 3 * torch.exp(-G2 / (4.0 * eta2)) / G2 * _weights(n)
    f[0, 0, 0] = 0.0
    want = float((f * (A2[0] - A2[1])).sum())
    assert abs(want) > 1e-10 * float((f * A2[1]).sum())
    assert abs((E[0] - E[1]) - want) <= 1e-12 * float((f * A2[1]).sum())
