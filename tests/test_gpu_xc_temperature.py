"""Exchange-correlation does not depend on the temperature: FP32 plans whose Thomas-Fermi term is
off or inverted in FP64, at temperatures where y = pi^2 n / (sqrt2 T^(3/2)) leaves the range of a float."""
import numpy as np
import pytest
import torch

from oracle import xc as xcmod
from paper_2601_23002_gb300 import Plan, TERM_TF, TERM_XC


# n on both sides of r_s = 1.  512 equal terms of a handful of FP32 operations: 3e-6, as in
# test_gpu_functional_tables.py.
@pytest.mark.gpu
@pytest.mark.parametrize("terms,fd64", [(TERM_XC, False), (TERM_XC, True), (TERM_TF | TERM_XC, True)])
@pytest.mark.parametrize("T", [1e-27, 0.4, 1e30])
@pytest.mark.parametrize("n", [0.03, 2.0])
def test_xc_at_any_temperature(n, T, terms, fd64):
    L = 4.0
    n = float(np.float32(n))
    plan = Plan(L, 8, np.array([n * L ** 3]), T, precision="fp32", terms=terms, fd64=fd64)
    plan.structure_factor(np.zeros((1, 3)))
    rho = torch.full((512,), n, dtype=torch.float32, device="cuda")
    v = torch.empty_like(rho)
    e = plan.energy_potential(rho, v)
    plan.close()
    exc, vxc = xcmod.lda_xc(np.array([n]))
    assert abs(e["E_xc"] - L ** 3 * n * float(exc[0])) <= 3e-6 * L ** 3 * n * abs(float(exc[0]))
    assert np.isfinite(e["F_TF"])
    if terms == TERM_XC:
        assert float((v.double() - float(vxc[0])).abs().max()) <= 3e-6 * abs(float(vxc[0]))
