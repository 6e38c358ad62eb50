"""The FP64 tables of the pointwise functional (Fermi-Dirac inversion and PZ81)
at their edges: uniform densities just inside and outside the tabulated ranges,
at an interval's end and at r_s = 1, against the oracle's quadrature and formulas."""
import math

import numpy as np
import pytest
import torch

from oracle import fermi_dirac as fd
from oracle import xc as xcmod
from paper_2601_23002_gb300 import Plan, TERM_TF, TERM_XC

N1 = 3.0 / (4.0 * math.pi)          # density of r_s = 1
EDGES = [(2.0 ** ey * f, 2.0 ** ex * g)
         for ey, ex in ((-14, -20), (0, 0), (17, 6))
         for f, g in ((1 - 1e-12, 1 - 1e-12), (1.0, 1.0), (1.0 + 1.0 / 16, 1.0 + 1.0 / 16), (0.25, 0.25), (8.0, 8.0))]


# Rounding: 512 equal terms and a handful of operations per point in FP64
# (1e-14), the oracle's Newton inversion 1e-14 in eta with f = n T (eta - p)
# and |eta| <= 1e4: 1e-11 relative to the terms is safe by two digits.
@pytest.mark.gpu
@pytest.mark.parametrize("precision,fd64,tol", [("fp64", False, 1e-11), ("fp32", True, 3e-6)])
@pytest.mark.parametrize("y,u", EDGES)
def test_uniform_density_at_the_tables_edges(precision, fd64, tol, y, u):
    if precision == "fp32":
        u = float(np.float32(u * N1)) / N1            # the density an FP32 plan holds
    n = u * N1
    # T with y = pi^2 n / (sqrt2 T^(3/2))
    T = (math.pi ** 2 * n / (math.sqrt(2.0) * y)) ** (2.0 / 3.0)
    L = 4.0
    plan = Plan(L, 8, np.array([n * L ** 3]), T, precision=precision, terms=TERM_TF | TERM_XC, fd64=fd64)
    plan.structure_factor(np.zeros((1, 3)))
    dt = torch.float64 if precision == "fp64" else torch.float32
    rho = torch.full((512,), n, dtype=dt, device="cuda")
    v = torch.empty_like(rho)
    e = plan.energy_potential(rho, v)
    plan.close()
    f, vt, _ = fd.tf_free_energy_density(np.array([n]), T)
    exc, vxc = xcmod.lda_xc(np.array([n]))
    _, _, eta = fd.tf_free_energy_density(np.array([n]), T)
    size = L ** 3 * n * T * max(1.0, abs(float(eta[0])))
    assert abs(e["F_TF"] - L ** 3 * float(f[0])) <= tol * size
    assert abs(e["E_xc"] - L ** 3 * n * float(exc[0])) <= tol * L ** 3 * n * abs(float(exc[0]))
    want = float(vt[0] + vxc[0])
    assert np.max(np.abs(v.double().cpu().numpy() - want)) <= tol * (T * max(1.0, abs(float(eta[0]))) + abs(float(vxc[0])))
