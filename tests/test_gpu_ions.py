"""Structure factor, Ewald energy and forces over the launch shapes of k_struct and
k_forces_g: grids that take each thread tile, ion counts around the 16-ion chunks,
one and two species, full S(G) and rows only, and cells on both sides of the
lengths where the Ewald sum needs images."""
import math

import numpy as np
import pytest
import torch

from oracle.cell import ewald_energy
from oracle.forces import forces as oracle_forces
from paper_2601_23002_gb300 import Plan, TERMS_ALL
from workloads.cells import Cell


def ions(n_ion, L, two):
    rng = np.random.default_rng([n_ion, int(10 * L)])
    pos = rng.uniform(0.0, L, (n_ion, 3))
    Z = np.ones(n_ion)
    if two:
        Z[::2] = 3.0
    return Z, pos


# FP64: sums of n_ion unit vectors, 1e-12 relative to sqrt(sum Z^2); FP32: phases
# rounded to 6e-8, products and sums of up to 300 terms: 1e-6 of sqrt(n_ion)
@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("n,n_ion", [(8, 1), (15, 2), (30, 15), (64, 16), (64, 17), (75, 33), (128, 40), (162, 5)])
def test_structure_factor(n, n_ion, two, precision, tol):
    L = 0.25 * n
    Z, pos = ions(n_ion, L, two)
    plan = Plan(L, n, Z, 0.3, precision=precision)
    ct = torch.complex64 if precision == "fp32" else torch.complex128
    S = torch.empty(n, n, n // 2 + 1, dtype=ct, device="cuda")
    plan.structure_factor(pos)
    plan.structure_factor(pos, S)
    plan.close()
    m = np.rint(np.fft.fftfreq(n) * n)
    ph = [torch.tensor(np.exp(-2j * math.pi * np.outer(pos[:, d] / L, m)), device="cuda") for d in range(3)]
    ref = (torch.einsum("ia,ib->abi", ph[0], ph[1]).reshape(n * n, -1) @ ph[2][:, :n // 2 + 1]).reshape(S.shape)
    assert float((S.to(torch.complex128) - ref).abs().max()) <= tol * math.sqrt(n_ion) * 4


# Ewald: both sides sum to 1e-16 of their largest terms; a few hundred terms of
# size Z^2 in FP64: 1e-11 relative.  FP32 plans cut the reciprocal sum at 1e-9.
@pytest.mark.gpu
@pytest.mark.parametrize("n,L,n_ion,two", [(16, 4.1, 3, True), (24, 6.2, 4, False), (24, 6.4, 5, True), (48, 12.5, 8, False),
                                           (50, 12.7, 9, True), (64, 16.0, 17, False)])
def test_ewald_and_forces(n, L, n_ion, two):
    Z, pos = ions(n_ion, L, two)
    cell = Cell(L=L, n=n, Z=Z, pos=pos, theta=0.5)
    rng = np.random.default_rng(1)
    x = np.arange(n) * (2 * np.pi / n)
    rho = cell.n_electrons / L ** 3 * (1.0 + 0.2 * np.cos(x)[:, None, None] + 0.1 * np.sin(2 * x)[None, :, None]
                                       + 0.15 * np.cos(x + 0.3)[None, None, :] * np.sin(x)[:, None, None])
    plan = Plan(L, n, Z, cell.T, precision="fp64", terms=TERMS_ALL)
    plan.structure_factor(pos)
    r = torch.tensor(rho, device="cuda").reshape(-1)
    e = plan.energy_potential(r)
    f = plan.forces(r)
    plan.close()
    ref = ewald_energy(Z, pos, L)
    assert abs(e["E_ion"] - ref) <= 1e-11 * (np.sum(Z * Z) + abs(ref))
    # coarse grids cut the forces' G sums at the grid's Nyquist |m| per axis
    # alike in the oracle's full grid and here, where the Gaussians allow it
    if math.pi * n / L > 12.6:
        fo = oracle_forces(cell, rho)
        assert np.max(np.abs(f - fo)) <= 1e-10 * max(1.0, np.max(np.abs(fo)))


# Positions outside [0, L) are wrapped: the same energy and forces (rounding of
# x + k L: 1e-16 |k| L in the positions times forces of a few hartree/bohr).
@pytest.mark.gpu
@pytest.mark.parametrize("shift", [3, -700, 90000])
def test_unwrapped_positions(shift):
    L, n = 9.0, 36
    Z, pos = ions(6, L, True)
    pos[1] = pos[0] + [L / 2, 0.0, 0.0]              # a pair at half a cell
    rho = torch.full((n ** 3,), float(np.sum(Z)) / L ** 3, dtype=torch.float64, device="cuda")
    got = []
    for s in (0, shift):
        p = pos.copy()
        p[::2, 0] += s * L
        p[1::3, 2] -= s * L
        plan = Plan(L, n, Z, 0.4, precision="fp64")
        plan.structure_factor(p)
        got.append((plan.energy_potential(rho)["E_ion"], plan.forces(rho)))
        plan.close()
    tol = 1e-11 + 1e-14 * abs(shift) * L
    assert abs(got[0][0] - got[1][0]) <= tol * 100
    assert np.max(np.abs(got[0][1] - got[1][1])) <= tol * 100
