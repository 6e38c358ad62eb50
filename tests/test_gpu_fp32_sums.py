"""Sums that FP32 plans form without FP32 rounding: the Ewald energy's reciprocal part, the
pressure's local and nonlocal parts, the forces' sums over G."""
import math

import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import Plan, TERM_LOC, TERMS_ALL


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


# Pressure, local part: of a uniform density 2^-4 the spectrum is n~(0) alone, exact in
# FP32 where every butterfly is (2 and 3 points), and P_loc = n V_loc(0) with V_loc(0)
# rounded to FP32: 3e-14 after a few operations on pairs of floats (48 bits).
@pytest.mark.gpu
@pytest.mark.parametrize("n", [16, 27, 72, 96])
def test_local_pressure_of_a_uniform_density(n):
    L, n_ion = 0.2 * n, 9
    plan = Plan(L, n, np.full(n_ion, 2.0), 0.3, rc=1.1, precision="fp32")
    plan.structure_factor(np.random.default_rng(n).uniform(0.0, L, (n_ion, 3)))
    p = plan.pressure(torch.full((n ** 3,), 0.0625, dtype=torch.float32, device="cuda"))
    plan.close()
    v0 = float(np.float32(math.pi * 1.1 * 1.1 / L ** 3 * 2.0 * n_ion))
    assert abs(p["loc"] - 0.0625 * v0) <= 3e-14 * 0.0625 * v0


# Nonlocal part: planes of density 1/4 and 1/16 in turn, mean wave 1/4 (N_e / L^3 = 1/16): every
# value of the transform of sqrt(n) is exact in FP32 and in FP64, and so is |n~|^2; the two
# plans' pressures then differ by some roundings of FP64 and of pairs of floats (48 bits).
@pytest.mark.gpu
@pytest.mark.parametrize("n", [16, 32, 64])
def test_nonlocal_pressure_of_an_exact_wave(n):
    rho = torch.full((n, n, n), 0.25, dtype=torch.float64)
    rho[1::2] = 0.0625
    got = []
    for precision in ("fp32", "fp64"):
        plan = Plan(8.0, n, np.full(32, 1.0), 0.4, precision=precision)
        plan.structure_factor(np.random.default_rng(n).uniform(0.0, 8.0, (32, 3)))
        got.append(plan.pressure(rho.to(plan.dtype).cuda().reshape(-1))["nl"])
        plan.close()
    assert abs(got[1]) > 1e-6
    assert abs(got[0] - got[1]) <= 1e-13 * abs(got[1])


# Forces without the local term: their G sums from the FP32 inputs the kernel has (w efac S_Z* and
# the kz phases, rounded) in FP64 here, the real-space part the FP64 plan's.  L = 0.6 n
# keeps every G of the grid in both plans' range.  The kernel's own roundings are two of the
# running sum U a term (restarted every second kz), one of V + kz U, one of each row
# product P; each is at most half a unit of 2^-23, evenly spread, and half of it shows in the
# imaginary part.  The mean square error over that is below 1 for each component (about
# 1/2, half a unit being that of the value's own binade; 36 ions: 5 standard deviations).
@pytest.mark.gpu
@pytest.mark.parametrize("n", [45, 96])
def test_force_sums_of_the_fp32_inputs(n):
    L, n_ion, nk = 0.6 * n, 3, n // 2 + 1
    tp = 2.0 * math.pi / L
    G2 = tp ** 2 * _m2(n)
    G2[0, 0, 0] = 1.0
    eta2 = (math.pi * n / L) ** 2 / (4.0 * 39.0)
    f = 4.0 * math.pi / L ** 3 * torch.exp(-G2 / (4.0 * eta2)) / G2 * _weights(n)
    f[0, 0, 0] = 0.0
    m = torch.tensor(np.rint(np.fft.fftfreq(n) * n), device="cuda")
    mz = m[:nk]
    plans = [Plan(L, n, np.ones(n_ion), 0.3, precision=p, terms=TERMS_ALL & ~TERM_LOC) for p in ("fp32", "fp64")]
    ratio = []
    for seed in range(12):
        pos = np.random.default_rng([n, seed]).uniform(0.0, L, (n_ion, 3))
        F, Q = [], []
        for plan in plans:
            ct = torch.complex64 if plan.dtype == torch.float32 else torch.complex128
            S = torch.empty(n, n, nk, dtype=ct, device="cuda")
            plan.structure_factor(pos, S)
            F.append(plan.forces(torch.full((n ** 3,), n_ion / L ** 3, dtype=plan.dtype, device="cuda")))
            Q.append((f * S.to(torch.complex128).conj()).to(ct).to(torch.complex128))
        for I in range(n_ion):
            e = [torch.exp(-2j * math.pi * (k * (pos[I, d] / L))) for d, k in enumerate((m, m, mz))]
            P = e[0][:, None] * e[1][None, :]
            t32 = Q[0] * e[2].to(torch.complex64).to(torch.complex128)
            im = (t32 * P[:, :, None]).imag - (Q[1] * e[2] * P[:, :, None]).imag
            want = -tp * np.array([float((im * k).sum()) for k in (m[:, None, None], m[None, :, None], mz)])
            t = torch.nn.functional.pad(t32, (0, nk % 2)).reshape(n, n, -1, 2)
            k0 = 2.0 * torch.arange(t.shape[2], device="cuda")
            u1 = t[..., 1]
            u2 = u1 + t[..., 0]
            vu = u1.abs() ** 2 + u2.abs() ** 2
            row = vu.sum(-1) + t32.sum(-1).abs() ** 2 / 4.0
            z = ((k0 + 1.0) ** 2 * vu + 0.5 * (k0 * u2 + u1).abs() ** 2).sum(-1) + (t32 * mz).sum(-1).abs() ** 2 / 4.0
            var = np.array([float((row * m[:, None] ** 2).sum()), float((row * m[None, :] ** 2).sum()), float(z.sum())])
            ratio.append(((F[0][I] - F[1][I]) - want) ** 2 / (tp ** 2 * 2.0 ** -48 / 3.0 * var))
    for plan in plans:
        plan.close()
    print("mean square error over that of the roundings, x y z:", np.mean(ratio, axis=0))
    assert np.all(np.mean(ratio, axis=0) <= 1.0)
