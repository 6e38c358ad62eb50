"""Performance cases of the orbital-free DFT library: what its users call, over the sizes they call it at.

A case is one operation of a `Plan` on one periodic cell:

  evaluate   energies and potential of a given density (an outer optimiser's or a
             response calculation's inner step)
  ions       new ion positions with the full structure factor S(G) written out
  forces     new ion positions and the Hellmann-Feynman forces at a density (a
             relaxation or an external molecular-dynamics driver)
  pressure   the pressure per term at a density (an equation-of-state table)
  shells     the electron-ion structure factor on |q| shells (a scattering analysis)
  minimize   L-BFGS from the uniform density, up to max_iter iterations (a snapshot,
             in one call or in slices between checkpoints)
  md         Born-Oppenheimer molecular dynamics: a cold minimisation and `steps` steps

Cells are hydrogen-like to Z = 4 at r_s of 1 to 3.2 bohr and theta = T/T_F of 0.1 to
2 on grids of 0.1 to 0.25 bohr spacing: the ranges of the workloads in
workloads/cells.py.  Ion positions and everything that follows from them come from
the seed; densities are superposed Gaussian ions over a background, as smooth and as
uneven as a minimised density of such cells.

Results that an FP32 plan hands over as Python or NumPy doubles carry FP32 accuracy;
they are returned here in the plan's own type.  The terms of an energy or a pressure
come as one vector, since a term (or their total) may vanish by cancellation.
"""
import math

import numpy as np
import torch

from paper_2601_23002_gb300 import Plan

ALL_TERMS = ("F_TF", "E_vW", "E_NL", "E_H", "E_loc", "E_xc", "E_ion")
ENERGIES = ALL_TERMS + ("F_total", "N_e", "mu", "residual")
PRESSURES = ("tf", "vw", "nl", "hartree", "loc", "xc", "ion", "total")
RC = 1.0                 # Gaussian smoothing radius of the local ion potential, bohr
PROTON = 1836.15267343   # electron masses


def _case(name, op, precision, n, n_ion, Z, rs, theta, **more):
    c = {"op": op, "precision": precision, "n": n, "n_ion": n_ion, "Z": Z, "rs": rs, "theta": theta}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the four-ion fcc-sized cell: one evaluation of a tiny grid, bound by launches and latency
        _case("evaluate_f32_n32", "evaluate", "fp32", 32, 4, 3.0, 2.06, 0.5),
        # an odd grid of the batched snapshots
        _case("evaluate_f32_n75", "evaluate", "fp32", 75, 40, 3.0, 2.3, 0.8),
        # 64 H at r_s = 2, theta = 1
        _case("evaluate_f32_n128", "evaluate", "fp32", 128, 64, 1.0, 2.0, 1.0),
        # the largest production cell, 1024 ions
        _case("evaluate_f32_n256", "evaluate", "fp32", 256, 1024, 3.0, 2.5, 0.3),
        # a hydrogen molecular-dynamics cell in full double precision (odd grid)
        _case("evaluate_f64_n45", "evaluate", "fp64", 45, 14, 1.0, 2.0, 1.0),
        # 64 H in full double precision
        _case("evaluate_f64_n128", "evaluate", "fp64", 128, 64, 1.0, 2.0, 1.0),
        # the structure factor of a served cell's new positions
        _case("ions_f32_n128", "ions", "fp32", 128, 300, 1.0, 2.6, 0.7),
        # forces of a mid-sized cell at new positions, as a relaxation calls them
        _case("forces_f32_n108", "forces", "fp32", 108, 128, 3.0, 2.2, 0.6),
        # an equation-of-state point in double precision
        _case("pressure_f64_n72", "pressure", "fp64", 72, 14, 1.0, 3.23, 1.0),
        # the scattering analysis of the largest cell
        _case("shells_f32_n256", "shells", "fp32", 256, 1024, 3.0, 2.5, 0.3, shells=200),
        # molecular dynamics of 32 H at r_s = 1 on its 30^3 grid (whole calls, small kernels)
        _case("md_f64_n30", "md", "fp64", 30, 32, 1.0, 1.0, 1.0, steps=2, dt=0.8),
        # a slice of the largest cell's minimisation (a whole call, history full)
        _case("minimize_f32_n256", "minimize", "fp32", 256, 1024, 3.0, 2.5, 0.3, max_iter=14),
    ]


def _smooth(k):
    for p in (2, 3, 5):
        while k % p == 0:
            k //= p
    return k == 1


def draw(rng):
    op = rng.choice(["evaluate"] * 8 + ["ions", "forces", "pressure", "shells", "md", "minimize", "minimize"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if op == "md":
        precision = "fp64"
    if op == "minimize":
        precision = "fp32"
    top = {"md": 72, "minimize": 160}.get(op, 256 if precision == "fp32" else 144)
    grids = [k for k in range(30, top + 1) if _smooth(k)]
    want = math.exp(rng.uniform(math.log(30), math.log(top)))
    n = min(grids, key=lambda k: abs(math.log(k / want)))
    Z = float(rng.choice([1, 1, 3, 4]))
    spacing = rng.uniform(0.2, 0.25)
    vol = (n * spacing) ** 3
    rs = rng.uniform(1.5, 3.0)
    n_ion = int(round(vol / (Z * 4.0 * math.pi / 3.0 * rs ** 3)))
    n_ion = max(2, min(1024, n_ion))
    rs = (vol / (n_ion * Z * 4.0 * math.pi / 3.0)) ** (1.0 / 3.0)
    more = {}
    if op == "evaluate":
        kind = rng.random()
        if kind < 0.08 and precision == "fp32":
            more["fd64"] = True                       # FP64 Fermi-Dirac inversion in an FP32 plan
        elif kind < 0.16 and Z == 1.0:
            more["alpha"] = 5.0 / 6.0                 # Wang-Teter exponent (three transformed fields)
    if op == "shells":
        more["shells"] = rng.choice([40, 100, 200])
    if op == "md":
        more.update(steps=rng.choice([1, 2]), dt=4.0)
    if op == "minimize":
        more["max_iter"] = rng.choice([6, 10, 14])
    return _case(None, op, precision, n, n_ion, Z, round(rs, 4), round(rng.uniform(0.1, 2.0), 3), **more)


# --------------------------------------------------------------------------- inputs

def _side(case):
    return (case["n_ion"] * case["Z"] * 4.0 * math.pi / 3.0 * case["rs"] ** 3) ** (1.0 / 3.0)


def _temperature(case):
    nbar = case["n_ion"] * case["Z"] / _side(case) ** 3
    return case["theta"] * 0.5 * (3.0 * math.pi ** 2 * nbar) ** (2.0 / 3.0)


def _positions(case, seed):
    """Uniform positions with a hard core, as a liquid's."""
    rng = np.random.default_rng([int(seed), case["n"], case["n_ion"]])
    L, ni = _side(case), case["n_ion"]
    core = min(0.8, 0.6 * case["rs"] * case["Z"] ** (1.0 / 3.0))
    pos = np.zeros((ni, 3))
    k = 0
    while k < ni:
        p = rng.uniform(0.0, L, size=3)
        d = pos[:k] - p
        d -= L * np.round(d / L)
        if k and np.min(np.einsum("ij,ij->i", d, d)) < core * core:
            continue
        pos[k] = p
        k += 1
    return pos


def _waves(n, device):
    """Integer wave numbers in FFT order: m = -n/2 .. n/2 - 1, odd n symmetric."""
    return torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=device).round()


def _phases(pos, L, m):
    """exp(-2 pi i m R_d / L) per axis d: three [n_ion, len(m)] complex128."""
    a = torch.as_tensor(pos, dtype=torch.float64, device=m.device) / L
    f = a[:, :, None] * m[None, None, :]
    f = f - f.round()
    return torch.polar(torch.ones_like(f), -2.0 * math.pi * f).unbind(1)


def _density(case, pos, dtype):
    """Gaussian ions over a background of 30%, normalised to N_e, on the GPU.  Range and gradient
    energy are those of minimised densities: 0.3 to 3.5 nbar and E_vW/N_e = 0.025 Ha for 64 H at
    r_s = 2 (0.022 minimised), 0.145 Ha for Z = 3 at r_s = 2.5 (0.145 minimised)."""
    n, L = case["n"], _side(case)
    m = _waves(n, "cuda")
    h = n // 2 + 1
    S = _structure(pos, n, L, True)
    m2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :h] ** 2
    width = 1.7 if case["Z"] == 1.0 else 1.45
    S *= torch.exp(-0.25 * (2.0 * math.pi / L * width) ** 2 * m2)
    rho = torch.fft.irfftn(S, s=(n, n, n))
    nbar = case["n_ion"] * case["Z"] / L ** 3
    rho = nbar * (0.3 + 0.7 * rho / rho.mean())
    rho.clamp_(min=1e-4 * nbar)
    rho *= nbar / rho.mean()
    return rho.to(dtype).reshape(-1).contiguous()


def prepare(case, seed):
    single = case["precision"] == "fp32"
    dtype = torch.float32 if single else torch.float64
    n, L = case["n"], _side(case)
    pos = _positions(case, seed)
    plan = Plan(L, n, np.full(case["n_ion"], case["Z"]), _temperature(case), rc=RC, precision=case["precision"],
                alpha=case.get("alpha", 0.5), fd64=case.get("fd64", False))
    plan.structure_factor(pos)
    s = {"op": case["op"], "plan": plan, "pos": pos, "case": dict(case), "host": np.float32 if single else np.float64}
    if case["op"] in ("evaluate", "forces", "pressure", "shells"):
        s["rho"] = _density(case, pos, dtype)
    if case["op"] == "evaluate":
        s["v"] = torch.empty_like(s["rho"])
    if case["op"] == "ions":
        s["S"] = torch.empty(n, n, n // 2 + 1, dtype=torch.complex64 if single else torch.complex128, device="cuda")
    if case["op"] in ("minimize", "md"):
        s["rho"] = torch.empty(n ** 3, dtype=dtype, device="cuda")
    if case["op"] == "md":
        rng = np.random.default_rng([int(seed), 77])
        mass = np.full(case["n_ion"], case["Z"] * PROTON)
        T = _temperature(case)
        vel = rng.normal(size=(case["n_ion"], 3)) * np.sqrt(T / mass)[:, None]
        s.update(mass=mass, T=T, vel=vel - vel.mean(axis=0))
    return s


def run(state):
    plan, case, op = state["plan"], state["case"], state["op"]
    if op == "evaluate":
        e = plan.energy_potential(state["rho"], state["v"])
        return {"energies": np.array([e[k] for k in ENERGIES], state["host"]), "v": state["v"]}
    if op == "ions":
        plan.structure_factor(state["pos"], state["S"])
        return state["S"]
    if op == "forces":
        plan.structure_factor(state["pos"])
        return plan.forces(state["rho"]).astype(state["host"])
    if op == "pressure":
        p = plan.pressure(state["rho"])
        return np.array([p[k] for k in PRESSURES], state["host"])
    if op == "shells":
        q, s = plan.sei_shells(state["rho"], case["shells"])
        return {"q": q, "s": s.astype(state["host"])}
    if op == "minimize":
        r = plan.minimize(state["rho"], start_uniform=True, max_iter=case["max_iter"])
        return {"rho": state["rho"], "energies": np.array([r[k] for k in ALL_TERMS + ("F_total", "mu")], state["host"])}
    r = plan.md_run(state["rho"], state["pos"], state["vel"], state["mass"], case["steps"], case["dt"],
                    T_ion=state["T"], tau=100.0 * case["dt"], start_uniform=True)
    return {"rho": state["rho"], "pos": r["pos"], "vel": r["vel"],
            "e_pot": r["frames"]["e_pot"], "conserved": r["frames"]["conserved"]}


def work(case):
    """Bytes: the inputs and outputs of the operation once (a minimisation's iteration also has its
    own vectors to read and write: psi, d, g and the pairs of the history).  Flops: the real
    transforms of the density and of sqrt(n) and back, and the pointwise functional."""
    N, w = float(case["n"]) ** 3, 4.0 if case["precision"] == "fp32" else 8.0
    ni = float(case["n_ion"])
    fft = 2.5 * N * math.log2(N)
    fields = 3 if case.get("alpha", 0.5) != 0.5 else 2
    point = 150.0 * N
    ev = {"bytes": 2.0 * N * w, "flops": 2.0 * fields * fft + point}
    L = _side(case)
    # wave vectors inside the local potential's Gaussian range, half spectrum
    ng = min(0.5 * N, 0.5 * 4.0 * math.pi / 3.0 * (math.sqrt(83.0 if w == 4.0 else 156.0) * L / (2.0 * math.pi)) ** 3)
    ions = 8.0 * ni * ng
    op = case["op"]
    if op == "evaluate":
        return ev
    if op == "ions":
        return {"bytes": N * w, "flops": 4.0 * ni * N}
    if op == "forces":
        return {"bytes": N * w, "flops": fft + ions + 20.0 * ni * ng}
    if op == "pressure":
        return {"bytes": N * w, "flops": 2.0 * fft + 2.0 * point}
    if op == "shells":
        return {"bytes": N * w, "flops": fft}
    if op == "minimize":
        it = case["max_iter"]
        pairs = sum(min(k, 8) for k in range(it))
        return {"bytes": (12.0 * it + 4.0 * pairs) * N * w, "flops": (it + 1) * (ev["flops"] + 2.0 * fft) + 16.0 * pairs * N}
    evals = 10.0 + 8.0 * case["steps"]
    return {"bytes": evals * 12.0 * N * w, "flops": evals * (ev["flops"] + 2.0 * fft) + case["steps"] * 30.0 * ni * ng}


# --------------------------------------------------------------------------- in 64 bits

def _fermi(eta, three_half=False, chunk=1 << 21):
    """(I_1/2, dI_1/2/deta[, I_3/2]) by the trapezoidal rule in t = sqrt(x): the integrands are even
    and analytic in a strip of half-width Im sqrt(eta + i pi), so the rule converges geometrically."""
    top = max(float(eta.max()), 0.0)
    d = (complex(top, math.pi) ** 0.5).imag
    h = 2.0 * math.pi * d / 42.0
    nodes = int(math.sqrt(top + 44.0) / h) + 1
    out = [torch.zeros_like(eta) for _ in range(3 if three_half else 2)]
    for a in range(0, eta.numel(), chunk):
        e = eta[a:a + chunk]
        acc = [torch.zeros_like(e) for _ in out]
        for k in range(nodes + 1):
            t2 = (k * h) ** 2
            f = torch.sigmoid(e - t2)
            acc[0].add_(f, alpha=2.0 * h * t2)
            acc[1].add_(f, alpha=h if k else 0.5 * h)
            if three_half:
                acc[2].add_(f, alpha=2.0 * h * t2 * t2)
        for o, v in zip(out, acc):
            o[a:a + chunk] = v
    return out


def _inverse_fermi(y):
    """eta with I_1/2(eta) = y, Newton on the logarithm."""
    u = y / math.gamma(1.5)
    eta = torch.where(y < 1.0, torch.log(u) + u / math.sqrt(8.0), (1.5 * y) ** (2.0 / 3.0))
    for _ in range(20):
        i, di = _fermi(eta)
        step = (torch.log(i) - torch.log(y)) * i / di
        eta = eta - step
        if float(step.abs().max()) < 1e-13 * max(1.0, float(eta.abs().max())):
            break
    return eta


def _xc(n):
    """Perdew-Zunger 1981, unpolarised; B and D from the continuity of e_c and de_c/dr_s at r_s = 1."""
    g, b1, b2, A, C = -0.1423, 1.0529, 0.3334, 0.0311, 0.0020
    den1 = 1.0 + b1 + b2
    D = -g * (0.5 * b1 + b2) / den1 ** 2 - A - C
    B = g / den1 - D
    rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    ex = -0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * n ** (1.0 / 3.0)
    sq = rs.sqrt()
    den = 1.0 + b1 * sq + b2 * rs
    lo = rs >= 1.0
    ln = torch.log(rs)
    ec = torch.where(lo, g / den, A * ln + B + C * rs * ln + D * rs)
    dec = torch.where(lo, -g * (0.5 * b1 / sq + b2) / den ** 2, A / rs + C * ln + C + D)
    return ex + ec, 4.0 / 3.0 * ex + ec - rs / 3.0 * dec


def _mean_density(nbar, T):
    y = torch.tensor([math.pi ** 2 * nbar / (math.sqrt(2.0) * T ** 1.5)], dtype=torch.float64, device="cuda")
    eta = _inverse_fermi(y)
    return T * float(eta), math.pi ** 2 / (math.sqrt(2.0 * T) * float(_fermi(eta)[1]))


def _kernel(L, nbar, T, alpha, m2, chunk=4096):
    """K on the integers m2 from the finite-temperature Lindhard function, by tanh-sinh quadrature on
    both sides of its logarithmic singularity k = q/2."""
    mu, dmu = _mean_density(nbar, T)
    kmax = math.sqrt(2.0 * max(mu + 45.0 * T, 45.0 * T))
    u = torch.linspace(-4.0, 4.0, 1601, dtype=torch.float64, device="cuda")
    s = 0.5 * math.pi * torch.sinh(u)
    near = 1.0 / (1.0 + torch.exp(2.0 * s))              # (1 - tanh)/2: distance to the upper end
    far = 1.0 / (1.0 + torch.exp(-2.0 * s))
    wgt = 0.25 * math.pi * torch.cosh(u) / torch.cosh(s) ** 2 * float(u[1] - u[0])
    out = []
    for q in (2.0 * math.pi / L * torch.sqrt(m2.to(torch.float64))).split(chunk):
        q = q[:, None].clamp(min=1e-300)
        c = 0.5 * q
        b = c.clamp(max=kmax)

        def part(k, dist, width):
            """k f(k) [ln|(2k+q)/(2k-q)| - 4k/q] with |k - q/2| = dist."""
            x = k / c
            small = x < 0.05
            ser = 2.0 * x ** 3 * (1 / 3 + x ** 2 * (1 / 5 + x ** 2 * (1 / 7 + x ** 2 * (1 / 9 + x ** 2 * (1 / 11 + x ** 2 / 13)))))
            e = torch.where(small, ser, torch.log((k + c) / dist.clamp(min=1e-300)) - 2.0 * x)
            return (k * torch.sigmoid((mu - 0.5 * k * k) / T) * e * wgt * width).sum(dim=1)

        tot = part(b * far, (c - b) + b * near, b)
        w = (kmax - c).clamp(min=0.0)
        tot = tot + part(c + w * far, w * far, w)
        q = q[:, 0]
        eps = tot * q / (4.0 * math.pi ** 2 * nbar)
        out.append(-q * q / (4.0 * nbar) * eps / (1.0 + eps))
    K = (torch.cat(out) - dmu) / (2.0 * alpha ** 2 * nbar ** (2.0 * alpha - 2.0))
    return torch.where(m2 == 0, torch.zeros_like(K), K)


def _spectrum(f):
    return torch.fft.fftn(f) / f.numel()


def _m2(n):
    m = _waves(n, "cuda")
    return m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2


def _structure(pos, n, L, half):
    m = _waves(n, "cuda")
    ex, ey, ez = _phases(pos, L, m)
    ez = ez[:, :n // 2 + 1] if half else ez
    S = torch.empty(n, n, ez.shape[1], dtype=torch.complex128, device="cuda")
    for a in range(0, n, 16):
        S[a:a + 16] = (torch.einsum("ia,ib->abi", ex[:, a:a + 16], ey).reshape(-1, len(pos)) @ ez).reshape(-1, n, ez.shape[1])
    return S


def _vloc(case, pos):
    """V_loc(G) on the full grid."""
    n, L, Z = case["n"], _side(case), case["Z"]
    G2 = (2.0 * math.pi / L) ** 2 * _m2(n)
    G2[0, 0, 0] = 1.0
    vt = -4.0 * math.pi * Z * torch.exp(-0.25 * RC * RC * G2) / G2
    vt[0, 0, 0] = math.pi * Z * RC * RC
    return vt * _structure(pos, n, L, False) / L ** 3


def _ewald(case, pos):
    """Ewald energy and forces; the splitting puts the real-space range at half the cell."""
    L, Z = _side(case), case["Z"]
    Om, eta = L ** 3, 12.4 / L
    x = torch.as_tensor(pos, dtype=torch.float64, device="cuda")
    d = x[:, None, :] - x[None, :, :]
    d = d - L * (d / L).round()
    r = d.norm(dim=2)
    own = torch.eye(len(pos), dtype=torch.bool, device="cuda")
    r = torch.where(own, torch.full_like(r, 1e3 * L), r)
    er = torch.erfc(eta * r) / r
    e = 0.5 * Z * Z * float(er.sum())
    f = Z * Z * (((er + 2.0 * eta / math.sqrt(math.pi) * torch.exp(-(eta * r) ** 2)) / (r * r))[:, :, None] * d).sum(dim=1)
    mm = int(math.ceil(2.0 * eta * 6.3 * L / (2.0 * math.pi)))
    m = torch.arange(-mm, mm + 1, dtype=torch.float64, device="cuda")
    ex, ey, ez = _phases(pos, L, m)
    A = (torch.einsum("ia,ib->abi", ex, ey).reshape(-1, len(pos)) @ ez).reshape(len(m), len(m), len(m)) * Z
    G2 = (2.0 * math.pi / L) ** 2 * (m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2)
    G2[mm, mm, mm] = 1.0
    w = torch.exp(-G2 / (4.0 * eta * eta)) / G2
    w[mm, mm, mm] = 0.0
    e += 2.0 * math.pi / Om * float((w * A.abs() ** 2).sum())
    f = f + 4.0 * math.pi / Om * Z * _moment(w * A.conj(), (ex, ey, ez), m * (2.0 * math.pi / L)) * -1.0
    ne = case["n_ion"] * Z
    e += -eta / math.sqrt(math.pi) * case["n_ion"] * Z * Z - math.pi * ne * ne / (2.0 * Om * eta * eta)
    return e, f


def _moment(W, phases, G):
    """sum_G G Im[W(G) exp(-i G.R_I)] per ion."""
    ex, ey, ez = phases
    na, nb, nc = W.shape
    plain = (W.reshape(-1, nc) @ ez.T).reshape(na, nb, -1)
    alongz = ((W * G).reshape(-1, nc) @ ez.T).reshape(na, nb, -1)
    fx = torch.einsum("abi,ib->ai", plain, ey)
    fy = torch.einsum("abi,ib->ai", plain, ey * G)
    fz = torch.einsum("abi,ib->ai", alongz, ey)
    return torch.stack([torch.einsum("ai,ia->i", fx, ex * G), torch.einsum("ai,ia->i", fy, ex),
                        torch.einsum("ai,ia->i", fz, ex)], dim=1).imag


def _evaluate(case, pos, rho):
    """Energies and potential in 64 bits; rho [n, n, n]."""
    n, L, T, a = case["n"], _side(case), _temperature(case), case.get("alpha", 0.5)
    Om, N = L ** 3, float(n) ** 3
    dV = Om / N
    nbar = case["n_ion"] * case["Z"] / Om
    nf = rho.clamp(min=1e-20)
    y = (math.pi ** 2 / (math.sqrt(2.0) * T ** 1.5)) * nf.reshape(-1)
    eta = _inverse_fermi(y)
    p = (2.0 / 3.0) * _fermi(eta, True)[2] / y
    eta, p = eta.reshape(rho.shape), p.reshape(rho.shape)
    e = {"F_TF": dV * float((nf * T * (eta - p)).sum())}
    exc, vxc = _xc(nf)
    e["E_xc"] = dV * float((rho * exc).sum())
    v = T * eta + vxc
    ptf, pxc = float((nf * T * p).sum()) / N, float((rho * (vxc - exc)).sum()) / N
    del eta, p, exc, vxc, y
    m2 = _m2(n)
    G2 = (2.0 * math.pi / L) ** 2 * m2
    cou = 4.0 * math.pi / torch.where(m2 > 0, G2, torch.full_like(G2, math.inf))
    nt = _spectrum(rho)
    Vl = _vloc(case, pos)
    e["E_H"] = 0.5 * Om * float((cou * nt.abs() ** 2).sum())
    e["E_loc"] = Om * float((nt.conj() * Vl).real.sum())
    cl = 1.0 - 0.5 * RC * RC * G2
    cl[0, 0, 0] = 3.0
    ploc = float(((nt.conj() * Vl).real * cl).sum()) / 3.0
    v += torch.fft.ifftn(cou * nt + Vl).real * N
    del Vl, cou, cl
    mi = m2.to(torch.int64)
    values = torch.arange(int(mi.max()) + 1, device="cuda")
    K = _kernel(L, nbar, T, a, values)
    na = nf ** a
    nat = _spectrum(na)
    e["E_NL"] = Om * float((K[mi] * nat.abs() ** 2).sum())
    v += 2.0 * a * nf ** (a - 1.0) * torch.fft.ifftn(K[mi] * nat).real * N
    phi = rho.clamp(min=0.0).sqrt()
    pt = _spectrum(phi)
    e["E_vW"] = 0.5 * Om * float((G2 * pt.abs() ** 2).sum())
    v += torch.fft.ifftn(G2 * pt).real * N / (2.0 * phi.clamp(min=1e-10))
    e["E_ion"], _ = _ewald(case, pos)
    e["F_total"] = sum(e[k] for k in ALL_TERMS)
    e["N_e"] = dV * float(rho.sum())
    e["mu"] = dV * float((v * rho).sum()) / e["N_e"]
    e["residual"] = math.sqrt(dV * float((rho * (v - e["mu"]) ** 2).sum()) / e["N_e"])
    return e, v, {"tf": ptf, "xc": pxc, "loc": ploc, "nat": nat, "K": K, "mi": mi}


def exact(case, seed):
    op, n, L = case["op"], case["n"], _side(case)
    if op in ("minimize", "md"):
        return None                     # where an iteration ends is not a value that 64 bits fix
    pos = _positions(case, seed)
    if op == "ions":
        return _structure(pos, n, L, True)
    dtype = torch.float32 if case["precision"] == "fp32" else torch.float64
    rho = _density(case, pos, dtype).to(torch.float64).reshape(n, n, n)
    if op == "evaluate":
        e, v, _ = _evaluate(case, pos, rho)
        return {"energies": np.array([e[k] for k in ENERGIES]), "v": v.reshape(-1)}
    if op == "forces":
        # only |G| inside the Gaussian's range: m up to 14 bohr^-1
        mm = min((n - 1) // 2, int(math.ceil(14.0 * L / (2.0 * math.pi))))
        m = torch.arange(-mm, mm + 1, dtype=torch.float64, device="cuda")
        at = m.to(torch.int64) % n
        nt = _spectrum(rho)[at][:, at][:, :, at]
        G2 = (2.0 * math.pi / L) ** 2 * (m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2)
        G2[mm, mm, mm] = 1.0
        vt = -4.0 * math.pi * case["Z"] * torch.exp(-0.25 * RC * RC * G2) / G2
        vt[mm, mm, mm] = 0.0
        f = -_moment(vt * nt.conj(), _phases(pos, L, m), m * (2.0 * math.pi / L)) + _ewald(case, pos)[1]
        return f.cpu().numpy()
    if op == "shells":
        # the first 200 shells end at |m|^2 = 241; even grids have m = -n/2 but not n/2
        m = torch.arange(-min(n // 2, 24), min((n - 1) // 2, 24) + 1, dtype=torch.float64, device="cuda")
        at = m.to(torch.int64) % n
        nt = _spectrum(rho)[at][:, at][:, :, at] * L ** 3
        ex, ey, ez = _phases(pos, L, m)
        S = (torch.einsum("ia,ib->abi", ex, ey).reshape(-1, len(pos)) @ ez).reshape(nt.shape)
        m2 = (m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2).to(torch.int64).reshape(-1)
        tot = torch.zeros(int(m2.max()) + 1, dtype=torch.float64, device="cuda")
        cnt = torch.zeros_like(tot)
        tot.index_add_(0, m2, (nt * S.conj()).real.reshape(-1))
        cnt.index_add_(0, m2, torch.ones_like(m2, dtype=torch.float64))
        there = torch.nonzero(cnt).reshape(-1)
        there = there[there > 0][:case["shells"]]
        s = tot[there] / cnt[there] / math.sqrt(case["n_ion"] * case["Z"] * case["n_ion"])
        return {"q": (2.0 * math.pi / L * there.to(torch.float64).sqrt()).cpu().numpy(), "s": s.cpu().numpy()}
    # pressure: -dF/dOmega under a dilation at fixed T and N_e, term by term
    e, _, x = _evaluate(case, pos, rho)
    Om, T, a = L ** 3, _temperature(case), case.get("alpha", 0.5)
    nbar = case["n_ion"] * case["Z"] / Om
    values = torch.arange(x["K"].numel(), device="cuda")

    def central(h):
        up, down = (_kernel(L * g, nbar / g ** 3, T, a, values) for g in (1.0 + h, 1.0 - h))
        return (up - down) / (2.0 * h)

    dK = (4.0 * central(1e-3) - central(2e-3)) / 3.0
    w2 = x["nat"].abs() ** 2
    p = {"tf": x["tf"], "xc": x["xc"], "loc": x["loc"], "vw": 2.0 * e["E_vW"] / (3.0 * Om),
         "hartree": e["E_H"] / (3.0 * Om), "ion": e["E_ion"] / (3.0 * Om),
         "nl": -float((w2 * ((3.0 - 6.0 * a) * x["K"] + dK)[x["mi"]]).sum()) / 3.0}
    p["total"] = sum(p.values())
    return np.array([p[k] for k in PRESSURES])
