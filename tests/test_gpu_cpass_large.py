"""The compile-time passes of FP32 grids above 160 points (planes over clusters of four and five
blocks, a three-stage even z transform at 250) in every role: preconditioning, three
fields, FP64 Fermi-Dirac inversion, forward-only; the plane pass on two-block clusters that
FP64 162^3 takes; and evaluations queued without a host round trip between them."""
import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import plan_for_cell
from workloads.cells import random_cell

from test_gpu_cpass import both, density

LARGE = [162, 225, 250]


def big_cell(n):
    cell = random_cell(7, 8, 1.0, 2.0, 0.8, n)
    cell.L *= 2.5
    cell.pos *= 2.5
    return cell


def three(monkeypatch, cell, go, **kw):
    """go(plan) of the FP64 plan, and of the FP32 plan with the compile-time and the tiled passes."""
    plan = plan_for_cell(cell, "fp64", alpha=kw.get("alpha", 0.5))
    ref = go(plan)
    plan.close()
    return ref, both(monkeypatch, cell, "fp32", go, **kw)


# Both round the psi transform (amplified by G^2) in another order: the error against
# the FP64 plan is not larger (1.5: two independent roundings).
@pytest.mark.gpu
@pytest.mark.parametrize("kw", [{"alpha": 5.0 / 6.0}, {"fd64": True}])
@pytest.mark.parametrize("n", LARGE)
def test_three_fields_and_fp64_inversion(monkeypatch, n, kw):
    cell = big_cell(n)
    rho = density(cell, torch.float32)

    def go(plan):
        r = rho.to(plan.dtype)
        v = torch.empty_like(r)
        plan.profile_enable(False)
        e = plan.energy_potential(r, v)
        return v.double(), e, set(plan.profile_read())

    (v64, e64, _), ((v1, e1, k1), (v0, e0, k0)) = three(monkeypatch, cell, go, **kw)
    assert "k_plane_c" in k1 and "k_plane_c" not in k0
    assert float((v1 - v64).norm()) <= 1.5 * float((v0 - v64).norm())
    size = max(abs(x) for x in e64.values())
    for k in e64:
        assert abs(e1[k] - e64[k]) <= max(1.5 * abs(e0[k] - e64[k]), 1e-6 * size), k


# Five L-BFGS iterations: the density's distance from the FP64 plan's, as above, or
# within FP32 rounding of it (1e-7 of the norm).
@pytest.mark.gpu
@pytest.mark.parametrize("n", LARGE)
def test_minimisation(monkeypatch, n):
    cell = big_cell(n)

    def go(plan):
        rho = torch.empty(n ** 3, dtype=plan.dtype, device="cuda")
        plan.profile_enable(False)
        plan.minimize(rho, max_iter=5)
        return rho.double(), set(plan.profile_read())

    (r64, _), ((r1, k1), (r0, k0)) = three(monkeypatch, cell, go)
    assert "k_plane_c" in k1 and "k_plane_c" not in k0
    assert float((r1 - r64).norm()) <= max(1.5 * float((r0 - r64).norm()), 1e-7 * float(r64.norm()))


# As in test_gpu_forward_views.py: sums over shells or all G of terms with 1e-7 errors.
@pytest.mark.gpu
@pytest.mark.parametrize("n", LARGE)
def test_forward_only_transforms(monkeypatch, n):
    cell = big_cell(n)
    rho = density(cell, torch.float32)
    (s1, f1, p1), (s0, f0, p0) = both(monkeypatch, cell, "fp32",
                                      lambda plan: (plan.sei_shells(rho, 40)[1], plan.forces(rho), plan.pressure(rho)))
    assert np.max(np.abs(s1 - s0)) <= 3e-6 * np.max(np.abs(s0))
    assert np.max(np.abs(f1 - f0)) <= 3e-6 * np.max(np.abs(f0))
    size = max(abs(v) for v in p0.values())
    assert all(abs(p1[k] - p0[k]) <= 3e-6 * size for k in p0)


# k_plane_prec2 is the preconditioning pass of FP64 162^3, and with OFDFT_CPASS=0 that of
# FP32 128^3; OFDFT_PREC2=0 takes the tiled chain or one block per plane there.  The FP32
# forms have one arithmetic (the same bits); the FP64 ones differ by roundings of 1e-16 in
# the preconditioned gradients, which five iterations carry to 1e-12 of the density.
@pytest.mark.gpu
@pytest.mark.parametrize("precision,n,cpass,tol", [("fp64", 162, "1", 1e-12), ("fp32", 128, "0", 0.0)])
def test_two_block_clusters(monkeypatch, precision, n, cpass, tol):
    cell = random_cell(7, 8, 1.0, 2.0, 0.8, n)
    monkeypatch.setenv("OFDFT_CPASS", cpass)
    out = []
    for v in ("1", "0"):
        monkeypatch.setenv("OFDFT_PREC2", v)
        plan = plan_for_cell(cell, precision)
        rho = torch.empty(n ** 3, dtype=plan.dtype, device="cuda")
        plan.profile_enable(False)
        plan.minimize(rho, max_iter=5)
        assert ("k_plane_prec2" in plan.profile_read()) == (v == "1")
        out.append(rho)
        plan.close()
    assert float((out[0] - out[1]).norm()) <= tol * float(out[1].norm())


# Evaluations queued one behind the other, their density rewritten on the stream in
# between, directly and as a captured graph: the bits of synchronous calls.
@pytest.mark.gpu
@pytest.mark.parametrize("precision,n", [("fp32", 16), ("fp32", 32), ("fp64", 45), ("fp32", 75), ("fp32", 162), ("fp32", 256)])
def test_queued_and_captured_evaluations(precision, n):
    cell = random_cell(7, 8, 1.0, 2.0, 0.8, n)
    plan = plan_for_cell(cell, precision)
    base = density(cell, plan.dtype)
    rhos = [base * (1.0 + 0.1 * k) for k in range(4)]
    v = torch.empty_like(base)
    want = []
    for r in rhos:
        e = plan.energy_potential(r, v)
        want.append((torch.tensor([e[k] for k in plan.ENERGY_KEYS], dtype=torch.float64), v.cpu()))

    def check(got):
        torch.cuda.synchronize()
        for (e, w), (e0, w0) in zip(got, want):
            assert torch.equal(e.cpu()[:6], e0[:6]) and torch.equal(w.cpu(), w0)

    rho, e = torch.empty_like(base), torch.empty(11, dtype=torch.float64, device="cuda")
    got = []
    for r in rhos:
        rho.copy_(r)
        plan.energy_potential_async(rho, v, e)
        got.append((e.clone(), v.clone()))
    check(got)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        plan.energy_potential_async(rho, v, e)
    got = []
    for r in rhos:
        rho.copy_(r)
        graph.replay()
        got.append((e.clone(), v.clone()))
    check(got)
    del graph
    plan.close()
