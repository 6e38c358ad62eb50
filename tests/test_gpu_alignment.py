"""Caller's buffers aligned to single values only: what an allocator of C doubles or a
slice of a longer array gives.  The results are those of aligned buffers."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import Plan
from paper_2601_23002_gb300.api import _check


# S(G) is written whole by the kernel or copied from the plan's: the same bytes.
@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("n", [8, 27, 64])
def test_structure_factor_at_a_single_values_alignment(n, two, precision):
    L, n_ion = 0.25 * n, 7
    pos = np.random.default_rng(n).uniform(0.0, L, (n_ion, 3))
    Z = np.ones(n_ion)
    if two:
        Z[::2] = 3.0
    real = torch.float32 if precision == "fp32" else torch.float64
    cnt = 2 * n * n * (n // 2 + 1)
    got = []
    for shift in (0, 1):
        buf = torch.zeros(cnt + 2, dtype=real, device="cuda")
        plan = Plan(L, n, Z, 0.3, precision=precision)
        ptr = ctypes.c_void_p(buf.data_ptr() + shift * buf.element_size())
        host = ctypes.c_void_p(np.ascontiguousarray(pos).ctypes.data)
        _check(plan.lib.ofdft_structure_factor(plan._p, host, 0, ptr, torch.cuda.current_stream().cuda_stream))
        rho = torch.full((n ** 3,), float(Z.sum()) / L ** 3, dtype=real, device="cuda")
        got.append((buf[shift:shift + cnt].clone(), plan.energy_potential(rho)["E_ion"]))
        assert float(buf[shift + cnt:].abs().max()) == 0.0 and float(buf[:shift].sum()) == 0.0
        plan.close()
    assert torch.equal(got[0][0], got[1][0]) and float(got[0][0].abs().max()) > 0.5
    assert got[0][1] == got[1][1]


def _density(n, nbar, dtype, shift):
    """A smooth density whose first value lies `shift` values into an aligned buffer."""
    x = np.arange(n) * (2 * np.pi / n)
    rho = 1.0 + 0.3 * np.cos(x)[:, None, None] * np.cos(2 * x)[None, :, None] + 0.2 * np.sin(x)[None, None, :]
    buf = torch.empty(n ** 3 + shift, dtype=dtype, device="cuda")[shift:]
    buf.copy_(torch.tensor(rho * nbar, dtype=dtype).reshape(-1))
    return buf


def _cell(n):
    L, n_ion = 0.22 * n, 8
    return L, np.ones(n_ion), np.random.default_rng(n).uniform(0.0, L, (n_ion, 3))


# Grids of the generic plane pass (16), the compile-time passes (75, 128, 162), the
# 256^3 passes and the tiled chain (270), and a tile schedule that takes the generic z
# passes: an unaligned density, and an unaligned potential.  Where another forward pass reads
# it (even compile-time grids, 256^3) the transforms round differently, and the
# potential is no further from the FP64 plan's (1.5: two independent roundings);
# elsewhere the same kernels run.
@pytest.mark.gpu
@pytest.mark.parametrize("n,tiles", [(16, None), (75, None), (75, (32, 16, 16)), (128, None), (128, (8, 16, 16)), (162, None),
                                     (256, None), (270, None)])
def test_fp32_density_at_a_single_values_alignment(n, tiles):
    L, Z, pos = _cell(n)
    got = {}
    for key, precision, shift in (("fp64", "fp64", 0), ("aligned", "fp32", 0), ("off", "fp32", 1)):
        plan = Plan(L, n, Z, 0.3, precision=precision)
        plan.structure_factor(pos)
        if tiles and precision == "fp32":
            plan.set_tiles(tiles)
        rho = _density(n, len(Z) / L ** 3, torch.float32, shift)
        if precision == "fp64":
            rho = rho.double()
        v = torch.empty(n ** 3 + shift, dtype=plan.dtype, device="cuda")[shift:]
        e = plan.energy_potential(rho, v)
        got[key] = (v.double(), e, plan.sei_shells(rho, 20)[1], plan.forces(rho), plan.pressure(rho))
        plan.close()
    v64 = got["fp64"][0]
    err = {k: float((got[k][0] - v64).norm() / v64.norm()) for k in ("aligned", "off")}
    assert err["off"] <= 1.5 * err["aligned"]
    if tiles or n in (16, 75, 270):
        assert torch.equal(got["off"][0], got["aligned"][0])
    size = max(abs(x) for x in got["fp64"][1].values())
    for k, x in got["aligned"][1].items():
        assert abs(got["off"][1][k] - x) <= 1e-6 * size, k
    # sums over shells or all G of terms with 1e-7 errors
    for i in (2, 3):
        assert np.max(np.abs(got["off"][i] - got["aligned"][i])) <= 3e-6 * np.max(np.abs(got["aligned"][i]))
    size = max(abs(x) for x in got["aligned"][4].values())
    assert all(abs(got["off"][4][k] - x) <= 3e-6 * size for k, x in got["aligned"][4].items())


# The minimiser reads and writes the caller's density, single values at a time.
@pytest.mark.gpu
@pytest.mark.parametrize("n", [16, 75, 128])
def test_minimisation_of_a_density_at_a_single_values_alignment(n):
    L, Z, pos = _cell(n)
    got = []
    for shift in (0, 1):
        plan = Plan(L, n, Z, 0.3, precision="fp32")
        plan.structure_factor(pos)
        rho = _density(n, len(Z) / L ** 3, torch.float32, shift)
        plan.minimize(rho, start_uniform=False, max_iter=4)
        got.append(rho.clone())
        plan.close()
    assert torch.equal(got[0], got[1])
