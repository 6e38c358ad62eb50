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
