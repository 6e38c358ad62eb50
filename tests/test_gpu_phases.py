"""Ion phases exp(-2 pi i m R / L): one sine and cosine each in FP64 plans, one rounding of
their products in FP32 plans."""
import numpy as np
import pytest
import torch

from paper_2601_23002_gb300 import Plan


def _structure(precision, n, pos):
    ct = torch.complex64 if precision == "fp32" else torch.complex128
    S = torch.empty(n, n, n // 2 + 1, dtype=ct, device="cuda")
    plan = Plan(16.0, n, np.ones(1), 0.3, precision=precision)
    out = []
    for p in pos:
        plan.structure_factor(p[None, :], S)
        out.append(S.cpu().numpy())
    plan.close()
    return out


# One ion: S on the axes is the axis phases themselves.  FP64 plans evaluate every m as
# m = 1: positions of 20 bits and L = 16 make m R / L exact, so the phase of m at R is
# that of 1 at m R (mod L), bit for bit.
@pytest.mark.gpu
@pytest.mark.parametrize("n", [27, 108, 160])
def test_fp64_phases_are_single_sines_and_cosines(n):
    pos = np.random.default_rng(n).integers(1, 1 << 20, 3) / (1 << 16)
    S = _structure("fp64", n, [pos])[0]
    h = (n - 1) // 2
    ones = _structure("fp64", n, [np.mod(m * pos, 16.0) for m in range(1, h + 1)])
    for m, one in zip(range(1, h + 1), ones):
        assert S[m, 0, 0] == one[1, 0, 0] and S[0, m, 0] == one[0, 1, 0] and S[0, 0, m] == one[0, 0, 1], m
        assert S[n - m, 0, 0] == np.conj(one[1, 0, 0])


# FP32: the kz = 0 plane of one ion's S is the product of the x and y phases, rounded to
# FP32 once: half a unit of the last place, plus 3e-14 for the pairs (48 bits: 2e-15 an
# operand, and FP32 sums of remainders of 6e-8: 4e-15 an operation).
@pytest.mark.gpu
@pytest.mark.parametrize("n", [24, 75, 128])
def test_fp32_phase_products_are_rounded_once(n):
    pos = np.random.default_rng(n).uniform(0.0, 16.0, (4, 3))
    for a, b in zip(_structure("fp32", n, pos), _structure("fp64", n, pos)):
        for x, y in ((a.real, b.real), (a.imag, b.imag)):
            x, y = x[:, :, 0], y[:, :, 0]
            half = 0.5 * np.spacing(np.abs(y).astype(np.float32)).astype(float)
            assert np.all(np.abs(x.astype(float) - y) <= half + 3e-14)
