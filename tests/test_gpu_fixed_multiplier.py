"""Complex multiplier entries whose imaginary part, as the 62-bit integer of the FP64 plans' column
pass, has the low half 0x80000000: a 32-bit value that is its own negation.  One entry in 2^23 is of
that form; here the kernel's scale is chosen so that a low-frequency entry is, with the imaginary
part's exponent at or below the real part's (then the integer is shifted first), in both signs, and
the plan is applied to that frequency's plane wave.

Tolerance: that of test_gpu_fixed.py (four transforms of at most 8192 points, each within 2.6e-16 of its
result's 2-norm, on each side, and a factor 2.5 from the 2-norm to the largest element): 5e-15.
"""
import numpy as np
import pytest
import torch

from paper_2107_03958_gb300.api import ConvPlan

pytestmark = pytest.mark.gpu

TOL = 5e-15


def _bits(x):
    return int(np.float64(abs(x)).view(np.uint64))


def _shift(g):
    """By how much the imaginary part's integer moves down to the entry's common exponent."""
    return max(0, (_bits(g.real) >> 52) - (_bits(g.imag) >> 52))


def _low_half_is_own_negation(g):
    m = ((_bits(g.imag) & ((1 << 52) - 1)) | (1 << 52)) << 9
    return (m >> _shift(g)) & 0xffffffff == 0x80000000


def _scale_for(g1, shifted):
    """A factor s near 1.3 for which the entry s g1 is of that form, shifted or not; None: there is none."""
    if g1.imag == 0.0:
        return None
    for d in range(30):
        width = 23 + d
        t = ((_bits(1.3 * g1.imag) >> width) << width) | (1 << (width - 1))
        for i in range(64):
            want = np.uint64(t + (i << width)).view(np.float64)
            s = want / abs(g1.imag)
            g = complex(s * g1.real, s * g1.imag)
            if _low_half_is_own_negation(g) and (_shift(g) > 0) == shifted:
                return float(s)
    return None


@pytest.mark.parametrize("n,period", [(64, 3), (256, 2), (512, 2)])  # runtime and compile-time lines
@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_multiplier_whose_low_half_is_its_own_negation(n, period, shifted, sign):
    def plan(scale):
        return ConvPlan("helmholtz", n=n, period=period, trunc_a=1.1 if period == 2 else 0.0, kappa=9.0, precision="fp64",
                        io="c2c", scale=scale)

    g1 = plan(1.0).ghat_quadrant()
    k2, k1 = next((i, j) for i in range(1, 12) for j in range(i, 12)
                  if _scale_for(g1[i, j], shifted))
    p = plan(sign * _scale_for(g1[k2, k1], shifted))
    g = p.ghat_quadrant()
    assert _low_half_is_own_negation(g[k2, k1])
    j = np.arange(n)
    u = (0.6 + 0.8j) * np.outer(np.exp(2j * np.pi * k1 * j / p.M), np.exp(2j * np.pi * k2 * j / p.M))
    k = np.minimum(np.arange(p.M), p.M - np.arange(p.M))
    ref = np.fft.ifft2(g[np.ix_(k, k)] * np.fft.fft2(u, (p.M, p.M)))[:n, :n]
    out = p.apply(torch.tensor(u, device="cuda")).cpu().numpy()
    assert np.max(np.abs(out - ref)) <= TOL * np.max(np.abs(ref))
