"""Errors of the FP64 plans' fixed-point passes against the convolution in long double (quadruple
precision on the GPU hosts) on the plan's own moment table: in the 2-norm and in the maximum norm no
larger than those of the FP64 stages (WSCONV_FUSED=2) on the same densities.  Smooth bumps,
spikes (every line one value) and white noise (dense lines; biases of the rounding add up over
its lines) on runtime and compile-time lines up to the longest.
"""
import math
import os

import numpy as np
import pytest
import scipy.fft as sf
import torch

from paper_2107_03958_gb300 import inputs
from paper_2107_03958_gb300.api import ConvPlan

pytestmark = pytest.mark.gpu


def _density(n, kind):
    if kind == "noise":
        return np.random.default_rng(n).standard_normal((n, n))
    if kind == "spikes":
        u = np.zeros((n, n))
        u[n // 3, n // 5], u[n // 2, n - 2] = 0.7, -0.3
        return u
    return inputs.bump_sums(n, 1, seed=n)[0]


CASES = [(n, io, kind) for n, io in ((64, "r2r"), (240, "r2r"), (256, "r2r"), (256, "c2c"), (512, "r2c"))
         for kind in ("bumps", "spikes", "noise")] + [(1024, "r2r", "noise"), (4096, "r2r", "noise")]


@pytest.mark.parametrize("n,io,kind", CASES)
def test_errors_are_not_above_the_fp64_stages(n, io, kind, monkeypatch):
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("long double is no wider than double")
    u = _density(n, kind)
    if io == "c2c":
        u = u + 1j * u[::-1]
    kw = dict(scale=-1 / (2 * math.pi)) if io == "r2r" else dict(kappa=20.0)
    L, err = 2 * n, {}
    k = np.minimum(np.arange(L), L - np.arange(L))
    ref = None
    for fused in ("1", "2"):
        monkeypatch.setenv("WSCONV_FUSED", fused)
        p = ConvPlan("log" if io == "r2r" else "helmholtz", n=n, period=2, trunc_a=1.1, precision="fp64", io=io, **kw)
        if ref is None:
            g, w = p.ghat_quadrant(), os.cpu_count()
            if io == "r2r":
                U = sf.rfft2(u.astype(np.longdouble), (L, L), workers=w)
                ref = sf.irfft2(U * g[k], (L, L), workers=w)[:n, :n]
            else:
                U = sf.fft2(u.astype(np.clongdouble), (L, L), workers=w)
                ref = sf.ifft2(U * g[np.ix_(k, k)], workers=w)[:n, :n]
        d = np.abs(p.apply(torch.tensor(u, device="cuda")).cpu().numpy() - ref)
        err[fused] = float(np.sqrt((d ** 2).sum())), float(d.max())
    assert err["1"][0] <= err["2"][0] and err["1"][1] <= err["2"][1]
