"""FP64 lines of 8192 points, the longest in fixed point (n = 4096, compact): the last stage's
quarter-turn twiddle table and the twiddles read from global memory run at this length alone.  Every io
mode, with mask, alpha and beta, against the FP64 stages of the same plan (WSCONV_FUSED=2).

Tolerance: that of test_gpu_fixed.py (four transforms of at most 8192 points, each within 2.6e-16 of its
result's 2-norm, on each side, and a factor 2.5 from the 2-norm to the largest element): 5e-15.
"""
import math

import numpy as np
import pytest
import torch

from paper_2107_03958_gb300 import inputs
from paper_2107_03958_gb300.api import ConvPlan

pytestmark = pytest.mark.gpu

TOL = 5e-15


@pytest.mark.parametrize("io", ["r2r", "r2c", "c2c"])
def test_lines_of_8192_match_the_fp64_stages(io, monkeypatch):
    n = 4096
    rng = np.random.default_rng(n)
    u = torch.tensor(inputs.bump_sums(n, 1, seed=n)[0] + 1e-3 * rng.standard_normal((n, n)), device="cuda")
    if io == "c2c":
        u = torch.complex(u, u.flip(0))
    mask = torch.tensor(rng.uniform(0.0, 1.0, (n, n)), device="cuda")
    kw = dict(scale=-1 / (2 * math.pi)) if io == "r2r" else dict(kappa=9.0)
    out = {}
    for fused in ("1", "2"):
        monkeypatch.setenv("WSCONV_FUSED", fused)
        p = ConvPlan("log" if io == "r2r" else "helmholtz", n=n, period=3, precision="fp64", io=io, compact=True, **kw)
        assert (p.info.static_len == 8192) == (fused == "1")
        out[fused] = [p.apply(u), p.apply(u, mask=mask, alpha=-0.3 if io == "r2r" else 0.2 - 1.7j, beta=1.5)]
        p.device_status()
    for ref, got in zip(out["2"], out["1"]):
        assert float((got - ref).abs().max()) <= TOL * float(ref.abs().max())
