"""FP64 plans' fixed-point passes (passes_fixed.cu) against the FP64 runtime-stage passes of the same
plan (WSCONV_FUSED=2 or 0) and the CPU oracle, at the edges of what they take: the shortest and longest
lines, one warp and several per line, every radix, odd n, each io mode, masks, alpha and beta, and
inputs of extreme size.

Tolerance: four transforms of at most 8192 points, each within 2.6e-16 of its result's 2-norm (the
error of FP64 transforms of that length), plus the other side's: 8 x 2.6e-16, and a factor 2.5 from
the 2-norm to the largest element: 5e-15.
"""
import ctypes
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2107_03958_gb300 import _native, inputs
from paper_2107_03958_gb300._native import ConvError
from paper_2107_03958_gb300.api import ConvPlan, multi_workspace_bytes

pytestmark = pytest.mark.gpu

TOL = 5e-15


def _plan(n, period, compact, io, batch=1):
    a = 1.1 if period == 2 else 0.0
    kw = dict(kappa=9.0) if io != "r2r" else dict(scale=-1 / (2 * math.pi))
    return ConvPlan("helmholtz" if io != "r2r" else "log", n=n, period=period, trunc_a=a, precision="fp64", io=io,
                    compact=compact, batch_max=batch, **kw)


def _table(plan):
    """The plan's own moment table on the whole M x M frequency grid, so that a comparison sees the
    transforms alone."""
    k = np.minimum(np.arange(plan.M), plan.M - np.arange(plan.M))
    return plan.ghat_quadrant()[np.ix_(k, k)]


def _apply(plan, u, **kw):
    return plan.apply(torch.tensor(u, device="cuda"), **kw).cpu().numpy()


def _err(ref, got):
    return float(np.max(np.abs(ref - got)) / np.max(np.abs(ref)))


# L = 32 and 48 (shortest), 450 (every odd radix), 512 (compile-time, one warp), 768, 960, 1250 (odd n),
# 1024 ... 4096 (compile-time, several warps), 6144 (longest of the runtime lengths' two buffers)
SHAPES = [(16, 2, False), (16, 3, False), (225, 2, False), (256, 3, True), (256, 3, False), (320, 3, False),
          (625, 2, False), (512, 2, False), (1024, 3, True), (2048, 2, False), (2048, 3, False)]


@pytest.mark.parametrize("io", ["r2r", "r2c", "c2c"])
@pytest.mark.parametrize("n,period,compact", SHAPES)
def test_fixed_point_passes_match_the_fp64_stages(n, period, compact, io, monkeypatch):
    B = 3 if n < 1000 else 1
    u = inputs.bump_sums(n, B, seed=n)
    rng = np.random.default_rng(n)
    u[0] += 1e-3 * rng.standard_normal((n, n))
    if io == "c2c":
        u = u + 1j * u[:, ::-1]
    mask = torch.tensor(rng.uniform(0.0, 1.0, (n, n)), device="cuda")
    out = {}
    for fused in ("1", "2"):
        monkeypatch.setenv("WSCONV_FUSED", fused)
        p = _plan(n, period, compact, io, B)
        out[fused] = [_apply(p, u), _apply(p, u, mask=mask, alpha=-0.3 if io == "r2r" else 0.2 - 1.7j, beta=1.5)]
        p.device_status()
    for ref, got in zip(out["2"], out["1"]):
        for i in range(B):
            assert _err(ref[i], got[i]) <= TOL


@pytest.mark.parametrize("scale", [2.0 ** -1015, 1e-290, 1e-150, 1.0, 1e150])
def test_lines_keep_their_own_exponent(scale):
    """Densities far from 1, rows of very different sizes and empty rows: each line has its own
    exponent, so the result scales with the density."""
    n = 64
    p = _plan(n, 2, False, "r2r")
    u = inputs.bump(n, (0.4, 0.6), 0.3)
    u[::7] *= 1e-9
    u[3::11] = 0.0
    ref = O.conv(u, p.M, _table(p)).real
    tol = TOL if scale > 2.0 ** -970 else 1e-9  # results of subnormal size carry fewer bits
    assert _err(ref, _apply(p, u * scale) / scale) <= tol
    assert np.array_equal(_apply(p, np.zeros((n, n))), np.zeros((n, n)))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n,compact", [(64, False), (512, True)])
def test_non_finite_input_is_not_hidden(bad, n, compact):
    p = _plan(n, 2 if not compact else 3, compact, "r2r", 2)
    u = inputs.bump_sums(n, 2, seed=1)
    good = _apply(p, u)
    u[0, n // 2, n // 3] = bad
    out = _apply(p, u)
    assert np.all(np.isnan(out[0])) and np.array_equal(out[1], good[1])


def test_non_power_of_two_scale_and_single_spike():
    """1/M^2 that is no power of two (the integer factor of the last pass) on a density whose every
    line is one value: the widest spread between a line's largest component and its L1 norm."""
    n = 60
    p = _plan(n, 2, False, "r2r")
    u = np.zeros((n, n))
    u[7, 53] = 0.7
    assert _err(O.conv(u, p.M, _table(p)).real, _apply(p, u)) <= TOL


@pytest.mark.parametrize("n,period,compact,B", [(256, 3, True, 8), (60, 4, False, 80), (60, 4, False, 95)])
def test_noalloc_without_room_for_scratch_lines(n, period, compact, B):
    """Helmholtz R2C whose spectra fit the fixed scratch array and whose parked spectra do not: taken on
    complex lines.  Two results, each within TOL of the exact one."""
    plan = _plan(n, period, compact, "r2c", batch=1)
    L = plan.info.transform_len
    spectra = (3 * (L // 2 + 1) * n + 1) * B * 16
    assert spectra <= 32 << 20 < plan.workspace_bytes(B)
    u = torch.tensor(inputs.bump_sums(n, B, seed=5), device="cuda")
    ref = plan.apply(u, workspace=torch.empty(plan.workspace_bytes(B) // 8 + 2, dtype=torch.float64, device="cuda"))
    out = torch.full_like(ref, float("nan"))
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = _native.load().conv_apply_noalloc(plan.handle, ctypes.c_void_p(u.data_ptr()), None,
                                           ctypes.c_void_p(out.data_ptr()), B, st)
    assert rc == 0, _native.load().conv_last_error()
    assert plan.info.r2c_split == 1
    r, o = ref.cpu().numpy(), out.cpu().numpy()
    assert np.max(np.abs(o - r)) <= 2 * TOL * np.max(np.abs(r))


@pytest.mark.parametrize("n,period,compact,taken", [(64, 5, False, False), (64, 3, False, True), (512, 3, True, True),
                                                    (100, 3, False, False), (256, 3, True, True)])
def test_multi_takes_the_lengths_of_its_domain(n, period, compact, taken):
    plans = [_plan(n, period, compact, "r2r") for _ in range(2)]
    if taken:
        assert multi_workspace_bytes(plans, 1) > 0
    else:
        with pytest.raises(ConvError, match="EUNSUPPORTED"):
            multi_workspace_bytes(plans, 1)
