"""conv_apply_noalloc changes nothing on its plan: while one thread runs it on a batch whose scratch
lines do not fit the fixed array (the call then runs on complex lines), another thread's
conv_workspace_size, conv_get_info and conv_apply with a workspace of its own answer on the same plan
as they do alone, conv_apply bitwise.
"""
import ctypes
import threading

import pytest
import torch

from paper_2107_03958_gb300 import _native, inputs
from paper_2107_03958_gb300.api import ConvPlan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,period,compact,B", [(256, 3, True, 8), (60, 4, False, 95)])
def test_noalloc_beside_other_calls_on_its_plan(n, period, compact, B):
    plan = ConvPlan("helmholtz", n=n, period=period, kappa=9.0, precision="fp64", io="r2c", compact=compact, batch_max=1)
    size = plan.workspace_bytes(B)
    assert (3 * (plan.info.transform_len // 2 + 1) * n + 1) * B * 16 <= 32 << 20 < size
    u = torch.tensor(inputs.bump_sums(n, B, seed=5), device="cuda")
    ws = torch.empty(size // 8 + 2, dtype=torch.float64, device="cuda")
    ref = plan.apply(u, workspace=ws)
    noalloc_out, out = torch.empty_like(ref), torch.empty_like(ref)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    lib, failed, done = _native.load(), [], threading.Event()

    def noalloc_calls():
        try:
            for _ in range(400):
                if lib.conv_apply_noalloc(plan.handle, ctypes.c_void_p(u.data_ptr()), None,
                                          ctypes.c_void_p(noalloc_out.data_ptr()), B, ctypes.c_void_p(other.cuda_stream)):
                    failed.append(lib.conv_last_error())
                    break
        finally:
            done.set()

    t = threading.Thread(target=noalloc_calls)
    t.start()
    sizes, splits, same = set(), set(), []
    while not done.is_set():
        sizes.update(plan.workspace_bytes(B) for _ in range(50))
        splits.add(plan._info().r2c_split)
        plan.apply(u, out=out, workspace=ws, stream=mine)
        mine.synchronize()
        same.append(torch.equal(out, ref))
    t.join()
    torch.cuda.synchronize()
    assert not failed and sizes == {size} and splits == {1} and all(same)
    assert float((noalloc_out - ref).abs().max()) <= 1e-14 * float(ref.abs().max())
