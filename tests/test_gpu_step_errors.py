"""What a step leaves behind when the CUDA runtime reports an error (GPU)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2609_10816_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu


def _leave_a_pending_error():
    # a box whose scratch (1.9 TB) cannot be allocated: the runtime keeps the error until it is read
    with pytest.raises(mhd.MHDError):
        mhd.Context((1290, 1290, 1290), (1.0, 1.0, 1.0))


@pytest.mark.parametrize("recon,fofc", [("ppm", True), ("plm_mc", False)])
def test_failed_step_leaves_the_state(gpu_lib, recon, fofc):
    shape = (12, 10, 8)
    cons, b, info = inputs.random_smooth(shape, seed=3, rough=0.02)
    ctx = mhd.Context(shape, info["h"])
    st = mhd.to_device(cons, b)
    sch = mhd.scheme(recon, "hlld", "q26", fofc=fofc)
    s = st.c()
    ctx.step(mhd.to_device(cons, b), 1e-3, sch)  # (a kernel's first launch clears a pending error)
    _leave_a_pending_error()
    assert mhd.lib().mhd_step(ctx._h, ctypes.byref(s), 1e-3, sch, 0.0) == mhd.ERR_CUDA
    torch.cuda.synchronize()
    assert np.array_equal(st.cons.cpu().numpy(), cons) and np.array_equal(st.b.cpu().numpy(), b)
    # reported once: the step taken again is the step
    ctx.step(st, 1e-3, sch)
    ref = mhd.to_device(cons, b)
    ctx.step(ref, 1e-3, sch)
    ctx.close()
    assert torch.equal(st.cons, ref.cons) and torch.equal(st.b, ref.b)
    assert not np.array_equal(st.cons.cpu().numpy(), cons)


def test_failed_noalloc_step_leaves_the_state(gpu_lib):
    shape = (12, 10, 8)
    cons, b, info = inputs.random_smooth(shape, seed=3, rough=0.02)
    f = mhd.lib().mhd_step_noalloc
    f.argtypes = [ctypes.POINTER(mhd._Config), ctypes.POINTER(mhd._State), ctypes.c_double, ctypes.c_int,
                  ctypes.c_double, ctypes.c_void_p]
    f.restype = ctypes.c_int
    st = mhd.to_device(cons, b)
    cfg = mhd._Config(*shape, *info["h"], 5.0 / 3.0, 3)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    other = mhd.to_device(cons, b)
    s, so = st.c(), other.c()
    sch = mhd.scheme("ppm", "hlld", "q26")
    assert f(ctypes.byref(cfg), ctypes.byref(so), 1e-3, sch, 0.0, stream) == mhd.OK
    _leave_a_pending_error()
    rc = f(ctypes.byref(cfg), ctypes.byref(s), 1e-3, sch, 0.0, stream)
    assert rc == mhd.ERR_CUDA
    torch.cuda.synchronize()
    assert np.array_equal(st.cons.cpu().numpy(), cons) and np.array_equal(st.b.cpu().numpy(), b)
