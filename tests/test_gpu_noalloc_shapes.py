"""mhd_step_noalloc's face sweeps, whose segments follow the box's size, against mhd_step's: the same bits
on boxes of one cell up to the fixed limit, long lines, short lines and sizes that divide nothing (GPU)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2609_10816_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (4096, 2, 2), (33, 31, 29), (2, 3, 300), (17, 130, 1), (32, 32, 32)])
@pytest.mark.parametrize("recon,rs", [("pc", "llf"), ("plm_mc", "hll"), ("ppm", "hlld"), ("ppm_ep", "hlld")])
def test_noalloc_step_is_the_step(gpu_lib, shape, recon, rs):
    h = (1.0 / max(shape),) * 3
    cons, b, _ = inputs.random_smooth(shape, seed=4, h=h, rough=0.03)
    f = mhd.lib().mhd_step_noalloc
    f.argtypes = [ctypes.POINTER(mhd._Config), ctypes.POINTER(mhd._State), ctypes.c_double, ctypes.c_int,
                  ctypes.c_double, ctypes.c_void_p]
    f.restype = ctypes.c_int
    sch, eta = mhd.scheme(recon, rs, "q26"), 1e-3
    ctx = mhd.Context(shape, h)
    ref, st = mhd.to_device(cons, b), mhd.to_device(cons, b)
    dt = ctx.max_dt(ref, 0.3, eta)
    ctx.step(ref, dt, sch, eta)
    ctx.close()
    cfg, s = mhd._Config(*shape, *h, 5.0 / 3.0, 3), st.c()
    rc = f(ctypes.byref(cfg), ctypes.byref(s), dt, sch, eta, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == mhd.OK, mhd.lib().mhd_create_error()
    torch.cuda.synchronize()
    assert torch.equal(st.cons, ref.cons) and torch.equal(st.b, ref.b)
    assert not np.array_equal(st.cons.cpu().numpy(), cons) or max(shape) == 1
