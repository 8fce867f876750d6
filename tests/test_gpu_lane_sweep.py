"""The x sweep by lanes (csrc/mhd_face.cuh: a batch's patches) against the walked one (a small single
box): the same bits, at a line's smallest length, with idle lanes in the last pass and in the last
group of lines, and with segments that end inside a line."""
import numpy as np
import pytest

from paper_2609_10816_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu
H = 1.0 / 32


@pytest.mark.parametrize("recon", ["pc", "plm_mc", "plm_minmod", "ppm", "ppm_ep"])
@pytest.mark.parametrize("emf,rs", [("q26", "hlld"), ("fs18", "hll")])
@pytest.mark.parametrize("seg", [8, 20, 64])
def test_lane_sweep_equals_walk(gpu_lib, recon, emf, rs, seg):
    dims = [(16, 5, 3), (45, 3, 7), (61, 1, 1), (64, 2, 9)]
    pats = [inputs.random_smooth(d, seed=k, h=(H,) * 3, rough=0.05)[:2] for k, d in enumerate(dims)]
    sch = mhd.scheme(recon, rs, emf)
    bt = mhd.Batch(dims, H)
    bt.set_schedule(seg=seg)
    bt.set_launches(3)
    cons, b = bt.pack(pats)
    bt.step(cons, b, 0.2, sch, 1e-3)
    dt = bt.last_dt()
    for p, d in enumerate(dims):
        ctx = mhd.Context(d, (H,) * 3)
        st = mhd.to_device(*pats[p])
        ctx.step(st, dt, sch, 1e-3)
        got = bt.unpack(cons, b, p)
        assert np.array_equal(got[0], st.cons.cpu().numpy()) and np.array_equal(got[1], st.b.cpu().numpy()), d
        ctx.close()
    bt.close()
