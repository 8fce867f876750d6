"""Which x sweeps run by lanes (csrc/mhd_face.cuh, face_by_lanes): line counts on either side of the rule,
and idle lanes in the last group of lines, give the bits of the walked sweep (GPU)."""
import numpy as np
import pytest

from paper_2609_10816_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu
H = 1.0 / 32


@pytest.mark.parametrize("recon", ["pc", "plm_mc", "plm_minmod", "ppm", "ppm_ep"])
@pytest.mark.parametrize("seg", [8, 64])
def test_line_counts(gpu_lib, recon, seg):
    # by lanes: 15 lines (one lane idle), 4, 27; walked: 1, 2, 13 lines
    dims = [(45, 3, 5), (61, 4, 1), (64, 3, 9), (131, 1, 1), (47, 2, 1), (32, 13, 1)]
    pats = [inputs.random_smooth(d, seed=k, h=(H,) * 3, rough=0.05)[:2] for k, d in enumerate(dims)]
    sch = mhd.scheme(recon, "hlld", "q26")
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


def test_single_lines_and_wide_boxes(gpu_lib):
    """Boxes above the size where lanes start: one line against the same box turned to y and z, whose sweeps
    are walked."""
    n = 1 << 17
    cons, b, _ = inputs.random_smooth((n, 1, 1), seed=2, h=(1.0 / n,) * 3, rough=0.02)
    sch, out = mhd.scheme("ppm", "hlld", "q26"), []
    for d in range(3):
        shape = tuple(n if k == d else 1 for k in range(3))
        c, f = cons.copy(), b.copy()
        for _ in range(d):  # x -> y -> z -> x for the vector components
            c[1:4], f = c[[3, 1, 2]].copy(), f[[2, 0, 1]].copy()
        c, f = c.reshape((5,) + shape[::-1]), f.reshape((3,) + shape[::-1])
        ctx = mhd.Context(shape, (1.0 / n,) * 3)
        st = mhd.to_device(np.ascontiguousarray(c), np.ascontiguousarray(f))
        ctx.step(st, 1e-7, sch)
        c, f = st.cons.cpu().numpy().reshape(5, -1), st.b.cpu().numpy().reshape(3, -1)
        ctx.close()
        for _ in range(d):
            c[1:4], f = c[[2, 3, 1]].copy(), f[[1, 2, 0]].copy()
        out.append((c, f))
    for c, f in out[1:]:
        assert np.abs(c - out[0][0]).max() <= 1e-12 * np.abs(c).max() and np.abs(f - out[0][1]).max() <= 1e-12
