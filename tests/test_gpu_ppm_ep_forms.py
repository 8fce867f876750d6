"""PPM-EP's interface offset on the integer pipe (csrc/mhd_device.cuh, ppm_ep_split: the face sweeps)
where its scale changes: smooth profiles, so that every value is the fourth-order one, whose
differences beside an inflection or an extremum pass through zero, down to those too small for the
fixed-point form. One step against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_2609_10816_gb300 import inputs, mhd
from tests.util import parity_failures

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amp", [0.2, 1e-3, 1e-9, 1e-290])
@pytest.mark.parametrize("shape", [(64, 5, 3), (24, 16, 7)])
@pytest.mark.parametrize("emf", ["q26", "b25a"])
def test_smooth_profiles(gpu_lib, amp, shape, emf):
    nx, ny, nz = shape
    x, y, z = inputs.Box(shape).coords()
    box = inputs.Box(shape)
    ph = 2 * np.pi * (x + 0.013)
    rho = 1.0 + 0.3 * np.sin(ph) + 0.05 * np.cos(2 * np.pi * y + 0.4)
    p = 1.0 + 0.2 * np.cos(ph) + 0.04 * np.sin(2 * np.pi * z + 0.7)
    # velocities of size amp: zero crossings at full relative precision
    u = [amp * np.sin(ph + 1.1 * d + 2 * np.pi * y) for d in range(3)]
    A = np.zeros((3,) + rho.shape)
    ex, ey, ez = box.edge_coords(2)
    A[2] = 0.05 * np.sin(2 * np.pi * ex + 0.3) * np.cos(2 * np.pi * ey + 0.2)
    b = inputs.curl_edges_to_faces(box, A)
    b[0] += 0.4
    b[2] += 0.1 + 0.02 * np.cos(2 * np.pi * (x - 0.5 / nx) + 0.9)
    cons = inputs.assemble(rho, u, p, b)
    cfg = oracle.Config(shape=shape, h=box.h, recon="ppm_ep", riemann="hlld", emf=emf)
    dt = oracle.max_dt(cfg, cons, b, 0.2)
    co, bo, _ = oracle.step(cfg, cons, b, dt)
    ctx = mhd.Context(shape, box.h)
    st = mhd.to_device(cons, b)
    ctx.step(st, dt, mhd.scheme("ppm_ep", "hlld", emf))
    got = st.cons.cpu().numpy(), st.b.cpu().numpy()
    ctx.close()
    assert not parity_failures(*got, co, bo)
