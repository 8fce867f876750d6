"""The CFL reduction's single-precision screening (csrc/mhd_cell.cuh, cfl_below) on magnetically
dominated cells whose face fields alternate in sign, so that the cell's field is a small difference of
large ones: the time step is the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2609_10816_gb300 import mhd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amp", [1.0, 10.0, 97.0, 1023.0, 5852.0, 33333.0])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_dt_where_face_fields_cancel(gpu_lib, amp, seed):
    # more cells than the grid has threads, the faster ones in the upper layers: they are judged against
    # the running maximum of the lower ones
    nx, ny, nz = 128, 96, 160
    rng = np.random.default_rng(seed)
    k = np.arange(nz)
    # means that depend on z alone, and b_x = -b_y = amp (-1)^(i+j) on top: no divergence
    size = 1e-4 * np.where(k < nz - 40, 0.5, 1.0) * rng.uniform(0.9, 1.0, nz)
    ang = rng.uniform(0.0, 2.0 * np.pi, nz)
    alt = amp * (1.0 - 2.0 * ((np.arange(ny)[:, None] + np.arange(nx)) % 2))
    b = np.zeros((3, nz, ny, nx))
    b[0] = (size * np.cos(ang))[:, None, None] + alt
    b[1] = (size * np.sin(ang))[:, None, None] - alt
    b[2] = 3e-5
    bc = [0.5 * (b[d] + np.roll(b[d], -1, axis=2 - d)) for d in range(3)]
    cons = np.zeros((5, nz, ny, nx))
    cons[0] = 1.0
    cons[4] = 5e-12 / (5.0 / 3.0 - 1.0) + 0.5 * (bc[0] ** 2 + bc[1] ** 2 + bc[2] ** 2)
    h = (1 / nx, 1 / ny, 1 / nz)
    ref = oracle.max_dt(oracle.Config(shape=(nx, ny, nz), h=h), cons, b, 0.3)
    ctx = mhd.Context((nx, ny, nz), h)
    st = mhd.to_device(cons, b)
    dt = ctx.max_dt(st, 0.3)
    ctx.step_cfl(st, 0.3, mhd.scheme("pc", "hll"))
    dt_step = ctx.last_dt()
    ctx.close()
    assert abs(dt - ref) <= 1e-14 * ref
    assert dt_step == dt
