"""The CFL reduction's single-precision screening (csrc/mhd_cell.cuh, cfl_below): whatever it settles,
the time step is the oracle's, on boxes whose largest speed sits in one cell that the screening has
to let through, and on states outside what it judges (huge and tiny units, a cell without pressure,
one that is not finite)."""
import numpy as np
import pytest

import oracle
from paper_2609_10816_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu


def _state(shape, seed, unit=1.0):
    cons, b, info = inputs.random_smooth(shape, seed=seed, rough=0.05)
    # the same flow in other units: velocities times `unit`
    cons[1:4] *= unit
    cons[4] *= unit**2
    return cons, b * unit, info["h"]


@pytest.mark.parametrize("unit", [1.0, 1e-7, 1e7, 1e-30, 1e30])
@pytest.mark.parametrize("excess", [1e-3, 1e-5, 1e-9])
def test_dt_with_one_fastest_cell(gpu_lib, unit, excess):
    shape = (96, 80, 64)
    cons, b, h = _state(shape, 3, unit)
    cfg = oracle.Config(shape=shape, h=h)
    # two far cells with almost the same, largest speed: the second is faster by `excess`
    for (k, j, i), f in (((60, 70, 90), 1.0), ((1, 2, 3), 1.0 + excess)):
        dm = 4.0 * unit * f * cons[0, k, j, i] - cons[1, k, j, i]
        cons[4, k, j, i] += 0.5 * ((cons[1, k, j, i] + dm) ** 2 - cons[1, k, j, i] ** 2) / cons[0, k, j, i]
        cons[1, k, j, i] += dm
    ctx = mhd.Context(shape, h)
    st = mhd.to_device(cons, b)
    dt = ctx.max_dt(st, 0.3)
    ctx.step_cfl(st, 0.3, mhd.scheme("plm_mc", "hll"))
    assert ctx.last_dt() == dt
    ctx.close()
    ref = oracle.max_dt(cfg, cons, b, 0.3)
    assert abs(dt - ref) <= 1e-14 * ref


def test_dt_of_states_it_does_not_judge(gpu_lib):
    shape = (32, 16, 16)
    cons, b, h = _state(shape, 5)
    cfg = oracle.Config(shape=shape, h=h)
    ctx = mhd.Context(shape, h)
    cold = cons.copy()
    cold[4, 3, 4, 5] *= 0.3  # no pressure there
    assert abs(ctx.max_dt(mhd.to_device(cold, b), 0.3) - oracle.max_dt(cfg, cold, b, 0.3)) <= 1e-14
    bad = cons.copy()
    bad[2, 9, 4, 5] = np.nan
    with pytest.raises(mhd.MHDError) as e:
        ctx.max_dt(mhd.to_device(bad, b), 0.3)
    assert e.value.code == mhd.ERR_NONFINITE
    ctx.close()
