"""How far an invalid cell reaches under PPM-EP: the signs of its curvatures beside a value that is not a
number (csrc/mhd_device.cuh, cmp_code). The counts are those of the signs of the rounded differences."""
import numpy as np
import pytest

from paper_2609_10816_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu
H = (1 / 32, 1 / 30, 1 / 28)
SMALL, LANES = (12, 11, 10), (64, 48, 44)  # (the second: the x sweep by lanes)


@pytest.mark.parametrize("shape,kind,emf,expected", [
    (SMALL, "nan_rho", "q26", (38, 215)), (SMALL, "nan_rho", "b25a", (41, 212)),
    (SMALL, "nan_b", "q26", (65, 253)), (SMALL, "nan_b", "b25a", (66, 259)),
    (SMALL, "nan_e", "q26", (38, 215)), (SMALL, "nan_e", "b25a", (34, 212)),
    (SMALL, "negative", "q26", (2, 391)), (SMALL, "negative", "b25a", (2, 381)),
    (LANES, "nan_rho", "q26", (44, 198)), (LANES, "nan_b", "q26", (51, 241)), (LANES, "nan_e", "b25a", (19, 174))])
def test_flagged_cells(gpu_lib, shape, kind, emf, expected):
    c, b = (np.array(x, copy=True) for x in inputs.random_smooth(shape, seed=3, h=H)[:2])
    if kind == "nan_rho":
        c[0][4, 5, 6] = np.nan
    elif kind == "nan_e":
        c[4][4, 5, 6] = np.nan
    elif kind == "nan_b":
        b[1][4, 5, 6] = np.nan
    else:
        c[0][2, 3, 4] = -0.5
        c[0][7, 8, 9] = -2.0
    ctx = mhd.Context(shape, H)
    st = mhd.to_device(c, b)
    ctx.step(st, 1e-5, mhd.scheme("ppm_ep", "hll", emf))
    flagged = ctx.stats()
    ctx.close()
    assert flagged == expected
