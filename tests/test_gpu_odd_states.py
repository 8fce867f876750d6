"""How far an invalid cell reaches in a stage: the face solve's speeds for a negative density
(csrc/mhd_device.cuh, fast_max) and PPM's limiter beside a value that is not a number."""
import numpy as np
import pytest

from paper_2609_10816_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu
N = (12, 11, 10)
H = (1 / 32, 1 / 30, 1 / 28)


def flags(c, b, recon, rs):
    ctx = mhd.Context(N, H)
    st = mhd.to_device(c, b)
    ctx.step(st, 1e-5, mhd.scheme(recon, rs, "q26"))
    first = ctx.stats()[0]
    ctx.close()
    return first


@pytest.mark.parametrize("recon", ["pc", "plm_mc", "plm_minmod", "ppm"])
def test_negative_density_flags_its_own_cell(gpu_lib, recon):
    # the face takes the other side's speed, so HLL's fluxes stay finite: only the two cells are flagged
    c, b = (np.array(x, copy=True) for x in inputs.random_smooth(N, seed=3, h=H)[:2])
    c[0][2, 3, 4] = -0.5
    c[0][7, 8, 9] = -2.0
    assert flags(c, b, recon, "hll") == 2


@pytest.mark.parametrize("rs", ["hll", "hlld"])
@pytest.mark.parametrize("recon", ["pc", "plm_mc", "ppm"])
def test_nan_reaches_its_faces_and_edges(gpu_lib, recon, rs):
    # limited values of the cells beside it stay finite, so its 6 faces' fluxes and its 12 edges' EMFs
    # are lost, and with them the fields of the faces at those edges: the cell, 6 and 12 neighbours
    c, b = (np.array(x, copy=True) for x in inputs.random_smooth(N, seed=3, h=H)[:2])
    c[0][4, 5, 6] = np.nan
    assert flags(c, b, recon, rs) == 19
