"""The rounding of the sum d/d(eta) of an adjoint step where the terms of different edges cancel (GPU)."""
import numpy as np
import pytest

from paper_2609_10816_gb300 import mhd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon,emf", [("ppm", "q26"), ("plm_mc", "fs18"), ("pc", "b25a")])
def test_eta_sum_of_opposite_components(gpu_lib, recon, emf):
    """b_z = f(x) + f(y) and its adjoint f(y) - f(x): the terms of the x edges, j_x^2 up to a factor, sum to
    S, those of the y edges to -S, and the sum is zero by the exchange of x and y."""
    n, dt = 64, 1e-4
    t = 2 * np.pi * (np.arange(n) + 0.5) / n
    f = 0.3 * np.sin(t) + 0.1 * np.cos(2 * t + 0.3)
    b, lb = np.zeros((3, n, n, n)), np.zeros((3, n, n, n))
    b[2] = f[None, :, None] + f[None, None, :]
    lb[2] = f[None, :, None] - f[None, None, :]
    cons = np.zeros((5, n, n, n))
    cons[0] = 1.0
    cons[4] = 1.5 + 0.5 * b[2] ** 2
    S = dt * (((np.roll(b[2], -1, 1) - b[2]) * n) ** 2).sum()
    ctx = mhd.Context((n, n, n), (1 / n,) * 3)
    st = mhd.to_device(cons, b)
    vals = [ctx.step_adjoint(st, mhd.to_device(np.zeros_like(cons), lb), dt, mhd.scheme(recon, "hlld", emf), 1e-3)
            for _ in range(5)]
    ctx.close()
    # one addition to the running sum per block of 128 cells and stage, off by 2^-53 / sqrt(3) of it rms;
    # the two components meet in a cell's own terms, so that with blocks in about their order it stays
    # below S / 16
    adds = 2 * n**3 / 128
    assert np.abs(vals).max() <= 3 * 2.0**-53 / 3**0.5 * adds**0.5 * S / 16
