"""The adjoint takes the branch that the forward step took where two branches of the method meet, so
that their values agree to rounding but their derivatives do not (GPU)."""
import numpy as np
import pytest
import torch

from paper_2609_10816_gb300 import mhd

pytestmark = pytest.mark.gpu
GAM = 5.0 / 3.0


def _gradient(ctx, cons, b, row, cell, dt, sch):
    """d(S^{n+1}[row, cell]) / d(cons) along the x line"""
    st = mhd.to_device(cons, b)
    lam = np.zeros_like(cons)
    lam[row, 0, 0, cell] = 1.0
    adj = mhd.to_device(lam, np.zeros_like(b))
    ctx.step_adjoint(st, adj, dt, sch)
    torch.cuda.synchronize()
    return adj.cons.cpu().numpy()[:, 0, 0, :]


@pytest.mark.parametrize("recon", ["pc", "plm_mc"])
def test_symmetric_collision(gpu_lib, recon):
    """Two gases of one density and pressure collide head-on: the contact's speed is zero up to rounding,
    and its sign says whose tangential velocity the HLLD flux carries. The left one's is exactly zero,
    so the momentum it receives is nonzero in just those steps whose flux (in either stage) came from
    the right, which are those in which that momentum depends on the normal momenta."""
    n, v = 8, 1e-10
    h, dt = 1.0 / n, 0.02
    ctx = mhd.Context((n, 1, 1), (h, h, h))
    sch = mhd.scheme(recon, "hlld", "q26")
    rng = np.random.default_rng(7)
    b = np.zeros((3, 1, 1, n))
    wrong, right = 0, 0
    for _ in range(150):
        rho, p, u = rng.uniform(0.5, 2.0), rng.uniform(0.5, 2.0), rng.uniform(0.2, 0.7)
        cons = np.zeros((5, 1, 1, n))
        cons[0] = rho
        cons[1, 0, 0] = rho * u * np.where(np.arange(n) < 4, 1.0, -1.0)
        cons[2, 0, 0, 4:] = rho * v  # (its kinetic energy is below the last bit of e)
        cons[4] = p / (GAM - 1.0) + 0.5 * rho * u * u
        st = mhd.to_device(cons, b)
        ctx.step(st, dt, sch)
        from_right = float(st.cons[2, 0, 0, 3]) != 0.0
        g = _gradient(ctx, cons, b, 2, 3, dt, sch)[1] / v
        depends = np.abs(g).max() > 1e-3
        wrong += from_right != depends
        right += from_right
    ctx.close()
    assert 10 < right < 140  # both branches are met
    assert wrong == 0


@pytest.mark.parametrize("k", [0.5, 1.0, 2.0, 3.0])
@pytest.mark.parametrize("scale", [0.0625, 0.25])
def test_ppm_ep_interface_value_on_the_cell_value(gpu_lib, k, scale):
    """PPM-EP's fourth-order value of the tangential velocity between cells of value 0 and 1 is exactly 0:
    7 (0 + 1) - (-k + 7 + k). The face sweep's fixed-point arithmetic is exact there, so the value is
    bounded by the cell's own, as it is when the value lies just beyond it: the gradients are the same."""
    n = 16
    h, dt = 1.0 / n, 0.01
    ctx = mhd.Context((n, 1, 1), (h, h, h))
    sch = mhd.scheme("ppm_ep", "hlld", "q26")
    b = np.zeros((3, 1, 1, n))

    def grad(eps):
        v = scale * np.array([-9.0, -8.2, -7.1, -6.3, -5.0, -4.1, -k, 0.0, 1.0, 7.0 + k + eps, 12.3, 13.1, 15.0, 11.0, 3.0,
                              -5.0])
        cons = np.zeros((5, 1, 1, n))
        cons[0] = 1.0
        cons[1] = 0.5  # (the flux takes the left state: the upper values of the cells)
        cons[2, 0, 0] = v
        cons[4] = 1.0 / (GAM - 1.0) + 0.5 * 0.25 + 0.5 * cons[2] ** 2
        return _gradient(ctx, cons, b, 2, 8, dt, sch)[2]

    at, beyond, inside = grad(0.0), grad(1e-5), grad(-1e-5)
    ctx.close()
    assert np.abs(inside - beyond).max() > 1e-2  # the two branches differ
    assert np.abs(at - beyond).max() < 1e-4
