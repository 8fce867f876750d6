"""PPM's fixed-point interface values (csrc/mhd_device.cuh, ppm_split) where its scale and its branches
change: neighbouring differences of very different size, of opposite sign and zero, and differences
too small for the fixed-point form (they take the FP64 form). One step against the CPU oracle.
PPM-EP takes the same differences in FP64; its switch at smooth extrema is discontinuous where
neighbours tie, so it is compared on the two kinds of state whose ties both sides resolve alike."""
import numpy as np
import pytest

import oracle
from paper_2609_10816_gb300 import inputs, mhd
from tests.util import parity_failures

pytestmark = pytest.mark.gpu


def _fields(kind, shape, rng):
    nx, ny, nz = shape
    s = (nz, ny, nx)
    sgn = lambda: rng.choice([-1.0, 1.0], s)  # noqa: E731
    rho, p = 1.0 + 0.2 * rng.uniform(-1, 1, s), 1.0 + 0.2 * rng.uniform(-1, 1, s)
    u = [0.3 * rng.uniform(-1, 1, s) for _ in range(3)]
    if kind == "jumps":  # differences from 1e-3 to 10 beside one another
        rho, p = 10.0 ** rng.uniform(-1, 1, s), 10.0 ** rng.uniform(-1, 1, s)
    elif kind == "binades":  # differences of one sign whose ratios are powers of two around the clamp at 2^3
        rho = 1.0 + 0.25 * np.cumsum(2.0 ** -rng.integers(0, 8, s), axis=2) / nx
        u = [v * 2.0 ** -rng.integers(0, 70, s) for v in u]
    elif kind == "zeros":  # equal neighbours, single steps, values of few bits
        rho, p = 1.0 + rng.integers(0, 2, s), 1.0 + 0.5 * rng.integers(0, 3, s)
        u = [0.25 * rng.integers(-1, 2, s) for _ in range(3)]
    elif kind == "tiny":  # differences below the fixed-point form's range, beside ordinary ones
        u = [np.where(rng.random(s) < 0.7, sgn() * 10.0 ** rng.uniform(-307, -265, s), v) for v in u]
    elif kind == "rounding":  # fields uniform up to their last bits
        rho, p = 1.0 + 2.0**-52 * rng.integers(0, 5, s), 1.0 + 2.0**-52 * rng.integers(0, 5, s)
    return rho, u, p


@pytest.mark.parametrize("recon,kind", [("ppm", k) for k in ("jumps", "binades", "zeros", "tiny", "rounding")]
                         + [("ppm_ep", k) for k in ("binades", "rounding")])
@pytest.mark.parametrize("shape", [(40, 9, 7), (5, 4, 33), (2, 1, 1)])
def test_step_matches_oracle(gpu_lib, recon, kind, shape):
    rng = np.random.default_rng(11)
    rho, u, p = _fields(kind, shape, rng)
    box = inputs.Box(shape)
    A = 0.02 * rng.uniform(-1, 1, (3,) + rho.shape) * min(box.h)
    b = inputs.curl_edges_to_faces(box, A)
    b[0] += 0.3
    b[2] -= 0.2
    cons = inputs.assemble(rho, u, p, b)
    cfg = oracle.Config(shape=shape, h=box.h, recon=recon, riemann="hlld", emf="q26")
    dt = oracle.max_dt(cfg, cons, b, 0.2)
    co, bo, _ = oracle.step(cfg, cons, b, dt)
    ctx = mhd.Context(shape, box.h)
    st = mhd.to_device(cons, b)
    ctx.step(st, dt, mhd.scheme(recon, "hlld", "q26"))
    got = st.cons.cpu().numpy(), st.b.cpu().numpy()
    ctx.close()
    assert not parity_failures(*got, co, bo)
