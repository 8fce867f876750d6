"""Performance cases of the constrained-transport MHD library: what its users have it do.

Each case goes through the public entry points of `paper_2609_10816_gb300` (`mhd.Context`,
`mhd.Batch`, `adjoint.evolve`). Inputs are made on the GPU from a seed. `exact` repeats the same
computation in plain torch, in 64 bits, from the method's definition (Sec. 2 of the paper), without
the library; gradients come from torch's own autograd.
"""
import math

import numpy as np
import torch

GAMMA = 5.0 / 3.0
DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------
def listed():
    def step(name, n, state, recon, riemann="hlld", emf="q26", eta=0.0, cfl=0.3, clock="cfl"):
        return {"name": name, "kind": "step", "nx": n[0], "ny": n[1], "nz": n[2], "state": state, "recon": recon,
                "riemann": riemann, "emf": emf, "eta": eta, "cfl": cfl, "clock": clock}

    return [
        # production size: one step of a resident decaying-turbulence box, the library's default scheme
        step("turbulence 256^3", (256, 256, 256), "turbulence", "ppm"),
        # the paper's throughput problem (its per-GPU weak-scaling size and reconstruction)
        step("alfven 128^3 ppm_ep", (128, 128, 128), "alfven", "ppm_ep"),
        # the two comparison EMF schemes, in the runs that compare them
        step("alfven 96^3 ppm_ep b25a", (96, 96, 96), "alfven", "ppm_ep", emf="b25a"),
        step("turbulence 128^3 fs18", (128, 128, 128), "turbulence", "ppm", emf="fs18"),
        # resistive reconnection in a thin slab, the limiter and solver its bench runs
        step("reconnection 512x512x4", (512, 512, 4), "harris", "plm_mc", eta=1e-4),
        # a convergence study's coarse wave: a small box, where latency and launches count
        step("fast wave 32^3", (32, 32, 32), "wave", "plm_mc", riemann="hll"),
        # a box whose sizes divide nothing, with resistivity and a time step set by the caller
        step("ragged 97x61x45", (97, 61, 45), "smooth", "ppm", eta=1e-3, clock="fixed"),
        # many uneven patches of one refinement level in one call
        {"name": "batch 96 patches", "kind": "batch", "npatch": 96, "edges": "16,24,32,48,64", "layout": 4,
         "recon": "ppm", "riemann": "hlld", "emf": "q26", "eta": 0.0, "cfl": 0.3, "tune": True},
        # reverse pass of one step of the differentiation workload's size
        {"name": "adjoint 64^3", "kind": "adjoint", "nx": 64, "ny": 64, "nz": 64, "recon": "ppm", "riemann": "hlld",
         "emf": "q26", "eta": 1e-3, "cfl": 0.3},
        # a whole gradient: forward and backward through several steps of a small box, checkpointed
        {"name": "evolve 32^3 4 steps", "kind": "evolve", "nx": 32, "ny": 32, "nz": 32, "recon": "ppm",
         "riemann": "hlld", "emf": "q26", "eta": 1e-3, "cfl": 0.3, "steps": 4, "every": 2},
        # a run's monitoring between outputs: the stable time step and the divergence check
        {"name": "diagnostics 192^3", "kind": "diag", "nx": 192, "ny": 192, "nz": 192, "state": "turbulence",
         "eta": 0.0, "cfl": 0.3},
    ]


def _size(rng, lo, hi, flat=False):
    """(nx, ny, nz) with the cell count spread over [lo, hi] by its logarithm, uneven and often odd."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nz = rng.randint(3, 8) if flat else None
    side = math.sqrt(cells / nz) if flat else cells ** (1.0 / 3.0)
    n = [max(6, int(side * math.exp(rng.uniform(-0.3, 0.3)))) for _ in range(2 if flat else 3)]
    if rng.random() < 0.4:  # the sizes people pick
        n = [max(8, 8 * round(k / 8)) for k in n]
    return tuple(n + [nz]) if flat else tuple(n)


def draw(rng):
    kind = rng.choices(["step", "batch", "adjoint", "evolve", "diag"], [10, 3, 3, 2, 1])[0]
    recon = rng.choices(["ppm", "ppm_ep", "plm_mc", "plm_minmod"], [5, 3, 3, 1])[0]
    c = {"kind": kind, "recon": recon, "riemann": rng.choices(["hlld", "hll"], [4, 1])[0],
         "emf": rng.choices(["q26", "fs18", "b25a"], [4, 1, 1])[0], "eta": rng.choice([0.0, 1e-4, 1e-3]),
         "cfl": rng.choice([0.2, 0.25, 0.3])}
    if kind == "step":
        c["state"] = rng.choice(["smooth", "smooth", "turbulence", "alfven", "harris"])
        n = _size(rng, 4e3, 4e6, flat=c["state"] == "harris")
        c["clock"] = rng.choice(["cfl", "cfl", "fixed"])
    elif kind == "batch":
        c.update(npatch=rng.randint(4, 60), edges=rng.choice(["16,24,32,48,64", "12,20,28,36", "8,16,32", "17,23,31,40"]),
                 layout=rng.randint(1, 10**6), tune=rng.random() < 0.5)
        return c
    elif kind == "adjoint":
        n = _size(rng, 2e3, 2.6e5)
    elif kind == "evolve":
        n = _size(rng, 2e3, 4e4)
        c.update(steps=rng.randint(2, 5), every=rng.randint(1, 3))
    else:
        n = _size(rng, 4e3, 1e7)
        c["state"] = rng.choice(["smooth", "turbulence"])
        for k in ("recon", "riemann", "emf"):
            del c[k]
    c.update(nx=n[0], ny=n[1], nz=n[2])
    return c


def _dims(case):
    edges = np.array([int(e) for e in case["edges"].split(",")])
    return [tuple(int(x) for x in d) for d in np.random.default_rng(case["layout"]).choice(edges, (case["npatch"], 3))]


# FP64 operations per cell and stage of one step: faces (three reconstructions and Riemann solves),
# edges (the EMF) and the update
_FACE = {"ppm": 860.0, "ppm_ep": 1300.0, "plm_mc": 650.0, "plm_minmod": 630.0}
_EDGE = {"q26": 345.0, "fs18": 700.0, "b25a": 560.0}


def work(case):
    """Bytes: every input read once and every output written once. Flops: the method's operations."""
    if case["kind"] == "batch":
        cells = float(sum(a * b * c for a, b, c in _dims(case)))
    else:
        cells = float(case["nx"]) * case["ny"] * case["nz"]
    if case["kind"] == "diag":
        return {"bytes": cells * 8 * 8, "flops": cells * 70}
    step = 2 * (_FACE[case["recon"]] + _EDGE[case["emf"]] + 140.0)
    if case["kind"] == "adjoint":  # state and cotangent in, cotangent out
        return {"bytes": cells * 8 * 24, "flops": cells * 4 * step}
    if case["kind"] == "evolve":
        return {"bytes": cells * 8 * 32, "flops": cells * 5 * step * case["steps"]}
    return {"bytes": cells * 8 * 16, "flops": cells * step}


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------
def _grid(n, h, stagger):
    """x, y, z of shape (1,1,nx), (1,ny,1), (nz,1,1)"""
    ax = [(torch.arange(n[d], device=DEV, dtype=F64) + stagger[d]) * h[d] for d in range(3)]
    return ax[0].view(1, 1, -1), ax[1].view(1, -1, 1), ax[2].view(-1, 1, 1)


def _edge_grid(n, h, e):
    return _grid(n, h, [0.5 if d == e else 0.0 for d in range(3)])


def _up(q, d, k=1):
    """q at the cell k further along direction d (periodic)"""
    return torch.roll(q, -k, 2 - d)


def _curl(A, h):
    out = []
    for d in range(3):
        a, c = (d + 1) % 3, (d + 2) % 3
        out.append((_up(A[c], a) - A[c]) / h[a] - (_up(A[a], c) - A[a]) / h[c])
    return torch.stack(out)


def _assemble(rho, u, p, b):
    bc = [0.5 * (b[d] + _up(b[d], d)) for d in range(3)]
    e = p / (GAMMA - 1) + 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2) + 0.5 * (bc[0] ** 2 + bc[1] ** 2 + bc[2] ** 2)
    return torch.stack([rho, rho * u[0], rho * u[1], rho * u[2], e]).contiguous()


def _full(n, v):
    return torch.full((n[2], n[1], n[0]), float(v), device=DEV, dtype=F64)


def _modes(rng, n, grid, size):
    """a smooth periodic scalar of largest size about `size`: a few random low-k modes"""
    x, y, z = grid
    f, norm = _full(n, 0.0), 0.0
    for _ in range(5):
        k = rng.integers(-2, 3, 3)
        k[rng.integers(0, 3)] = rng.integers(1, 3)
        a = rng.uniform(0.4, 1.0)
        f += a * torch.cos(2 * math.pi * (k[0] * x + k[1] * y + k[2] * z) + rng.uniform(0, 2 * math.pi))
        norm += a
    return f * (size / norm)


def _smooth(n, seed):
    """smooth flow with small cell-to-cell noise: rho in about [0.5, 2], |u| < 1, p about 1"""
    rng = np.random.default_rng([seed, *n])
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    h = [1.0 / k for k in n]
    noise = lambda: torch.rand((n[2], n[1], n[0]), device=DEV, dtype=F64, generator=gen) * 2 - 1  # noqa: E731
    g = _grid(n, h, (0.5, 0.5, 0.5))
    rho = (1.25 + _modes(rng, n, g, 0.7)) * (1 + 0.01 * noise())
    u = [_modes(rng, n, g, 0.8) + 0.01 * noise() for _ in range(3)]
    p = (1.0 + _modes(rng, n, g, 0.5)) * (1 + 0.01 * noise())
    A = torch.stack([_modes(rng, n, _edge_grid(n, h, e), 0.08) for e in range(3)])
    b = _curl(A, h) + torch.tensor([0.3, -0.2, 0.4], device=DEV, dtype=F64).view(3, 1, 1, 1)
    return _assemble(rho, u, p, b), b.contiguous(), h


def _turbulence(n, seed, v_rms=5.0):
    """decaying-turbulence start: rho = 1, c_s = 1, b0 = (0, 0, 0.5), solenoidal Gaussian velocity on 1 <= |k| <= 3"""
    rng = np.random.default_rng([seed, 2])
    h = [1.0 / k for k in n]
    x, y, z = _grid(n, h, (0.5, 0.5, 0.5))
    u = [_full(n, 0.0) for _ in range(3)]
    for kx in range(-3, 4):
        for ky in range(-3, 4):
            for kz in range(0, 4):
                k = np.array([kx, ky, kz], float)
                kk = np.linalg.norm(k)
                if not 1 <= kk <= 3 or (kz == 0 and (ky < 0 or (ky == 0 and kx < 0))):
                    continue
                a = kk**-2 * (rng.normal(size=3) + 1j * rng.normal(size=3))
                a = a - k * (k @ a) / kk**2
                ph = 2 * math.pi * (kx * x + ky * y + kz * z)
                c, s = torch.cos(ph), torch.sin(ph)
                for d in range(3):
                    u[d] += a[d].real * c - a[d].imag * s
    rms = torch.sqrt((u[0] ** 2 + u[1] ** 2 + u[2] ** 2).mean())
    u = [v * (v_rms / rms) for v in u]
    b = torch.stack([_full(n, 0.0), _full(n, 0.0), _full(n, 0.5)])
    rho = _full(n, 1.0)
    return _assemble(rho, u, rho / GAMMA, b), b, h


def _alfven(n, seed):
    """the oblique linear Alfven wave of the paper's throughput runs, at a phase of the seed's"""
    h = [1.0 / k for k in n]
    phase = np.random.default_rng([seed, 5]).uniform(0, 2 * math.pi)
    k = 2 * math.pi * np.array([1.0, 2.0, 3.0])
    kk = np.linalg.norm(k)
    nk = k / kk
    npol = np.cross((0.0, 0.0, 1.0), nk)
    npol /= np.linalg.norm(npol)
    e2 = np.cross(nk, npol)
    e2 = e2 if e2[2] > 0 else -e2
    nb = math.cos(math.pi / 4) * nk + math.sin(math.pi / 4) * e2
    amp = 1e-6
    x, y, z = _grid(n, h, (0.5, 0.5, 0.5))
    A = amp * torch.cos(k[0] * x + k[1] * y + k[2] * z + phase)
    coef = np.cross(npol, k) / kk**2 * amp
    pot = []
    for e in range(3):
        ex, ey, ez = _edge_grid(n, h, e)
        pot.append(coef[e] * torch.sin(k[0] * ex + k[1] * ey + k[2] * ez + phase))
    b = _curl(torch.stack(pot), h) + torch.tensor(nb, device=DEV, dtype=F64).view(3, 1, 1, 1)
    u = [-A * float(npol[d]) for d in range(3)]
    return _assemble(_full(n, 1.0), u, _full(n, 1.0 / GAMMA), b), b.contiguous(), h


def _wave(n, seed):
    """fast magnetosonic eigenmode along the box diagonal, at a phase of the seed's"""
    from paper_2609_10816_gb300 import inputs

    cons, b, info = inputs.fast_wave(n, t=float(np.random.default_rng([seed, 7]).uniform(0, 1)))
    return torch.tensor(cons, device=DEV), torch.tensor(b, device=DEV), list(info["h"])


def _harris(n, seed):
    """periodic double current sheet in pressure balance with velocity noise"""
    hx = 1.0 / n[0]
    h = [hx, 1.0 / n[1], hx]
    w = 0.05
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    _, ey, _ = _edge_grid(n, h, 2)
    ey = ey - 0.5

    def F(y):
        c = lambda s: torch.log(torch.cosh(s))  # noqa: E731
        return w * (c((y + 0.25) / w) - c((y - 0.25) / w))

    half = torch.tensor(0.5, device=DEV, dtype=F64)
    m = F(half) - F(-half)
    A = torch.stack([_full(n, 0.0), _full(n, 0.0), _full(n, 0.0) + F(ey) - m * ey])
    b = _curl(A, h)
    bc = 0.5 * (b[0] + _up(b[0], 0))
    p = 0.1 + 0.5 * (1.0 - bc**2)
    u = [1e-3 * torch.randn((n[2], n[1], n[0]), device=DEV, dtype=F64, generator=gen) for _ in range(3)]
    return _assemble(_full(n, 1.0), u, p, b), b.contiguous(), h


_STATES = {"smooth": _smooth, "turbulence": _turbulence, "alfven": _alfven, "wave": _wave, "harris": _harris}


def _inputs(case, seed):
    """(cons, b, h) of a box, or lists of them per patch"""
    if case["kind"] == "batch":
        return [_patch(d, [seed, i]) for i, d in enumerate(_dims(case))]
    n = (case["nx"], case["ny"], case["nz"])
    return _STATES[case.get("state", "smooth")](n, seed)


H_BATCH = 1.0 / 64


def _patch(n, seed):
    """smooth patch: rho in about [0.5, 2], |u| < 1, p = 1, b = curl of a low-k potential; cell width 1/64"""
    rng = np.random.default_rng(seed)
    h = [H_BATCH] * 3
    unit = [1.0 / k for k in n]  # modes periodic over the patch
    g = _grid(n, unit, (0.5, 0.5, 0.5))
    rho = 1.25 + _modes(rng, n, g, 0.75)
    u = [_modes(rng, n, g, 0.55) for _ in range(3)]
    b = _curl(torch.stack([_modes(rng, n, _edge_grid(n, unit, e), 0.1) for e in range(3)]), h)
    return _assemble(rho, u, _full(n, 1.0), b), b.contiguous(), h


def _cotangent(case, seed):
    n = (case["nx"], case["ny"], case["nz"])
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
    return [torch.randn((k, n[2], n[1], n[0]), device=DEV, dtype=F64, generator=gen) for k in (5, 3)]


def _fixed_dt(cons, b, h, cfl, eta):
    return float(_ref_dt(cons, b, h, cfl, eta))


def prepare(case, seed):
    from paper_2609_10816_gb300 import mhd

    kind = case["kind"]
    data = _inputs(case, seed)
    s = dict(case)
    if kind != "diag":
        s["scheme"] = mhd.scheme(case["recon"], case["riemann"], case["emf"])
    if kind == "batch":
        s["batch"] = mhd.Batch(_dims(case), H_BATCH)
        s["cons"] = torch.cat([c.reshape(-1) for c, _, _ in data])
        s["b"] = torch.cat([b.reshape(-1) for _, b, _ in data])
        if case["tune"]:
            s["batch"].tune(s["cons"], s["b"], case["cfl"], s["scheme"], case["eta"])
        return s
    cons, b, h = data
    s["ctx"] = mhd.Context((case["nx"], case["ny"], case["nz"]), h)
    s["state"] = mhd.State(cons, b)
    if kind in ("adjoint", "evolve") or case.get("clock") == "fixed":
        # a caller's own step, held over the run: well inside the first state's limit
        s["dt"] = _fixed_dt(cons, b, h, (0.5 if kind == "step" else 1.0) * case["cfl"], case["eta"])
    if kind in ("adjoint", "evolve"):
        s["gcons"], s["gb"] = _cotangent(case, seed)
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        if s["clock"] == "fixed":
            s["ctx"].step(s["state"], s["dt"], s["scheme"], s["eta"])
        else:
            s["ctx"].step_cfl(s["state"], s["cfl"], s["scheme"], s["eta"])
        return {"cons": s["state"].cons, "b": s["state"].b}
    if kind == "batch":
        s["batch"].step(s["cons"], s["b"], s["cfl"], s["scheme"], s["eta"])
        return {"cons": s["cons"], "b": s["b"]}
    if kind == "diag":
        dt = s["ctx"].max_dt(s["state"], s["cfl"], s["eta"])
        return {"dt": dt, "max_b": s["ctx"].divb(s["state"])[1]}
    if kind == "adjoint":
        from paper_2609_10816_gb300 import mhd

        lam = mhd.State(s["gcons"].clone(), s["gb"].clone())
        deta = s["ctx"].step_adjoint(s["state"], lam, s["dt"], s["scheme"], s["eta"])
        return {"cons": lam.cons, "b": lam.b, "eta": deta}
    from paper_2609_10816_gb300 import adjoint

    c0 = s["state"].cons.detach().requires_grad_()
    b0 = s["state"].b.detach().requires_grad_()
    eta = torch.tensor(s["eta"], dtype=F64, requires_grad=True)
    c1, b1 = adjoint.evolve(c0, b0, eta, s["ctx"], [s["dt"]] * s["steps"], s["scheme"], s["every"])
    g = torch.autograd.grad([c1, b1], [c0, b0, eta], [s["gcons"], s["gb"]])
    return {"cons": c1.detach(), "b": b1.detach(), "gcons": g[0], "gb": g[1], "geta": g[2]}


# ------------------------------------------------------------------------------------------
# The method in plain torch
# ------------------------------------------------------------------------------------------
class _Invalid(Exception):
    """a cell needs first-order flux correction, which this reference leaves out"""


def _sqrt(x):
    pos = x > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, x, 1.0)), 0.0)


def _same(a, b):
    return ((a > 0) & (b > 0)) | ((a < 0) & (b < 0))


def _min(*v):
    m = v[0]
    for x in v[1:]:
        m = torch.minimum(m, x)
    return m


def _mono(a, aL, aR):
    """Colella & Woodward 1984, Eq. 1.10"""
    s1, s2 = aR - a, a - aL
    flat = ~_same(s1, s2)
    fl = ~flat & (s2.abs() > 2 * s1.abs())
    fr = ~flat & (2 * s2.abs() < s1.abs())
    L = torch.where(flat, a, torch.where(fl, 3 * a - 2 * aR, aL))
    R = torch.where(flat, a, torch.where(fr, 3 * a - 2 * aL, aR))
    return L, R


def _cell_states(q, d, kind):
    """lower and upper value of every point along d"""
    dq = _up(q, d) - q          # q[j+1] - q[j]
    dl = _up(dq, d, -1)         # q[j] - q[j-1]
    if kind.startswith("plm"):
        same = _same(dl, dq)
        if kind == "plm_mc":
            m = _min(dl.abs(), dq.abs(), 0.25 * (dl + dq).abs())
        else:
            m = 0.5 * _min(dl.abs(), dq.abs())
        s = torch.where(same, torch.where(dl > 0, m, -m), 0.0)
        return q - s, q + s
    if kind == "ppm":
        t = dl + dq
        m = _min(t.abs(), 4 * dl.abs(), 4 * dq.abs())
        d2 = torch.where(_same(dl, dq), torch.where(t > 0, m, -m), 0.0)
        f = q + 0.5 * dq - (_up(d2, d) - d2) / 12  # at j + 1/2
        return _mono(q, _up(f, d, -1), f)
    # extremum-preserving PPM
    q1 = _up(q, d)
    f = (7 * (q + q1) - (_up(q, d, -1) + _up(q, d, 2))) / 12
    dn = _up(dq, d)
    opp = lambda x, y: (x * y.sign()) < 0  # noqa: E731
    ext = opp(dl, dq) | opp(dq, dn) | opp(dl, dn)       # interface j + 1/2 at an extremum
    D = dq - dl                                          # curvature of point j
    smooth = _same(D, _up(D, d))
    med = torch.maximum(torch.minimum(q, q1), torch.minimum(torch.maximum(q, q1), f))
    f = torch.where(ext & smooth, f, med)
    fl = _up(f, d, -1)
    keep = (ext | _up(ext, d, -1)) & smooth & _up(smooth, d, -1)
    L, R = _mono(q, fl, f)
    return torch.where(keep, fl, L), torch.where(keep, f, R)


def _recon(q, d, kind):
    """left and right value of the interface at j - 1/2"""
    lo, hi = _cell_states(q, d, kind)
    return _up(hi, d, -1), lo


def _prim(U, B):
    rho = U[0]
    u = [U[1 + d] / rho for d in range(3)]
    b = [0.5 * (B[d] + _up(B[d], d)) for d in range(3)]
    p = (GAMMA - 1) * (U[4] - 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
                       - 0.5 * (b[0] ** 2 + b[1] ** 2 + b[2] ** 2))
    return rho, u, p, b


def _speed2(rho, p, b2, bn):
    S = GAMMA * p + b2
    return (S + _sqrt(torch.clamp(S * S - 4 * bn * bn * GAMMA * p, min=0.0))) / (2 * rho)


def _ref_dt(U, B, h, cfl, eta):
    rho, u, p, b = _prim(U, B)
    b2 = b[0] ** 2 + b[1] ** 2 + b[2] ** 2
    hm = min(h)
    s = max(float(((u[d].abs() + torch.sqrt(_speed2(rho, p, b2, b[d]))) * (hm / h[d])).max()) for d in range(3))
    return cfl * hm / max(s, 2 * eta / hm)


def _side(left, l, r):
    return [torch.where(left, x, y) for x, y in zip(l, r)]


def _star(q, b2, S, SM, pt, ptS, bn, energy=None):
    """star state of one side (Miyoshi & Kusano 2005, Eqs. 43-48)"""
    rho, u, v, w, p, by, bz = q
    su, ssm = S - u, S - SM
    rs = rho * su / ssm
    dd = rho * su * ssm - bn * bn
    tang = dd.abs() > 1e-12 * (rho * su * su + bn * bn)
    dd = torch.where(tang, dd, 1.0)
    cv = torch.where(tang, bn * (SM - u) / dd, 0.0)
    cb = torch.where(tang, (rho * su * su - bn * bn) / dd, 1.0)
    vs, ws, bys, bzs = v - by * cv, w - bz * cv, by * cb, bz * cb
    es = vbs = None
    if energy is not None:
        vb = u * bn + v * by + w * bz
        vbs = SM * bn + vs * bys + ws * bzs
        es = (su * energy - pt * u + ptS * SM + bn * (vb - vbs)) / ssm
    return rs, vs, ws, bys, bzs, es, vbs


def _flux(q, bn):
    rho, u, v, w, p, by, bz = q
    b2 = bn * bn + by * by + bz * bz
    pt = p + 0.5 * b2
    e = p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v + w * w) + 0.5 * b2
    ub = u * bn + v * by + w * bz
    U = [rho, rho * u, rho * v, rho * w, e]
    F = [rho * u, rho * u * u + pt - bn * bn, rho * u * v - bn * by, rho * u * w - bn * bz, (e + pt) * u - ub * bn]
    return U, F, pt, e


def _riemann(l, r, bn, kind):
    """flux of (rho, m_n, m_t1, m_t2, e), alpha+, alpha- and the Q26 face velocity"""
    b2l = bn * bn + l[5] ** 2 + l[6] ** 2
    b2r = bn * bn + r[5] ** 2 + r[6] ** 2
    c = torch.sqrt(torch.maximum(_speed2(l[0], l[4], b2l, bn), _speed2(r[0], r[4], b2r, bn)))
    SL = torch.minimum(l[1], r[1]) - c
    SR = torch.maximum(l[1], r[1]) + c
    ap, am = torch.clamp(SR, min=0.0), torch.clamp(-SL, min=0.0)
    us = (ap * l[1] + am * r[1]) / (ap + am)
    Ul, Fl, ptl, el = _flux(l, bn)
    Ur, Fr, ptr, er = _flux(r, bn)
    if kind == "hll":
        F = [(ap * a + am * b - ap * am * (x - y)) / (ap + am) for a, b, x, y in zip(Fl, Fr, Ur, Ul)]
        return F, ap, am, us
    fan = ~(SL > 0) & ~(SR < 0)
    mL, mR = (SL - l[1]) * l[0], (SR - r[1]) * r[0]
    den = torch.where(fan, mR - mL, 1.0)
    SM = (mR * r[1] - mL * l[1] + ptl - ptr) / den
    ptS = (mR * ptl - mL * ptr + mL * mR * (r[1] - l[1])) / den
    left = torch.where(fan, SM >= 0, SL > 0)
    # outside the fan, a harmless stand-in keeps every quotient finite
    SM = torch.where(fan, SM, 0.0)
    a_S = torch.where(fan, torch.where(left, SL, SR), torch.where(left, -1.0, 1.0))
    b_S = torch.where(fan, torch.where(left, SR, SL), torch.where(left, 1.0, -1.0))
    q, qo = _side(left, l, r), _side(left, r, l)
    P_U, P_F = _side(left, Ul, Ur), _side(left, Fl, Fr)
    safe = lambda s: [torch.where(fan, x, y) for x, y in zip(s, (1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0))]  # noqa: E731
    bnf = torch.where(fan, bn, 0.0)
    rs, vs, ws, bys, bzs, es, vbs = _star(safe(q), None, a_S, SM, torch.where(left, ptl, ptr), ptS, bnf, P_U[4])
    Us = [rs, rs * SM, rs * vs, rs * ws, es]
    Fs = [f + a_S * (x - y) for f, x, y in zip(P_F, Us, P_U)]
    rot = fan & torch.where(left, SM * SM * rs < bn * bn, SM * SM * rs <= bn * bn)
    rso, vso, wso, byso, bzso, _, _ = _star(safe(qo), None, b_S, SM, None, None, bnf)
    one = torch.ones_like(rs)
    sa = torch.sqrt(torch.where(rot, rs, one))
    sb = torch.sqrt(torch.where(rot, rso, one))
    sg = torch.where(bn < 0, -1.0, 1.0)
    sgl = torch.where(left, sg, -sg)  # differences below are right minus left
    inv = 1.0 / (sa + sb)
    vss = (sa * vs + sb * vso + sgl * (byso - bys)) * inv
    wss = (sa * ws + sb * wso + sgl * (bzso - bzs)) * inv
    byss = (sa * byso + sb * bys + sgl * sa * sb * (vso - vs)) * inv
    bzss = (sa * bzso + sb * bzs + sgl * sa * sb * (wso - ws)) * inv
    vbss = SM * bn + vss * byss + wss * bzss
    S2 = SM - torch.where(left, one, -one) * bn.abs() / sa
    Uss = [rs, rs * SM, rs * vss, rs * wss, es - torch.where(left, sg, -sg) * sa * (vbs - vbss)]
    F = [torch.where(fan, torch.where(rot, f + S2 * (x - y), f), g) for f, x, y, g in zip(Fs, Uss, Us, P_F)]
    return F, ap, am, us


def _current(B, h, e):
    a, c = (e + 1) % 3, (e + 2) % 3
    return (B[c] - _up(B[c], a, -1)) / h[a] - (B[a] - _up(B[a], c, -1)) / h[c]


def _fluxes(U, B, h, sch, eta):
    """face fluxes [3][5] and edge EMFs [3] of a state"""
    recon, riemann, emf, resistive = sch
    rho, u, p, bc = _prim(U, B)
    Fs, ap, am, us, VL, VR = [], [], [], [], [], []
    for d in range(3):
        a, c = (d + 1) % 3, (d + 2) % 3
        lr = [_recon(q, d, recon) for q in (rho, u[d], u[a], u[c], p, bc[a], bc[c])]
        l, r = [x[0] for x in lr], [x[1] for x in lr]
        F, p1, m1, s1 = _riemann(l, r, B[d], riemann)
        if resistive:
            ja, jc = _current(B, h, a), _current(B, h, c)
            ea, ec = 0.5 * eta * (ja + _up(ja, c)), 0.5 * eta * (jc + _up(jc, a))
            four = lambda q, k: 0.25 * (_up(q, d, -1) + q + _up(_up(q, d, -1), k) + _up(q, k))  # noqa: E731
            F[4] = F[4] + ea * four(B[c], c) - ec * four(B[a], a)
        out = [None] * 5
        out[0], out[1 + d], out[1 + a], out[1 + c], out[4] = F
        Fs.append(out)
        ap.append(p1), am.append(m1), us.append(s1)
        if emf == "fs18":
            VL.append({d: l[1], a: l[2], c: l[3]})
            VR.append({d: r[1], a: r[2], c: r[3]})
    Es = []
    for e in range(3):
        a, c = (e + 1) % 3, (e + 2) % 3
        baB, baT = _recon(B[a], c, recon)
        bcL, bcR = _recon(B[c], a, recon)
        if emf == "q26":
            uaB, uaT = _recon(us[a], c, recon)
            ucL, ucR = _recon(us[c], a, recon)
            eLB, eRB = -uaB * bcL + ucL * baB, -uaB * bcR + ucR * baB
            eLT, eRT = -uaT * bcL + ucL * baT, -uaT * bcR + ucR * baT
        elif emf == "fs18":
            def corner(k):  # velocity component k at LB, RB, LT, RT: mean of both orders
                o1 = [_recon(VL[a][k], c, recon), _recon(VR[a][k], c, recon)]
                o2 = [_recon(VL[c][k], a, recon), _recon(VR[c][k], a, recon)]
                return [0.5 * (o1[s][t] + o2[t][s]) for t in range(2) for s in range(2)]

            ua, uc = corner(a), corner(c)
            eLB, eRB = -ua[0] * bcL + uc[0] * baB, -ua[1] * bcR + uc[1] * baB
            eLT, eRT = -ua[2] * bcL + uc[2] * baT, -ua[3] * bcR + uc[3] * baT
        else:
            eps = -u[a] * bc[c] + u[c] * bc[a]
            o1 = [_recon(f, c, recon) for f in _recon(eps, a, recon)]
            o2 = [_recon(f, a, recon) for f in _recon(eps, c, recon)]
            eLB, eRB, eLT, eRT = [0.5 * (o1[s][t] + o2[t][s]) for t in range(2) for s in range(2)]
        pa, ma = torch.maximum(_up(ap[a], c, -1), ap[a]), torch.maximum(_up(am[a], c, -1), am[a])
        pc, mc = torch.maximum(_up(ap[c], a, -1), ap[c]), torch.maximum(_up(am[c], a, -1), am[c])
        E = (pc * (pa * eLB + ma * eRB) + mc * (pa * eLT + ma * eRT)) / ((pa + ma) * (pc + mc))
        E = E + pa * ma / (pa + ma) * (bcR - bcL) - pc * mc / (pc + mc) * (baT - baB)
        if resistive:
            E = E + eta * _current(B, h, e)
        Es.append(E)
    return Fs, Es


def _update(U, B, F, E, dt, h):
    cells = torch.stack([U[v] + sum((F[d][v] - _up(F[d][v], d)) * (dt / h[d]) for d in range(3)) for v in range(5)])
    faces = []
    for d in range(3):
        a, c = (d + 1) % 3, (d + 2) % 3
        faces.append(B[d] + (E[c] - _up(E[c], a)) * (dt / h[a]) + (_up(E[a], c) - E[a]) * (dt / h[c]))
    faces = torch.stack(faces)
    rho, _, p, _ = _prim(cells.detach(), faces.detach())
    if not bool(((rho > 0) & (p > 0) & torch.isfinite(p)).all()):
        raise _Invalid
    return cells, faces


def _ref_step(U, B, dt, h, sch, eta):
    F1, E1 = _fluxes(U, B, h, sch, eta)
    Uh, Bh = _update(U, B, F1, E1, dt, h)
    F2, E2 = _fluxes(Uh, Bh, h, sch, eta)
    F = [[0.5 * (x + y) for x, y in zip(f, g)] for f, g in zip(F1, F2)]
    return _update(U, B, F, [0.5 * (x + y) for x, y in zip(E1, E2)], dt, h)


def exact(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    cfl, eta = case["cfl"], case["eta"]
    if kind == "diag":
        cons, b, h = data
        return {"dt": float(_ref_dt(cons, b, h, cfl, eta)), "max_b": float(b.abs().max())}
    sch = (case["recon"], case["riemann"], case["emf"], eta != 0.0)
    try:
        if kind == "batch":
            dt = min(_ref_dt(c, b, h, cfl, eta) for c, b, h in data)
            with torch.no_grad():
                out = [_ref_step(c, b, dt, h, sch, eta) for c, b, h in data]
            return {"cons": torch.cat([c.reshape(-1) for c, _ in out]), "b": torch.cat([b.reshape(-1) for _, b in out])}
        cons, b, h = data
        if kind == "step":
            with torch.no_grad():
                dt = _ref_dt(cons, b, h, (0.5 if case["clock"] == "fixed" else 1.0) * cfl, eta)
                c1, b1 = _ref_step(cons, b, dt, h, sch, eta)
            return {"cons": c1, "b": b1}
        gc, gb = _cotangent(case, seed)
        dt = _fixed_dt(cons, b, h, cfl, eta)
        c0, b0 = cons.requires_grad_(), b.requires_grad_()
        et = torch.tensor(eta, dtype=F64, device=DEV, requires_grad=True)
        c1, b1 = c0, b0
        sch = sch[:3] + (True,)  # the derivative in eta is wanted at eta = 0 too
        for _ in range(case.get("steps", 1)):
            c1, b1 = _ref_step(c1, b1, dt, h, sch, et)
        g = torch.autograd.grad([c1, b1], [c0, b0, et], [gc, gb])
        if kind == "adjoint":
            # with eta = 0 the library runs the ideal scheme, whose derivative in eta it gives as 0
            return {"cons": g[0], "b": g[1], "eta": float(g[2]) if eta else None}
        return {"cons": c1.detach(), "b": b1.detach(), "gcons": g[0], "gb": g[1], "geta": g[2] if eta else None}
    except _Invalid:
        return None
