"""The work a user of the multipole Poisson solver has it do, as timed cases.

A case names one call through the public binding (``paper_2602_02507_gb300.multipole``):

* ``solve``    one Poisson solve of a density resident on the device (``Mesh.solve``), with
               the moments of the solve copied out where the caller wants them too;
* ``batch``    several meshes of different sizes and l_max solved by one ``Batch.solve``;
* ``gravity``  the momentum and energy source terms from a potential, a density and a velocity;
* ``coarsen``  the averaging of several fields over the coarsening blocks of one mesh.

The solver comes in a float64 precision and two split-bf16 ones; all three are used in
earnest (the spheroid study and reference solutions in float64, evolutions in bf16x3, rough
densities in bf16x6).  Sizes are those of this repository's workloads, studies and tests.

Inputs are made on the GPU from the seed alone.  ``exact`` evaluates the paper's formulas
(GenASiS II, Sec. 2.2; the gravitational sources of Sec. 3; the block means of Sec. 2.3) with
torch in float64 and uses nothing of the library.
"""
import math

import numpy as np
import torch

from paper_2602_02507_gb300 import multipole as mpl

TWO_PI = 2.0 * math.pi
G_CGS = 6.674e-8
DEV = "cuda"


# ------------------------------------------------------------------------------ cases
def _solve(name, n_r, n_theta, n_phi, l_max, precision, density, radii, angles="even", moments=False):
    case = {"do": "solve", "n_r": n_r, "n_theta": n_theta, "n_phi": n_phi, "l_max": l_max, "precision": precision,
            "density": density, "radii": radii, "angles": angles, "moments": moments}
    return {"name": name, **case} if name else case


def listed():
    return [
        # the smallest 3-D solve users run: the homogeneous-spheroid check of a fresh set-up;
        # launches and latency decide it
        _solve("spheroid_small_bf16x3", 64, 32, 64, 8, "bf16x3", "spheroid", "ball"),
        # the convergence study's everyday form: axisymmetric (one azimuthal cell), float64
        _solve("spheroid_2d_fp64", 471, 128, 1, 20, "fp64", "spheroid", "paper"),
        # self-gravity of a presupernova core once per time step of an evolution
        _solve("core_bf16x3", 512, 128, 256, 16, "bf16x3", "core", "shells"),
        # the same step in reference precision, with its moments (they are what is analysed)
        _solve("core_fp64_moments", 512, 128, 256, 16, "fp64", "core", "shells", moments=True),
        # a convective, turbulent star: rough in every shell, higher degrees
        _solve("rough_bf16x3", 1024, 256, 512, 32, "bf16x3", "rough", "shells"),
        # its reference solution
        _solve("rough_fp64", 1024, 256, 512, 32, "fp64", "rough", "shells"),
        # odd sizes and unevenly spaced cells in every coordinate, with the six-product precision
        _solve("ragged_bf16x6_moments", 301, 99, 180, 21, "bf16x6", "rough", "shells", angles="uneven", moments=True),
        # the convergence study's 3-D mesh (an origin shell, widths growing outward) in float64
        _solve("spheroid_3d_fp64", 353, 96, 192, 20, "fp64", "spheroid", "paper"),
        # the largest solve one device is used for: a billion cells, l_max = 64
        _solve("core_large_bf16x3", 2048, 512, 1024, 64, "bf16x3", "core", "shells"),
        # a survey: stars of several resolutions solved together
        {"name": "survey_batch_bf16x3", "do": "batch", "count": 8, "precision": "bf16x3", "largest": 768},
        # what the fluid solver takes from the potential in every step
        {"name": "gravity_sources", "do": "gravity", "n_r": 512, "n_theta": 128, "n_phi": 256},
        # the fluid's conserved fields averaged near the axis and the origin, once per step
        {"name": "coarsen_fields", "do": "coarsen", "n_theta": 192, "n_fields": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["solve"] * 7 + ["batch", "gravity", "coarsen"])
    if do == "batch":
        return {"do": "batch", "count": rng.randint(3, 8), "precision": rng.choice(["bf16x3", "bf16x6"]),
                "largest": rng.choice([256, 512, 768])}
    if do == "gravity":
        n_theta = _log_int(rng, 24, 200)
        return {"do": "gravity", "n_r": _log_int(rng, 40, 700), "n_theta": n_theta,
                "n_phi": rng.choice([1, 2 * n_theta, 2 * n_theta + 1, _log_int(rng, 32, 400)])}
    if do == "coarsen":
        return {"do": "coarsen", "n_theta": 32 * rng.randint(2, 6), "n_fields": rng.randint(1, 4)}
    precision = rng.choice(["bf16x3", "bf16x3", "bf16x6", "fp64", "fp64", "fp64"])
    density, radii = rng.choice([("core", "shells"), ("rough", "shells"), ("spheroid", "paper"), ("spheroid", "ball")])
    angles = rng.choice(["even", "even", "even", "uneven"])
    while True:
        n_theta = _log_int(rng, 24, 512)
        n_phi = rng.choice([2 * n_theta, 2 * n_theta, _log_int(rng, 32, 1024)])
        if precision == "fp64" and density == "spheroid" and rng.random() < 0.3:
            n_phi = 1
        elif precision != "fp64":
            n_phi += n_phi % 2  # the split precisions take an even number of azimuthal cells
        # next to the origin the midpoint rule weighs a shell's own moments by about 2^l: the
        # studies on such meshes stop at l_max = 20
        l_max = min(_log_int(rng, 4, 64 if radii == "shells" else 20), n_theta // 2)
        n_r = int(3.68 * n_theta) if radii == "paper" else _log_int(rng, 48, 2048)
        cells = n_r * n_theta * n_phi
        if cells <= 1024 * 256 * 512 and (precision != "fp64" or cells * (2 * l_max + 1) <= 1024 * 256 * 512 * 65):
            # thin shells (r_{i+1} / r_i moderate), as the midpoint rule of the method needs
            if radii != "shells" or n_r >= 3 * l_max:
                break
    return _solve(None, n_r, n_theta, n_phi, l_max, precision, density, radii, angles,
                  radii == "shells" and rng.random() < 0.5)


# ------------------------------------------------------------------------------ meshes
def _stretched(n, span, angles):
    """n + 1 edges over [0, span]; uneven ones grow along the range by a factor of about 1.5."""
    x = np.arange(n + 1, dtype=np.float64) / n
    if angles == "uneven":
        x = x + 0.2 * x * (x - 1.0)
    e = span * x
    e[0], e[-1] = 0.0, span
    return e


def _paper_radii(n_theta, n_r):
    """Uniform cells inside r = 0.25, then widths growing in proportion to r (Sec. 2.1)."""
    n_core = (25 * n_theta) // 32
    dr = 0.25 / n_core
    e = [dr * i for i in range(n_core)] + [0.25]
    for _ in range(n_core, n_r):
        e.append(e[-1] * (1.0 + dr / 0.25))
    return np.array(e[:n_r + 1], dtype=np.float64)


def _edges(case):
    if case["radii"] == "paper":
        r = _paper_radii(case["n_theta"], case["n_r"])
    elif case["radii"] == "ball":
        r = _stretched(case["n_r"], 1.5, "even")
    else:
        # five decades, or fewer where few shells would leave them thick
        decades = min(5.0, case["n_r"] * 0.02)
        r = 1e10 * 10.0 ** (-decades * (1.0 - np.arange(case["n_r"] + 1) / case["n_r"]))
    return r, _stretched(case["n_theta"], math.pi, case["angles"]), _stretched(case["n_phi"], TWO_PI, case["angles"])


def _gravitational_constant(case):
    return G_CGS if case["radii"] == "shells" else 1.0


def _mid(e):
    return 0.5 * (e[:-1] + e[1:])


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


# ------------------------------------------------------------------------------ densities
def _legendre(l_max, x):
    """P~_l^m(x), m <= l <= l_max, with the (-1)^m phase and unit norm on the sphere together
    with exp(i m phi): [l][m] -> tensor shaped like x."""
    s = torch.sqrt(torch.clamp(1.0 - x * x, min=0.0))
    P = [[None] * (l + 1) for l in range(l_max + 1)]
    pmm = torch.full_like(x, math.sqrt(1.0 / (4.0 * math.pi)))
    for m in range(l_max + 1):
        if m:
            pmm = -math.sqrt((2.0 * m + 1.0) / (2.0 * m)) * s * pmm
        P[m][m] = pmm
        if m < l_max:
            P[m + 1][m] = math.sqrt(2.0 * m + 3.0) * x * pmm
        for l in range(m + 2, l_max + 1):
            a = math.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
            b = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1.0) ** 2 - 1.0))
            P[l][m] = a * (x * P[l - 1][m] - b * P[l - 2][m])
    return P


def _angular(rng, n, l_max, amplitudes, thc, phc):
    """n random fields sum_{1 <= l <= l_max} amplitude_l N(0, 1) Y_lm on the cell centres."""
    P = _legendre(l_max, torch.cos(_dev(thc)))
    n_t, n_p = len(thc), len(phc)
    B = torch.zeros(n, n_t, 2 * l_max + 1, dtype=torch.float64, device=DEV)
    trig = torch.ones(2 * l_max + 1, n_p, dtype=torch.float64, device=DEV)
    for m in range(l_max + 1):
        ls = list(range(max(1, m), l_max + 1))
        leg = torch.stack([P[l][m] * amplitudes[l] for l in ls])
        for a in range(1 if m == 0 else 2):
            c = torch.randn(n, len(ls), dtype=torch.float64, device=DEV, generator=rng)
            p = 0 if m == 0 else 2 * m - 1 + a
            B[:, :, p] = c @ leg
            if m:
                trig[p] = math.sqrt(2.0) * (torch.cos(m * _dev(phc)) if a == 0 else torch.sin(m * _dev(phc)))
    return (B.reshape(n * n_t, -1) @ trig).reshape(n, n_t, n_p)


def _core_profile(rc, outer, central, radius):
    return _dev(central / (1.0 + (rc * (1e10 / outer) / radius) ** 2) ** 1.5)


def _density(case, seed, edges):
    r, th, ph = edges
    rng = torch.Generator(device=DEV)
    rng.manual_seed(int(seed))
    u = torch.rand(4, dtype=torch.float64, device=DEV, generator=rng).tolist()
    rc, thc, phc = _mid(r), _mid(th), _mid(ph)
    n_r, n_t, n_p = len(rc), len(thc), len(phc)
    if case["density"] == "spheroid":
        # homogeneous oblate spheroid; cells that its surface cuts carry their volume fraction
        a1 = (0.9 + 0.1 * u[0]) * (1.0 if case["radii"] == "ball" else 6.5)
        a3 = a1 * (0.5 + 0.4 * u[1])
        sub = (torch.arange(8, dtype=torch.float64, device=DEV) + 0.5) / 8
        r3, mu = _dev(r) ** 3, torch.cos(_dev(th))
        rs = (r3[:-1, None] + sub * (r3[1:] - r3[:-1])[:, None]) ** (1.0 / 3.0)
        ms = mu[:-1, None] + sub * (mu[1:] - mu[:-1])[:, None]
        surface = 1.0 / torch.sqrt((1.0 - ms * ms) / a1 ** 2 + ms * ms / a3 ** 2)
        frac = torch.zeros(n_r, n_t, dtype=torch.float64, device=DEV)
        for k in range(8):
            frac += (rs[:, None, :, None] < surface[None, :, None, k:k + 1]).double().mean(dim=(2, 3)) / 8
        rho = (1e-3 if case["radii"] == "paper" else 1.0) * frac
        return rho[:, :, None].expand(n_r, n_t, n_p).contiguous()
    profile = _core_profile(rc, r[-1], 10.0 ** (9.0 + 2.0 * u[0]), 5e7 * 4.0 ** u[1])
    if case["density"] == "core":
        amp = [1e-2 if 1 <= l <= 4 else 1e-3 for l in range(65)]
        ang = 1.0 + _angular(rng, 1, 64, amp, thc, phc)[0]
        return profile[:, None, None] * ang
    # log-normal with a unit-variance exponent, C_l ~ l^-2, drawn for every shell
    cl = [0.0] + [float(l) ** -2 for l in range(1, 65)]
    norm = sum(c * (2 * l + 1) / (4.0 * math.pi) for l, c in enumerate(cl))
    amp = [math.sqrt(c / norm) for c in cl]
    rho = torch.empty(n_r, n_t, n_p, dtype=torch.float64, device=DEV)
    for i in range(0, n_r, 256):
        n = min(256, n_r - i)
        rho[i:i + n] = _angular(rng, n, 64, amp, thc, phc).sub_(0.5).exp_() * profile[i:i + n, None, None]
    return rho


# ------------------------------------------------------------------------------ prepare and run
def _batch_members(case, seed):
    """The meshes of a survey: sizes and l_max do not depend on the seed, the stars do."""
    shapes = [s for s in [(256, 64, 128), (512, 128, 256), (768, 192, 384)] if s[0] <= case["largest"]]
    out = []
    for k in range(case["count"]):
        n_r, n_t, n_p = shapes[(len(shapes) - 1 - k) % len(shapes)]
        sub = _solve(None, n_r, n_t, n_p, [16, 8, 32, 16, 8][k % 5], case["precision"], "core", "shells")
        out.append((sub, 1000 * int(seed) + k))
    return out


def _mesh(case, edges):
    return mpl.Mesh(*edges, case["l_max"], _gravitational_constant(case), precision=case["precision"])


def _gravity_mesh(case):
    n = {"n_r": case["n_r"], "n_theta": case["n_theta"], "n_phi": case["n_phi"]}
    return _edges({**n, "radii": "shells", "angles": "even"})


def _gravity_inputs(case, seed, edges):
    """A potential with the shape of a core's, the density and a velocity field."""
    r, th, ph = edges
    rng = torch.Generator(device=DEV)
    rng.manual_seed(int(seed))
    n_r, n_t, n_p = case["n_r"], case["n_theta"], case["n_phi"]
    rc = _dev(_mid(r))
    u = torch.rand(2, dtype=torch.float64, device=DEV, generator=rng).tolist()
    amp = [0.0] + [1e-2 / l for l in range(1, 9)]
    ang = 1.0 + _angular(rng, 1, 8, amp, _mid(th), _mid(ph))[0]
    phi = -(1e19 + 1e19 * u[0]) / (1.0 + (rc / 1e8) ** 2).sqrt()[:, None, None] * ang
    rho = _core_profile(_mid(r), r[-1], 1e10, 1e8)[:, None, None] * (1.0 + _angular(rng, 1, 8, amp, _mid(th), _mid(ph))[0])
    v = torch.randn(3, n_r, n_t, n_p, dtype=torch.float64, device=DEV, generator=rng)
    v[0] *= 1e8
    v[1:] *= (1e7 / rc)[None, :, None, None]
    return phi.contiguous(), rho.contiguous(), v


def _coarsen_mesh(case):
    n_t = case["n_theta"]
    return _edges({"n_r": int(3.68 * n_t), "n_theta": n_t, "n_phi": 2 * n_t, "radii": "paper", "angles": "even"})


def _coarsen_fields(case, seed, edges):
    n_r, n_t, n_p = (len(e) - 1 for e in edges)
    rng = torch.Generator(device=DEV)
    rng.manual_seed(int(seed))
    f = torch.rand(case["n_fields"], n_r, n_t, n_p, dtype=torch.float64, device=DEV, generator=rng)
    f += 0.5
    return f * (1.0 / (1.0 + (_dev(_mid(edges[0])) / 2.0) ** 2))[None, :, None, None]


def prepare(case, seed):
    if case["do"] == "solve":
        edges = _edges(case)
        rho = _density(case, seed, edges)
        s = {"case": case, "mesh": _mesh(case, edges), "rho": rho, "phi": torch.empty_like(rho)}
        s["mesh"].set_density(rho)
        s["mesh"].set_phi_output(s["phi"])
        if case["moments"]:
            n_r, K = case["n_r"], (case["l_max"] + 1) ** 2
            for key, rows in (("ang", n_r), ("mr", n_r + 1), ("mi", n_r + 1)):
                s[key] = torch.empty(rows, K, dtype=torch.float64, device=DEV)
        return s
    if case["do"] == "batch":
        members = []
        for sub, sub_seed in _batch_members(case, seed):
            members.append(prepare(sub, sub_seed))
        return {"case": case, "members": members, "batch": mpl.Batch([m["mesh"] for m in members])}
    if case["do"] == "gravity":
        edges = _gravity_mesh(case)
        phi, rho, v = _gravity_inputs(case, seed, edges)
        mesh = mpl.Mesh(*edges, 2, G_CGS, precision="fp64")
        return {"case": case, "mesh": mesh, "phi": phi, "rho": rho, "v": v, "S": torch.empty_like(v),
                "E": torch.empty_like(phi)}
    edges = _coarsen_mesh(case)
    return {"case": case, "mesh": mpl.Mesh(*edges, 2, 1.0, precision="fp64"),
            "fields": _coarsen_fields(case, seed, edges)}


def run(state):
    case = state["case"]
    if case["do"] == "solve":
        state["mesh"].solve()
        if not case["moments"]:
            return {"phi": state["phi"]}
        state["mesh"].get_moments(state["ang"], state["mr"], state["mi"])
        return {"phi": state["phi"], "ang": state["ang"], "mr": state["mr"], "mi": state["mi"]}
    if case["do"] == "batch":
        state["batch"].solve()
        return [m["phi"] for m in state["members"]]
    if case["do"] == "gravity":
        state["mesh"].gravity_sources(phi=state["phi"], rho=state["rho"], v=state["v"], S=state["S"], E=state["E"])
        return {"S": state["S"], "E": state["E"]}
    state["mesh"].coarsen(state["fields"], n_fields=case["n_fields"])
    return state["fields"]


# ------------------------------------------------------------------------------ work
def _solve_work(case):
    """The density in, the potential (and the moments) out; the separable sums as products."""
    n_r, n_t, n_p, L = case["n_r"], case["n_theta"], case["n_phi"], case["l_max"]
    K = (L + 1) ** 2
    nbytes = 16 * n_r * n_t * n_p + (8 * K * (3 * n_r + 2) if case["moments"] else 0)
    flops = 2 * 2 * n_r * n_t * (n_p * (2 * L + 1) + K)
    return nbytes, flops


def work(case):
    if case["do"] == "solve":
        b, f = _solve_work(case)
    elif case["do"] == "batch":
        parts = [_solve_work(sub) for sub, _ in _batch_members(case, 0)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif case["do"] == "gravity":
        cells = case["n_r"] * case["n_theta"] * case["n_phi"]
        b, f = 72 * cells, 14 * cells
    else:
        edges = _coarsen_mesh(case)
        c_t, c_p = _block_sizes(edges)
        cells = case["n_fields"] * int(np.sum((c_t[:, None] > 1) | (c_p > 1))) * (len(edges[2]) - 1)
        b, f = 16 * cells, 4 * cells
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------ exact values
def _theta_integrals(l_max, th):
    """Integrals of P~_l^m sin(theta) over the polar cells, [l][m] -> [n_theta]."""
    x, w = np.polynomial.legendre.leggauss(32)
    half = _dev(0.5 * np.diff(th))
    t = _dev(_mid(th))[:, None] + half[:, None] * _dev(x)
    wt = half[:, None] * _dev(w) * torch.sin(t)
    P = _legendre(l_max, torch.cos(t))
    return [[(P[l][m] * wt).sum(1) for m in range(l + 1)] for l in range(l_max + 1)]


def _exact_solve(case, rho, edges):
    r, th, ph = edges
    n_r, n_t, n_p, L = case["n_r"], case["n_theta"], case["n_phi"], case["l_max"]
    G, K = _gravitational_constant(case), (case["l_max"] + 1) ** 2
    It = _theta_integrals(L, th)
    dmu = _dev(2.0 * np.sin(_mid(th)) * np.sin(0.5 * np.diff(th)))
    mid, half = _dev(_mid(ph)), _dev(0.5 * np.diff(ph))
    Ip = torch.empty(2 * L + 1, n_p, dtype=torch.float64, device=DEV)
    Ip[0] = 2.0 * half
    for m in range(1, L + 1):
        s = 2.0 * torch.sin(m * half) / m
        Ip[2 * m - 1], Ip[2 * m] = torch.cos(m * mid) * s, torch.sin(m * mid) * s
    # angular moments
    F = (rho.reshape(n_r * n_t, n_p) @ Ip.T).reshape(n_r, n_t, 2 * L + 1)
    A = torch.empty(n_r, K, dtype=torch.float64, device=DEV)
    for m in range(L + 1):
        W = torch.stack([It[l][m] for l in range(m, L + 1)])
        for p in ([0] if m == 0 else [2 * m - 1, 2 * m]):
            q = torch.tensor([l * l + p for l in range(m, L + 1)], device=DEV)
            A[:, q] = 4.0 * math.pi * G * (F[:, :, p] @ W.T)
    # shell integrals of r^2 r^l and r^2 r^-(l+1), r in units of r_ref
    r_ref = math.sqrt((r[0] if r[0] > 0 else r[1]) * r[-1])
    x0, x1 = r[:-1] / r_ref, r[1:] / r_ref
    WR, WI = np.empty((n_r, L + 1)), np.zeros((n_r, L + 1))
    own = slice(0 if x0[0] > 0 else 1, None)
    lr = np.log1p((x1[own] - x0[own]) / x0[own])

    def diff(p):
        return x0[own] ** p * np.expm1(p * lr)

    for l in range(L + 1):
        WR[own, l] = r_ref ** 3 * diff(l + 3.0) / (l + 3.0)
        WI[own, l] = r_ref ** 2 * (lr if l == 2 else diff(2.0 - l) / (2.0 - l))
        if x0[0] == 0:
            WR[0, l] = r_ref ** 3 * x1[0] ** (l + 3.0) / (l + 3.0)
            WI[0, l] = r_ref ** 2 * x1[0] ** (2.0 - l) / (2.0 - l) if l < 2 else 0.0
    vol = np.empty(n_r)
    vol[own] = (r[:-1][own] ** 3) * np.expm1(3.0 * lr) / 3.0
    if x0[0] == 0:
        vol[0] = r[1] ** 3 / 3.0
    deg = torch.tensor([l for l in range(L + 1) for _ in range(2 * l + 1)], device=DEV)
    two = torch.tensor([1.0 if p == 0 else 2.0 for l in range(L + 1) for p in range(2 * l + 1)], dtype=torch.float64,
                       device=DEV)
    wr, wi = _dev(WR)[:, deg], _dev(WI)[:, deg]
    zero = torch.zeros(1, K, dtype=torch.float64, device=DEV)
    MR = torch.cat([zero, torch.cumsum(wr * A, 0)])
    MI = torch.cat([torch.flip(torch.cumsum(torch.flip(wi * A, [0]), 0), [0]), zero])
    h = -0.5 / (2.0 * deg.double() + 1.0)
    v = _dev(vol)[:, None]
    C = h * (wr / v * (MI[:-1] + MI[1:]) + wi / v * (MR[:-1] + MR[1:]))
    if x0[0] == 0:  # the shell at the origin: its own degrees l >= 2 as a uniform ball's
        ball = h * 2.0 * (wr[0] / v[0] * MI[1] + 6.0 * r[1] ** 2 / (5.0 * (deg.double() + 3.0)) * A[0])
        C[0] = torch.where(deg >= 2, ball, C[0])
    C *= two
    del F, wr, wi
    # potential
    Gm = torch.empty(n_r, n_t, 2 * L + 1, dtype=torch.float64, device=DEV)
    for m in range(L + 1):
        W = torch.stack([It[l][m] / dmu for l in range(m, L + 1)])
        for p in ([0] if m == 0 else [2 * m - 1, 2 * m]):
            q = torch.tensor([l * l + p for l in range(m, L + 1)], device=DEV)
            Gm[:, :, p] = C[:, q] @ W
    phi = (Gm.reshape(n_r * n_t, -1) @ (Ip / (2.0 * half))).reshape(n_r, n_t, n_p)
    if not case["moments"]:
        return {"phi": phi}
    return {"phi": phi, "ang": A, "mr": MR, "mi": MI}


def _difference(f, dim, edges, wraps):
    xc = _dev(_mid(edges))
    n = f.shape[dim]
    if n == 1:
        return torch.zeros_like(f)
    k = torch.arange(n, device=DEV)
    if wraps:
        lo, hi = (k - 1) % n, (k + 1) % n
        dx = xc[hi] + TWO_PI * (k == n - 1).double() - (xc[lo] - TWO_PI * (k == 0).double())
    else:
        lo, hi = (k - 1).clamp(min=0), (k + 1).clamp(max=n - 1)
        dx = xc[hi] - xc[lo]
    w = torch.where(lo == hi, torch.zeros_like(dx), 1.0 / dx)
    return (f.index_select(dim, hi) - f.index_select(dim, lo)) * w.reshape([-1 if d == dim else 1 for d in range(3)])


def _block_sizes(edges):
    """Cells per coarsening block: polar [n_r], azimuthal [n_r][n_theta] (Sec. 2.1)."""
    r, th, ph = edges
    dr, rc, tc = float(np.min(np.diff(r))), _mid(r), _mid(th)
    n_t, n_p = len(tc), len(ph) - 1

    def block(need, n):
        p = 1
        while p <= n:
            if n % p == 0 and p >= need:
                return p
            p *= 2
        return n

    polar = dr / (rc * float(np.min(np.diff(th))))
    azim = dr / (rc[:, None] * np.sin(tc)[None, :] * float(np.min(np.diff(ph))))
    c_t = np.array([block(p, n_t) for p in polar])
    c_p = np.empty((len(rc), n_t), dtype=np.int64)
    for i, ct in enumerate(c_t):
        for j in range(0, n_t, ct):
            c_p[i, j:j + ct] = block(float(np.max(azim[i, j:j + ct])), n_p)
    return c_t, c_p


def _exact_coarsen(case, f, edges):
    n_r, n_t, n_p = (len(e) - 1 for e in edges)
    c_t, c_p = _block_sizes(edges)
    dmu, dph = _dev(-np.diff(np.cos(edges[1]))), _dev(np.diff(edges[2]))
    for i in range(n_r):
        ct = int(c_t[i])
        of_block = c_p[i, ::ct]
        x = f[:, i].reshape(case["n_fields"], n_t // ct, ct, n_p)
        for cp in np.unique(of_block):
            if ct == 1 and cp == 1:
                continue
            at = torch.as_tensor(np.nonzero(of_block == cp)[0], device=DEV)
            y = x[:, at].reshape(case["n_fields"], len(at), ct, n_p // int(cp), int(cp))
            w = dmu.reshape(-1, ct)[at][:, :, None, None] * dph.reshape(1, 1, -1, int(cp))
            mean = (y * w).sum((2, 4), keepdim=True) / w.sum((1, 3), keepdim=True)
            x[:, at] = mean.expand_as(y).reshape(case["n_fields"], len(at), ct, n_p)
    return f


def exact(case, seed):
    if case["do"] == "solve":
        edges = _edges(case)
        return _exact_solve(case, _density(case, seed, edges), edges)
    if case["do"] == "batch":
        return [exact(sub, sub_seed)["phi"] for sub, sub_seed in _batch_members(case, seed)]
    if case["do"] == "gravity":
        edges = _gravity_mesh(case)
        phi, rho, v = _gravity_inputs(case, seed, edges)
        g = [_difference(phi, d, edges[d], d == 2) for d in range(3)]
        S = torch.stack([-rho * x for x in g])
        return {"S": S, "E": (v * S).sum(0)}
    edges = _coarsen_mesh(case)
    return _exact_coarsen(case, _coarsen_fields(case, seed, edges), edges)
