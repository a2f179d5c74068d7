"""The performance cases: the work that users of this framework have it do, each
as one pass through the public entry points (``RadioProcess``, ``RadioTraces``,
``Batch``), with its inputs, its least traffic and arithmetic, and the same
result in 64 bits from plain torch.

A case is a dict of plain values:

* ``op``: "traces" (push a shower, fetch the traces), "step" (traces and every
  gradient of a loss through ``RadioTraces``) or "batch" (many uneven showers);
* ``formalism``, ``precision``, ``medium``, ``deposit``: as the framework names them;
* ``tracks``, ``layout`` ("line", "star" or "grid"), ``antennas``, ``hills`` (m,
  antenna altitudes spread over that range; 0: a flat array), ``zenith`` (degrees),
  ``bins``, ``dt`` (ns); for "batch": ``showers``, and ``tracks`` is the most of one.

The showers have the shape of the framework's own benchmark showers: start height
N(4 km, 1.5 km) within [0.5, 10] km, lateral offset Exp(30 m), directions 5 degrees
about the axis, lengths U[0.5, 5] m, Lorentz factors log-uniform in [10, 1e4], and
55 % electrons; each trace starts 50 ns before the shower front arrives.
"""
import math

import numpy as np
import torch

from paper_2309_03717_gb300 import c8r

C_NS = 0.299792458               # m/ns
C_SI = 299792458.0
EPS0 = 8.8541878128e-12
QE = 1.602176634e-19
K_ENDPOINT = QE / (4.0 * math.pi * EPS0 * C_SI)
K_ZHS = QE / (4.0 * math.pi * EPS0 * C_SI)  # mu0 e c / (4 pi), mu0 = 1/(eps0 c^2)
EPS_CHERENKOV = 1e-3
MEDIA = {
    "uniform": {"kind": "uniform", "n": 1.000292},
    "exponential": {"kind": "exponential", "N0": 3.25e-4, "H": 8000.0},
    "exponential_spherical": {"kind": "exponential_spherical", "N0": 3.25e-4, "H": 8000.0, "R_E": 6.371e6},
    "exponential_ray": {"kind": "exponential_ray", "N0": 3.25e-4, "H": 8000.0},
}
TRACK = c8r.TRACK_FIELDS
GRADS = c8r.GRAD_FIELDS


def _case(name, op="traces", formalism="endpoint", precision="mixed", medium="exponential", deposit="bin",
          tracks=1000, layout="star", antennas=160, hills=0.0, zenith=0.0, bins=4096, dt=0.2, showers=0):
    c = dict(op=op, formalism=formalism, precision=precision, medium=medium, deposit=deposit, tracks=tracks,
             layout=layout, antennas=antennas, hills=hills, zenith=zenith, bins=bins, dt=dt, showers=showers)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small event on a few antennas, fetched at once: launches and latency count
        _case("small_event", tracks=3000, layout="line", antennas=8),
        # the reference-precision run on an east line: FP64 Endpoint, uniform air
        _case("line16_fp64", precision="fp64", medium="uniform", tracks=100_000, layout="line", antennas=16),
        # reference-precision ZHS traces of a thinned shower on the star array
        _case("star160_zhs_fp64", formalism="zhs", precision="fp64", tracks=100_000),
        # a vertical shower on the 160-antenna star, one chunk of tracks
        _case("star160_endpoint", tracks=4_000_000),
        # the whole vertical shower on the star array, vector potentials
        _case("star160_zhs", formalism="zhs", tracks=20_000_000),
        # an inclined shower on the large next-generation array, one streamed chunk
        _case("grid1024_inclined", tracks=4_000_000, layout="grid", antennas=1024, zenith=60.0, bins=8192, dt=0.1),
        # one step of a fit: traces and the gradient of every input, Endpoint
        _case("fit_endpoint", op="step", tracks=1_000_000, antennas=64, bins=2048),
        # the same with ZHS on hilly ground, ragged sizes
        _case("fit_zhs_hills", op="step", formalism="zhs", tracks=300_007, antennas=61, hills=150.0, zenith=30.0,
              bins=2048),
        # a library of uneven showers in one launch
        _case("batch64", op="batch", tracks=100_000, antennas=512, showers=64),
        # traces that are continuous in the arrival times (two-bin deposits)
        _case("star160_linear", deposit="linear", tracks=1_000_000),
        # the Earth's curvature in the propagator, inclined shower, large array
        _case("grid1024_spherical_zhs", formalism="zhs", medium="exponential_spherical", tracks=250_000,
              layout="grid", antennas=1024, zenith=60.0, bins=8192, dt=0.1),
        # refracted rays in the propagator, inclined shower
        _case("grid256_ray_zhs", formalism="zhs", medium="exponential_ray", tracks=250_000, layout="grid",
              antennas=256, zenith=60.0, bins=8192, dt=0.1),
    ]


# pairs per millisecond that the cap on a drawn case's size reckons with, by kind
_PAIRS_PER_MS = {"fp64": 2e6, "step": 1.5e7, "exponential_spherical": 4e7, "exponential_ray": 2.5e7, "linear": 4e7}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "fp64", "fp64", "mixed", "mixed", "mixed", "mixed", "step", "step", "batch", "linear",
                       "heavy"])
    c = _case(None)
    c["formalism"] = rng.choice(["endpoint", "zhs"])
    c["layout"] = rng.choice(["line", "star", "grid"])
    c["zenith"] = rng.choice([0.0, round(rng.uniform(0.0, 65.0), 1)])
    c["hills"] = rng.choice([0.0, 0.0, 0.0, round(rng.uniform(10.0, 150.0), 1)])
    c["bins"], c["dt"] = rng.choice([(1000, 0.5), (2048, 0.2), (4096, 0.2), (4096, 0.2), (8192, 0.1)])
    c["medium"] = rng.choice(["uniform", "exponential", "exponential"])
    most_tracks, most_ant, rate = 4_000_000, 1024, 6e7
    if kind == "small":
        most_tracks, most_ant = 10_000, 32
        c["precision"] = rng.choice(["mixed", "mixed", "fp64"])
    elif kind == "fp64":
        c["precision"] = "fp64"
        most_tracks, most_ant, rate = 400_000, 200, _PAIRS_PER_MS["fp64"]
    elif kind == "step":
        c["op"] = "step"
        most_tracks, most_ant, rate = 1_000_000, 128, _PAIRS_PER_MS["step"]
    elif kind == "linear":
        c["deposit"] = "linear"
        rate = _PAIRS_PER_MS["linear"]
    elif kind == "heavy":
        # the costlier propagators, with the formalism whose traces are
        # continuous in the arrival time
        c["medium"] = rng.choice(["exponential_spherical", "exponential_ray"])
        c["formalism"] = "zhs"
        most_tracks, rate = 1_000_000, _PAIRS_PER_MS[c["medium"]]
    elif kind == "batch":
        c.update(op="batch", showers=rng.randint(2, 64), hills=0.0, zenith=0.0, layout="star")
        c["tracks"] = _log_int(rng, 2_000, 200_000)
        c["antennas"] = rng.randint(16, 512)
        return c
    if c["layout"] == "line":
        most_ant = min(most_ant, 64)
    c["antennas"] = _log_int(rng, 1, most_ant)
    # at most ~20 ms of work: the largest listed case takes about twice that
    cap = min(most_tracks, 20.0 * rate / c["antennas"])
    c["tracks"] = _log_int(rng, min(1000, cap), max(1001, cap))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _antennas(layout, count, hills, seed):
    if layout == "line":
        x = 25.0 * np.arange(1, count + 1)
        pos = np.stack([x, np.zeros_like(x), np.zeros_like(x)], 1)
    elif layout == "star":
        per_arm = max(1, math.ceil(count / 8))
        radii = np.linspace(10.0, 400.0, per_arm) if per_arm > 1 else np.array([100.0])
        ang = 2.0 * math.pi * np.arange(8) / 8
        pos = np.stack([np.outer(np.cos(ang), radii).ravel(), np.outer(np.sin(ang), radii).ravel(),
                        np.zeros(8 * per_arm)], 1)[:count]
    else:
        side = math.ceil(math.sqrt(count))
        c = (np.arange(side) - (side - 1) / 2.0) * 50.0
        X, Y = np.meshgrid(c, c, indexing="ij")
        pos = np.stack([X.ravel(), Y.ravel(), np.zeros(side * side)], 1)[:count]
    if hills:
        pos[:, 2] = np.random.default_rng(seed + 77).uniform(0.0, hills, size=len(pos))
    return np.ascontiguousarray(pos)


def _starts(pos, zenith):
    z = math.radians(zenith)
    return (10000.0 - (pos[:, 0] * math.sin(z) + pos[:, 2] * math.cos(z))) / C_NS - 50.0


def _shower(n, seed, zenith, dtype):
    """n shower-like tracks on the GPU (a dict of tensors of the framework's track fields)."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))

    def u():
        return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)

    def normal():
        return torch.randn(n, generator=g, device="cuda", dtype=torch.float64)

    lo, hi = (0.5 * math.erfc(-v / math.sqrt(2.0)) for v in ((500.0 - 4000.0) / 1500.0, (10000.0 - 4000.0) / 1500.0))
    h = (4000.0 + 1500.0 * torch.special.ndtri(lo + (hi - lo) * u())).clamp(500.0, 10000.0)
    r = -30.0 * torch.log(1.0 - u())
    phi = 2.0 * math.pi * u()
    sig = math.radians(5.0)
    ax, ay = sig * normal(), sig * normal()
    length = 0.5 + 4.5 * u()
    gamma = torch.exp(math.log(10.0) + math.log(1e3) * u())
    q = torch.where(u() < 0.55, -1.0, 1.0)
    ux, uy, uz = -torch.cos(ax) * torch.sin(ay), torch.sin(ax), -torch.cos(ax) * torch.cos(ay)
    norm = torch.sqrt(ux * ux + uy * uy + uz * uz)
    d = [ux / norm, uy / norm, uz / norm]
    x = [r * torch.cos(phi), r * torch.sin(phi), h]
    if zenith:
        c, s = math.cos(math.radians(zenith)), math.sin(math.radians(zenith))
        x = [c * x[0] + s * x[2], x[1], c * x[2] - s * x[0]]
        d = [c * d[0] + s * d[2], d[1], c * d[2] - s * d[0]]
    bmag = torch.sqrt(1.0 - 1.0 / (gamma * gamma))
    b = torch.stack([v * bmag for v in d]).to(dtype)
    if dtype == torch.float32:
        # rounding may bring |beta| to 1: scale those down
        for _ in range(8):
            over = (b.double() ** 2).sum(0) >= 1.0
            b = torch.where(over, (b.double() * (1.0 - 2e-7)).to(dtype), b)
    bn = torch.sqrt((b.double() ** 2).sum(0))
    t0 = (10000.0 - h) / C_NS
    t1 = t0 + length / (bn * C_NS)
    f = [x[0], x[1], x[2], x[0] + d[0] * length, x[1] + d[1] * length, x[2] + d[2] * length, t0, t1, b[0], b[1], b[2],
         q]
    return {k: v.to(dtype).contiguous() for k, v in zip(TRACK, f)}


def _batch_plan(case):
    """(tracks, antennas, zenith, layout) of each shower: log-uniform tracks over two decades
    up to the case's most, antennas uniform from 16 up to the case's; the same for every seed."""
    rng = np.random.default_rng(9_000_000 + case["tracks"] + 1000 * case["showers"] + case["antennas"])
    plan = []
    for s in range(case["showers"]):
        n = int(round(case["tracks"] * 10.0 ** rng.uniform(-2.0, 0.0)))
        a = int(rng.integers(16, max(17, case["antennas"] + 1)))
        plan.append((max(n, 1), a, float(rng.uniform(0.0, 65.0)), "grid" if s % 2 else "star"))
    return plan


def _cotangent(case, seed, antennas):
    """dL/dtraces of a loss of order one."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
    scale = 1e9 if case["formalism"] == "endpoint" else 1e18
    return scale * torch.randn((antennas, 3, case["bins"]), generator=g, device="cuda", dtype=torch.float32)


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _inputs(case, seed):
    if case["op"] == "batch":
        plan = _batch_plan(case)
        showers = []
        for s, (n, a, zen, layout) in enumerate(plan):
            pos = _antennas(layout, a, 0.0, seed)
            showers.append(dict(n_tracks=n, ant_xyz=pos, t_start_ns=_starts(pos, zen),
                                tracks=_shower(n, 1000 * seed + s, zen, torch.float32)))
        return showers
    pos = _antennas(case["layout"], case["antennas"], case["hills"], seed)
    return dict(ant_xyz=pos, t_start_ns=_starts(pos, case["zenith"]),
                tracks=_shower(case["tracks"], seed, case["zenith"], _dtype(case)))


def prepare(case, seed):
    medium = MEDIA[case["medium"]]
    if case["op"] == "batch":
        showers = _inputs(case, seed)
        tracks = {f: torch.cat([s["tracks"][f] for s in showers]) for f in TRACK}
        batch = c8r.Batch([{k: s[k] for k in ("n_tracks", "ant_xyz", "t_start_ns")} for s in showers], medium,
                          case["bins"], case["dt"], case["formalism"])
        return dict(op="batch", batch=batch, tracks=tracks, out=batch.new_output())
    w = _inputs(case, seed)
    p = c8r.RadioProcess(medium, w["ant_xyz"], w["t_start_ns"], case["bins"], case["dt"], case["formalism"],
                         case["precision"], deposit=case["deposit"])
    state = dict(op=case["op"], process=p, tracks=w["tracks"])
    if case["op"] == "step":
        n0 = medium["N0"] if "N0" in medium else medium["n"] - 1.0
        state["N0"] = torch.tensor(n0, dtype=torch.float64, device="cuda", requires_grad=True)
        state["ant"] = torch.from_numpy(w["ant_xyz"]).cuda().requires_grad_(True)
        for f in GRADS:
            state["tracks"][f].requires_grad_(True)
        state["G"] = _cotangent(case, seed, len(w["ant_xyz"]))
    return state


def run(state):
    if state["op"] == "batch":
        out = state["out"].zero_()
        state["batch"].run(state["tracks"], out)
        return out
    p, tracks = state["process"], state["tracks"]
    if state["op"] == "traces":
        p.push(tracks)
        return p.traces(reset=True)
    leaves = [state["N0"], state["ant"]] + [tracks[f] for f in GRADS]
    tr = c8r.RadioTraces.apply(p, state["N0"], *[tracks[f] for f in TRACK], state["ant"])
    grads = torch.autograd.grad(tr, leaves, state["G"])
    return {"traces": tr.detach(), "N0": grads[0], "antennas": grads[1],
            **{f: g for f, g in zip(GRADS, grads[2:])}}


def work(case):
    if case["op"] == "batch":
        plan = _batch_plan(case)
        n, a = sum(p[0] for p in plan), sum(p[1] for p in plan)
        pairs = sum(p[0] * p[1] for p in plan)
    else:
        n, a = case["tracks"], case["antennas"]
        pairs = n * a
    es = 8 if case["precision"] == "fp64" else 4
    nbytes = 12 * es * n + 32 * a + 3 * es * a * case["bins"]
    # operations of the plain formulas per (track, antenna) pair
    ops = 62 if case["formalism"] == "endpoint" else 54
    if case["op"] == "step":
        # the cotangent and the tracks read, every gradient written
        nbytes += 3 * 4 * a * case["bins"] + (12 + 11) * es * n + 24 * a
        ops += 184
    return {"bytes": float(nbytes), "flops": float(ops * pairs)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, plain torch
# ---------------------------------------------------------------------------
_NODES, _WEIGHTS = (torch.from_numpy(v) for v in np.polynomial.legendre.leggauss(16))


class _Medium:
    def __init__(self, spec, n0):
        self.kind, self.n0 = spec["kind"], n0
        self.H, self.RE = spec.get("H", 1.0), spec.get("R_E", 0.0)

    def nu(self, x, y, z):
        """n - 1 at a point."""
        if self.kind == "uniform":
            return self.n0
        if self.kind == "exponential_spherical":
            z = torch.sqrt(x * x + y * y + (z + self.RE) ** 2) - self.RE
        return self.n0 * torch.exp(-z / self.H)

    def path(self, e, a):
        """Distance, unit direction at the emission point, n there and optical path from e to a."""
        d = [a[k] - e[k] for k in range(3)]
        R = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        rh = [v / R for v in d]
        nu_e = self.nu(*e)
        if self.kind == "uniform":
            return R, rh, 1.0 + nu_e, R + nu_e * R
        if self.kind == "exponential_spherical":
            mean = 0.0
            for s, w in zip(_NODES.tolist(), _WEIGHTS.tolist()):
                f = 0.5 * (1.0 + s)
                mean = mean + 0.5 * w * self.nu(*[e[k] + f * d[k] for k in range(3)])
            return R, rh, 1.0 + nu_e, R + mean * R
        x = d[2] / self.H
        small = x.abs() < 1e-2
        xs = torch.where(small, torch.ones_like(x), x)
        ratio = torch.where(small, 1 + x * (-1 / 2 + x * (1 / 6 + x * (-1 / 24 + x * (1 / 120 + x * (-1 / 720 + x / 5040))))),
                            -torch.expm1(-xs) / xs)
        opt = R + nu_e * ratio * R
        if self.kind == "exponential_ray":
            rho = torch.sqrt(d[0] ** 2 + d[1] ** 2)
            adz = d[2].abs()
            bent = (rho > 0) & (adz >= 1e-3 * R)
            S = rho / R
            nus = [nu_e * torch.exp(-0.5 * (1.0 + s) * x) for s in _NODES.tolist()]
            p = S * (1.0 + nu_e * ratio)
            for _ in range(5):  # Newton's method on the end-point condition
                f, df = -rho / adz, 0.0
                for nu, w in zip(nus, _WEIGHTS.tolist()):
                    c = torch.sqrt((1.0 + nu) ** 2 - p * p)
                    f = f + 0.5 * w * p / c
                    df = df + 0.5 * w * (1.0 + nu) ** 2 / c ** 3
                p = p - f / df
            ray = 0.0
            for nu, w in zip(nus, _WEIGHTS.tolist()):
                ray = ray + 0.5 * w * (1.0 + nu) ** 2 / torch.sqrt((1.0 + nu) ** 2 - p * p)
            opt = torch.where(bent, ray * adz, opt)
            st = p / (1.0 + nu_e)
            ct = torch.sqrt(1.0 - st * st) * torch.sign(d[2])
            safe = torch.where(rho > 0, rho, torch.ones_like(rho))
            rh = [torch.where(bent, v, o) for v, o in zip((st * d[0] / safe, st * d[1] / safe, ct), rh)]
        return R, rh, 1.0 + nu_e, opt


def _rows(t, ant, t_start):
    """Track columns [n, 1] and antenna rows [1, A]."""
    v = {f: t[f][:, None] for f in TRACK}
    return v, [ant[None, :, k] for k in range(3)], t_start[None, :]


def _field(b, rh, n):
    c = b[0] * rh[0] + b[1] * rh[1] + b[2] * rh[2]
    return [c * rh[k] - b[k] for k in range(3)], 1.0 - n * c


def _deposits(case, med, t, ant, t_start, keep):
    """The deposits of a chunk: a list of (weight vector [n, A] x 3, bin [n, A], use [n, A]),
    and of boxes (vector, first bin, last bin, use), every quantity differentiable with the bins held fixed."""
    v, a, ts = _rows(t, ant, t_start)
    dt = case["dt"]
    e0, e1 = [v[f] for f in ("x0", "y0", "z0")], [v[f] for f in ("x1", "y1", "z1")]
    em = [0.5 * (p + r) for p, r in zip(e0, e1)]
    b = [v[f] for f in ("bx", "by", "bz")]
    t0, t1, q = v["t0"], v["t1"], v["q"]
    N = case["bins"]
    keep = keep[:, None]
    one, box = [], []

    def point(u, vec, use):
        """A point deposit: in its bin, or spread over a bin's width."""
        if case["deposit"] == "bin":
            one.append((vec, torch.floor(u.detach()), use))
            return
        k = torch.floor(u.detach() - 0.5)
        f = u - 0.5 - k
        one.append(([x * (1.0 - f) for x in vec], k, use))
        one.append(([x * f for x in vec], k + 1.0, use))

    if case["formalism"] == "endpoint":
        K = q * K_ENDPOINT / (dt * 1e-9)
        (R0, r0, n0, o0), (R1, r1, n1, o1) = med.path(e0, a), med.path(e1, a)
        (V0, D0), (V1, D1) = _field(b, r0, n0), _field(b, r1, n1)
        near = torch.minimum(D0.abs(), D1.abs()).detach() < EPS_CHERENKOV
        far = keep & ~near
        u0, u1 = ((t0 - ts) + o0 / C_NS) / dt, ((t1 - ts) + o1 / C_NS) / dt
        point(u0, [K / (D0 * R0) * x for x in V0], far)
        point(u1, [-K / (D1 * R1) * x for x in V1], far)
        # near the Cherenkov angle: midpoint, linearised arrivals
        near = near & keep
        Rm, rm, nm, om = med.path(em, a)
        Vm, Dm = _field(b, rm, nm)
        um = (0.5 * (t0 + t1) - ts + om / C_NS) / dt
        h = Dm * (t1 - t0) / (2.0 * dt)
        ua, ub = um - h, um + h
        shift = 0.0 if case["deposit"] == "bin" else 0.5
        ka, kb = torch.floor(ua.detach() + shift), torch.floor(ub.detach() + shift)
        same = near & (ka == kb)
        if case["deposit"] == "linear":
            B = K * ((t1 - t0) / dt) / Rm
            one.append(([B * x for x in Vm], ka - 1.0, same))
            one.append(([-B * x for x in Vm], ka, same))
        apart = near & (ka != kb)
        s = K / (torch.where(apart, Dm, torch.ones_like(Dm)) * Rm)
        point(ua, [s * x for x in Vm], apart)
        point(ub, [-s * x for x in Vm], apart)
        return one, box
    # ZHS: the step potential over the interval u_m -/+ |D| (t1 - t0)/(2 dt)
    Rm, rm, nm, om = med.path(em, a)
    Vm, Dm = _field(b, rm, nm)
    A = q * K_ZHS * (t1 - t0) / dt / Rm
    vec = [-A * x for x in Vm]
    um = (0.5 * (t0 + t1) - ts + om / C_NS) / dt
    h = Dm.abs() * (t1 - t0) / (2.0 * dt)
    lo, hi = um - h, um + h
    shift = 0.0 if case["deposit"] == "bin" else 0.5
    klo, khi = torch.floor(lo.detach() + shift), torch.floor(hi.detach() + shift)
    single, multi = keep & (klo == khi), keep & (klo != khi)
    W = torch.where(multi, 2.0 * h, torch.ones_like(h))
    if case["deposit"] == "bin":
        one.append((vec, klo, single))
        wl, wh = (klo + 1.0 - lo) / W, (hi - khi) / W
        one.append(([x * wl for x in vec], klo, multi))
        one.append(([x * wh for x in vec], khi, multi))
        box.append(([x / W for x in vec], klo + 1.0, khi - 1.0, multi & (khi - klo >= 2)))
        return one, box
    f = um + 0.5 - klo
    one.append(([x * (1.0 - f) for x in vec], klo - 1.0, single))
    one.append(([x * f for x in vec], klo, single))
    # two-bin deposits averaged over the interval: by cells [J - 1/2, J + 1/2], each
    # shared between bins J - 1 and J
    sl, sh = lo + 0.5 - klo, hi + 0.5 - khi
    for w, k in ((0.5 * (1.0 - sl) ** 2, klo - 1.0), (0.5 * (1.0 - sl * sl), klo),
                 (sh * (1.0 - 0.5 * sh), khi - 1.0), (0.5 * sh * sh, khi)):
        one.append(([x * w / W for x in vec], k, multi))
    whole = multi & (khi - klo >= 2)
    half = [0.5 * x / W for x in vec]
    box.append((half, klo, khi - 2.0, whole))      # each whole cell J: 1/2 to bin J - 1
    box.append((half, klo + 1.0, khi - 1.0, whole))  # and 1/2 to bin J
    return one, box


def _kept(t):
    ok = (t["q"] != 0) & (t["t1"] > t["t0"])
    ok &= (t["x1"] != t["x0"]) | (t["y1"] != t["y0"]) | (t["z1"] != t["z0"])
    s = t["bx"] ** 2 + t["by"] ** 2 + t["bz"] ** 2
    return ok & (s > 0) & (s < 1)


def _exact_traces(case, med, tracks, ant, t_start, tr, edge):
    N, A = case["bins"], ant.shape[0]
    rows = (torch.arange(A, device="cuda") * (3 * N))[None, :]
    n = tracks["x0"].numel()
    step = max(1, 4_000_000 // A)
    for i in range(0, n, step):
        t = {f: tracks[f][i:i + step] for f in TRACK}
        one, box = _deposits(case, med, t, ant, t_start, _kept(t))
        for vec, k, use in one:
            use = (use & (k >= 0) & (k < N)).expand(-1, A)
            at = (rows + k.long())[use]
            for c in range(3):
                tr.index_add_(0, at + c * N, vec[c].expand_as(use)[use])
        for vec, k0, k1, use in box:
            k0, k1 = k0.clamp(min=0), k1.clamp(max=N - 1)
            use = (use & (k0 <= k1)).expand(-1, A)
            first = (rows + k0.long())[use]
            after = (rows + k1.long() + 1)[use]
            inside = (k1 + 1 < N).expand_as(use)[use]
            for c in range(3):
                x = vec[c].expand_as(use)[use]
                edge.index_add_(0, first + c * N, x)
                edge.index_add_(0, after[inside] + c * N, -x[inside])


def _exact_grads(case, med_spec, n0, tracks, ant, t_start, G):
    """The gradients of sum(G traces) with the bins held fixed."""
    N, A = case["bins"], ant.shape[0]
    P = torch.cat([torch.zeros((A, 3, 1), dtype=torch.float64, device="cuda"), torch.cumsum(G, 2)], 2)
    rows = torch.arange(A, device="cuda")[None, :]
    n0 = n0.clone().requires_grad_(True)
    ant = ant.clone().requires_grad_(True)
    got = [torch.zeros_like(n0), torch.zeros_like(ant)]
    parts = {f: [] for f in GRADS}
    n = tracks["x0"].numel()
    step = max(1, 2_000_000 // A)
    for i in range(0, n, step):
        t = {f: tracks[f][i:i + step].clone().requires_grad_(f != "q") for f in TRACK}
        med = _Medium(med_spec, n0)
        one, box = _deposits(case, med, t, ant, t_start, _kept({f: x.detach() for f, x in t.items()}))
        loss = 0.0
        for vec, k, use in one:
            use = (use & (k >= 0) & (k < N)).expand(-1, A)
            kk = torch.where(use, k, torch.zeros_like(k)).long()
            for c in range(3):
                loss = loss + (torch.where(use, vec[c], 0.0) * G[rows, c, kk]).sum()
        for vec, k0, k1, use in box:
            k0, k1 = k0.clamp(min=0), k1.clamp(max=N - 1)
            use = (use & (k0 <= k1)).expand(-1, A)
            a0 = torch.where(use, k0, torch.zeros_like(k0)).long()
            a1 = torch.where(use, k1 + 1.0, torch.zeros_like(k1)).long()
            for c in range(3):
                loss = loss + (torch.where(use, vec[c], 0.0) * (P[rows, c, a1] - P[rows, c, a0])).sum()
        leaves = [n0, ant] + [t[f] for f in GRADS]
        g = torch.autograd.grad(loss, leaves, allow_unused=True)
        g = [torch.zeros_like(x) if y is None else y for x, y in zip(leaves, g)]
        got[0] += g[0]
        got[1] += g[1]
        for f, x in zip(GRADS, g[2:]):
            parts[f].append(x)
    return got[0], got[1], {f: torch.cat(parts[f]) for f in GRADS}


def exact(case, seed):
    if work(case)["flops"] > 1e11:
        return None  # tens of seconds
    spec = MEDIA[case["medium"]]
    n0 = torch.tensor(spec["N0"] if "N0" in spec else spec["n"] - 1.0, dtype=torch.float64, device="cuda")
    med = _Medium(spec, n0)
    w = _inputs(case, seed)
    showers = w if case["op"] == "batch" else [w]
    outs = []
    for s in showers:
        ant = torch.from_numpy(s["ant_xyz"]).cuda()
        ts = torch.from_numpy(np.ascontiguousarray(s["t_start_ns"])).cuda()
        tracks = {f: x.double() for f, x in s["tracks"].items()}
        tr = torch.zeros(ant.shape[0] * 3 * case["bins"], dtype=torch.float64, device="cuda")
        edge = torch.zeros_like(tr)
        _exact_traces(case, med, tracks, ant, ts, tr, edge)
        outs.append(tr.view(-1, 3, case["bins"]) + torch.cumsum(edge.view(-1, 3, case["bins"]), 2))
    traces = torch.cat(outs)
    if case["op"] != "step":
        return traces
    g0, ga, gt = _exact_grads(case, spec, n0, tracks, ant, ts, _cotangent(case, seed, ant.shape[0]).double())
    return {"traces": traces, "N0": g0, "antennas": ga, **gt}
