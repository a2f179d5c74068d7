"""The series of the curved-ray and spherical-Earth propagators for flat antenna
arrays: on the host, the ray series in FP64 against the exact solve inside the range
the kernels take it in (T^2 b < 4e-3 and b < 1e-2), and on the GPU the arrivals
against the quadrature's in media where the range ends: dense and steep atmospheres,
small spheres."""
import numpy as np
import pytest

from _util import built_lib, oracle_arrivals, to_device
from paper_2309_03717_gb300 import synth

GATE_T2B, GATE_B = 4e-3, 1e-2
_s, _w = np.polynomial.legendre.leggauss(8)
SIGMA, WEIGHT = np.longdouble(0.5) * (1 + _s.astype(np.longdouble)), np.longdouble(0.5) * _w.astype(np.longdouble)


def exact_change(C, nu_e, x):
    """Optical path of the refracted ray less the straight line's, per metre of the
    straight line, and C Q, for the line at cosine C to the vertical from a point of
    refractivity nu_e over x scale heights: Snell's constant p = n sin(theta) by
    Newton's method on the end-point condition, at the same nodes."""
    nu = np.longdouble(nu_e) * np.exp(-SIGMA * x)
    n, C = 1 + nu, np.longdouble(C)
    S = np.sqrt(1 - C * C)
    p = S * (1 + (WEIGHT * nu).sum())
    for _ in range(60):
        c = np.sqrt(n * n - p * p)
        step = ((WEIGHT * p / c).sum() - S / C) / (WEIGHT * n * n / c ** 3).sum()
        p = p - step
        if abs(step) < 1e-18:
            break
    # n ds - straight = 2 n sin^2((theta - theta_s)/2)/C, free of cancellation
    turn = np.arcsin(p / n) - np.arctan2(S, C)
    change = -2 * (WEIGHT * n * np.sin(turn / 2) ** 2).sum()
    return change, C * np.sin(np.arcsin(p / (1 + np.longdouble(nu_e))) - np.arctan2(S, C)) / S


def series_change(C, nu_e, x):
    nu = np.longdouble(nu_e) * np.exp(-SIGMA * x)
    r = nu / (1 + nu)
    mean = (WEIGHT * r).sum()
    inv_abar = 1 / (1 - mean)
    b = (mean - r) * inv_abar
    B2, B3, B4 = ((WEIGHT * b ** k).sum() for k in (2, 3, 4))
    be = (mean - nu_e / (1 + np.longdouble(nu_e))) * inv_abar
    nu_a = np.longdouble(nu_e) * np.exp(np.longdouble(-x))
    bmax = max(abs(be), abs((mean - nu_a / (1 + nu_a)) * inv_abar))
    T2 = 1 / np.longdouble(C) ** 2 - 1
    t = -T2 / 2 * (3 * B2 + B3 * (1 + 5 * T2))
    v = B2 / 2 + B3 * (T2 / 2 - 0.5) + (T2 * (T2 * 0.625 - 0.375) + 0.5) * B4 - 1.125 * (T2 * B2) ** 2
    e = t + (1 + t) * be
    return -T2 * inv_abar * v, e * (1 + T2 / 2 * e * (1 + T2 * e)), bmax


def test_ray_series_inside_its_range():
    """Path change and turn within 1e-6 of the exact ones (16 FP32 roundings, what the
    kernels' arithmetic leaves anyway); beyond the range of b the path is not."""
    worst, beyond = 0.0, 0.0
    for N0 in (3e-4, 1e-3, 5e-3, 0.01, 0.02, 0.05, 0.1, 0.4):
        for x in (-5.0, -1.5, -0.7, -0.3, -0.1, 0.1, 0.3, 1.5):
            nu_e = N0 * np.exp(min(x, 0.0))
            b = series_change(0.5, nu_e, x)[2]
            if b < 3e-5:
                continue  # a change of 1e-9: longdouble's cancellation shows in the exact one
            for q in (1e-5, 1e-4, 1e-3, 0.999 * GATE_T2B):
                C = 1 / np.sqrt(1 + q / float(b))
                d0, Q0 = exact_change(C, nu_e, x)
                d1, Q1, _ = series_change(C, nu_e, x)
                err = max(abs(d1 / d0 - 1), abs(Q1 / Q0 - 1))
                if b < GATE_B:
                    worst = max(worst, float(err))
                else:
                    beyond = max(beyond, float(err))
    assert worst < 1e-6, worst
    assert beyond > 1e-3, beyond


RAYS = [{"kind": "exponential_ray", "N0": N0, "H": H} for N0, H in ((3.25e-4, 8000.0), (0.01, 2000.0), (0.3, 1000.0),
                                                                    (0.4, 77.0), (0.78, 100.0))]
SPHERES = [{"kind": "exponential_spherical", "N0": 3.25e-4, "H": 8000.0, "R_E": R} for R in (6.371e6, 2.0e6, 2.0e4, 5.0e3)]


@pytest.mark.gpu
@pytest.mark.parametrize("medium", RAYS + SPHERES)
def test_arrivals_of_a_flat_array(medium):
    """The ZHS interval ends of a flat array's pairs (series in its range) against the
    same antennas next to one at another altitude (the quadrature, pair by pair), in
    bins of 0.2 ns: within 40 FP32 roundings of what the medium changes in them, the
    difference to the plain exponential atmosphere, and the listing's own rounding."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()
    from paper_2309_03717_gb300 import c8r
    rng = np.random.default_rng(4)
    n, n_ant, dt = 301, 40, 0.2
    top = min(4000.0, 4.0 * medium["H"])
    vals = {f: np.zeros(n) for f in synth.FIELDS}
    z = rng.uniform(0.1 * top, top, n)
    for e, k in (("0", 0.0), ("1", -2.0)):
        vals["x" + e], vals["y" + e], vals["z" + e] = rng.normal(size=n) * 5.0, rng.normal(size=n) * 5.0, z + k
    vals["t0"][:], vals["t1"][:], vals["bz"][:], vals["q"][:] = 0.0, 7.0, -0.99, -1.0
    tracks = {f: x.astype(np.float32) for f, x in vals.items()}
    reach = 3.0 * top
    if "R_E" in medium:  # the range of the sphere's series
        reach = min(reach, 0.99 * np.sqrt(0.02 * medium["R_E"] * medium["H"]))
    r = reach * np.geomspace(1e-3, 1.0, n_ant)
    a = 2.4 * np.arange(n_ant)
    ant = np.stack([r * np.cos(a), r * np.sin(a), np.zeros(n_ant)], 1)
    _, u = oracle_arrivals(tracks, ant, np.zeros(n_ant), 1, dt, medium, "zhs")
    u = u.reshape(n, n_ant, 2)
    _, plain = oracle_arrivals(tracks, ant, np.zeros(n_ant), 1, dt, dict(medium, kind="exponential"), "zhs")
    plain = plain.reshape(n, n_ant, 2)
    # (rays: where one arrives, and inside the series' range of T^2 b; the quadrature's
    # own iteration is not made for the others in the dense media)
    ok = np.isfinite(u).all(-1)
    if medium["kind"] == "exponential_ray":
        b = np.array([series_change(0.5, medium["N0"] * np.exp(-h / medium["H"]), -h / medium["H"])[2] for h in z - 1.0])
        ok &= (r[None] / (z - 1.0)[:, None]) ** 2 * b[:, None].astype(float) < 0.9 * GATE_T2B
    start = np.floor(np.where(ok[..., None], u, np.inf).min((0, 2))) - 3.0
    start = np.where(np.isfinite(start), start, 0.0)
    N = int(np.where(ok[..., None], u - start[None, :, None], 0.0).max()) + 5
    got = []
    for extra in (0, 1):
        k = n_ant + extra
        p = c8r.RadioProcess(medium, np.concatenate([ant, ant[:1] + [0.0, 0.0, 0.5]])[:k],
                             np.concatenate([start, start[:1]])[:k] * dt, N, dt, "zhs", "mixed")
        _, bins, frac = p.arrivals(to_device(tracks))
        got.append((bins.cpu().numpy() + frac.double().cpu().numpy())[:, :n_ant])
        p.close()
    change = np.abs(u - plain)[ok]
    diff = np.abs(got[0] - got[1])[ok]
    assert ok.mean() > 0.2 and change.max() > 0
    assert (diff <= 40 * 2.0 ** -24 * change + 2.0 ** -22).all(), (diff - 40 * 2.0 ** -24 * change).max()
