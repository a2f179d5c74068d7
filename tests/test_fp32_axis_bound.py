"""Host check (numpy FP32) of the FP32 arrival along an axis: w = -(d . A) with A
an FP32 vector of unit length up to rounding, x = |d x A|^2/(R + w) where w >= 0
and R - w elsewhere, T = t/dt + k (position . A)/|A| for track endpoints and
antennas.  As test_fp32_arrival_bound does for the vertical and direct forms:
every step rounded once, approximations perturbed within 2 ulp, against the
oracle's arrivals; every endpoint inside its bound, and few in-window endpoints
left undecided on an inclined shower."""
import numpy as np
import pytest

import oracle
from test_fp32_arrival_bound import C_M_PER_NS, F32, F64, U, fma, perturb, r, split
from paper_2309_03717_gb300 import synth


def emulated_axis_arrivals(w, tracks, axis, mode, rng):
    dt, med = w["dt_ns"], w["medium"]
    expo = med["kind"] == "exponential"
    kc = 1.0 / (C_M_PER_NS * dt)
    k = kc if expo else med["n"] * kc
    kh, _ = split(k)
    A = r(axis)
    L = np.linalg.norm(A.astype(F64))
    kA = [F64(p) + F64(q) for p, q in (split(k * F64(a) / L) for a in A)]
    P = np.asarray(w["ant_xyz"], F64)
    ph = [split(P[:, c]) for c in range(3)]
    Ta = np.asarray(w["t_start_ns"], F64) / dt + sum(kA[c] * P[:, c] for c in range(3))
    Tah, Tal = split(Ta)
    nmax = 1.0 + med["N0"] if expo else med["n"]
    al = np.sqrt(sum(l.astype(F64) ** 2 for _, l in ph))
    fb_abs = r(r(2.02 * nmax * kc * al + 16.0 * U * U * np.abs(w["t_start_ns"] / dt + k * P[:, 2]) + 1e-6).astype(F64)
               + 16.0 * U * U * np.abs(Tah))
    if expo:
        N0, H = med["N0"], med["H"]
        cNh, _ = split(N0 * H * kc)
        invHh, _ = split(1.0 / H)
        fb_rel_v = r(1.01 * np.abs(ph[2][1].astype(F64)) / (0.999e-3 * H))
        Eah, Eal = split(np.exp(-P[:, 2] / H))
    else:
        fb_rel_v = np.zeros(len(P), F32)
    out = []
    for j in "01":
        pos = [tracks[c + j].astype(F32)[:, None] for c in "xyz"]
        Te = tracks["t" + j].astype(F64) / dt + sum(kA[c] * tracks["xyz"[c] + j].astype(F64) for c in range(3))
        Teh, Tel = (v[:, None] for v in split(Te))
        s = [r(ph[c][0][None] - pos[c]) for c in range(3)]
        rho2 = fma(s[0], s[0], r(s[1].astype(F64) * s[1]))
        S = fma(s[2], s[2], rho2)
        y = perturb(1.0 / np.sqrt(S.astype(F64)), mode, rng)
        R = r(S.astype(F64) * y)
        c = [fma(s[1], A[2], -r(s[2].astype(F64) * A[1])), fma(s[2], A[0], -r(s[0].astype(F64) * A[2])),
             fma(s[0], A[1], -r(s[1].astype(F64) * A[0]))]
        Pc = fma(c[0], c[0], fma(c[1], c[1], r(c[2].astype(F64) * c[2])))
        wa = -fma(s[0], A[0], fma(s[1], A[1], r(s[2].astype(F64) * A[2])))
        with np.errstate(divide="ignore", invalid="ignore"):
            x = perturb(Pc.astype(F64) / r(R.astype(F64) + wa).astype(F64), mode, rng)
            x = np.where(wa >= 0, x, r(R.astype(F64) - wa))
        q = r(x.astype(F64) * kh)
        Td = r(r(Teh.astype(F64) - Tah[None]).astype(F64) + r(Tel.astype(F64) - Tal[None]))
        v = np.zeros_like(q)
        if expo:
            z = tracks["z" + j].astype(F64)
            Eeh, Eel = (e[:, None] for e in split(np.exp(-z / H)))
            xq = r(s[2].astype(F64) * invHh)
            num = r(r(Eeh.astype(F64) - Eah[None]).astype(F64) + r(Eel.astype(F64) - Eal[None]))
            with np.errstate(divide="ignore", invalid="ignore"):
                big = perturb(num.astype(F64) / s[2], mode, rng)
            f = r(xq.astype(F64) * fma(xq, fma(xq, r(-1.0 / 24.0), r(1.0 / 6.0)), r(-0.5)))
            small = r(r(Eeh.astype(F64) * invHh).astype(F64) * r(1.0 + f.astype(F64)))
            qv = np.where(np.abs(xq) > F32(1e-3), big, small)
            v = r(r(qv.astype(F64) * R).astype(F64) * cNh)
        uf = r(r(Td.astype(F64) + q).astype(F64) + v)
        tail = fma(r(2.25 * U), np.abs(Td),
                   fma(fma(r(22.0), r(U), fb_rel_v[None]), np.abs(v), fma(r(3.25 * U), np.abs(uf), fb_abs[None])))
        # c_q = 72, and 3/8 u k R (w >= 0) or 10 u k R
        kR = np.where(wa >= 0, r(0.375 * U * F64(kh)), r(10.0 * U * F64(kh)))
        eps = fma(r(72.0 * U), q, fma(kR, R, tail))
        out.append((uf, eps))
    return out


def workload(name):
    if name == "dense":
        w = synth.workload(0, n_tracks=1500)
        w["medium"] = {"kind": "uniform", "n": 1.78}
        zenith = 20.0
    else:
        w = synth.workload(1, n_tracks=1500, n_ant=64)
        zenith = float(name)
        w["zenith"] = zenith
        w["t_start_ns"] = synth.trace_start_ns(w["ant_xyz"], zenith)
    w["dtype"] = np.float32
    tracks = synth.make_tracks(1500, 77, w["zenith"])
    if name == "dense":
        _, u0 = oracle.arrivals(oracle.tracks_from_ns(tracks), w["ant_xyz"], np.zeros(len(w["ant_xyz"])), 1,
                                w["dt_ns"] * 1e-9, w["medium"], oracle.ENDPOINT)
        w["t_start_ns"] = np.median(u0[..., 0], axis=0) * w["dt_ns"] - 300.0
    return w, tracks, synth.shower_axis_up(zenith)


@pytest.mark.parametrize("name", ["12", "30", "60", "75", "dense"])
@pytest.mark.parametrize("tilt", [0.0, 0.3, 2.0])
def test_axis_arrival_within_its_bound(name, tilt):
    """Also along a wrong axis (tilted from the shower's, or pointing away from it)."""
    w, tracks, axis = workload(name)
    if tilt:
        c, s = np.cos(tilt), np.sin(tilt)
        axis = np.array([c * axis[0] - s * axis[2], 0.2 * s, s * axis[0] + c * axis[2]])
        axis = axis / np.linalg.norm(axis)
    br, u = oracle.arrivals(oracle.tracks_from_ns(tracks), w["ant_xyz"], w["t_start_ns"] * 1e-9, w["n_bins"],
                            w["dt_ns"] * 1e-9, w["medium"], oracle.ENDPOINT)
    two = br == 0
    rng = np.random.default_rng(9)
    worst = 0.0
    for mode in ("up", "down", "random"):
        for j, (uf, eps) in enumerate(emulated_axis_arrivals(w, tracks, axis, mode, rng)):
            ratio = (np.abs(uf.astype(F64) - u[..., j]) / eps)[two]
            assert np.all(np.isfinite(ratio))
            worst = max(worst, float(ratio.max()))
            inwin = two & (u[..., j] > 0) & (u[..., j] < w["n_bins"])
            undecided = (np.floor(uf - eps) != np.floor(uf + eps))[inwin].mean()
    assert worst <= 1.0, worst
    if tilt == 0.0 and name != "dense":
        assert undecided < 0.03, undecided
