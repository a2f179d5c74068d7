"""The one-bin Endpoint kernels evaluate a pair's two endpoints together, the
ZHS forward kernels two tracks, and both redo the rare pair (an emission point
near the antenna's altitude or below it, an antenna behind the track) half by
half.  Antennas spread through the shower's
own heights make those pairs common, next to usual ones; track counts around the
128-track tile and antenna counts around the 32-antenna tile.  Traces and
adjoint against the oracle at the mixed bar (1e-4 relative L2)."""
import numpy as np
import pytest

import oracle
from _util import built_lib, drop_tracks, oracle_arrivals, oracle_traces, rel_l2, to_device, unambiguous
from paper_2309_03717_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 1e-4
UNIFORM = {"kind": "uniform", "n": 1.000292}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()


def among_the_tracks(n, n_ant, medium):
    """A shower and n_ant antennas 60-460 m from its axis at heights from below to above its tracks."""
    w = synth.workload(1, n_tracks=n + 60, n_ant=n_ant)
    w["n_bins"], w["medium"] = 2048, medium or w["medium"]
    tracks = synth.workload_tracks(w)
    r = np.linspace(60.0, 460.0, n_ant)
    a = 2.4 * np.arange(n_ant)
    z = np.quantile(tracks["z0"], np.linspace(0.0, 1.0, n_ant + 2)[1:-1]).astype(np.float64)
    w["ant_xyz"] = np.stack([r * np.cos(a), r * np.sin(a), z], 1)
    zero = np.zeros(n_ant)
    _, u0 = oracle_arrivals(tracks, w["ant_xyz"], zero, 1, w["dt_ns"], w["medium"], "endpoint")
    w["t_start_ns"] = np.median(u0.reshape(n + 60, n_ant, 2)[..., 0], axis=0) * w["dt_ns"] - 200.0
    keep = unambiguous(tracks, w["ant_xyz"], w["t_start_ns"], w["n_bins"], w["dt_ns"], w["medium"], "endpoint")
    tracks = {f: x[:n] for f, x in drop_tracks(tracks, keep).items()}
    assert len(tracks["x0"]) == n
    return w, {f: np.ascontiguousarray(x) for f, x in tracks.items()}


@pytest.mark.parametrize("form", ["split", "direct"])
@pytest.mark.parametrize("medium", [None, UNIFORM])
@pytest.mark.parametrize("n,n_ant", [(1, 1), (127, 31), (128, 32), (129, 33), (700, 5)])
def test_traces_and_adjoint_with_antennas_among_the_tracks(n, n_ant, medium, form):
    from paper_2309_03717_gb300 import c8r
    w, tracks = among_the_tracks(n, n_ant, medium)
    p = c8r.RadioProcess(w["medium"], w["ant_xyz"], w["t_start_ns"], w["n_bins"], w["dt_ns"], "endpoint", "mixed")
    p.set_arrival_form(form)
    dev = to_device(tracks)
    p.push(dev)
    ref, kept = oracle_traces(tracks, w["ant_xyz"], w["t_start_ns"], w["n_bins"], w["dt_ns"], w["medium"], "endpoint")
    assert kept == n
    assert rel_l2(p.traces().cpu().numpy(), ref) <= TOL
    G = torch.from_numpy(np.random.default_rng(n).normal(size=ref.shape).astype(np.float32)).cuda()
    tg = {f: torch.zeros(n, dtype=torch.float32, device="cuda") for f in c8r.GRAD_FIELDS}
    ag = torch.zeros((n_ant, 3), dtype=torch.float64, device="cuda")
    dn = torch.zeros(1, dtype=torch.float64, device="cuda")
    c8r.c8r_backward(p.ctx, dev, G, tg, ag, dn)
    got = np.stack([tg[f].double().cpu().numpy() for f in c8r.GRAD_FIELDS], axis=1)
    p.close()
    tg_ref, ag_ref, _ = oracle.backward(oracle.tracks_from_ns(tracks), w["ant_xyz"], w["t_start_ns"] * 1e-9,
                                        w["n_bins"], w["dt_ns"] * 1e-9, w["medium"], G.double().cpu().numpy())
    assert rel_l2(got[:, 0:6], tg_ref[:, 0:6]) <= TOL
    assert rel_l2(got[:, 8:11], tg_ref[:, 8:11]) <= TOL
    assert rel_l2(ag.cpu().numpy(), ag_ref) <= TOL


@pytest.mark.parametrize("form", ["split", "direct"])
@pytest.mark.parametrize("n,n_ant,height", [(1, 1, 0.0), (129, 33, 0.0), (700, 5, None)])
def test_flat_arrays_give_what_uneven_ones_do(n, n_ant, height, form):
    """A flat array's kernels form the refractivity quotient per track; one more
    antenna at another altitude (its dL/dtrace is zero) sends the same antennas
    through the kernels that form it per pair.  Same bins and roundings: what is
    left is the order of up to 2 x 700 additions, 1400 x 2^-24 at most of the sum
    of magnitudes and its square root of them as a rule (2e-6).  Ground below the
    tracks, and at their median height (None), where some quotients are series."""
    from paper_2309_03717_gb300 import c8r
    w, tracks = among_the_tracks(n, n_ant, None)
    if height is None:
        height = float(np.median(tracks["z0"]))
    ant = w["ant_xyz"].copy()
    ant[:, 2] = height
    _, u0 = oracle_arrivals(tracks, ant, np.zeros(n_ant), 1, w["dt_ns"], w["medium"], "endpoint")
    t_start = np.median(u0.reshape(n, n_ant, 2)[..., 0], axis=0) * w["dt_ns"] - 200.0
    G = np.random.default_rng(n).normal(size=(n_ant + 1, 3, w["n_bins"])).astype(np.float32)
    G[-1] = 0.0
    dev, out = to_device(tracks), []
    for extra in (0, 1):
        k = n_ant + extra
        p = c8r.RadioProcess(w["medium"], np.concatenate([ant, ant[:1] + [0.0, 0.0, 900.0]])[:k],
                             np.concatenate([t_start, t_start[:1]])[:k], w["n_bins"], w["dt_ns"], "endpoint", "mixed")
        p.set_arrival_form(form)
        p.push(dev)
        tg = {f: torch.zeros(n, dtype=torch.float32, device="cuda") for f in c8r.GRAD_FIELDS}
        ag = torch.zeros((k, 3), dtype=torch.float64, device="cuda")
        dn = torch.zeros(1, dtype=torch.float64, device="cuda")
        c8r.c8r_backward(p.ctx, dev, torch.from_numpy(G[:k]).cuda(), tg, ag, dn)
        out.append((p.traces().cpu().numpy()[:n_ant], ag.cpu().numpy()[:n_ant],
                    np.stack([tg[f].double().cpu().numpy() for f in c8r.GRAD_FIELDS], axis=1)))
        p.close()
    for flat, uneven in zip(*out):
        assert np.abs(uneven).max() > 0
        assert rel_l2(flat, uneven) <= 2e-5


@pytest.mark.parametrize("deposit", ["bin", "linear"])
@pytest.mark.parametrize("medium", [None, UNIFORM])
@pytest.mark.parametrize("n,n_ant,n_bins", [(1, 1, 2048), (2, 3, 7), (127, 31, 2048), (129, 33, 2048), (700, 5, 1),
                                            (33, 2, (1 << 21) + 5)])
def test_zhs_traces_with_antennas_among_the_tracks(n, n_ant, n_bins, medium, deposit):
    from paper_2309_03717_gb300 import c8r
    w, tracks = among_the_tracks(n, n_ant, medium)
    if n_bins < 2048:
        w["t_start_ns"] = w["t_start_ns"] + 200.0  # around the arrivals
    tracks["q"][n // 2 :: 7] = 0.0  # filtered tracks next to kept ones
    p = c8r.RadioProcess(w["medium"], w["ant_xyz"], w["t_start_ns"], n_bins, w["dt_ns"], "zhs", "mixed",
                         deposit=deposit)
    p.push(to_device(tracks))
    got = p.traces().cpu().numpy()
    p.close()
    ref, _ = oracle.forward(oracle.tracks_from_ns(tracks), w["ant_xyz"], w["t_start_ns"] * 1e-9, n_bins,
                            w["dt_ns"] * 1e-9, w["medium"], oracle.ZHS,
                            deposit=oracle.DEPOSIT_LINEAR if deposit == "linear" else oracle.DEPOSIT_BIN)
    assert rel_l2(got, ref) <= TOL


HEAVY = [{"kind": "exponential_spherical", "N0": 3.25e-4, "H": 8000.0, "R_E": 6.371e6},
         {"kind": "exponential_ray", "N0": 3.25e-4, "H": 8000.0},
         {"kind": "exponential_ray", "N0": 5e-3, "H": 2000.0}]


@pytest.mark.parametrize("deposit", ["bin", "linear"])
@pytest.mark.parametrize("medium", HEAVY)
@pytest.mark.parametrize("reach,z", [(400.0, 0.0), (12_000.0, 120.0), (60_000.0, 0.0), (3_000.0, None)])
def test_zhs_over_a_sphere_and_along_rays(reach, z, medium, deposit):
    """Flat arrays take the propagators' series in the pairs where those hold
    (steep lines of sight, sites within 32 km), the quadrature elsewhere: sites
    from the shower axis out to where only the latter is left, and uneven ground
    (z None), where no pair takes the series."""
    from paper_2309_03717_gb300 import c8r
    n, n_ant = 301, 33
    w = synth.workload(1, n_tracks=n, n_ant=n_ant)
    tracks = synth.workload_tracks(w)
    tracks["q"][5::11] = 0.0  # filtered tracks next to kept ones
    x = np.concatenate([[0.0], np.geomspace(reach / 1000.0, reach, n_ant - 1)])
    heights = np.linspace(0.0, 200.0, n_ant) if z is None else np.full(n_ant, z)
    ant = np.stack([x, 0.3 * x, heights], 1)
    _, u0 = oracle_arrivals(tracks, ant, np.zeros(n_ant), 1, w["dt_ns"], medium, "zhs")
    t_start = np.median(u0.reshape(n, n_ant, 2)[..., 0], axis=0) * w["dt_ns"] - 200.0
    # (in the steep atmosphere no direct ray reaches the farthest sites: no start time there)
    ant, t_start = ant[np.isfinite(t_start)], t_start[np.isfinite(t_start)]
    n_ant = len(ant)
    assert n_ant >= 25
    p = c8r.RadioProcess(medium, ant, t_start, 2048, w["dt_ns"], "zhs", "mixed", deposit=deposit)
    p.push(to_device(tracks))
    got = p.traces().cpu().numpy()
    p.close()
    ref, _ = oracle.forward(oracle.tracks_from_ns(tracks), ant, t_start * 1e-9, 2048, w["dt_ns"] * 1e-9, medium,
                            oracle.ZHS,
                            deposit=oracle.DEPOSIT_LINEAR if deposit == "linear" else oracle.DEPOSIT_BIN)
    for a in range(n_ant):
        if np.abs(ref[a]).max() > 0:
            assert rel_l2(got[a], ref[a]) <= TOL, a


@pytest.mark.parametrize("medium", [None, UNIFORM])
@pytest.mark.parametrize("zenith,hills,offset", [(35.0, 0.0, 0.0), (60.0, 0.0, 0.0), (60.0, 150.0, 0.0),
                                                 (78.0, 0.0, 1.0e6), (50.0, 0.0, None)])
def test_axis_form_gives_the_bins_of_the_others(zenith, hills, offset, medium):
    """Windows placed along an inclined front: the automatic form (along the
    front's axis) against the pinned direct one, traces and adjoint, which take
    the same bins and so differ by the order of additions only.  Also with a time
    origin 1e6 ns early, and (offset None) with antennas far up the axis, behind
    most of the tracks."""
    from paper_2309_03717_gb300 import c8r
    n = 4001
    tracks = synth.make_tracks(n, 31, zenith)
    ant = synth.antennas_star(8, n_radii=9)[:67].copy()
    ant[:, 2] = np.linspace(0.0, hills, len(ant))
    if offset is None:
        ant[::3] += 5000.0 * synth.shower_axis_up(zenith)
    t_start = synth.trace_start_ns(ant, zenith)
    if offset:
        t_start = t_start + offset
        for f in ("t0", "t1"):
            tracks[f] = (tracks[f].astype(np.float64) + offset).astype(np.float32)
    out = []
    for form in ("auto", "direct"):
        p = c8r.RadioProcess(medium or synth.AIR_EXPONENTIAL, ant, t_start, 4096, 0.2, "endpoint", "mixed")
        p.set_arrival_form(form)
        dev = to_device(tracks)
        p.push(dev)
        tr = p.traces().cpu().numpy()
        G = torch.from_numpy(np.random.default_rng(3).normal(size=tr.shape).astype(np.float32)).cuda()
        tg = {f: torch.zeros(n, dtype=torch.float32, device="cuda") for f in c8r.GRAD_FIELDS}
        ag = torch.zeros((len(ant), 3), dtype=torch.float64, device="cuda")
        dn = torch.zeros(1, dtype=torch.float64, device="cuda")
        c8r.c8r_backward(p.ctx, dev, G, tg, ag, dn)
        out.append((tr, np.stack([tg[f].cpu().numpy() for f in c8r.GRAD_FIELDS]), ag.cpu().numpy()))
        p.close()
    assert np.abs(out[1][0]).max() > 0
    for a, d in zip(*out):
        assert rel_l2(a, d) <= 2e-6


@pytest.mark.parametrize("medium", [synth.AIR_EXPONENTIAL, UNIFORM])
@pytest.mark.parametrize("hills", [0.0, 150.0])
def test_batch_groups_showers_by_arrival_form(hills, medium):
    """Showers from the vertical to 75 degrees in one batch, each with the axis
    of its own windows, an empty one, and one whose windows open together, so
    that no front orders them: every shower's traces as its own process in the
    direct form gives them, to the order of the additions."""
    from paper_2309_03717_gb300 import c8r
    showers, tracks = [], []
    for k, (zenith, n) in enumerate([(75.0, 700), (0.0, 129), (50.0, 1), (60.0, 0), (35.0, 3000), (70.0, 1500)]):
        ant = synth.antennas_star(8, n_radii=5)[: 5 + 7 * k].copy()
        ant[:, 2] = np.linspace(0.0, hills, len(ant))
        t_start = synth.trace_start_ns(ant, zenith)
        if k == 5:
            t_start = np.full(len(ant), t_start.min())
        showers.append({"n_tracks": n, "ant_xyz": ant, "t_start_ns": t_start})
        tracks.append({f: x[:n] for f, x in synth.make_tracks(max(n, 1), 50 + k, zenith).items()})
    b = c8r.Batch(showers, medium, 8192, 0.2, "endpoint")
    out = b.new_output()
    b.run(to_device({f: np.concatenate([t[f] for t in tracks]) for f in synth.FIELDS}), out)
    b.sync()
    got, off = out.cpu().numpy(), 0
    b.close()
    for s, t in zip(showers, tracks):
        k = len(s["ant_xyz"])
        if s["n_tracks"]:
            p = c8r.RadioProcess(medium, s["ant_xyz"], s["t_start_ns"], 8192, 0.2, "endpoint", "mixed")
            p.set_arrival_form("direct")
            p.push(to_device(t))
            ref = p.traces().cpu().numpy()
            p.close()
            assert np.abs(ref).max() > 0
            assert rel_l2(got[off:off + k], ref) <= 2e-6
        else:
            assert not got[off:off + k].any()
        off += k
