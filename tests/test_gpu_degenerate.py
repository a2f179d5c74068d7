"""Pairs whose geometry has no finite form: an antenna exactly on a track's endpoint
(R = 0), and an emission point so far away that the square of its distance
overflows.  Such an endpoint deposits nothing; everything else stays finite and as
it is without it."""
import numpy as np
import pytest

from _util import built_lib, to_device
from paper_2309_03717_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

UNIFORM = {"kind": "uniform", "n": 1.000292}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()


def gradients(p, tracks, G):
    from paper_2309_03717_gb300 import c8r
    n = len(tracks["x0"])
    dev = to_device(tracks)
    p.push(dev)
    gdt = torch.float64 if p.precision == "fp64" else torch.float32
    tg = {f: torch.zeros(n, dtype=gdt, device="cuda") for f in c8r.GRAD_FIELDS}
    ag = torch.zeros((p.n_ant, 3), dtype=torch.float64, device="cuda")
    dn = torch.zeros(1, dtype=torch.float64, device="cuda")
    c8r.c8r_backward(p.ctx, dev, G, tg, ag, dn)
    out = {f: tg[f].cpu().numpy() for f in c8r.GRAD_FIELDS}
    out.update(traces=p.traces().cpu().numpy(), antennas=ag.cpu().numpy(), N0=dn.cpu().numpy())
    p.close()
    return out


@pytest.mark.parametrize("form", ["split", "direct", "auto"])
@pytest.mark.parametrize("medium", [synth.AIR_EXPONENTIAL, UNIFORM])
@pytest.mark.parametrize("hills", [0.0, 150.0])
@pytest.mark.parametrize("end", [0, 1])
def test_antenna_on_a_track_end(end, hills, medium, form):
    """The end on the antenna has no deposit there and no part in any gradient, the
    other end keeps its own.  The reference is the same shower with that one end
    moved 30 km up: it arrives 1e5 ns late, outside every window, deposits nothing
    either, and the other end's deposit does not depend on it.  The loss looks at
    that antenna only.  What is left is rounding: the order of at most 2 x 301
    additions (600 x 2^-24 of the largest value)."""
    from paper_2309_03717_gb300 import c8r
    n, zenith = 301, 60.0 if form == "auto" else 0.0  # auto: windows along an inclined front
    tracks = synth.make_tracks(n, 31, zenith)
    ant = synth.antennas_star(8, n_radii=2)[:9].copy()
    ant[:, 2] = np.linspace(0.0, hills, len(ant))
    j, a = 150, 4
    here, other = str(end), str(1 - end)
    ant[a] = ant[a].astype(np.float32)  # FP32-exact
    t_start = synth.trace_start_ns(ant, zenith)
    for c, v in zip("xyz", ant[a]):
        tracks[c + here][j] = tracks[c + other][j] = v
    tracks["x" + other][j] += 40.0
    tracks["bx"][j], tracks["by"][j], tracks["bz"][j] = -0.9 if end else 0.9, 0.05, 0.02
    tracks["t0"][j] = t_start[a] + 20.0
    tracks["t1"][j] = t_start[a] + 20.0 + 40.0 / 0.27
    moved = {f: x.copy() for f, x in tracks.items()}
    moved["z" + here][j] += 3.0e4
    G = np.zeros((len(ant), 3, 2048), np.float32)
    G[a] = np.random.default_rng(3).normal(size=G[a].shape)
    out = []
    for t in (tracks, moved):
        p = c8r.RadioProcess(medium, ant, t_start, 2048, 0.2, "endpoint", "mixed")
        p.set_arrival_form(form)
        out.append(gradients(p, t, torch.from_numpy(G).cuda()))
    got, ref = out
    assert np.abs(ref["x" + other][j]) > 0  # its deposit lies in the window
    got["traces"], ref["traces"] = got["traces"][a], ref["traces"][a]
    for f in got:
        assert np.isfinite(got[f]).all(), f
        assert np.abs(got[f] - ref[f]).max() <= 600 * 2.0 ** -24 * np.abs(ref[f]).max(), f


@pytest.mark.parametrize("medium", [synth.AIR_EXPONENTIAL, UNIFORM])
@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
@pytest.mark.parametrize("hills", [0.0, 150.0])
def test_fp64_emission_point_whose_distance_overflows(hills, formalism, medium):
    """Tracks at 1e200 m pass the track filter; they arrive after every window."""
    from paper_2309_03717_gb300 import c8r
    n = 200
    tracks = {f: x.astype(np.float64) for f, x in synth.make_tracks(n, 31, 0.0).items()}
    ant = synth.antennas_star(8, n_radii=2)[:9].copy()
    ant[:, 2] = np.linspace(0.0, hills, len(ant))
    t_start = synth.trace_start_ns(ant, 0.0)
    out = []
    for far in (False, True):
        t = {f: x.copy() for f, x in tracks.items()}
        if far:
            t["x0"][::7] = 1.0e200
            t["x1"][::7] = 1.1e200
        else:
            t["q"][::7] = 0.0
        p = c8r.RadioProcess(medium, ant, t_start, 1024, 0.2, formalism, "fp64")
        dev = to_device(t)
        p.push(dev)
        assert p.stats()["tracks_kept"] == (n if far else n - len(t["q"][::7]))
        out.append(p.traces().cpu().numpy())
        if far:
            _, bins, _ = p.arrivals(dev)
            assert (bins[::7] == 1024).all()
        p.close()
    assert np.abs(out[0]).max() > 0 and np.isfinite(out[1]).all()
    assert np.abs(out[1] - out[0]).max() <= 1e-12 * np.abs(out[0]).max()


@pytest.mark.parametrize("medium", [synth.AIR_EXPONENTIAL, UNIFORM])
@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
@pytest.mark.parametrize("precision,far", [("fp64", 1.0e200), ("mixed", 1.0e25)])
def test_adjoint_of_emission_points_out_of_range(precision, far, formalism, medium):
    """Tracks whose squared distance overflows pass the filter and have no part in
    any gradient: as with those tracks dropped, to the order of the additions (FP32:
    200 of them; FP64: 1e-12)."""
    from paper_2309_03717_gb300 import c8r
    dtype = np.float64 if precision == "fp64" else np.float32
    tracks = {f: x.astype(dtype) for f, x in synth.make_tracks(200, 31, 0.0).items()}
    ant = synth.antennas_star(8, n_radii=2)[:9].copy()
    G = torch.from_numpy(np.random.default_rng(3).normal(size=(len(ant), 3, 1024)).astype(dtype)).cuda()
    out = []
    for dropped in (True, False):
        t = {f: x.copy() for f, x in tracks.items()}
        if dropped:
            t["q"][::7] = 0.0
        else:
            t["x0"][::7] = far
            t["x1"][::7] = 1.1 * far
        p = c8r.RadioProcess(medium, ant, synth.trace_start_ns(ant, 0.0), 1024, 0.2, formalism, precision)
        out.append(gradients(p, t, G))
    for f in out[0]:
        assert np.isfinite(out[1][f]).all(), f
        tol = 1e-12 if precision == "fp64" else 200 * 2.0 ** -24
        assert np.abs(out[1][f] - out[0][f]).max() <= tol * np.abs(out[0][f]).max(), f
