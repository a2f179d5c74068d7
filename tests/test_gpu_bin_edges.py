"""Arrivals within rounding of a bin edge: the forward pass, the arrival listing
and the adjoint form them by the same arithmetic, so they put every deposit in the
same bin, wherever a rounding leaves it.  One track and many antennas, each with a
window that opens a whole number of bins before the track's arrival there (the
oracle's, in FP64), so that about half of the arrivals fall on either side."""
import numpy as np
import pytest

from _util import built_lib, oracle_arrivals, to_device
from paper_2309_03717_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

UNIFORM = {"kind": "uniform", "n": 1.000292}
SPHERE = {"kind": "exponential_spherical", "N0": 3.25e-4, "H": 8000.0, "R_E": 6.371e6}
RAY = {"kind": "exponential_ray", "N0": 3.25e-4, "H": 8000.0}
K = 40  # the bin whose lower edge the arrivals lie on


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()


def on_the_edge(formalism, medium, hills, dt, n_ant, dtype, K=K, spread=1e-9):
    """A 4 m track 3 km up and n_ant antennas, the first arrival of each on edge K."""
    rng = np.random.default_rng(11)
    b = np.array([0.02, 0.01, -0.999])
    x0 = np.array([30.0, -20.0, 3000.0])
    t0 = 7.0 / 0.299792458
    t1 = t0 + 4.0 / (np.linalg.norm(b) * 0.299792458)
    x1 = x0 + 4.0 * b / np.linalg.norm(b)
    vals = [*x0, *x1, t0, t1, *b, -1.0]
    tracks = {f: np.array([v], dtype) for f, v in zip(synth.FIELDS, vals)}
    r, a = rng.uniform(700.0, 1500.0, n_ant), rng.uniform(0.0, 2.0 * np.pi, n_ant)
    ant = np.stack([r * np.cos(a), r * np.sin(a), rng.uniform(0.0, 1.0, n_ant) * hills], 1)
    exact = {f: x.astype(np.float64) for f, x in tracks.items()}
    br, u = oracle_arrivals(exact, ant, np.zeros(n_ant), 1, dt, medium, formalism)
    u = u.reshape(n_ant, 2)
    assert (br.ravel() == (0 if formalism == "endpoint" else 3)).all()
    assert (np.abs(u[:, 1] - u[:, 0]) > 3.0).all()
    # moved by a rounding or two of an arrival (FP64: 2e-12 ns; float-float: `spread` bins)
    jitter = rng.normal(size=n_ant) * (3e-12 if dtype is np.float64 else spread * dt)
    return tracks, ant, (u.min(1) - K) * dt + jitter, int(np.argmin(u[0]))


def forward_listing_adjoint(formalism, precision, medium, hills, dt, adjoint=True, n_ant=1500, N=512, K=K,
                            spread=1e-9):
    from paper_2309_03717_gb300 import c8r
    dtype = np.float64 if precision == "fp64" else np.float32
    tracks, ant, t_start, first = on_the_edge(formalism, medium, hills, dt, n_ant, dtype, K, spread)
    dev = to_device(tracks)
    p = c8r.RadioProcess(medium, ant, t_start, N, dt, formalism, precision)
    p.push(dev)
    below = p.traces()[:, :, K - 1].abs().amax(1).cpu().numpy() > 0
    bins = p.arrivals(dev)[1].cpu().numpy()[0, :, first]
    ag = None
    if adjoint:
        # dL/dtrace in bin K - 1 only: an antenna has a gradient when its deposit is there
        G = torch.zeros((n_ant, 3, N), dtype=p.trace_dtype, device="cuda")
        G[:, :, K - 1] = torch.tensor([1.0, -2.0, 3.0], dtype=p.trace_dtype, device="cuda") * 1e9
        gdt = torch.float64 if precision == "fp64" else torch.float32
        tg = {f: torch.zeros(1, dtype=gdt, device="cuda") for f in c8r.GRAD_FIELDS}
        ag = torch.zeros((n_ant, 3), dtype=torch.float64, device="cuda")
        dn = torch.zeros(1, dtype=torch.float64, device="cuda")
        c8r.c8r_backward(p.ctx, dev, G, tg, ag, dn)
        ag = ag.cpu().numpy()
    p.close()
    assert 0.05 < below.mean() < 0.95  # both sides of the edge are reached
    return below, bins, ag


@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
@pytest.mark.parametrize("medium", [synth.AIR_EXPONENTIAL, UNIFORM])
@pytest.mark.parametrize("hills", [0.0, 150.0])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_forward_listing_and_adjoint_agree(precision, hills, medium, formalism):
    below, bins, ag = forward_listing_adjoint(formalism, precision, medium, hills, 0.05)
    assert np.array_equal(bins == K - 1, below)
    assert np.array_equal(np.abs(ag).max(1) > 0, below)


@pytest.mark.parametrize("medium", [SPHERE, RAY])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
@pytest.mark.parametrize("hills", [0.0, 150.0])
def test_forward_and_listing_agree_in_the_costlier_media(hills, formalism, precision, medium):
    below, bins, _ = forward_listing_adjoint(formalism, precision, medium, hills, 0.05, adjoint=False)
    assert np.array_equal(bins == K - 1, below)


@pytest.mark.parametrize("medium", [synth.AIR_EXPONENTIAL, SPHERE, UNIFORM])
@pytest.mark.parametrize("N,K", [((1 << 21) + 300, (1 << 21) + 9), ((1 << 23) + 5, (1 << 23) - 90), (1 << 24, (1 << 24) - 95)])
def test_long_windows(N, K, medium):
    """Windows beyond 2^21 bins, where the FP32 spacing of an arrival reaches a bin:
    a tent of bins in front of the window's end."""
    below, bins, _ = forward_listing_adjoint("zhs", "mixed", medium, 0.0, 0.05, adjoint=False, n_ant=24, N=N, K=K,
                                             spread=1e-6)
    assert np.array_equal(bins == K - 1, below)


@pytest.mark.parametrize("medium", [SPHERE, RAY, synth.AIR_EXPONENTIAL, UNIFORM])
@pytest.mark.parametrize("z", [0.0, 5.0])
def test_a_filtered_neighbour_changes_no_arrival(z, medium):
    """The ZHS kernels take tracks two at a time: the arrivals of one are the same
    bit for bit whether the other passes the filter or not."""
    from paper_2309_03717_gb300 import c8r
    n = 257
    ant = synth.antennas_star(8, n_radii=3)[:17].copy()
    ant[:, 2] = z
    tracks = synth.make_tracks(n, 31, 40.0)
    p = c8r.RadioProcess(medium, ant, synth.trace_start_ns(ant, 40.0) - 100.0, 4096, 0.2, "zhs", "mixed")
    want = [x.cpu().numpy() for x in p.arrivals(to_device(tracks))]
    assert (want[1] >= 0).any()
    for first in (0, 1):
        t = {f: x.copy() for f, x in tracks.items()}
        t["q"][1 - first::2] = 0.0
        t["x0"][1 - first::2] = np.nan
        got = [x.cpu().numpy() for x in p.arrivals(to_device(t))]
        assert (got[0][1 - first::2] == -1).all()
        for g, w in zip(got, want):
            assert np.array_equal(g[first::2], w[first::2])
    p.close()
