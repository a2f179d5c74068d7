"""The accumulator's memory: what a layout takes of the device, and that the copies
and the row of box edges are a help, not a need: without room for them the traces
are the same."""
import json

import numpy as np
import pytest

import oracle
from _util import built_lib, rel_l2, to_device
from paper_2309_03717_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SPHERE = {"kind": "exponential_spherical", "N0": 3.25e-4, "H": 8000.0, "R_E": 6.371e6}
RAY = {"kind": "exponential_ray", "N0": 3.25e-4, "H": 8000.0}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()


def process(medium, ant, n_bins, deposit="bin"):
    from paper_2309_03717_gb300.c8r import RadioProcess
    return RadioProcess(medium, ant, synth.trace_start_ns(ant), n_bins, 0.2, "zhs", "fp64", deposit=deposit)


def reference(medium, ant, n_bins, tracks, deposit="bin"):
    ref, _ = oracle.forward(oracle.tracks_from_ns(tracks), ant, synth.trace_start_ns(ant) * 1e-9, n_bins, 0.2e-9,
                            medium, oracle.ZHS,
                            deposit=oracle.DEPOSIT_LINEAR if deposit == "linear" else oracle.DEPOSIT_BIN)
    return ref


def shower(n):
    return {f: x.astype(np.float64) for f, x in synth.make_tracks(n, 5, 0.0).items()}


@pytest.mark.parametrize("medium,deposit", [(SPHERE, "bin"), (RAY, "bin"), (synth.AIR_EXPONENTIAL, "linear")])
def test_fp64_zhs_without_boxes_takes_one_row(medium, deposit):
    """Only the one-bin deposit of the plain media adds boxes: the others take 32
    bytes per bin and antenna (256 antennas x 32768 bins: 256 MB), also after a push."""
    ant = synth.antennas_grid(16)
    tracks = to_device(shower(64))
    process(medium, ant[:70], 64, deposit).close()  # the library's own first-use memory
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    p = process(medium, ant, 32768, deposit)
    p.push(tracks)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    p.close()
    assert taken < 1.25 * 256 * 32768 * 32, taken


@pytest.mark.parametrize("late", [False, True])
@pytest.mark.parametrize("n_ant", [1, 9, 70])
def test_fp64_zhs_without_room_for_the_edges(n_ant, late):
    """The row of box edges cannot be had: the boxes go in bin by bin."""
    from paper_2309_03717_gb300 import c8r
    n_bins, n = 1000, 3000
    ant = synth.antennas_grid(9)[:n_ant]
    tracks = shower(n)
    ref = reference(synth.AIR_EXPONENTIAL, ant, n_bins, tracks)
    dev = to_device(tracks)
    try:
        # the context's counters and error word, the antenna table, then the
        # accumulator with its edges (and, that failing, without); in another medium
        # first, the edges after a push's scratch
        if late:
            p = process(SPHERE, ant, n_bins)
            p.medium = dict(synth.AIR_EXPONENTIAL)
            p._apply_medium()
            c8r.c8r_inject_alloc_failures(1, 1)
        else:
            c8r.c8r_inject_alloc_failures(3, 1)
            p = process(synth.AIR_EXPONENTIAL, ant, n_bins)
        p.push(dev)
    finally:
        c8r.c8r_inject_alloc_failures(0, 0)
    for _ in range(2):
        assert rel_l2(p.traces(reset=True).cpu().numpy(), ref) < 1e-9
        assert not p.traces().any()
        p.push(dev)
    p.close()


def test_fp64_zhs_media_and_deposits_in_turn():
    """Pushes with and without boxes into one accumulator, and resets between."""
    from paper_2309_03717_gb300 import c8r
    n_bins, n = 1000, 3000
    ant = synth.antennas_grid(3)[:7]
    tracks = shower(n)
    dev = to_device(tracks)
    p = process(SPHERE, ant, n_bins)
    parts = [(SPHERE, "bin"), (synth.AIR_EXPONENTIAL, "bin"), (synth.AIR_EXPONENTIAL, "linear")]
    refs = [reference(m, ant, n_bins, tracks, d) for m, d in parts]

    def push(k):
        p.medium = dict(parts[k][0])
        p._apply_medium()
        c8r.c8r_set_deposit(p.ctx, {"bin": c8r.C8R_DEPOSIT_BIN, "linear": c8r.C8R_DEPOSIT_LINEAR}[parts[k][1]])
        p.push(dev)

    for order in ([0], [0, 1], [1, 2], [2], [2, 1, 0]):
        for k in order:
            push(k)
        assert rel_l2(p.traces(reset=len(order) > 1).cpu().numpy(), sum(refs[k] for k in order)) < 1e-9
        p.reset()
        assert not p.traces().any()
    push(1)
    p.set_antenna_positions(ant + [0.5, 0.0, 0.0])
    assert not p.traces().any()
    p.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
def test_captured_pushes_and_fetches(formalism, precision):
    """Pushes, fetches and resets from graphs captured at different times, next to
    eager ones that use more copies: nothing is left out, nothing left behind.
    Against one eager push, to the order of the additions."""
    from paper_2309_03717_gb300.c8r import RadioProcess
    dtype = torch.float64 if precision == "fp64" else torch.float32
    ant = synth.antennas_star(8, n_radii=1)[:2]
    many = to_device(synth.make_tracks(60_000, 5, 0.0), dtype)
    few = {f: x[:500].contiguous() for f, x in many.items()}
    p = RadioProcess(synth.AIR_EXPONENTIAL, ant, synth.trace_start_ns(ant), 1000, 0.5, formalism, precision)
    out = torch.empty((2, 3, 1000), dtype=dtype, device="cuda")
    # a fetch captured before anything was pushed
    torch.cuda.synchronize()
    fetch = torch.cuda.CUDAGraph()
    with torch.cuda.graph(fetch):
        p.traces(reset=True, out=out)
    p.push(many)
    all_tracks = p.traces(reset=True).double().cpu().numpy()
    p.push(few)
    some = p.traces(reset=True).double().cpu().numpy()
    tol = 1e-13 if precision == "fp64" else 2e-6
    assert rel_l2(all_tracks, 0 * all_tracks) > 0
    torch.cuda.synchronize()
    push = torch.cuda.CUDAGraph()
    with torch.cuda.graph(push):
        p.push(few)
    for eager in (False, True):
        p.push(many)
        push.replay()
        if eager:
            got = p.traces(reset=True)
        else:
            fetch.replay()
            got = out
        assert rel_l2(got.double().cpu().numpy(), all_tracks + some) < tol
        assert not p.traces().any()
        push.replay()
        push.replay()
        assert rel_l2(p.traces().double().cpu().numpy(), 2.0 * some) < tol
        p.reset()
        assert not p.traces().any()
    push.replay()
    p.set_antenna_positions(ant + [0.5, 0.0, 0.0])
    assert not p.traces().any()
    p.set_antenna_positions(ant)
    push.replay()
    fetch.replay()
    assert rel_l2(out.double().cpu().numpy(), some) < tol
    p.close()


def test_moving_antennas_zeroes_the_copies_in_use(tmp_path):
    """64 antennas x 2048 bins keep 16 copies of 2 MB, of which a push of 3000 tracks
    uses two: moving the antennas afterwards zeroes those (and a few counters)."""
    from torch.profiler import ProfilerActivity, profile
    from paper_2309_03717_gb300.c8r import RadioProcess
    ant = synth.antennas_star(8, n_radii=8)
    p = RadioProcess(synth.AIR_EXPONENTIAL, ant, synth.trace_start_ns(ant), 2048, 0.2, "endpoint", "mixed")
    tracks = to_device(synth.make_tracks(3000, 5, 0.0))
    for _ in range(2):  # (the profiler's first session can come up empty)
        p.push(tracks)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            p.set_antenna_positions(p.ant_xyz + [0.5, 0.0, 0.0])
            torch.cuda.synchronize()
    path = str(tmp_path / "trace.json")
    prof.export_chrome_trace(path)
    sets = [e["args"]["bytes"] for e in json.load(open(path))["traceEvents"] if e.get("cat") == "gpu_memset"]
    if not sets:
        pytest.skip("the profiler records no device activity here")
    assert max(sets) == 2 * 64 * 2048 * 16, sets
    assert not p.traces().any()
    p.close()
