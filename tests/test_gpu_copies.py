"""The copies of the trace accumulator (one to sixteen, by the antennas and by
the tracks of a push): pushes of sizes around the steps of the count, windows
that end inside a fetch round, resets by either fetch path and by c8r_reset, and
pushes replayed from a CUDA graph, whose copies the host does not see used.
Against the oracle at the mixed bar (1e-4 relative L2)."""
import numpy as np
import pytest

from _util import built_lib, drop_tracks, endpoint_unambiguous, oracle_traces, rel_l2, to_device
from paper_2309_03717_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 1e-4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()


def setup(formalism, n_tracks, n_ant, n_bins):
    from paper_2309_03717_gb300.c8r import RadioProcess
    w = synth.workload(1, n_tracks=n_tracks, n_ant=n_ant)
    t = synth.workload_tracks(w)
    if formalism == "endpoint":
        t = drop_tracks(t, endpoint_unambiguous(t, w["ant_xyz"], w["t_start_ns"], n_bins, w["dt_ns"], w["medium"]))
    ref, _ = oracle_traces(t, w["ant_xyz"], w["t_start_ns"], n_bins, w["dt_ns"], w["medium"], formalism)
    p = RadioProcess(w["medium"], w["ant_xyz"], w["t_start_ns"], n_bins, w["dt_ns"], formalism, "mixed")
    p.set_arrival_form("split")
    return p, to_device(t), ref


@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
@pytest.mark.parametrize("n_tracks,n_ant,n_bins", [(1, 3, 1000), (1999, 3, 1000), (2000, 3, 1000), (16500, 3, 1021),
                                                   (9000, 65, 1025), (5000, 2, 4097), (300, 1, 1)])
def test_traces_and_resets(formalism, n_tracks, n_ant, n_bins):
    p, t, ref = setup(formalism, n_tracks, n_ant, n_bins)
    few = {f: x[:max(1, len(x) // 40)].contiguous() for f, x in t.items()}
    for reset in ("fetch", "host", "reset"):
        p.push(t)
        if reset == "host":
            got = torch.empty(ref.shape, dtype=torch.float32)
            p.traces(reset=True, out=got)
        else:
            got = p.traces(reset=reset == "fetch").cpu()
            if reset == "reset":
                p.reset()
        assert rel_l2(got.numpy(), ref) < TOL
        # zero everywhere, also to a push that uses fewer copies
        assert not p.traces().any()
        p.push(few)
        p.reset()
        assert not p.traces().any()
    p.close()


@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
def test_push_replayed_from_a_graph(formalism):
    p, t, ref = setup(formalism, 16500, 3, 1000)
    p.push(t)  # allocates the scratch
    p.traces(reset=True)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        p.push(t)
    p.reset()
    g.replay()
    g.replay()
    assert rel_l2(p.traces(reset=True).cpu().numpy(), 2.0 * ref) < TOL
    g.replay()
    assert rel_l2(p.traces().cpu().numpy(), ref) < TOL
    p.reset()
    assert not p.traces().any()
    p.close()


@pytest.mark.parametrize("formalism", ["endpoint", "zhs"])
@pytest.mark.parametrize("n_tracks,n_ant,n_bins", [(1, 1, 1000), (16500, 1, 1000), (16500, 3, 1021), (9000, 32, 1025),
                                                   (9000, 33, 1025)])
def test_copies_of_the_fp64_accumulator(formalism, n_tracks, n_ant, n_bins):
    """Few antennas on the FP64 path: traces, both kinds of reset and pushes
    replayed from a graph, against the oracle at the FP64 bar (1e-9)."""
    from paper_2309_03717_gb300.c8r import RadioProcess
    w = synth.workload(1, n_tracks=n_tracks, n_ant=n_ant)
    tr = synth.workload_tracks(w)
    if formalism == "endpoint":
        tr = drop_tracks(tr, endpoint_unambiguous(tr, w["ant_xyz"], w["t_start_ns"], n_bins, w["dt_ns"], w["medium"]))
    ref, _ = oracle_traces(tr, w["ant_xyz"], w["t_start_ns"], n_bins, w["dt_ns"], w["medium"], formalism)
    p = RadioProcess(w["medium"], w["ant_xyz"], w["t_start_ns"], n_bins, w["dt_ns"], formalism, "fp64")
    t = to_device({f: x.astype(np.float64) for f, x in tr.items()})
    for _ in range(2):
        p.push(t)
        assert rel_l2(p.traces(reset=True).cpu().numpy(), ref) < 1e-9
    p.push(t)
    p.reset()
    assert not p.traces().any()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        p.push(t)
    p.reset()
    g.replay()
    g.replay()
    assert rel_l2(p.traces().cpu().numpy(), 2.0 * ref) < 1e-9
    p.close()
