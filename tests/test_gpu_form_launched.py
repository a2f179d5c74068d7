"""Which of the one-bin Endpoint kernels a push, an adjoint and a batch launch: the
form of the FP32 arrival is the fourth template argument of their arithmetic
(OpsMixed: formalism, medium, deposit, form, flat), read from the profiler's kernel
names.  The forms give the same bins, so no result tells them apart."""
import re

import numpy as np
import pytest

from _util import built_lib, to_device
from paper_2309_03717_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DIRECT, SPLIT, AXIS = 0, 1, 2
NO_FRONT = "no front"
warm = False


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()


def launched(work, kernel):
    from torch.profiler import ProfilerActivity, profile
    global warm
    if not warm:  # the profiler's first session can come up empty
        with profile(activities=[ProfilerActivity.CUDA]):
            torch.zeros(1, device="cuda")
            torch.cuda.synchronize()
        warm = True
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        work()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events()]
    if not names:
        pytest.skip("the profiler records no kernels here")
    forms = set()
    for n in names:
        m = re.search(kernel + r"<c8r::OpsMixed<[^>]*>", n)
        if m:
            args = re.findall(r"true|false|\d+", m.group(0).split("OpsMixed<")[1])
            forms.add(int(args[3]))
    assert forms, names
    return forms


def process(zenith, start_zenith, hills=0.0):
    from paper_2309_03717_gb300 import c8r
    tracks = to_device(synth.make_tracks(2001, 31, zenith))
    ant = synth.antennas_star(8, n_radii=5)[:37].copy()
    ant[:, 2] = np.linspace(0.0, hills, len(ant))
    t_start = synth.trace_start_ns(ant, zenith if start_zenith == NO_FRONT else start_zenith)
    if start_zenith == NO_FRONT:
        t_start[:] = t_start.min()
    return c8r.RadioProcess(synth.AIR_EXPONENTIAL, ant, t_start, 4096, 0.2, "endpoint", "mixed"), tracks


@pytest.mark.parametrize("zenith,start_zenith,hills,first,then", [
    (0.0, 0.0, 0.0, SPLIT, SPLIT), (15.0, 15.0, 0.0, SPLIT, SPLIT), (35.0, 35.0, 0.0, AXIS, AXIS),
    (60.0, 60.0, 0.0, AXIS, AXIS), (60.0, 60.0, 150.0, AXIS, AXIS), (78.0, 78.0, 0.0, AXIS, AXIS),
    (70.0, NO_FRONT, 0.0, SPLIT, DIRECT),  # windows that open together follow no inclined front
    (0.0, 60.0, 0.0, AXIS, SPLIT)])        # a front that the tracks do not come from: until their count is in
def test_form_of_pushes_and_adjoints(zenith, start_zenith, hills, first, then):
    from paper_2309_03717_gb300 import c8r
    p, tracks = process(zenith, start_zenith, hills)
    assert launched(lambda: p.push(tracks), "k_forward") == {first}
    p.stats()  # waits for the count of the tracks seen from above
    assert launched(lambda: p.push(tracks), "k_forward") == {then}
    n = tracks["x0"].numel()
    tg = {f: torch.zeros(n, dtype=torch.float32, device="cuda") for f in c8r.GRAD_FIELDS}
    ag = torch.zeros((p.n_ant, 3), dtype=torch.float64, device="cuda")
    dn = torch.zeros(1, dtype=torch.float64, device="cuda")
    G = torch.ones((p.n_ant, 3, p.n_bins), dtype=torch.float32, device="cuda")
    assert launched(lambda: c8r.c8r_backward(p.ctx, tracks, G, tg, ag, dn), "k_backward") == {then}
    for form, code in (("direct", DIRECT), ("split", SPLIT)):
        p.set_arrival_form(form)
        assert launched(lambda: p.push(tracks), "k_forward") == {code}
    p.close()


@pytest.mark.parametrize("zeniths,forms", [((0.0, 10.0), {SPLIT}), ((50.0, 65.0), {AXIS}),
                                           ((0.0, 60.0, NO_FRONT), {SPLIT, AXIS, DIRECT})])
def test_forms_of_a_batch(zeniths, forms):
    from paper_2309_03717_gb300 import c8r
    showers, tracks = [], []
    for k, z in enumerate(zeniths):
        zenith = 70.0 if z == NO_FRONT else z
        ant = synth.antennas_star(8, n_radii=5)[:30 + k].copy()
        t_start = synth.trace_start_ns(ant, zenith)
        if z == NO_FRONT:
            t_start[:] = t_start.min()
        showers.append({"n_tracks": 900 + k, "ant_xyz": ant, "t_start_ns": t_start})
        tracks.append(synth.make_tracks(900 + k, 50 + k, zenith))
    b = c8r.Batch(showers, synth.AIR_EXPONENTIAL, 4096, 0.2, "endpoint")
    out = b.new_output()
    dev = to_device({f: np.concatenate([t[f] for t in tracks]) for f in synth.FIELDS})
    b.run(dev, out, use_graph=False)
    assert launched(lambda: b.run(dev, out, use_graph=False), "k_batch") == forms
    b.sync()
    b.close()
