"""Each gradient that RadioTraces returns is a tensor of its own: it holds no other
gradient's memory, and what autograd allows on a plain tensor (detach_, resize)
works on it."""
import numpy as np
import pytest

from _util import built_lib, to_device
from paper_2309_03717_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_gradients_do_not_share_memory(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()
    from paper_2309_03717_gb300 import c8r
    dtype = torch.float64 if precision == "fp64" else torch.float32
    tracks = to_device(synth.make_tracks(1001, 3, 0.0), dtype)
    ant = synth.antennas_star(8, n_radii=2)[:5]
    p = c8r.RadioProcess(synth.AIR_EXPONENTIAL, ant, synth.trace_start_ns(ant), 256, 0.5, "endpoint", precision)
    N0 = torch.tensor(3.25e-4, dtype=torch.float64, device="cuda", requires_grad=True)
    pos = torch.from_numpy(np.ascontiguousarray(ant)).cuda().requires_grad_(True)
    for f in c8r.GRAD_FIELDS:
        tracks[f].requires_grad_(True)
    leaves = [tracks[f] for f in c8r.GRAD_FIELDS] + [pos, N0]
    tr = c8r.RadioTraces.apply(p, N0, *[tracks[f] for f in c8r.TRACK_FIELDS], pos)
    grads = torch.autograd.grad(tr, leaves, torch.full_like(tr, 1e9))
    starts = set()
    for leaf, g in zip(leaves, grads):
        assert g.shape == leaf.shape and g.dtype == leaf.dtype and g.is_contiguous()
        assert g.untyped_storage().nbytes() == g.numel() * g.element_size()
        starts.add(g.untyped_storage().data_ptr())
        g.detach_()
    assert len(starts) == len(leaves)
    assert grads[0].any() and grads[-2].any() and grads[-1].any()
    p.close()
