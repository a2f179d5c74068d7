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


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [0, 1, 3, 5, 1023, 70_001])
def test_zero_gradients(n, precision):
    """All of the outputs and nothing beside them, on a 16-byte boundary or not."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    built_lib()
    from paper_2309_03717_gb300 import c8r
    dtype = torch.float64 if precision == "fp64" else torch.float32
    ant = synth.antennas_star(8, n_radii=2)[:5]
    p = c8r.RadioProcess(synth.AIR_EXPONENTIAL, ant, synth.trace_start_ns(ant), 256, 0.5, "endpoint", precision)
    rows = [torch.ones(n + 8, dtype=dtype, device="cuda") for _ in c8r.GRAD_FIELDS]
    tg = {f: rows[k][k % 4:k % 4 + n] for k, f in enumerate(c8r.GRAD_FIELDS)}
    ag, dn = torch.ones(17, dtype=torch.float64, device="cuda"), torch.ones(3, dtype=torch.float64, device="cuda")
    c8r.c8r_zero_gradients(p.ctx, tg, ag[1:16].view(5, 3), dn[1:2])
    p.close()
    for k, row in enumerate(rows):
        want = torch.ones_like(row)
        want[k % 4:k % 4 + n] = 0.0
        assert torch.equal(row, want)
    assert ag.tolist() == [1.0] + [0.0] * 15 + [1.0] and dn.tolist() == [1.0, 0.0, 1.0]
