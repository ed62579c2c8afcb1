"""Calls on one surface enqueued on a stream of the caller's without waits (needs a GPU).

Record lengths, and the tile shapes of batched and single calls, change from call to
call while the earlier ones are still pending behind a delay on the stream: the tables
that go with them (observer windows, panel-set plans) must reach the device in the
stream's order.  Every result against the same call made alone, to the rounding of the
FP64 output sums (1e-12 of the largest value; gradients, without atomics here, to the
same)."""
import pytest
import torch

from fwh_inputs.geometry import observers_circle, uv_sphere

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("prec,shape", [("mixed", 2), ("mixed", 10), ("fp64", 3)])
def test_tables_follow_the_stream(dev, prec, shape):
    from paper_2312_16263_gb300 import FWH, batch_forward
    sf = uv_sphere(0.5, 10, 20)

    def surface():
        return FWH(sf.centroids, sf.normals, sf.areas, 0.4, 0.1, 0.02, prec,
                   observers=observers_circle(30.0, 5))

    dtype = torch.float64 if prec == "fp64" else torch.float32
    g = torch.Generator(device=dev).manual_seed(9)
    lengths = (700, 90, 400, 91, 700)
    fields = [torch.randn((nt, 5, 200), dtype=dtype, device=dev, generator=g) * 1e-3 for nt in lengths]
    grads = [torch.randn((5, nt), dtype=torch.float64, device=dev, generator=g) for nt in lengths]
    alone, refs, grad_refs = surface(), [], []
    for f, gp in zip(fields, grads):
        refs.append(alone.forward(f).clone())
        grad_refs.append(alone.backward(f, gp).clone())
        torch.cuda.synchronize()
    lead, s = surface(), surface()
    s.set_tile_config(shape)                 # its single calls; batches run the lead's shape
    batch_forward([lead, s], [fields[0], fields[0]])
    s.forward(fields[0])
    s.backward(fields[0], grads[0])          # every buffer at its full size
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(int(4e8))          # about 0.2 s: all that follows is enqueued behind it
        outs, got_grads = [], []
        for f, gp in zip(fields, grads):
            outs.append((s.forward(f), batch_forward([lead, s], [f, f])))
            got_grads.append(s.backward(f, gp))
    stream.synchronize()
    s.check()
    lead.check()
    for (one, pair), ref in zip(outs, refs):
        top = ref.abs().max().item()
        assert top > 0
        torch.testing.assert_close(one, ref, rtol=0, atol=(1e-12 if prec == "fp64" else 1e-5) * top)
        for p in pair:
            torch.testing.assert_close(p, ref, rtol=1e-12, atol=1e-12 * top)
    for a, b in zip(got_grads, grad_refs):
        torch.testing.assert_close(a, b, rtol=0, atol=(1e-12 if prec == "fp64" else 1e-5) * b.abs().max().item())
    for h in (alone, lead, s):
        h.close()
