"""Batched calls replayed after something changed under their graph (needs a GPU).

A batched call is captured once and replayed for the same arguments.  Between two
calls a surface may run by itself under another tile shape, which plans its records
for other windows; every batched call then needs its own plan back.  And a surface
that took a closed one's place needs a graph of its own.  Against one fwh_forward
call per surface, to the rounding of the FP64 output sums (1e-12 of the largest
value)."""
import numpy as np
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


def _surface(i, prec, aoa=0.1):
    from paper_2312_16263_gb300 import FWH
    sf = uv_sphere(1.0 + 0.3 * i, 12, 20, center=(i, 0, 0))
    return FWH(sf.centroids, sf.normals, sf.areas, 0.35, aoa, 0.02, prec,
               observers=observers_circle(30.0, 5))


def _fields(prec, dev, nt=300):
    g = torch.Generator(device=dev).manual_seed(4)
    dtype = torch.float64 if prec == "fp64" else torch.float32
    return [torch.randn((nt, 5, 240), dtype=dtype, device=dev, generator=g) * 1e-3 for _ in range(2)]


def _close(outs, refs):
    for a, b in zip(outs, refs):
        assert b.abs().max().item() > 0
        torch.testing.assert_close(a, b, rtol=1e-12, atol=1e-12 * b.abs().max().item())


@pytest.mark.parametrize("form", ["pipelined", "grid", "persistent"])
@pytest.mark.parametrize("prec,shape", [("mixed", 2), ("mixed", 10), ("fp64", 1),
                                        ("fp64", 3)])
def test_another_tile_shape_between_two_batches(dev, prec, shape, form):
    from paper_2312_16263_gb300 import batch_forward
    fields = _fields(prec, dev)
    refs = []
    for i in range(2):
        s = _surface(i, prec)
        refs.append(s.forward(fields[i]))
        s.check()
        s.close()
    surfs = [_surface(i, prec) for i in range(2)]
    surfs[0].set_batch_options(0, form)
    outs = batch_forward(surfs, fields)
    _close(outs, refs)
    surfs[1].set_tile_config(shape)          # plans the records of surface 1 for that shape
    other = surfs[1].forward(fields[1])
    torch.testing.assert_close(other, refs[1], rtol=0, atol=1e-5 * refs[1].abs().max().item())
    for p in outs:
        p.zero_()
    _close(batch_forward(surfs, fields, outs), refs)  # the same arguments: replayed
    surfs[0].check()
    for s in surfs:
        s.close()


def test_another_surface_in_the_place_of_a_closed_one(dev):
    """A new surface may get the address and the buffers of one that was closed; it
    must not get its graph (here: its angle of attack)."""
    from paper_2312_16263_gb300 import batch_forward
    fields = _fields("mixed", dev)
    outs = [torch.empty((5, 300), dtype=torch.float64, device=dev) for _ in range(2)]
    first = _surface(0, "mixed")
    for aoa in (0.1, -0.4, 0.3, 0.0):
        second = _surface(1, "mixed", aoa)
        batch_forward([first, second], fields, outs)
        first.check()
        refs = [first.forward(fields[0]), second.forward(fields[1])]
        _close(outs, refs)
        second.close()
    first.close()
