"""Records whose last round of a series ring starts at the record's end (needs a GPU).

A ring keeps the series of R time segments (252 intervals mixed, 128 samples
FP64, 512 in FP64's copy-pipeline shape) and prepares each round's rows anew.  An
FP64 record of 128 m - 1 or 128 m samples ends in a round of one or two rows, the
last sample and the ghost after it.  Record lengths around every such edge, in both
precisions and every launch form, against one fwh_forward call per surface on
handles of their own, to the rounding of the FP64 output sums (1e-12 of the largest
value).  The series buffers hold a longer record of larger fields first, so a row
left unwritten shows; the small surfaces leave nearly the whole record valid."""
import numpy as np
import pytest
import torch

from fwh_inputs.geometry import observers_circle, uv_sphere

pytestmark = pytest.mark.gpu

F64 = (255, 256, 257, 383, 384, 511, 512, 513)
F64_PIPE = (511, 512, 1022, 1023, 1024, 1025, 1535, 1536)
MIXED = (252, 253, 254, 255, 256, 504, 505, 512, 756, 757)


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("form", ["pipelined", "grid", "persistent"])
@pytest.mark.parametrize("prec,cfg,ring,nts", [
    ("fp64", -1, 128, F64), ("fp64", -1, 256, F64), ("fp64", 1, 512, F64_PIPE),
    ("mixed", -1, 256, MIXED), ("mixed", -1, 512, MIXED)])
def test_rounds_at_the_record_end(dev, prec, cfg, ring, nts, form):
    from paper_2312_16263_gb300 import FWH, batch_forward
    rng = np.random.default_rng(7)

    def handles():
        out = []
        for i in range(2):
            sf = uv_sphere(0.02 + 0.01 * i, 7, 11)
            s = FWH(sf.centroids, sf.normals, sf.areas, 0.4, 0.1, 0.03, prec,
                    observers=observers_circle(6.0 + i, 3))
            s.set_tile_config(cfg)
            out.append(s)
        return out

    def fields(nt, scale):
        return torch.as_tensor(rng.normal(size=(nt, 5, 77)) * scale, device=dev).to(
            torch.float64 if prec == "fp64" else torch.float32)

    batch, single = handles(), handles()
    batch[0].set_batch_options(ring, form)
    for nt in nts:
        fs = [fields(nt, 1e-3), fields(nts[-1] - nt + nts[0], 1e-3)]
        for s in batch:  # larger values in every row of the series buffer
            s.forward(fields(2100, 0.1))
        outs = batch_forward(batch, fs)
        batch[0].check()
        for s, f, p in zip(single, fs, outs):
            ref = s.forward(f)
            s.check()
            _, nv = s.window(f.shape[0])
            assert min(nv) >= f.shape[0] - 4, (nt, nv)
            torch.testing.assert_close(p, ref, rtol=1e-12, atol=1e-12 * ref.abs().max().item())
    for s in batch + single:
        s.close()
