"""Work items of batched calls (needs a GPU).

Panel sets smaller than the number of parts a set is cut into.

65 panels, 64 close together and one apart, make panel sets of 64 and 1, and a
launch with few items cuts each set into several parts: the lone panel then
leaves parts without panels, hundreds of consecutive work items with no
pipeline step.  Every launch form of a batched call (for the persistent one both
precisions' copy-pipeline shapes) against one fwh_forward call per surface, to
the rounding of the FP64 output sums (the partial sums are the same): 1e-12 of
the largest value."""
import numpy as np
import pytest
import torch

from fwh_inputs.geometry import observers_circle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


def _cluster_and_one(rng):
    pos = np.concatenate([0.01 * rng.random((64, 3)), [[6.0, 0.0, 0.0]]])
    nrm = rng.normal(size=(65, 3))
    return pos, nrm / np.linalg.norm(nrm, axis=1, keepdims=True), rng.uniform(0.5, 1.5, 65)


@pytest.mark.parametrize("form", ["pipelined", "grid", "persistent"])
@pytest.mark.parametrize("prec,cfg,seg", [("mixed", -1, 252), ("mixed", 2, 496), ("fp64", 1, 512)])
@pytest.mark.parametrize("n_obs,n_segs", [(4, 113), (40, 56), (3, 2)])
def test_sets_smaller_than_their_parts(dev, prec, cfg, seg, form, n_obs, n_segs):
    from paper_2312_16263_gb300 import FWH, batch_forward
    rng = np.random.default_rng(65)
    pos, nrm, area = _cluster_and_one(rng)
    nt = n_segs * seg - 5
    surfs, fields, singles = [], [], []
    for i in range(2):
        s = FWH(pos, nrm, area, 0.4, 0.1, 0.02, prec,
                observers=observers_circle(40.0 + i, n_obs) + rng.normal(size=(n_obs, 3)))
        s.set_tile_config(cfg)
        f = torch.randn((nt, 5, 65), dtype=s.dtype, device=dev,
                        generator=torch.Generator(device=dev).manual_seed(i)) * 1e-3
        surfs.append(s)
        fields.append(f)
        singles.append(s.forward(f).clone())
        s.check()
    surfs[0].set_batch_options(0, form)
    for _ in range(2):  # the second call replays the captured graph
        outs = batch_forward(surfs, fields)
        surfs[0].check()
        for a, b in zip(outs, singles):
            assert b.abs().max().item() > 0
            torch.testing.assert_close(a, b, rtol=1e-12, atol=1e-12 * b.abs().max().item())
    for s in surfs:
        s.close()


@pytest.mark.parametrize("ring", [0, 512])
@pytest.mark.parametrize("prec,cfg", [("mixed", -1), ("mixed", 2), ("fp64", 1)])
def test_persistent_surfaces_with_unlike_observer_counts(dev, prec, cfg, ring):
    """The compute warps of a persistent CTA go from item to item on their own, so
    neighbours may work on surfaces with unlike numbers of observers a warp; their
    windows must not meet.  Against one fwh_forward call per surface (1e-12 of the
    largest value)."""
    from paper_2312_16263_gb300 import FWH, batch_forward
    rng = np.random.default_rng(12)
    surfs, fields, singles = [], [], []
    for i, (n, nt, n_obs) in enumerate([(700, 1300, 36), (300, 900, 3), (500, 1100, 20), (65, 1300, 9),
                                        (400, 700, 28), (200, 1500, 1)]):
        d = rng.normal(size=(n, 3))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        s = FWH(2.0 * d, d, rng.uniform(0.5, 1.5, n), 0.4, 0.1, 0.02, prec,
                observers=observers_circle(60.0 + i, n_obs))
        s.set_tile_config(cfg)
        f = torch.randn((nt, 5, n), dtype=s.dtype, device=dev,
                        generator=torch.Generator(device=dev).manual_seed(i)) * 1e-3
        surfs.append(s)
        fields.append(f)
        singles.append(s.forward(f).clone())
        s.check()
    surfs[0].set_batch_options(ring, "persistent")
    outs = None
    for _ in range(20):
        outs = batch_forward(surfs, fields, outs)
        surfs[0].check()
        for a, b in zip(outs, singles):
            torch.testing.assert_close(a, b, rtol=1e-12, atol=1e-12 * b.abs().max().item())
    for s in surfs:
        s.close()
