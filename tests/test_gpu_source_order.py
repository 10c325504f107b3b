"""The spatial order that a large source is put into before its rounds, against
the same source in the caller's order (a traced registration is not reordered):
the same poses bit for bit, since the node moments are exact integer sums.
Sizes at the edges of a tile of 2,048 points and of the sorting CTAs' ranges;
clouds spread over the grid's cells, inside one cell, and far outside the
target (the grid repeats), with starting poses other than the identity."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,depth", [("scene", 1 << 20, 4), ("scene", (1 << 20) + 1, 5), ("blob", (1 << 20) + 2047, 3),
                                          ("far", (1 << 20) + 777, 2), ("scene", (1 << 21) + 4097, 4)])
def test_order_of_a_large_source_changes_nothing(kind, n, depth):
    import torch
    from paper_1807_02587_gb300 import binding as B
    rng = synth.make_rng(n)
    scene = synth.primitive_scene(rng)
    tgt, _ = PT.device_cloud(synth._sample_primitives(rng, scene, 100000, 0.005))
    P = synth._sample_primitives(rng, scene, 250000, 0.005)
    P = P[rng.integers(0, len(P), n)] + 1e-3 * rng.normal(size=(n, 3))
    if kind == "blob":
        P[n // 50:] = P[0] + 1e-3 * rng.normal(size=(n - n // 50, 3))
    elif kind == "far":
        P[::3] = 1e3 * rng.normal(size=P[::3].shape)
        P[7] = 1e30
    src, _ = PT.device_cloud(P)
    T0 = torch.from_numpy(synth.rigid(synth.random_rotation(rng, 20.0), rng.uniform(-0.1, 0.1, 3)).reshape(16)).cuda()
    tree = B.Tree(n, depth)
    tree.build(tgt, depth)
    hists = []
    for traced in (False, True):
        B.hgmm_trace(tree.handle, traced)
        hist = torch.zeros((4, 4, 4), dtype=torch.float64, device="cuda")
        tree.register(src, T_init=T0, iters=4, T_hist=hist)
        tree.sync()
        hists.append(hist.cpu().numpy())
    assert np.isfinite(hists[0]).all()
    assert np.array_equal(hists[0], hists[1])
