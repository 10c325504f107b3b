"""The flat model's table of group maxima: bounded memory, and the same bits
where a call is too large for it."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu


def test_memory_of_a_large_model_is_bounded():
    """2^20 points x 4,680 components: 256 MB of table, and the components
    (0.4 KB each), points (4 bytes) and partial sums (13 MB) beside it."""
    import torch
    from paper_1807_02587_gb300 import binding as B
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    flat = B.Flat(1 << 20, B.hgmm_node_count(4))
    used = before - torch.cuda.mem_get_info()[0]
    flat.close()
    assert used <= (256 + 64) << 20, used


def test_same_bits_without_the_table():
    """A depth-5 tree whose deepest level is all dead has the same components
    cut at its last two levels, but the deeper cut's 37,448 candidates are too
    many for the table with 60,000 points."""
    import torch
    from paper_1807_02587_gb300 import binding as B
    p = synth.primitive_pair(8, 60000)
    tgt, _ = PT.device_cloud(p["tgt"])
    src, _ = PT.device_cloud(p["src"])
    tree = B.Tree(60000, 5)
    tree.build(tgt, 5, B.params(n_min=300.0))
    tree.sync()
    assert not tree.export(4)["live"].any()
    flat = B.Flat(60000, B.hgmm_node_count(5))
    out = []
    for level in (3, 4):
        flat.from_tree(tree, level)
        hist = torch.zeros((4, 16), dtype=torch.float64, device="cuda")
        flat.register(src, iters=4, T_hist=hist)
        flat.sync()
        J = len(flat.export()["pi"])
        moments = flat.moments()
        flat.fit(tgt, 2)
        flat.sync()
        e = flat.export()
        out.append((J, hist.cpu().numpy(), moments, e["pi"], e["mu"], e["Sigma"]))
    assert out[0][0] == out[1][0] > 64
    for a, b in zip(out[0][1:], out[1][1:]):
        assert np.array_equal(a, b)
