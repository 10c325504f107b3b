"""The flat model's components against the records of the tree they come from,
for cuts whose candidates one launch writes (8 and 72) and for larger ones."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, depth", [(300, 1), (300, 2), (20000, 2), (20000, 3), (300, 4), (20000, 4)])
def test_components(n, depth):
    """mu and Sigma are copies; the weights are products of at most four numbers
    and one division: a few roundings of 2^-53."""
    from paper_1807_02587_gb300 import binding as B
    dev, _ = PT.device_cloud(synth.primitive_pair(2, n)["tgt"])
    tree = B.Tree(n, depth)
    tree.build(dev, depth)
    tree.sync()
    lv = [tree.export(l) for l in range(depth)]
    flat = B.Flat(n, B.hgmm_node_count(depth))
    for cut in range(depth):
        w, node = [], []
        path = np.ones(1)
        for l in range(cut + 1):
            path = np.repeat(path, 8) * np.where(lv[l]["live"], lv[l]["pi"], 0.0)
            leaf = lv[l]["live"].astype(bool).copy()
            if l < cut:
                leaf &= ~lv[l + 1]["live"].astype(bool).reshape(-1, 8).any(axis=1)
            for i in np.flatnonzero(leaf):
                w.append(path[i])
                node.append((l, i))
        flat.from_tree(tree, cut)
        flat.sync()
        e = flat.export()
        assert [tuple(x) for x in e["node"]] == node
        np.testing.assert_allclose(e["pi"], np.array(w) / np.sum(w), rtol=1e-13)
        for k, (l, i) in enumerate(node):
            assert np.array_equal(e["mu"][k], lv[l]["mu"][i]) and np.array_equal(e["Sigma"][k], lv[l]["Sigma"][i])
