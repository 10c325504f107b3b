"""The flat E-step's and moments' skipped components: per point, groups of 32
components that lie more than 127 binary orders below the point's likelihood
add nothing to any FP32 sum.  Clouds of separated blobs, where most groups are
skipped, next to one blob, where none is; point counts at the edges of the
moments' stage (2,048 points), component counts below, at and across a group.
One EM iteration and the first registration round's moments against the FP64
oracle, with the tolerances of tests/test_gpu_flat.py."""
import numpy as np
import pytest

from oracle import hgmm_oracle as O
from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu


def _cloud(blobs, n):
    rng = synth.make_rng(31 * blobs + n)
    c = rng.uniform(-20.0, 20.0, size=(blobs, 3))
    k = rng.integers(0, blobs, size=n)
    return c[k] + rng.normal(size=(n, 3)) * rng.uniform(0.05, 0.6, size=(blobs, 3))[k]


def _oracle(flat, eps):
    e = flat.export()
    return O.Flat(pi=e["pi"], mu=e["mu"], Sigma=e["Sigma"], node=e["node"], eps=eps)


@pytest.mark.parametrize("blobs,n,depth", [(1, 2047, 1), (40, 2048, 2), (40, 2049, 3), (6, 4097, 3), (60, 33, 1),
                                           (60, 20001, 4)])
def test_skipped_groups_change_nothing(blobs, n, depth):
    import torch
    from paper_1807_02587_gb300 import binding as B
    dev, Z = PT.device_cloud(_cloud(blobs, n))
    tree = B.Tree(n, depth)
    tree.build(dev, depth)
    eps = tree.root()["eps"]
    flat = B.Flat(n, int(B.hgmm_node_count(depth)))
    flat.from_tree(tree)
    if not tree.export(0)["pi"].any():  # too few points in every node: no component to register to
        with pytest.raises(B.HgmmError):
            flat.sync()
        return
    flat.sync()
    before = _oracle(flat, eps)
    flat.register(dev, T_init=torch.eye(4, dtype=torch.float64, device="cuda").reshape(16), iters=1)
    flat.sync()
    g = flat.moments()
    M0, M1 = O.flat_moments(before, Z)
    assert abs(g[:, 0].sum() - n) < 1e-5 * n
    big = M0 > 1.0
    assert (np.abs(g[big, 0] - M0[big]) / M0[big]).max() < 1e-4
    err = np.linalg.norm(M1[big] / M0[big, None] - g[big, 1:] / g[big, :1], axis=1)
    assert (err / tree.root()["extent"]).max() < 1e-5
    flat.fit(dev, 1)
    flat.sync()
    cur = _oracle(flat, eps)
    want, _ = O.flat_em(Z, before, 1, n_min=8.0)
    live = want.pi > 0
    assert np.array_equal(live, cur.pi > 0)
    scale = np.maximum(np.linalg.norm(want.mu[live], axis=1),
                       np.sqrt(np.trace(want.Sigma[live], axis1=1, axis2=2)))
    assert (np.linalg.norm(cur.mu[live] - want.mu[live], axis=1) / scale).max() < PT.MEAN_TOL
    assert (np.linalg.norm(cur.Sigma[live] - want.Sigma[live], axis=(1, 2))
            / np.linalg.norm(want.Sigma[live], axis=(1, 2))).max() < PT.COV_TOL
    assert np.abs(cur.pi[live] - want.pi[live]).max() < PT.PI_TOL
