"""The registration's two descents (trees whose levels are all staged in shared
memory, up to depth 3; deeper ones) against the descent variant that searches
the same best path node by node from the nodes' own records: the same moments,
at point counts around a warp and a CTA, every depth on both sides of the line
and thresholds that stop early, late and never; and points so far away that the
squares of a level's scores overflow, at the first level and further down."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu


def _moments(B, tree, src, lam_c, rounds=(1, 3)):
    """Pose and last round's node moments after each number of rounds, both ways."""
    out = []
    for k in rounds:
        T = tree.register(src, iters=k, lam_c=lam_c)
        a = (T.cpu().numpy().reshape(16), tree.reg_moments())
        T = tree.register_descent(src, B.HGMM_DESCENT_ML_LOCAL, iters=k, lam_c=lam_c)
        out.append((a, (T.cpu().numpy().reshape(16), tree.reg_moments())))
    return out


@pytest.mark.parametrize("n", [1, 31, 33, 257, 5000, 90001])
@pytest.mark.parametrize("depth", [1, 2, 3, 4])
def test_moments_and_pose(depth, n):
    """Both convert every point's moments to the same 64-bit quanta (2^-32) from
    FP32 terms that differ by a few roundings of 2^-24, one point per quantum
    sum: 1e-6 of the mass, 1e-5 of a node's moment (mass times extent)."""
    from paper_1807_02587_gb300 import binding as B
    p = synth.primitive_pair(11, 90001)
    tgt, _ = PT.device_cloud(p["tgt"])
    src, _ = PT.device_cloud(p["src"][:n])
    tree = B.Tree(90001, depth)
    tree.build(tgt, depth)
    tree.sync()
    ext = tree.root()["extent"]
    for lam_c in (-1.0, 0.0, 0.05):
        for i, ((Ta, ma), (Tb, mb)) in enumerate(_moments(B, tree, src, lam_c)):
            if i == 0:
                big = mb[:, 0] > 0
                assert np.array_equal(ma[:, 0] > 0, big)
                assert abs(ma[:, 0].sum() - mb[:, 0].sum()) <= 1e-6 * n
                assert np.all(np.abs(ma[:, 0] - mb[:, 0]) <= 1e-6 * np.maximum(mb[:, 0], 1.0))
                assert np.all(np.abs(ma[:, 1:] - mb[:, 1:]) <= 1e-5 * ext * np.maximum(mb[:, :1], 1.0))
            if n >= 5000:  # a few points do not determine a pose
                assert np.max(np.abs(Ta - Tb)) <= 1e-5
    try:
        tree.sync()
    except B.HgmmError as e:
        assert e.code == B.HGMM_EDEGENERATE and n < 5000


@pytest.mark.parametrize("depth", [2, 3, 4])
def test_scores_that_overflow(depth):
    """A score is a sum of squares of W (z - mu) with W about 0.85 / sigma: at
    1e25 metres every square overflows FP32 at the first level (the point has no
    node); at 1e18 it does not for the first level's Gaussians (sigma of tenths
    of a metre: 1e37) and does for deeper ones of a few centimetres' thickness
    (1e39), and the point stays with the node above."""
    import torch
    from paper_1807_02587_gb300 import binding as B
    p = synth.primitive_pair(11, 60000)
    tgt, _ = PT.device_cloud(p["tgt"])
    tree = B.Tree(60000, depth)
    tree.build(tgt, depth)
    tree.sync()
    rng = np.random.default_rng(3)
    d = rng.normal(size=(4096, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    for scale, near in ((1e25, 0), (1e18, 0), (1e18, 2048), (1e25, 2048)):
        P = np.zeros((4096, 4), np.float32)
        P[:, :3] = d * scale
        P[:near, :3] = p["src"][:near]
        P = P[rng.permutation(4096)]
        src = torch.from_numpy(P).cuda()
        (_, ma), (_, mb) = _moments(B, tree, src, 0.0, rounds=(1,))[0]
        assert np.array_equal(ma[:, 0] > 0, mb[:, 0] > 0)
        assert np.all(np.abs(ma[:, 0] - mb[:, 0]) <= 1e-6 * np.maximum(mb[:, 0], 1.0))
        mass = ma[:, 0].sum()
        if scale == 1e25:
            assert near == 0 and mass == 0.0 or near and mass <= near * (1 + 1e-6)
        else:
            # some stopped above the last level without a stop flag (lam_c = 0): the case this is about
            assert ma[: B.hgmm_node_count(depth) - 8 ** depth, 0].sum() > 0
    try:
        tree.sync()
    except B.HgmmError as e:
        assert e.code == B.HGMM_EDEGENERATE


def test_registrations_around_a_variant():
    """A variant with another threshold between two registrations leaves no
    trace: the blocks are those of the registration's own threshold."""
    from paper_1807_02587_gb300 import binding as B
    p = synth.primitive_pair(5, 20000)
    tgt, _ = PT.device_cloud(p["tgt"])
    src, _ = PT.device_cloud(p["src"])
    want = {}
    for lam_c in (-1.0, 0.0, 0.2):
        tree = B.Tree(20000, 4)
        tree.build(tgt, 4)
        want[lam_c] = tree.register(src, iters=5, lam_c=lam_c).cpu().numpy()
    tree = B.Tree(20000, 4)
    tree.build(tgt, 4)
    for lam_c, other in ((0.0, 0.2), (0.2, 0.0), (-1.0, 0.0), (0.0, -1.0)):
        tree.register_descent(src, B.HGMM_DESCENT_MULTIPATH, tau=0.1, iters=2, lam_c=other)
        assert np.array_equal(tree.register(src, iters=5, lam_c=lam_c).cpu().numpy(), want[lam_c])
    tree.sync()
