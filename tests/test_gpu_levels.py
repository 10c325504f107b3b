"""The one-launch build of the tree's levels at the sizes where its split of
the points changes: less than one item, the edges of an item and of a run,
one and several items per chunk, runs reduced directly and in slices, several
runs of one parent in a CTA, and the first size that the level-wide launches
take.  One EM iteration at a time against the FP64 oracle (teacher forcing,
Eq. 2-3), with the tolerance of tests/test_gpu_build.py."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu

CHUNKS = 3 * 152  # chunks of a level-wide E-step on 152 SMs


def _cloud(kind, n):
    rng = synth.make_rng(n + 17)
    if kind == "scene":
        return synth._sample_primitives(rng, synth.primitive_scene(rng), n, 0.005)
    # a dense blob far below the covariance regulariser: its points stay in
    # one node per level, so a deep parent holds most of the cloud
    k = n // 4
    P = np.concatenate([rng.uniform(-1.0, 1.0, size=(k, 3)), 0.3 + 1e-4 * rng.normal(size=(n - k, 3))])
    return P[rng.permutation(n)]


@pytest.mark.parametrize("kind,n,depth", [
    ("scene", 8, 1), ("scene", 255, 2), ("scene", 257, 3), ("scene", 1024, 3), ("scene", 1025, 4),
    ("scene", 256 * CHUNKS, 2), ("scene", 256 * CHUNKS + 1, 2), ("scene", 512 * CHUNKS + 1, 2),
    ("scene", 409600, 2), ("blob", 150001, 4),
    # the level-wide E-step: two threads per point, whole and ragged items
    ("scene", 409601, 3), ("blob", 700001, 4)])
def test_em_iterations_of_every_level(kind, n, depth):
    from paper_1807_02587_gb300 import binding as B
    dev, Z = PT.device_cloud(_cloud(kind, n))
    steps = [(l, k) for l in range(depth) for k in ((1, 8) if n < 10000 or l == depth - 1 else (2,))]
    for r in PT.check_em_steps(B, dev, Z, depth, steps):
        print(kind, n, r)
        assert r["live_mismatch"] == 0, r
        assert r["mu"] < 1e-5 and r["S"] < 1e-5 and r["pi"] < 1e-5, r


@pytest.mark.parametrize("precision", [0, 1])  # 1: the level-wide launches at every size
@pytest.mark.parametrize("kind,n,depth", [("scene", 8, 2), ("scene", 300, 3), ("scene", 256 * CHUNKS + 1, 3),
                                          ("blob", 60000, 4), ("scene", 20000, 5), ("scene", 409601, 2)])
def test_segments_partition_the_points(kind, n, depth, precision):
    """After every hand-off each node's segment holds exactly the points
    labelled with it, children inside their parent, every point with its best
    child under the level's parameters (near-ties aside), and two builds agree."""
    from paper_1807_02587_gb300 import binding as B
    dev, Z = PT.device_cloud(_cloud(kind, n))
    prm = B.params(precision=precision)
    tree = B.Tree(n, depth)
    tree.build(dev, depth, prm)
    tree.sync()
    prev = np.zeros(n, np.int64)
    first = []
    for l in range(depth):
        lab = tree.labels(l).astype(np.int64)
        assert np.array_equal(lab // 8, prev), l
        g = tree.export(l)
        assert np.array_equal(np.bincount(lab, minlength=8 ** (l + 1)), g["count"]), l
        if n <= 100000:
            ref, margin = PT.handoff_check(Z, prev, g)
            assert not np.any((lab != ref) & (margin >= PT.TIE_MARGIN)), l
        first.append((lab, g))
        prev = lab
    tree.build(dev, depth, prm)
    tree.sync()
    for l in range(depth):
        assert np.array_equal(tree.labels(l), first[l][0])
        for k, v in tree.export(l).items():
            assert np.array_equal(v, first[l][1][k]), (l, k)
