"""The level-wide launches at the sizes where their kernels change (one item per
chunk and per CTA, up to four items per chunk, more; a parent's items over
several chunks and several parents in one), against the cooperative EM, which
runs the general E-step over the same chunks: the same bits.

Precision 0 reaches them at these sizes when the device refuses the one-launch
build (hgmm_debug_refuse_build), and always from about 410,000 points on."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu

CHUNKS = 3 * 152  # chunks of the E-step's grid on 152 SMs


def _cloud(n):
    """A scene with a dense blob in it, so that parents of a few and of most
    points lie side by side."""
    rng = synth.make_rng(n)
    k = n // 3
    P = np.concatenate([synth._sample_primitives(rng, synth.primitive_scene(rng), n - k, 0.005),
                        0.3 + 1e-3 * rng.normal(size=(k, 3))])
    return P[rng.permutation(n)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n, depth", [(8, 1), (255, 2), (257, 3), (5000, 4), (256 * (CHUNKS - 8), 2),
                                      (256 * CHUNKS, 3), (700 * CHUNKS + 3, 3), (1024 * (CHUNKS - 2), 2),
                                      (1024 * CHUNKS + 1, 3), (600001, 4)])
def test_per_iteration_launches_equal_the_cooperative_em(n, depth, precision):
    from paper_1807_02587_gb300 import binding as B
    dev, _ = PT.device_cloud(_cloud(n))
    out = []
    for flags in (0, B.HGMM_FLAG_EM_COOPERATIVE):
        tree = B.Tree(n, depth)
        B.hgmm_debug_refuse_build(tree.handle, True)
        tree.profile(True)
        tree.build(dev, depth, B.params(flags=flags, precision=precision))
        tree.sync()
        p = tree.profile_read()
        assert p["build_levels"][1] == 0 and (p["mstep"][1] == 0) == (flags != 0)
        out.append([(tree.export(l), tree.labels(l)) for l in range(depth)])
    for (a, la), (b, lb) in zip(*out):
        for k in ("pi", "mu", "Sigma", "live", "count", "lam"):
            assert np.array_equal(a[k], b[k])
        assert np.array_equal(la, lb)
