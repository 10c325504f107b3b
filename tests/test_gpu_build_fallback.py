"""A device that refuses the build's cooperative launch (a context that owns
part of the SMs): the level-wide launches build the same tree.

The refusal is the runtime's own: the launch asks for more CTAs than the device
can hold, returns an error and runs nothing.  The two builds add the same FP32
run sums in another order, in compensated pairs whose rounding is about 2^-48
of a sum; eight iterations per level pass that on.  Records are held to 1e-10
of the extent (squared for covariances), labels to one point in a thousand."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_1807_02587_gb300 import binding
    return binding


def _build(B, dev, depth, refuse, profile=False):
    tree = B.Tree(dev.shape[0], depth)
    B.hgmm_debug_refuse_build(tree.handle, refuse)
    tree.profile(profile)
    tree.build(dev, depth)
    tree.sync()
    return tree


# one chunk per CTA, parents of many runs, and a depth whose last level the one-launch build leaves over
@pytest.mark.parametrize("n, depth", [(1000, 2), (30000, 4), (150000, 3), (60000, 5)])
def test_refused_launch_builds_the_same_tree(B, n, depth):
    dev, _ = PT.device_cloud(synth.primitive_pair(3, n)["tgt"])
    a, b = _build(B, dev, depth, False), _build(B, dev, depth, True)
    ext = a.root()["extent"]
    assert abs(b.root()["extent"] - ext) <= 1e-6 * ext
    for l in range(depth):
        x, y = a.export(l), b.export(l)
        assert np.array_equal(x["live"], y["live"])
        for k, s in (("pi", 1.0), ("mu", ext), ("Sigma", ext * ext)):
            assert np.max(np.abs(x[k] - y[k])) <= 1e-10 * s, (l, k)
        assert np.mean(a.labels(l) != b.labels(l)) <= 1e-3


def test_the_level_wide_launches_ran(B):
    """The profile names what ran: no one-launch build when it is refused, no
    level-wide E-step when it is not."""
    dev, _ = PT.device_cloud(synth.corner_pair(1)["tgt"])
    one = _build(B, dev, 3, False, profile=True).profile_read()
    wide = _build(B, dev, 3, True, profile=True).profile_read()
    assert one["build_levels"][1] == 1 and one["estep"][1] == 0
    assert wide["build_levels"][1] == 0 and wide["estep"][1] > 0

