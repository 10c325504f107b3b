"""The registration descent's sibling blocks: the moments of the first round
against the FP64 oracle at the edges of a warp's 32 points, for every depth
(staged levels only, one and two levels read from the cache), with stop flags
for none, some and most nodes, in both builds of the kernel's inputs (a large
source is recorded and reordered), and for points far outside the model.
Tolerances as in tests/test_gpu_register.py."""
import numpy as np
import pytest

from oracle import hgmm_oracle as O
from paper_1807_02587_gb300 import synth
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,depth,lam_c", [(8, 1, 0.0), (31, 2, 0.01), (32, 3, 0.1), (33, 4, 0.01), (257, 5, 0.0),
                                           (20001, 5, 0.01), (77825, 4, 0.3), (300000, 3, 0.01)])
def test_first_round_moments(n, depth, lam_c):
    import torch
    from paper_1807_02587_gb300 import binding as B
    rng = synth.make_rng(n + depth)
    scene = synth.primitive_scene(rng)
    tgt, _ = PT.device_cloud(synth._sample_primitives(rng, scene, 60000, 0.005))
    P = synth._sample_primitives(rng, scene, n, 0.005)
    P[::17] += rng.normal(size=P[::17].shape) * 50.0  # some far outside
    src, Zs = PT.device_cloud(P[rng.permutation(n)])
    tree = B.Tree(60000, depth)
    tree.build(tgt, depth, B.params(lam_c=lam_c))
    tree.sync()
    extent = tree.root()["extent"]
    ot = PT.tree_from_gpu(tree, PT.oracle_params(B.params(lam_c=lam_c), depth), extent)
    tree.register(src, T_init=torch.eye(4, dtype=torch.float64, device="cuda").reshape(16), iters=1)
    tree.sync()
    E = O.e_step_adaptive(ot, Zs)
    M0, M1 = np.concatenate(E["M0"]), np.concatenate(E["M1"])
    g = tree.reg_moments()
    dM0 = np.abs(g[:, 0] - M0)
    assert dM0.sum() <= 1e-4 * n + 1.0, dM0.sum()
    assert np.isclose(g[:, 0].sum(), M0.sum(), rtol=1e-5)
    big = M0 > 5.0
    if big.any():
        err = np.linalg.norm(M1[big] / M0[big, None] - g[big, 1:] / g[big, :1], axis=1) / extent
        assert np.median(err) < 1e-6, np.median(err)
