"""The batch's second sort of a large source before its seventh round (runs of
18 rounds and more): the node moments are exact integer sums, so the poses of
the rounds that a shorter run shares with a longer one are the same bit for
bit.  Source sizes at the threshold of the sorts, every extreme of the cluster
shape."""
import numpy as np
import pytest

from paper_1807_02587_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [1, 8])
def test_a_second_sort_changes_no_pose(shape):
    import torch
    from paper_1807_02587_gb300 import binding as B
    sizes = [16383, 16384, 40001]
    pairs = [synth.primitive_pair(50 + n, n, max_deg=8.0, max_t=0.05) for n in sizes]
    clouds = [synth.to_float4(p["tgt"]) for p in pairs] + [synth.to_float4(p["src"]) for p in pairs]
    off = np.concatenate([[0], np.cumsum([len(c) for c in clouds])]).astype(np.int64)
    pts = torch.from_numpy(np.concatenate(clouds)).cuda()
    bat = B.Batch(int(np.diff(off).max()), 4, len(sizes))
    B.hgmm_batch_plan(bat.handle, off[:4], off[3:], [3, 4, 4])
    B.hgmm_batch_set_shape(bat.handle, shape)
    hist = {}
    for iters in (5, 17, 18, 30):
        T = torch.zeros((len(sizes), 16), dtype=torch.float64, device="cuda")
        h = torch.zeros((len(sizes), iters, 16), dtype=torch.float64, device="cuda")
        st = torch.full((len(sizes),), 99, dtype=torch.int32, device="cuda")
        B.hgmm_batch_register(bat.handle, pts, T, iters=iters, pair_status=st, T_hist=h)
        torch.cuda.synchronize()
        assert np.all(st.cpu().numpy() == 0)
        hist[iters] = h.cpu().numpy()
        assert np.array_equal(hist[iters][:, -1], T.cpu().numpy())
    for iters in (5, 17, 18):
        assert np.array_equal(hist[iters], hist[30][:, :iters])
