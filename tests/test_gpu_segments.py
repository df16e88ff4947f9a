"""Segment totals in tensor memory against exact distances: small integers without centring are
exact in BF16 and their sums in FP32 whatever the segment length, so calls of several segments
must equal the oracle and the call of one segment bitwise (a wrong accumulator, a segment left
out or added twice shows in every distance)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_02059_gb300 as m
    return m


@pytest.mark.parametrize("prec", ["split_bf16", "bf16"])
@pytest.mark.parametrize("N,D,L,k,seg,groups", [
    (700, 800, 5, 10, 256, 0), (700, 800, 5, 10, 64, 1), (1500, 130, 1, 33, 32, 0),
    (600, 640, 3, 64, 96, 0), (900, 200, 17, 5, 64, 1), (300, 400, 2, 4, 32, 0)])
def test_segment_totals_are_exact(tk, prec, N, D, L, k, seg, groups):
    import torch
    X = np.random.default_rng(N + D).integers(0, 4, (N, D)).astype(np.float32)
    e = L - 1
    oidx, odist, _ = oracle.knn_scores(X, L, k, e)
    Xd = torch.from_numpy(X).cuda()
    got = []
    for s in (seg, 0):
        hd = tk.Handle()
        hd.set_option("segment_k", s)
        hd.set_option("epi_groups", groups)
        kw = dict(precision=prec, center=False, handle=hd)
        got.append(tk.knn_scores(Xd, L, k, e, embed="never", **kw))
        got += tk.knn_scores_multi(Xd, [(L, k, e), (max(1, L - 1), k, e)], **kw)[:1]
        assert hd.sync_status() == 0
        hd.close()
    for idx, dist, score in got:
        assert np.array_equal(dist.cpu().numpy(), odist.astype(np.float32))
        assert np.array_equal(idx.cpu().numpy(), oidx)
        assert torch.equal(score, got[0][2])
