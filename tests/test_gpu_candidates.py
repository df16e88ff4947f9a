"""Candidate lists, shared minima and bounds of the symmetric kernels where they can go
wrong: few-valued integer fields, whose distances tie by the hundred (lists, column records
and the merge's buffer overflow, and the order among ties decides), every range of k with its
own number of shared minima, exclusion zones wider than the band, and two epilogue groups
with a window. Small integers are exact in BF16 and their sums in FP32, so without centring
the neighbour sets and distances must equal the oracle's, ties included."""
import numpy as np
import pytest

import oracle
from synth import make_slp_like

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_02059_gb300 as m
    return m


def _integers(N, D, top, seed):
    return np.random.default_rng(seed).integers(0, top + 1, (N, D)).astype(np.float32)


@pytest.mark.parametrize("prec", ["split_bf16", "bf16"])
@pytest.mark.parametrize("N,D,top,L,k,e", [
    (700, 3, 1, 1, 1, 0), (700, 3, 1, 2, 5, 1), (700, 4, 2, 1, 20, 0), (1300, 3, 1, 5, 33, 4),
    (700, 4, 3, 3, 41, 2), (700, 3, 1, 17, 64, 16), (2600, 4, 2, 2, 20, 1),
    (1500, 4, 3, 2, 10, 400), (1500, 4, 3, 1, 40, 700), (129, 2, 1, 2, 64, 1)])
def test_ties_and_wide_exclusion_equal_the_oracle(tk, prec, N, D, top, L, k, e):
    import torch
    X = _integers(N, D, top, seed=N + k)
    oidx, odist, _ = oracle.knn_scores(X, L, k, e)
    for embed in ("never", "always") if L > 1 else ("never",):
        idx, dist, _ = tk.knn_scores(torch.from_numpy(X).cuda(), L, k, e, precision=prec,
                                     center=False, embed=embed)
        assert np.array_equal(dist.cpu().numpy(), odist.astype(np.float32))
        assert np.array_equal(idx.cpu().numpy(), oidx)


@pytest.mark.parametrize("N,D,top,L,k,e", [
    (700, 3, 1, 1, 1, 0), (700, 4, 2, 1, 20, 0), (1300, 3, 1, 5, 33, 4), (700, 3, 1, 17, 64, 16),
    (1500, 4, 3, 2, 10, 400), (129, 70, 3, 2, 64, 1), (384, 600, 1, 4, 5, 3)])
def test_fp32_upper_triangle_equals_the_oracle(tk, N, D, top, L, k, e):
    """Small integers again (exact in FP32): single, batched and several-settings calls."""
    import torch
    X = _integers(N, D, top, seed=N + k)
    Xd = torch.from_numpy(X).cuda()
    L2 = max(1, L - 1)
    ref = [oracle.knn_scores(X, l, k, e)[:2] for l in (L, L2)]
    got = [(tk.knn_scores(Xd, L, k, e, precision="fp32", center=False), 0)]
    got += zip(tk.knn_scores_batched([(Xd, L, k, e), (Xd, L2, k, e)], precision="fp32",
                                     center=False), (0, 1))
    got += zip(tk.knn_scores_multi(Xd, [(L, k, e), (L2, k, e)], precision="fp32",
                                   center=False), (0, 1))
    for (idx, dist, _), b in got:
        assert np.array_equal(dist.cpu().numpy(), ref[b][1].astype(np.float32))
        assert np.array_equal(idx.cpu().numpy(), ref[b][0])


@pytest.mark.parametrize("N,h,w,L,k,e", [(1500, 20, 32, 5, 20, 4), (2000, 36, 41, 2, 10, 1),
                                         (900, 30, 33, 17, 32, 16), (385, 20, 40, 3, 1, 2),
                                         (3000, 45, 50, 4, 12, 3)])
def test_two_epilogue_groups_with_a_window_equal_one(tk, N, h, w, L, k, e):
    """The second group starts its windows from columns it reads itself, the first one a
    tile's from the columns the second group read: bitwise the same distances."""
    import torch
    X = torch.from_numpy(make_slp_like(N, h, w, seed=N + L)[0]).cuda()
    for prec in ("split_bf16", "bf16"):
        got = []
        for groups in (0, 1):
            hd = tk.Handle()
            hd.set_option("epi_groups", groups)
            got.append(tk.knn_scores(X, L, k, e, precision=prec, embed="never", handle=hd))
            got.append(tk.knn_scores_multi(X, [(L, k, e), (max(1, L - 1), k, e)],
                                           precision=prec, handle=hd)[0])
            torch.cuda.synchronize()
            assert hd.sync_status() == 0
        for a, b in ((got[0], got[2]), (got[1], got[3])):
            for x, y in zip(a, b):
                assert torch.equal(x, y)


@pytest.mark.parametrize("N,h,w,L,k,sym,seg", [
    (1500, 9, 14, 5, 10, True, 0), (700, 9, 14, 2, 41, True, 0), (130, 9, 14, 3, 5, True, 0),
    (900, 20, 40, 17, 20, False, 0), (1000, 20, 40, 1, 64, True, 0), (1100, 20, 40, 5, 20, True, 256),
    (9000, 8, 9, 4, 10, True, 64)])
def test_pairs_of_ctas_equal_two_groups(tk, N, h, w, L, k, sym, seg):
    """Pairs of CTAs (one epilogue group) on single, split and host-array calls: odd numbers
    of strips, parts that start on odd strips, both triangles, several segments; against two
    epilogue groups on single CTAs where k allows them, else against the FP32 path."""
    import torch
    X = torch.from_numpy(make_slp_like(N, h, w, seed=N + k)[0])
    Xd, e = X.cuda(), L - 1
    one, two = tk.Handle(), tk.Handle()
    one.set_option("epi_groups", 1)
    for hd in (one, two):
        hd.set_option("segment_k", seg)
    kw = dict(symmetric=sym, embed="never", handle=one)
    got = [tk.knn_scores(Xd, L, k, e, **kw)]
    if sym:
        got.append(tk.knn_scores_host(X, L, k, e, **kw))
        P = 3
        parts = [tk.knn_partial(Xd, L, k, e, p, P, handle=one) for p in range(P)]
        got.append(tk.merge_partials(torch.stack([p[0] for p in parts]),
                                     torch.stack([p[1] for p in parts]), handle=one))
    ref = tk.knn_scores(Xd, L, k, e, symmetric=sym, embed="never", handle=two) if k <= 32 else \
        tk.knn_scores(Xd, L, k, e, precision="fp32", handle=two)
    torch.cuda.synchronize()
    assert one.sync_status() == 0 and two.sync_status() == 0
    for g in got:
        if k <= 32:
            assert all(torch.equal(x.cpu(), y.cpu()) for x, y in zip(g, ref))
        else:
            rel = (g[1].cpu() - ref[1].cpu()).abs() / ref[1].cpu()
            assert rel.max().item() <= 2e-4
            assert all(torch.equal(x.cpu(), y.cpu()) for x, y in zip(g, got[0]))


@pytest.mark.parametrize("N,count", [(125000, 1), (90000, 2)])
def test_fp32_calls_with_too_many_column_lists_equal_exact_rows(tk, N, count):
    """Column-side lists above 32 GB (k = 64): one series goes to both triangles, two go one
    after the other. Small integers, so rows compare exactly, ties included."""
    import torch
    k, e = 64, 3
    X = _integers(N, 4, 200, seed=N)
    Xd = torch.from_numpy(X).cuda()
    got = tk.knn_scores_batched([(Xd, 1, k, e)] * count, precision="fp32", center=False)
    Xi = X.astype(np.int64)
    for t in (0, 1, N // 2, N - 1, 127, 128, 77777):
        d = ((Xi - Xi[t]) ** 2).sum(axis=1)
        d[max(0, t - e):t + e + 1] = np.iinfo(np.int64).max
        order = np.argsort(d, kind="stable")[:k]
        for idx, dist, _ in got:
            assert np.array_equal(idx[t].cpu().numpy(), order)
            assert np.array_equal(dist[t].cpu().numpy(), d[order].astype(np.float32))


@pytest.mark.parametrize("N,D,L", [(301, 1100, 1), (129, 40, 1), (1003, 600, 1), (333, 90, 4),
                                   (4100, 700, 1)])
def test_rows_that_are_trajectories_equal_the_oracle(tk, N, D, L):
    """L = 1 and embedded operands: the operand preparation writes the window sums and clears
    the bounds, for few and many groups per row and ragged blocks, on used workspaces too."""
    import torch
    for seed in (N, N + 1):
        X = _integers(N, D, 3, seed=seed)
        oidx, odist, _ = oracle.knn_scores(X, L, 7, 2)
        Xd = torch.from_numpy(X).cuda()
        for prec in ("split_bf16", "bf16"):
            got = [tk.knn_scores(Xd, L, 7, 2, precision=prec, center=False, embed="always")]
            if L == 1:
                got += tk.knn_scores_batched([(Xd, L, 7, 2)], precision=prec, center=False)
            for idx, dist, _ in got:
                assert np.array_equal(dist.cpu().numpy(), odist.astype(np.float32))
                assert np.array_equal(idx.cpu().numpy(), oidx)
