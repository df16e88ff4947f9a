"""Days with NaN values, without centring: a NaN distance is below no bound, so trajectories
that touch no such day keep their neighbours among the others, whatever path evaluates them.
The values are small integers (exact in BF16, their sums in FP32), so those rows compare
exactly, ties included; enough NaN days lie in one strip to overfill a column's record."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_02059_gb300 as m
    return m


def _input(N, D, L, seed):
    X = np.random.default_rng(seed).integers(0, 4, (N, D)).astype(np.float32)
    bad = np.zeros(N, bool)
    bad[20:90] = True
    bad[N // 2::37] = True
    X[bad, seed % D] = np.nan
    M = N - L + 1
    touched = np.array([bad[t:t + L].any() for t in range(M)])
    return X, touched


def _expected(X, touched, L, k, e):
    M = len(touched)
    T = np.stack([X[t:t + L].ravel() for t in range(M)]).astype(np.float64)
    rows = np.nonzero(~touched)[0]
    sq = (T[rows] ** 2).sum(1)
    d = sq[:, None] + sq[None, :] - 2.0 * T[rows] @ T[rows].T
    d[np.abs(rows[:, None] - rows[None, :]) <= e] = np.inf
    order = np.argsort(d, axis=1, kind="stable")[:, :k]
    return rows, rows[order], np.take_along_axis(d, order, axis=1)


def _check(got, want):
    rows, idx, dist = want
    assert np.isfinite(dist).all()
    assert np.array_equal(got[1].cpu().numpy()[rows], dist.astype(np.float32))
    assert np.array_equal(got[0].cpu().numpy()[rows], idx)


@pytest.mark.parametrize("N,D,L,k,e", [(700, 4, 1, 5, 0), (1300, 6, 2, 20, 1), (1300, 6, 2, 40, 1),
                                       (900, 5, 3, 64, 2), (700, 900, 1, 5, 0)])
@pytest.mark.parametrize("prec", ["split_bf16", "bf16", "fp32"])
def test_rows_without_nan_days_keep_their_neighbours(tk, prec, N, D, L, k, e):
    import torch
    X, touched = _input(N, D, L, seed=N + k)
    want = _expected(X, touched, L, k, e)
    Xd = torch.from_numpy(X).cuda()
    kw = dict(precision=prec, center=False)
    for embed in ("never", "always"):
        _check(tk.knn_scores(Xd, L, k, e, embed=embed, **kw), want)
    for got in tk.knn_scores_multi(Xd, [(L, k, e), (L, k, e)], **kw):
        _check(got, want)
    hd = tk.Handle()
    hd.set_option("epi_groups", 1)
    _check(tk.knn_scores(Xd, L, k, e, embed="never", handle=hd, **kw), want)
    assert hd.sync_status() == 0
    hd.close()
