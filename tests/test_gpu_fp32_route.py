"""FP32 calls beside the tensor-core path: plain asynchronous launches on a workspace of their
own, whatever the shape and however many series, that a caller can capture, and that neither
the tensor-core path's options nor its plans and graphs concern."""
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


def _integers(N, D, top, seed):
    import torch
    return torch.from_numpy(
        np.random.default_rng(seed).integers(0, top + 1, (N, D)).astype(np.float32)).cuda()


def _outs(M, k):
    import torch
    return (torch.empty((M, k), dtype=torch.int32, device="cuda"),
            torch.empty((M, k), dtype=torch.float32, device="cuda"),
            torch.empty((M,), dtype=torch.float32, device="cuda"))


def _equal(a, b):
    return all(x.equal(y) for x, y in zip(a, b))


def test_autotune_leaves_fp32_calls_alone(tk):
    X = _integers(1500, 300, 5, seed=1)
    counts = []
    for tune in (0, 1):
        hd = tk.Handle()
        hd.set_option("autotune", tune)
        tk.knn_scores(X, 3, 5, 2, precision="fp32", handle=hd)
        assert hd.sync_status() == 0
        counts.append(hd.launch_count())
        hd.close()
    assert counts[0] == counts[1]


def _captured(hd, call):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    g.replay()
    assert hd.sync_status() == 0


def test_fp32_batched_calls_can_be_captured(tk):
    import torch
    shapes = [(1500, 5, 8), (1301, 3, 20), (1200, 1, 4)]
    Xs = [_integers(N, 40, 5, seed=N) for N, _, _ in shapes]
    series = [(X, L, k, L - 1) for X, (_, L, k) in zip(Xs, shapes)]
    ref = [tk.knn_scores(X, L, k, e, precision="fp32") for X, L, k, e in series]
    outs = [_outs(N - L + 1, k) for N, L, k in shapes]
    hd = tk.Handle()
    kw = dict(precision="fp32", handle=hd, outs=outs)
    tk.knn_scores_batched(series, **kw)
    assert hd.sync_status() == 0
    for o in outs:
        for t in o:
            t.zero_()
    torch.cuda.synchronize()
    _captured(hd, lambda: tk.knn_scores_batched(series, **kw))
    assert all(_equal(o, r) for o, r in zip(outs, ref))
    hd.close()


def _asynchronous(call):
    """Whether `call` returns while work enqueued before it still runs."""
    import torch
    torch.cuda.synchronize()
    torch.cuda._sleep(int(1e9))  # about half a second
    ev = torch.cuda.Event()
    ev.record()
    call()
    running = not ev.query()
    torch.cuda.synchronize()
    return running


def test_fp32_calls_of_changing_shapes_are_asynchronous(tk):
    hd = tk.Handle()
    kw = dict(precision="fp32", handle=hd)
    calls = [(_integers(N, D, 5, seed=N), L, k) for N, D, L, k in
             [(4000, 300, 5, 20), (2000, 300, 3, 10), (3001, 40, 1, 33), (1500, 290, 17, 5)]]
    ref = [tk.knn_scores(X, L, k, **kw) for X, L, k in calls]
    outs = [_outs(X.shape[0] - L + 1, k) for X, L, k in calls]
    for (X, L, k), o, r in zip(calls, outs, ref):
        assert _asynchronous(lambda: tk.knn_scores(X, L, k, out=o, **kw))
        assert hd.sync_status() == 0 and _equal(o, r)
    hd.close()


def test_fp32_calls_of_new_shapes_and_many_series_can_be_captured(tk):
    big = _integers(3000, 100, 5, seed=2)
    hd = tk.Handle()
    kw = dict(precision="fp32", handle=hd)
    tk.knn_scores(big, 3, 30, **kw)  # sizes the workspace
    X = _integers(1700, 60, 5, seed=3)
    ref = tk.knn_scores(X, 4, 12, precision="fp32")
    out = _outs(1697, 12)
    _captured(hd, lambda: tk.knn_scores(X, 4, 12, out=out, **kw))
    assert _equal(out, ref)
    # more series than one launch sequence takes
    Xs = [_integers(60 + b, 60, 5, seed=b) for b in range(70)]
    ref = [tk.knn_scores(x, 2, 3, precision="fp32") for x in Xs]
    outs = [_outs(59 + b, 3) for b in range(70)]
    series = [(x, 2, 3, 1) for x in Xs]
    _captured(hd, lambda: tk.knn_scores_batched(series, outs=outs, **kw))
    assert all(_equal(o, r) for o, r in zip(outs, ref))
    hd.close()


def test_fp32_calls_keep_the_graphs_of_batched_calls(tk):
    hd = tk.Handle()
    series = [(_integers(1500, 40, 5, seed=b), 3, 7, 2) for b in range(3)]
    outs = [_outs(1498, 7) for _ in range(3)]

    def batched():
        tk.knn_scores_batched(series, handle=hd, outs=outs)

    batched()
    tk.knn_scores(series[0][0], 3, 7, precision="fp32", handle=hd)
    assert _asynchronous(batched)  # a first call would capture, and wait
    assert hd.sync_status() == 0
    hd.close()


def _fill_device(leave):
    """All of the device's free memory but `leave` bytes."""
    import torch
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(max(0, free - leave), dtype=torch.uint8, device="cuda")


def test_fp32_calls_without_room_for_lists_stay_asynchronous(tk):
    """About 1 GB of lists and 0.5 GB left: both triangles, without freeing the workspace and
    asking for the memory again on every call."""
    import torch
    X = _integers(27394, 32, 40, seed=4)
    ref = tk.knn_scores(X, 5, 20, precision="fp32", center=False)
    out = _outs(27390, 20)
    hd = tk.Handle()
    kw = dict(precision="fp32", center=False, handle=hd)
    torch.cuda.synchronize()
    fill = _fill_device(500 << 20)
    try:
        tk.knn_scores(X, 5, 20, out=out, **kw)
        assert hd.sync_status() == 0 and _equal(out, ref)
        assert _asynchronous(lambda: tk.knn_scores(X, 5, 20, out=out, **kw))
        assert hd.sync_status() == 0 and _equal(out, ref)
    finally:
        del fill
        torch.cuda.empty_cache()
        hd.close()


def test_fp32_lists_stay_within_their_bound(tk):
    """150,000 days: 45 GB of row-side lists with units of two tiles."""
    import torch
    N, k, e = 150000, 20, 3
    X = _integers(N, 70, 100, seed=5)
    hd = tk.Handle()
    out = _outs(N, k)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    tk.knn_scores(X, 1, k, e, precision="fp32", center=False, handle=hd, out=out)
    assert hd.sync_status() == 0
    assert before - torch.cuda.mem_get_info()[0] <= 1.125 * 32e9 + 1e9
    Xi = X.cpu().numpy().astype(np.int64)
    for t in (0, 1, N // 2, N - 1, 127, 128, 77777):
        d = ((Xi - Xi[t]) ** 2).sum(axis=1)
        d[max(0, t - e):t + e + 1] = np.iinfo(np.int64).max
        order = np.argsort(d, kind="stable")[:k]
        assert np.array_equal(out[0][t].cpu().numpy(), order)
        assert np.array_equal(out[1][t].cpu().numpy(), d[order].astype(np.float32))
    hd.close()
