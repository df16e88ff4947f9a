"""Several settings of one record whose candidate lists are too large for one sweep, by the
bound on them or for want of memory: several sweeps, the same results. Small integers without
centring, so that they compare bitwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
N, D, K = 27394, 32, 20


@pytest.fixture(scope="module")
def tk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_02059_gb300 as m
    return m


def _integers(seed):
    import torch
    return torch.from_numpy(
        np.random.default_rng(seed).integers(0, 41, (N, D)).astype(np.float32)).cuda()


def _equal(a, b):
    return all(x.equal(y) for p, q in zip(a, b) for x, y in zip(p, q))


def test_settings_without_memory_for_one_sweep(tk):
    import torch
    X, settings = _integers(1), [(L, K, L - 1) for L in (5, 2, 4, 3)]
    one = tk.Handle()
    ref = tk.knn_scores_multi(X, settings, center=False, handle=one)
    assert one.sync_status() == 0
    one.close()
    hd = tk.Handle()
    torch.cuda.empty_cache()
    # one sweep takes 14 GB
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (6 << 30), dtype=torch.uint8, device="cuda")
    try:
        for _ in range(2):
            got = tk.knn_scores_multi(X, settings, center=False, handle=hd)
            assert hd.sync_status() == 0 and _equal(got, ref)
        torch.cuda._sleep(int(1e9))
        ev = torch.cuda.Event()
        ev.record()
        tk.knn_scores_multi(X, settings, center=False, handle=hd)
        assert not ev.query()  # the sweeps' plans are kept: nothing waits for the device
        torch.cuda.synchronize()
    finally:
        del fill
        torch.cuda.empty_cache()
        hd.close()


def test_settings_beyond_the_bound_of_the_lists(tk):
    """Twelve settings: 44 GB of lists in one sweep."""
    import torch
    X, settings = _integers(2), [(1 + q % 5, K, q) for q in range(12)]
    hd = tk.Handle()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    got = tk.knn_scores_multi(X, settings, center=False, handle=hd)
    assert hd.sync_status() == 0
    taken = before - torch.cuda.mem_get_info()[0]
    assert taken <= 1.125 * 32e9 + 1e9
    for g, (L, k, e) in zip(got, settings):
        assert _equal([g], [tk.knn_scores(X, L, k, e, center=False, embed="never")])
    hd.close()
