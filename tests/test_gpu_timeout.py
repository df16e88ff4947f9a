"""A bounded wait that runs out, on a workspace that earlier calls have used: the units of the
CTA that gave up leave their list counts unwritten, so the merge meets whatever lay there. The
call must report the timeout and nothing else, and the next one must be right again."""
import time

import pytest

from synth import make_slp_like

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_02059_gb300 as m
    return m


def _timeout_then_right(tk, N, h, w, L, k, prec, **options):
    import torch
    X = torch.from_numpy(make_slp_like(N, h, w, seed=N + k)[0]).cuda()
    kw = dict(precision=prec, embed=options.pop("embed", "never"))
    fresh, used = tk.Handle(), tk.Handle()
    for hd in (fresh, used):
        for name, v in options.items():
            hd.set_option(name, v)
    ref = tk.knn_scores(X, L, k, L - 1, handle=fresh, **kw)
    # other shapes first: operands, lists and bounds of theirs fill the workspace
    big = torch.from_numpy(make_slp_like(3000, 40, 50, seed=1)[0]).cuda()
    tk.knn_scores(big, 2, 30, 1, handle=used, **kw)
    tk.knn_scores(big[:, :700].contiguous(), 5, 60, 4, handle=used, **kw)
    assert used.sync_status() == 0
    used.set_option("wait_limit_ms", 100)
    used.set_option("debug_withhold", 1)
    for _ in range(2):
        t0 = time.monotonic()
        tk.knn_scores(X, L, k, L - 1, handle=used, **kw)
        assert used.sync_status() == 5
        # the band pre-pass and the main pass each wait for their own limit, and once
        assert 0.19 < time.monotonic() - t0 < 2.0
    used.set_option("debug_withhold", 0)
    got = tk.knn_scores(X, L, k, L - 1, handle=used, **kw)
    assert used.sync_status() == 0 and fresh.sync_status() == 0
    assert all(torch.equal(a, b) for a, b in zip(got, ref))
    fresh.close()
    used.close()


@pytest.mark.parametrize("prec", ["split_bf16", "bf16"])
@pytest.mark.parametrize("N,h,w,L,k,embed", [(400, 6, 6, 3, 4, "always"), (700, 9, 14, 5, 20, "never"),
                                             (1500, 8, 8, 1, 10, "never")])
def test_timeout_of_single_ctas_on_a_used_workspace(tk, prec, N, h, w, L, k, embed):
    _timeout_then_right(tk, N, h, w, L, k, prec, embed=embed)


@pytest.mark.parametrize("prec", ["split_bf16", "bf16"])
@pytest.mark.parametrize("N,h,w,L,k,seg", [(400, 6, 6, 3, 4, 0), (700, 20, 40, 5, 20, 256),
                                           (1300, 9, 14, 2, 64, 0)])
def test_timeout_of_pairs_of_ctas(tk, prec, N, h, w, L, k, seg):
    """The first CTA of a pair withholds a stage that the second one fills."""
    _timeout_then_right(tk, N, h, w, L, k, prec, epi_groups=1, segment_k=seg)
