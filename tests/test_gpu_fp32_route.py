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
