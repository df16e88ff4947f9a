"""Rows beside the edges of the work units that the 75-year workload really takes (units of one
Gram tile on the tensor cores, of two on the CUDA cores) against the oracle."""
import pytest

from parity import check_sampled, structural_rows, tc_unit_bounds
from synth import config_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tiles,tol", [("split_bf16", 1, 2e-4), ("fp32", 2, 1e-5)])
def test_rows_beside_unit_edges(prec, tiles, tol):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_02059_gb300 as tk
    X, _, cfg = config_inputs("euro_75y_46x81")
    L, k, e = cfg["L"], cfg["k"], cfg["exclusion"]
    hd = tk.Handle()
    idx, dist, score = tk.knn_scores(torch.from_numpy(X).cuda(), L, k, e, precision=prec, handle=hd)
    assert hd.sync_status() == 0
    if prec != "fp32":
        assert hd.work_shape()[0] == tiles
    hd.close()
    M = X.shape[0] - L + 1
    rows = structural_rows(M, L, n_random=0, strip_every=M, col_bounds=tc_unit_bounds(M, L, tiles))
    check_sampled(X, L, k, e, rows, idx.cpu().numpy(), dist.cpu().numpy(), score.cpu().numpy(), tol)
