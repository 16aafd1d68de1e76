"""Outlier budgets far below one entry per row: most rows keep nothing."""
import numpy as np
import pytest
import torch

from paper_2309_01885_gb300 import inputs, qe
from tests.test_gpu_parity import _outlier_replay

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


@pytest.mark.parametrize("rows", [[0], [699], [350], [0, 0, 699], [3, 4, 300, 698]])
def test_few_kept_entries(rows):
    """Large weights planted in a few rows, with gaps of empty rows before, between and after
    them: those entries are kept, and every iteration is the oracle's."""
    q, p, bits, iters, power_iters = 700, 192, 3, 3, 200
    W = inputs.layer_weights(q, p, dtype=torch.bfloat16, seed=47, device="cuda")
    cols = [7 + 31 * k for k in range(len(rows))]
    for k, (r, c) in enumerate(zip(rows, cols)):
        W[r, c] = 1.0 + k
    X = inputs.calib_inputs(p, 2048, dtype=torch.bfloat16, seed=47, device="cuda", heavy_frac=0.02, heavy_mult=30.0)
    Sg = qe.qe_build_sigma(X)
    out = qe.qe_quantize_layer_outlier(W, Sg, bits, iters, len(rows), power_iters=power_iters, record_sweeps=True)
    assert qe.qe_sync_status() == qe.QE_OK
    assert out["H_idx"].tolist() == sorted(r * p + c for r, c in zip(rows, cols))
    assert int(out["H_nnz"].item()) == len(rows)
    assert _outlier_replay(W, Sg, bits, iters, len(rows), power_iters, False, out) == 0
    assert np.all(np.isfinite(out["obj"].cpu().numpy()))


def test_one_kept_entry_costs_no_more_than_none():
    """A tall narrow layer with a budget of one entry takes no longer than with none (within a
    fifth; the row pointers behind the last kept entry, written by one thread, made it half
    as long again)."""
    q, p = 1 << 18, 32
    W = inputs.layer_weights(q, p, dtype=torch.bfloat16, seed=1, device="cuda")
    W[0, 0] = 1.0
    X = inputs.calib_inputs(p, 2048, dtype=torch.bfloat16, seed=1, device="cuda", heavy_frac=0.01, heavy_mult=30.0)
    Sg = qe.qe_build_sigma(X)
    ws = torch.empty(qe.qe_workspace_size(q, p, outlier=True), dtype=torch.uint8, device="cuda")
    ms = {0: [], 1: []}
    for n in range(6):
        for b in (0, 1):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            qe.qe_quantize_layer_outlier(W, Sg, 3, 10, b, workspace=ws)
            e[1].record()
            torch.cuda.synchronize()
            if n:
                ms[b].append(e[0].elapsed_time(e[1]))
    assert qe.qe_sync_status() == qe.QE_OK
    assert min(ms[1]) < 1.2 * min(ms[0]), ms
