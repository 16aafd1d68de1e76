"""Weights as a view: rows of every alignment give the result of a contiguous copy."""
import pytest
import torch

from paper_2309_01885_gb300 import inputs, qe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("q,p,offset,extra", [(70, 320, 1, 0), (70, 320, 2, 0), (70, 320, 0, 1), (33, 257, 0, 1), (33, 258, 0, 2),
                                              (300, 511, 3, 4)])
def test_view_of_weights(dtype, q, p, offset, extra):
    full = inputs.layer_weights(q, p + offset + extra, dtype=dtype, seed=9, device="cuda")
    W = full[:, offset:offset + p]
    X = inputs.calib_inputs(p, 2048, dtype=torch.bfloat16, seed=9, device="cuda", heavy_frac=0.02, heavy_mult=30.0)
    S = qe.qe_build_sigma(X)
    a = qe.qe_quantize_layer(W, S, 4, 3, want_norm=True)
    b = qe.qe_quantize_layer(W.contiguous(), S, 4, 3, want_norm=True)
    assert qe.qe_sync_status() == qe.QE_OK
    assert torch.equal(a["codes"], b["codes"]) and torch.equal(a["scales"], b["scales"])
    # the objective kernels' wide and narrow forms add the terms of a row in different orders
    assert torch.allclose(a["obj"], b["obj"], rtol=1e-6) and torch.allclose(a["wx_norm2"], b["wx_norm2"], rtol=1e-6)
