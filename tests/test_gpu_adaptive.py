"""The adaptive schedule decides on the device: what its calls promise."""
import time

import pytest
import torch

from paper_2309_01885_gb300 import inputs, qe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


def _layer(q, p, seed):
    W = inputs.layer_weights(q, p, dtype=torch.bfloat16, seed=seed, device="cuda")
    X = inputs.calib_inputs(p, 4096, dtype=torch.bfloat16, seed=seed, device="cuda", heavy_frac=0.01, heavy_mult=30.0)
    return W, qe.qe_build_sigma(X)


def test_adaptive_calls_return_before_the_gpu_is_done():
    """Calls are asynchronous: behind half a second of other work on the stream, four layers
    with dense sweeps throughout are enqueued in a fraction of that time."""
    W, S = _layer(150, 700, 19)
    ws = torch.empty(qe.qe_workspace_size(150, 700), dtype=torch.uint8, device="cuda")
    kw = dict(switch_below=1, workspace=ws)
    ref = qe.qe_quantize_layer(W, S, 3, 6, **kw)["codes"]
    clock = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda._sleep(1 << 20)
    clock[0].record()
    torch.cuda._sleep(1 << 24)
    clock[1].record()
    torch.cuda.synchronize()
    per_ms = (1 << 24) / clock[0].elapsed_time(clock[1])
    torch.cuda._sleep(int(500 * per_ms))
    t0 = time.perf_counter()
    outs = [qe.qe_quantize_layer(W, S, 3, 6, **kw)["codes"] for _ in range(4)]
    host_ms = 1e3 * (time.perf_counter() - t0)
    busy = not torch.cuda.current_stream().query()
    assert qe.qe_sync_status() == qe.QE_OK
    assert busy and host_ms < 250, host_ms
    assert all(torch.equal(c, ref) for c in outs)
