"""Calls from several host threads, each on its own stream."""
import ctypes
import threading

import pytest
import torch

from paper_2309_01885_gb300 import inputs, qe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


def test_layers_of_different_heights_from_threads():
    """Layers of 2100 and 4200 rows (14 and 28 rows per SM: the same kernels with different
    amounts of shared memory) quantized at once: every call succeeds and gives the codes of a
    call on its own.  The calls go straight to the C ABI with everything allocated before, so
    that the threads spend their time inside the library."""
    p, calls, bits, iters = 64, 4000, 3, 2
    lib = qe.load()
    X = inputs.calib_inputs(p, 2048, dtype=torch.bfloat16, seed=3, device="cuda", heavy_frac=0.01, heavy_mult=30.0)
    S = qe.qe_build_sigma(X)
    jobs = []
    for q in (2100, 4200):
        W = inputs.layer_weights(q, p, dtype=torch.bfloat16, seed=q, device="cuda")
        ref = qe.qe_quantize_layer(W, S, bits, iters)["codes"]
        for _ in range(2):
            ws = torch.empty(qe.qe_workspace_size(q, p), dtype=torch.uint8, device="cuda")
            out = [torch.zeros(q, p, dtype=torch.uint8, device="cuda"), torch.zeros(q, device="cuda"),
                   torch.zeros(q, device="cuda"), torch.zeros(iters, dtype=torch.float64, device="cuda")]
            jobs.append((q, W, ref, ws, out, torch.cuda.Stream()))
    torch.cuda.synchronize()
    bad = {}
    start = threading.Barrier(len(jobs))

    def work(n):
        q, W, _, ws, out, stream = jobs[n]
        o = qe.QEOpts(workspace=ws.data_ptr(), workspace_bytes=ws.numel())
        ptr = [ctypes.c_void_p(x.data_ptr()) for x in (W, S, *out)]
        args = (ptr[0], qe.QE_BF16, q, p, p, ptr[1], bits, iters, ctypes.byref(o), *ptr[2:],
                ctypes.c_void_p(stream.cuda_stream))
        start.wait()
        bad[n] = [st for st in (lib.qe_quantize_layer(*args) for _ in range(calls)) if st != qe.QE_OK]

    threads = [threading.Thread(target=work, args=(n,)) for n in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert qe.qe_sync_status() == qe.QE_OK
    assert all(bad[n] == [] for n in range(len(jobs))), {n: len(b) for n, b in bad.items()}
    for _, _, ref, _, out, _ in jobs:
        assert torch.equal(out[0], ref)
