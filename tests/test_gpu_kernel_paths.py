"""Kernel branches at the sizes where they can go wrong: ragged tiles and blocks, unaligned
rows, and the rare paths (near-tie checks, window overflow) made common.  Each is compared
with the fp64 oracle or with another form that must agree bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2309_01885_gb300 import inputs
from paper_2309_01885_gb300 import qe
from tests import parity

pytestmark = pytest.mark.gpu
O = oracle.get()


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


def _layer(q, p, n, seed, dtype=torch.bfloat16):
    W = inputs.layer_weights(q, p, dtype=dtype, seed=seed, device="cuda")
    X = inputs.calib_inputs(p, n, dtype=torch.bfloat16, seed=seed, device="cuda", heavy_frac=0.01, heavy_mult=30.0)
    return W, qe.qe_build_sigma(X)


@pytest.mark.parametrize("q,p,dtype,block", [(40, 331, torch.bfloat16, 0), (40, 512, torch.bfloat16, 0),
                                             (33, 200, torch.float32, 64), (33, 260, torch.bfloat16, 128)])
def test_every_near_tie_checked(q, p, dtype, block):
    """A tie threshold of 0.2 grid steps sends two decisions in five through the near-tie
    checks (the first sweep's check of a whole CTA with rows that go through a block many
    times, the list sweeps' recompute): every code after every sweep is the oracle's."""
    W, Sg = _layer(q, p, 4096, 7, dtype)
    out = qe.qe_quantize_layer(W, Sg, 3, 4, record_sweeps=True, tie_eps=0.2, block_width=block)
    assert qe.qe_sync_status() == qe.QE_OK
    W64, S64 = parity.f64(W), parity.f64(Sg)
    s, z = parity.check_grid(out["scales"], out["zeros"], W64, 3)
    ref = O.alg1(W64, S64, s, z, 3, 4, record=True)
    assert np.array_equal(out["sweep_codes"].cpu().numpy(), ref["sweep_codes"])
    parity.check_obj(out["obj"].cpu().numpy(), ref["obj"])


@pytest.mark.parametrize("q,p,block", [(311, 1003, 0), (311, 1024, 0), (311, 1003, 64), (311, 904, 128),
                                       (2100, 1003, 0), (1, 512, 0)])
def test_free_rows_match_lockstep(q, p, block):
    """Rows on their own from the second list sweep on (windows that outgrow shared memory
    included: 5-bit grids over few tokens change many codes) against rows in lockstep; with
    few and (2100 rows) many rows per SM, whose kernels keep different numbers of changes
    in flight."""
    W, Sg = _layer(q, p, 2048, 11)
    runs = [qe.qe_quantize_layer(W, Sg, 5, 8, record_sweeps=True, free_changes=f, block_width=block)
            for f in (-1, 0, 1 << 20)]
    assert qe.qe_sync_status() == qe.QE_OK
    changes = (runs[0]["sweep_codes"][2] != runs[0]["sweep_codes"][1]).sum(dim=1)
    assert q == 1 or int(changes.max()) > 128   # the windows do overflow
    for r in runs[1:]:
        assert torch.equal(r["sweep_codes"], runs[0]["sweep_codes"])
        assert torch.equal(r["obj"], runs[0]["obj"])


@pytest.mark.parametrize("below,form", [(1 << 40, "lists at once"), (1, "dense throughout"), (0, "in between")])
def test_adaptive_loop_matches_gated_launches(below, form):
    """The adaptive schedule's dense sweeps as a loop on the device (the plain call) against
    the gated launches it enqueues with a record of every sweep and under a stream capture:
    codes, objectives and forms, for a switch at once, never and midway; 40 sweeps, so the
    lists take more than one launch."""
    W, Sg = _layer(150, 700, 4096, 19)
    if below == 0:   # midway: between the changes of two sweeps
        sc = qe.qe_quantize_layer(W, Sg, 3, 6, record_sweeps=True, dense_sweeps=6)["sweep_codes"]
        ch = [int((sc[t] != sc[t - 1]).sum()) for t in range(1, 6)]
        below = (ch[2] + ch[1]) // 2
    kw = dict(switch_below=below, record_forms=True)
    gated = qe.qe_quantize_layer(W, Sg, 3, 40, record_sweeps=True, **kw)
    plain = qe.qe_quantize_layer(W, Sg, 3, 40, **kw)
    ws = torch.empty(qe.qe_workspace_size(150, 700), dtype=torch.uint8, device="cuda")
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=stream):
        captured = qe.qe_quantize_layer(W, Sg, 3, 40, workspace=ws, **kw)
    graph.replay()
    torch.cuda.synchronize()
    assert qe.qe_sync_status() == qe.QE_OK
    forms = gated["sweep_forms"].tolist()
    first_list = forms.index(2) if 2 in forms else 40
    assert {"lists at once": first_list == 2, "dense throughout": first_list >= 3,
            "in between": 2 < first_list < 40}[form]
    for r in (plain, captured):
        assert r["sweep_forms"].tolist() == forms
        assert torch.equal(r["codes"], gated["codes"])
        assert torch.equal(r["obj"], gated["obj"])


@pytest.mark.parametrize("p,n,token_major,ld_extra", [(1, 1, False, 0), (64, 128, False, 0), (65, 1000, True, 0),
                                                      (130, 257, False, 3), (200, 4100, True, 1), (768, 300, True, 4)])
def test_sigma_fp32_split(p, n, token_major, ld_extra):
    """fp32 Sigma over ragged tiles, unaligned rows and every split of the tokens, against
    binary64; accumulation on top of an earlier Sigma; the same bits on a second run.  Every
    sum of n products, split or not, is within n rounding errors of its terms' magnitudes."""
    rows, cols = (n, p) if token_major else (p, n)
    g = torch.Generator(device="cuda").manual_seed(p + n)
    X = torch.randn(rows, cols + ld_extra, generator=g, device="cuda")[:, :cols]
    layout = qe.QE_TOKEN_MAJOR if token_major else qe.QE_FEATURE_MAJOR
    S = qe.qe_build_sigma(X, layout)
    F = (X.t() if token_major else X).double()
    ref, mag = F @ F.t(), F.abs() @ F.abs().t()
    tol = 2.0 ** -24 * (n + 1) * mag
    assert torch.all((S.double() - ref).abs() <= tol)
    assert torch.equal(S, S.t()) and torch.equal(S, qe.qe_build_sigma(X, layout))
    S2 = qe.qe_build_sigma(X, layout, Sigma=S.clone(), accumulate=True)
    assert torch.equal(S2, S + S)


@pytest.mark.parametrize("q,p,bits", [(1, 1, 3), (3, 511, 3), (5, 513, 5), (2, 4096, 1), (3, 4097, 7), (4, 8200, 8), (70000, 33, 2),
                                      (7, 32, 6), (9, 96, 7), (5, 160, 3), (300, 64, 4)])
@pytest.mark.parametrize("extra", [0, 5, 16])
def test_pack_codes_row_pieces(q, p, bits, extra):
    """Rows of every alignment and of more than one piece, against numpy's bit packing."""
    g = torch.Generator(device="cuda").manual_seed(q + p)
    codes = torch.randint(0, 1 << bits, (q, p + extra), generator=g, device="cuda", dtype=torch.uint8)[:, :p]
    packed = qe.qe_pack_codes(codes, bits)
    c = codes.cpu().numpy()
    ref = np.packbits(((c[:, :, None] >> np.arange(bits)) & 1).reshape(q, -1), axis=1, bitorder="little")
    assert np.array_equal(packed.cpu().numpy(), ref)
    assert torch.equal(qe.qe_unpack_codes(packed, p, bits), codes)


@pytest.mark.parametrize("p,n,ld_extra,offset", [(8, 1, 0, 0), (64, 64, 0, 0), (72, 200, 0, 0), (136, 63, 8, 0), (264, 1000, 0, 0),
                                                (520, 129, 16, 8), (131, 300, 0, 0), (264, 300, 0, 3)])
def test_sigma_token_major_as_it_lies(p, n, ld_extra, offset):
    """bf16 token-major X against its feature-major copy (the same products, summed in the
    same order along the tokens: equal bits up to 8192 tokens, where the staged form starts a
    new chunk) over ragged tiles; unaligned rows (odd p, an offset base) take the staged
    form.  Accumulated on an earlier Sigma as well, and through the call that never allocates."""
    g = torch.Generator(device="cuda").manual_seed(p + n)
    Xt = torch.randn(n, p + ld_extra + offset, generator=g, device="cuda").bfloat16()[:, offset:offset + p]
    Xf = torch.zeros(p, (n + 7) // 8 * 8, dtype=torch.bfloat16, device="cuda")[:, :n]
    Xf.copy_(Xt.t())
    S = qe.qe_build_sigma(Xt, qe.QE_TOKEN_MAJOR)
    assert torch.equal(S, qe.qe_build_sigma(Xf))
    assert torch.equal(S, qe.qe_build_sigma_static(Xt, qe.QE_TOKEN_MAJOR))
    assert torch.equal(qe.qe_build_sigma(Xt, qe.QE_TOKEN_MAJOR, Sigma=S.clone(), accumulate=True), S + S)
    ref = Xt.double().t() @ Xt.double()
    assert torch.all((S.double() - ref).abs() <= 1e-5 * torch.sqrt(torch.outer(ref.diagonal(), ref.diagonal())) + 1e-30)


def test_few_rows_per_sm_match_many():
    """The list kernel of layers with few rows per SM against the one for many: the rows of a
    layer of 300 take the same codes as the first 300 rows of one of 2100."""
    W, Sg = _layer(2100, 900, 4096, 23)
    many = qe.qe_quantize_layer(W, Sg, 4, 8, record_sweeps=True)["sweep_codes"][:, :300]
    few = qe.qe_quantize_layer(W[:300], Sg, 4, 8, record_sweeps=True)["sweep_codes"]
    assert qe.qe_sync_status() == qe.QE_OK
    assert torch.equal(few, many)
