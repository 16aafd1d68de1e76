"""Performance cases: the calls a user of the library makes, at the sizes they make them.

A case is a dict of plain values; ``prepare`` builds what a calling program holds before the
call, ``run`` is one pass through the public entry points (``paper_2309_01885_gb300.qe``),
``work`` the bytes and flops the pass cannot do without, ``exact`` the same results in binary64
with plain torch.  The layers are synthetic (``paper_2309_01885_gb300/inputs.py`` describes the
distributions): W ~ N(0, 0.02^2), X ~ N(0, 1) with a fraction of heavy channels.
"""
from __future__ import annotations

import math

import torch

from paper_2309_01885_gb300 import inputs, qe

GROUP = 256          # columns per group of the grouped-grid cases
BLOCK = 256          # columns per block of the binary64 reference
POWER_ITERS = 64     # the library's default power-method steps for lambda_max


def listed():
    return [
        # Sigma of a LLaMA-7B attention projection from the whole calibration set (128 sequences
        # of 2048 tokens), activations collected feature-major in bf16: the largest Gram matrix
        # product a 7B model asks for at this width.
        dict(name="sigma_proj", kind="sigma", p=4096, n=262144, seqs=1, dtype="bf16", layout="feature"),
        # The calibration loop of a running model: eight sequences of 2048 tokens, token-major as
        # the model emits them, each added to Sigma as it comes.
        dict(name="sigma_tokens", kind="sigma", p=4096, n=2048, seqs=8, dtype="bf16", layout="token"),
        # fp32 activations of an OPT-125m-sized layer (two sequences of 2048 tokens).
        dict(name="sigma_fp32", kind="sigma", p=768, n=4096, seqs=1, dtype="f32", layout="feature"),
        # The smallest layer, where launches and latency count: OPT-125m-sized, fp32 weights, the
        # plain call (no caller workspace).
        dict(name="layer_opt125m", kind="layer", q=768, p=768, n=4096, dtype="f32", bits=4, iters=5, group=0,
             workspace=False),
        # LLaMA-7B attention projection, 3 bits, 20 sweeps, the caller's workspace kept over layers.
        dict(name="layer_proj", kind="layer", q=4096, p=4096, n=262144, dtype="bf16", bits=3, iters=20, group=0,
             workspace=True),
        # LLaMA-7B MLP up projection: many rows over a Sigma that fits L2.
        dict(name="layer_up", kind="layer", q=11008, p=4096, n=262144, dtype="bf16", bits=4, iters=20, group=0,
             workspace=True),
        # LLaMA-7B MLP down projection: a Sigma wider than L2.
        dict(name="layer_down", kind="layer", q=4096, p=11008, n=262144, dtype="bf16", bits=4, iters=20, group=0,
             workspace=True),
        # Falcon-180B QKV projection: the largest layer of the list.
        dict(name="layer_qkv", kind="layer", q=15360, p=14848, n=65536, dtype="bf16", bits=3, iters=10, group=0,
             workspace=True),
        # A layer whose sizes fit no tile (2-bit codes, fp32 weights).
        dict(name="layer_ragged", kind="layer", q=1531, p=2050, n=16384, dtype="f32", bits=2, iters=10, group=0,
             workspace=False),
        # Grouped grids (one scale and zero-point per row and 256 columns).
        dict(name="layer_grouped", kind="layer", q=4096, p=4096, n=262144, dtype="bf16", bits=4, iters=20,
             group=GROUP, workspace=True),
        # The outlier-aware variant: 3 bits, 1% of the entries kept in full precision.
        dict(name="outlier_proj", kind="outlier", q=4096, p=4096, n=262144, dtype="bf16", bits=3, iters=20,
             budget=0.01, workspace=True),
        # Storage of a quantized layer: codes to bit streams and back.
        dict(name="codes_up", kind="codes", q=11008, p=4096, bits=3),
    ]


def _log_int(rng, lo, hi, even):
    """Log-uniform in [lo, hi]; `even`: rounded to a multiple of 64."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(64, v // 64 * 64) if even else v


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "layer", "layer", "layer", "grouped", "outlier", "codes"])
    even = rng.random() < 0.5
    if kind == "sigma":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        layout = rng.choice(["feature", "token"])
        p = _log_int(rng, 192, 2048 if dtype == "f32" else 11008, even)
        n = _log_int(rng, 512, 16384 if dtype == "f32" else 65536, even)
        seqs = rng.choice([1, 1, 2, 4])
        return dict(kind="sigma", p=p, n=max(64, n // seqs), seqs=seqs, dtype=dtype, layout=layout)
    if kind == "codes":
        return dict(kind="codes", q=_log_int(rng, 64, 11008, even), p=_log_int(rng, 64, 11008, even),
                    bits=rng.choice([2, 3, 4, 8]))
    dtype = rng.choice(["bf16", "bf16", "f32"])
    bits = rng.choice([2, 3, 3, 4, 4, 8])
    iters = rng.choice([5, 10, 20])
    workspace = rng.random() < 0.5
    if kind == "outlier":
        q, p = _log_int(rng, 192, 4096, even), _log_int(rng, 192, 4096, even)
        n = min(262144, max(4096, _log_int(rng, 2 * p, 32 * p, True)))
        return dict(kind="outlier", q=q, p=p, n=n, dtype=dtype, bits=min(bits, 4), iters=iters,
                    budget=rng.choice([0.005, 0.01, 0.02]), workspace=workspace)
    grouped = kind == "grouped"
    q = _log_int(rng, 64, 15360, even)
    p = _log_int(rng, 600 if grouped else 192, 8192 if grouped else 11008, even)
    n = min(262144, max(4096, _log_int(rng, 2 * p, 32 * p, True)))
    return dict(kind="layer", q=q, p=p, n=n, dtype=dtype, bits=bits, iters=iters,
                group=rng.choice([GROUP, 2 * GROUP]) if grouped else 0, workspace=workspace)


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000 * int(seed) + stream)
    return g


def _channel_scale(p, seed):
    """0.5% heavy channels (at least one), x30."""
    s = torch.ones(p, 1, device="cuda")
    k = max(1, round(0.005 * p))
    s[torch.randperm(p, generator=_gen(seed, 3), device="cuda")[:k]] = 30.0
    return s


def _activations(case, seed):
    """The activations of each sequence, in the case's type and layout."""
    p, n = case["p"], case["n"]
    g, scale = _gen(seed, 2), _channel_scale(p, seed)
    out = []
    for _ in range(case["seqs"]):
        if case["layout"] == "feature":
            X = torch.empty(p, n, dtype=_dtype(case), device="cuda")
            for c0 in range(0, n, 16384):
                c1 = min(n, c0 + 16384)
                X[:, c0:c1] = torch.randn(p, c1 - c0, generator=g, device="cuda") * scale
        else:
            X = (torch.randn(n, p, generator=g, device="cuda") * scale.t()).to(_dtype(case))
        out.append(X)
    return out


def _calibration_sigma(p, n, seed):
    """Sigma (fp32, exactly symmetric) of n tokens of bf16 activations, by torch: bf16 values are
    exact in TF32, so the products are exact and the sums fp32."""
    g, scale = _gen(seed, 2), _channel_scale(p, seed)
    S = torch.zeros(p, p, device="cuda")
    tf32 = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = True
    try:
        for c0 in range(0, n, 16384):
            c1 = min(n, c0 + 16384)
            X = (torch.randn(p, c1 - c0, generator=g, device="cuda") * scale).to(torch.bfloat16).float()
            S.addmm_(X, X.t())
    finally:
        torch.backends.cuda.matmul.allow_tf32 = tf32
    U = torch.triu(S, 1)
    return U + U.t() + torch.diag(torch.diagonal(S))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sigma":
        return dict(case=case, X=_activations(case, seed))
    if kind == "codes":
        g = _gen(seed, 7)
        codes = torch.randint(0, 1 << case["bits"], (case["q"], case["p"]), generator=g, device="cuda",
                              dtype=torch.uint8)
        return dict(case=case, codes=codes)
    q, p = case["q"], case["p"]
    planted = case.get("budget", 0.0)
    W = inputs.layer_weights(q, p, dtype=_dtype(case), seed=seed, device="cuda", planted_frac=planted)
    st = dict(case=case, W=W, Sigma=_calibration_sigma(p, case["n"], seed), workspace=None)
    if case["workspace"]:
        size = qe.qe_workspace_size(q, p, outlier=kind == "outlier", group_size=case.get("group", 0))
        st["workspace"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sigma":
        layout = qe.QE_FEATURE_MAJOR if case["layout"] == "feature" else qe.QE_TOKEN_MAJOR
        S = None
        for X in state["X"]:
            S = qe.qe_build_sigma(X, layout, Sigma=S, accumulate=S is not None)
        return S
    if kind == "codes":
        packed = qe.qe_pack_codes(state["codes"], case["bits"])
        return packed, qe.qe_unpack_codes(packed, case["p"], case["bits"])
    if kind == "layer":
        return qe.qe_quantize_layer(state["W"], state["Sigma"], case["bits"], case["iters"],
                                    group_size=case["group"], workspace=state["workspace"])
    return qe.qe_quantize_layer_outlier(state["W"], state["Sigma"], case["bits"], case["iters"], _budget(case),
                                        workspace=state["workspace"])


def _budget(case):
    return int(round(case["budget"] * case["q"] * case["p"]))


def work(case):
    kind, p = case["kind"], case["p"]
    if kind == "sigma":
        n = case["n"] * case["seqs"]
        return {"bytes": p * n * (2 if case["dtype"] == "bf16" else 4) + 4 * p * p, "flops": p * (p + 1) * n}
    q = case["q"]
    if kind == "codes":
        packed = q * ((p * case["bits"] + 7) // 8)
        return {"bytes": 2 * q * p + 2 * packed, "flops": 0}
    # The first sweep moves every coordinate, and each move reaches every other column of its row:
    # 2 q p^2.  How many coordinates later sweeps move is up to the data: not counted.  The
    # outlier variant adds lambda_max (a product with Sigma per step) and, per iteration, what each
    # kept entry adds to its row.
    flops = 2 * q * p * p
    out = q * p
    if kind == "outlier":
        flops += 2 * p * p * POWER_ITERS + case["iters"] * 2 * _budget(case) * p
        out += 12 * _budget(case)
    return {"bytes": 4 * p * p + q * p * (2 if case["dtype"] == "bf16" else 4) + out, "flops": flops}


# ---- the same results in binary64 ------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "codes":
        return None
    if kind == "sigma":
        p = case["p"]
        if p * p * case["n"] * case["seqs"] > 5e12:
            return None
        S = torch.zeros(p, p, dtype=torch.float64, device="cuda")
        for X in _activations(case, seed):
            X = X if case["layout"] == "feature" else X.t()
            for c0 in range(0, X.shape[1], 16384):
                Xc = X[:, c0:c0 + 16384].double()
                S.addmm_(Xc, Xc.t())
        return S
    # about 10 s on the GPU at these sizes; beyond them it takes too long
    if case["q"] * case["p"] ** 2 * case["iters"] > 4e12 or case["p"] * case["iters"] > 90000:
        return None
    st = prepare(dict(case, workspace=False), seed)
    return _exact_layer(case, st["W"], st["Sigma"])


def _grid(W, bits, group):
    """(scales in binary64; the grid itself, scale and zero-point of each column, in binary32:
    the zero-point is an integer that the library's binary32 division decides)."""
    q, p = W.shape
    G = group if 0 < group < p else p
    maxq = float((1 << bits) - 1)
    s64, s_col, z_col = [], torch.empty(q, p, device="cuda"), torch.empty(q, p, device="cuda")
    for j0 in range(0, p, G):
        w = W[:, j0:j0 + G]
        lo, hi = w.amin(1).clamp(max=0.0), w.amax(1).clamp(min=0.0)
        s64.append((hi.double() - lo.double()) / maxq)
        s = (hi - lo) / torch.full_like(hi, maxq)
        s_col[:, j0:j0 + G] = s[:, None]
        z_col[:, j0:j0 + G] = torch.round(-lo / s)[:, None]
    return (torch.stack(s64, 1) if len(s64) > 1 else s64[0]), s_col, z_col


def _sweep64(V, Gr, S, d, s_col, z_col, maxq, zf):
    """One cyclic sweep: every column to its nearest level of the closed-form minimiser.  V = What,
    Gr = (What + H - W) Sigma, kept current; V and Gr change in place."""
    q, p = V.shape
    for b0 in range(0, p, BLOCK):
        b1 = min(p, b0 + BLOCK)
        g = Gr[:, b0:b1].t().contiguous()          # block x q: a column is one contiguous row
        v = V[:, b0:b1].t().contiguous()
        v0 = v.clone()
        s, z = s_col[:, b0:b1].t().contiguous(), z_col[:, b0:b1].t().contiguous()
        Sb = S[b0:b1, b0:b1]
        for j in range(b1 - b0):
            t = torch.sub(v[j], g[j] * zf[b0 + j]).div_(s[j]).add_(z[j]).clamp_(0.0, maxq).round_()
            t.sub_(z[j]).mul_(s[j])
            delta = t - v[j]
            v[j] = t
            if j + 1 < b1 - b0:
                g[j + 1:].addr_(Sb[j, j + 1:], delta)
        D = (v - v0).t()
        V[:, b0:b1] = v.t()
        Gr.addmm_(D, S[b0:b1])


def _exact_layer(case, W, Sigma):
    q, p = W.shape
    bits, iters = case["bits"], case["iters"]
    W, S = W.double(), Sigma.double()
    d = torch.diagonal(S).contiguous()
    inv = 1.0 / d
    maxq = float((1 << bits) - 1)
    outlier = case["kind"] == "outlier"
    H = torch.zeros_like(W)

    def keep(T):
        """The entries of largest magnitude, as many as the budget; ties to the smaller index."""
        k = _budget(case)
        flat = T.reshape(-1)
        idx = torch.argsort(flat.abs(), descending=True, stable=True)[:k]
        out = torch.zeros_like(flat)
        out[idx] = flat[idx]
        return out.view(q, p)

    if outlier:
        H = keep(W)
        y = torch.ones(p, dtype=torch.float64, device="cuda") / math.sqrt(p)
        for _ in range(POWER_ITERS):
            y = S @ (y / y.norm())
        y = y / y.norm()
        eta = 1.0 / (2.0 * float(y @ (S @ y)))
    scales, s_col, z_col = _grid((W - H).float(), bits, case.get("group", 0))
    s_col, z_col = s_col.double(), z_col.double()
    V = W - H                                   # the descent starts at What = W (- H)
    Gr = torch.zeros_like(W)
    obj, obj_cd = [], []
    for _ in range(iters):
        _sweep64(V, Gr, S, d, s_col, z_col, maxq, inv)
        if outlier:
            obj_cd.append(torch.sum((V + H - W) * Gr))
            Hn = keep(H - (2.0 * eta) * Gr)
            Gr.addmm_(Hn - H, S)
            H = Hn
        obj.append(torch.sum((V + H - W) * Gr))
    out = dict(codes=None, scales=scales, zeros=None, obj=torch.stack(obj))
    if outlier:
        # the kept values are listed by their indices, so one entry tied at the threshold shifts
        # all that follow: no value is given for them
        out.update(obj_cd=torch.stack(obj_cd), H_val=None, H_idx=None, H_nnz=None)
    return out
