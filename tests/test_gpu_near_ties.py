"""Near-tie refinement where binary32 is wrong often: layers made so that the binary32 value of
some columns is a few hundredths of a grid step off, while every exact value is known.

Most columns of such a layer ("plain") have a huge Sigma_kk, so they stay on the level next to
their weight, a quarter step away.  A few ("hubs", at most four per column block) have
Sigma_jj = 1 and large couplings to the plain columns that cancel in pairs: beta~ / s + z is of
order one, a sum of terms of order 2^13 each.  All numbers are dyadic and short, so binary64
(and any exact arithmetic) gives the hubs' values without rounding, and the right codes are
compared without a tolerance.
"""
import numpy as np
import pytest
import torch

from paper_2309_01885_gb300 import qe

pytestmark = pytest.mark.gpu

BITS, ZERO = 3, 3          # levels -3 .. 4 around the zero-point
TIE_EPS = 0.2              # far above the hubs' binary32 error, below the plain columns' quarter


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qe.load()


class HubLayer:
    """W (q x p, zero-point 3; scale 1, or with groups a power of two per group) and Sigma;
    c: the plain columns' codes; t_first, t_later: the hubs' exact beta~ / s + z in the first
    sweep (columns to their left decided, the others still at W) and in every later one.
    outliers: one weight of 32 in a plain column of every row, the entries that H keeps."""

    def __init__(self, q, p, seed, hubs_per_block=3, couple=2 ** 15, group=0, outliers=False):
        rng = np.random.default_rng(seed)
        edge = {k + e for k in range(0, p, group or p) for e in (0, 1)}   # -3 and 4 steps: the range
        hubs = [j for b0 in range(0, p, 256) for j in sorted(rng.choice(np.arange(b0 + 16, min(b0 + 250, p - 2)),
                                                                         hubs_per_block, replace=False))]
        hubs = [j for j in hubs if j < p]
        plain = [k for k in range(p) if k not in edge and k not in hubs]
        c = np.zeros((q, p), np.int64)
        D = np.zeros((q, p))
        c[:, sorted(edge)[0::2]], c[:, sorted(edge)[1::2]] = 0, 7
        sc = 2.0 ** -(np.arange(p) // (group or p) % 3)
        S = np.zeros((p, p))
        np.fill_diagonal(S, 2.0 ** 40)
        for a, b in zip(plain[0::2], plain[1::2]):
            c[:, a] = c[:, b] = rng.integers(1, 7, q)
            D[:, a] = D[:, b] = np.where(rng.random(q) < 0.5, 0.25, -0.25)
        for k in plain[len(plain) // 2 * 2:]:
            c[:, k] = rng.integers(1, 7, q)
        for j in hubs:
            S[j, j] = 1.0
            for n, (a, b) in enumerate(zip(plain[0::2], plain[1::2])):
                if a < j < b:
                    continue
                if n % 8 == 7:                                    # small couplings: the low bits
                    x = rng.integers(-2 ** 21, 2 ** 21) * 2.0 ** -24
                    y = 0.0
                else:                                             # a pair that nearly cancels
                    x = rng.integers(couple * 256, couple * 512) * 2.0 ** -9
                    y = -x + rng.integers(-2 ** 9, 2 ** 9) * 2.0 ** -9
                S[a, j] = S[j, a] = x * sc[j] / sc[a]
                S[b, j] = S[j, b] = y * sc[j] / sc[b]
        if outliers:
            pair = rng.integers(0, len(plain) // 2, q)            # (its other column on its level)
            self.out_cols = np.array(plain)[2 * pair]
            c[np.arange(q), self.out_cols] = ZERO
            D[np.arange(q), self.out_cols] = D[np.arange(q), np.array(plain)[2 * pair + 1]] = 0.0
        W = ((c - ZERO) + D) * sc
        W[:, hubs] = 0.0
        if outliers:
            W[np.arange(q), self.out_cols] = 32.0
        assert np.array_equal(S, S.astype(np.float32))
        self.W, self.S, self.hubs, self.c = W, S, np.array(hubs), c
        self.M = S[:, hubs] * sc[:, None] / sc[hubs] * (1 - np.eye(p)[:, hubs])   # couplings in grid steps
        left = np.tri(p, p, -1).T[:, hubs]                        # k < j
        self.t_first, self.t_later = ZERO + D @ (self.M * left), ZERO + D @ self.M

    def device(self, dtype=torch.bfloat16):
        W = torch.tensor(self.W, dtype=torch.float32, device="cuda").to(dtype)
        assert torch.equal(W.double().cpu(), torch.tensor(self.W))
        return W, torch.tensor(self.S, dtype=torch.float32, device="cuda")

    def codes(self, t):
        out = self.c.copy()
        out[:, self.hubs] = np.clip(np.rint(t), 0, 2 ** BITS - 1)
        return out.astype(np.uint8)

    def check(self, sweeps):
        for n, got in enumerate(sweeps.cpu().numpy()):
            want = self.codes(self.t_first if n == 0 else self.t_later)
            bad = np.argwhere(got != want)
            assert bad.size == 0, (n, len(bad), bad[:4].tolist())


@pytest.mark.parametrize("q,p,group", [(6144, 512, 0), (6144, 509, 0), (6144, 512, 256)])
def test_dense_sweeps_decide_wrong_rows_again(q, p, group):
    """Dense sweeps: rows whose binary32 decision is wrong decide again from the block's start.
    With more wrong rows than CTAs some CTA takes two and more of them, one after another: each
    has to be found by every thread of the CTA before the first warp replaces its codes."""
    L = HubLayer(q, p, 5, group=group)
    W, S = L.device()
    rough = qe.qe_quantize_layer(W, S, BITS, 2, record_sweeps=True, dense_sweeps=2, tie_eps=-1.0, group_size=group)
    wrong = (rough["sweep_codes"][1].cpu().numpy() != L.codes(L.t_later))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = qe.qe_quantize_layer(W, S, BITS, 4, record_sweeps=True, dense_sweeps=4, tie_eps=TIE_EPS,
                               group_size=group)
    assert qe.qe_sync_status() == qe.QE_OK
    assert int(wrong[:, :256].sum()) > sms or group, int(wrong[:, :256].sum())
    assert wrong.any()
    L.check(out["sweep_codes"])


@pytest.mark.parametrize("q,p,group,dtype", [(6144, 512, 0, torch.bfloat16), (600, 1024, 0, torch.bfloat16),
                                             (600, 1021, 0, torch.bfloat16), (600, 512, 0, torch.float32),
                                             (600, 1024, 256, torch.bfloat16), (2500, 512, 256, torch.float32)])
def test_first_and_list_sweeps(q, p, group, dtype):
    """The first sweep's check of a CTA with many rows, a few of them wrong, and the list
    sweeps' recompute, in lockstep and row by row, with few and many rows per SM, over per-row
    and grouped grids, rows of whole 16-byte pieces and others, bf16 and fp32 weights."""
    L = HubLayer(q, p, 7, group=group)
    W, S = L.device(dtype)
    kw = dict(record_sweeps=True, group_size=group)
    rough = qe.qe_quantize_layer(W, S, BITS, 4, tie_eps=-1.0, **kw)["sweep_codes"].cpu().numpy()
    assert (rough[0] != L.codes(L.t_first)).any() and (rough[2] != L.codes(L.t_later)).any()
    for free in (-1, 0, 1 << 20):
        out = qe.qe_quantize_layer(W, S, BITS, 4, tie_eps=TIE_EPS, free_changes=free, **kw)
        assert qe.qe_sync_status() == qe.QE_OK
        L.check(out["sweep_codes"])


@pytest.mark.parametrize("q,p", [(2500, 1024), (300, 1021)])
def test_outlier_variant(q, p):
    """The same with H: its entries leave the target, in the first sweep exactly, then as the IHT
    steps have moved them (from a run that stops there; the hubs' values then hold within
    binary64's rounding, and those within 1e-9 of a midpoint are left out)."""
    L = HubLayer(q, p, 11, couple=2 ** 12, outliers=True)
    W, S = L.device()
    runs = [qe.qe_quantize_layer_outlier(W, S, BITS, n, q, record_sweeps=True, tie_eps=TIE_EPS) for n in (1, 2, 3)]
    rough = qe.qe_quantize_layer_outlier(W, S, BITS, 1, q, record_sweeps=True, tie_eps=-1.0)["sweep_codes"]
    assert qe.qe_sync_status() == qe.QE_OK
    rows = np.arange(q)
    want = L.codes(L.t_first)
    assert np.array_equal(runs[2]["sweep_codes"][0].cpu().numpy(), want)
    assert (rough[0].cpu().numpy() != want).any()
    for n in (1, 2):
        assert int(runs[n - 1]["H_nnz"].item()) == q
        assert np.array_equal(runs[n - 1]["H_idx"].cpu().numpy(), rows * p + L.out_cols)
        H = runs[n - 1]["H_val"].double().cpu().numpy()
        t = L.t_later + (32.0 - H)[:, None] * L.M[L.out_cols]
        got = runs[2]["sweep_codes"][n].cpu().numpy()
        clear = np.abs(np.abs(t - np.floor(t)) - 0.5) > 1e-9
        assert np.array_equal(got[:, L.hubs][clear], np.clip(np.rint(t), 0, 7)[clear])
        plain = np.delete(got == want, L.hubs, axis=1)
        assert plain.all()


def _two_sweeps(W, S, tie_eps=TIE_EPS):
    W, S = (torch.tensor(x, dtype=torch.float32, device="cuda") for x in (W, S))
    sweeps = qe.qe_quantize_layer(W.bfloat16(), S, BITS, 2, record_sweeps=True, tie_eps=tie_eps)["sweep_codes"]
    assert qe.qe_sync_status() == qe.QE_OK
    return sweeps.cpu().numpy()


def test_recompute_keeps_small_terms_beside_large_ones():
    """The recompute's sum, lane by lane: four terms of +-2^25, then 112 terms of 1 + 2^-20, then
    the large ones back.  The small terms' last bits must outlive the large partial sum: the
    code of column j turns on 1584 units of 2^-20 of a sum of 3584.  (A sum whose low part is
    not folded back into the high one loses 3072 of these units.)  First sweep: the CTA-wide
    recompute; second: the list sweeps'."""
    p, j, u = 4096, 3940, 2.0 ** -20
    k = np.arange(3840)
    sign = np.where(k // 4 % 2 == 0, 1.0, -1.0)          # (lanes cancel each other in the GEMMs' sums)
    x = np.where(k < 128, sign * 2.0 ** 25, np.where(k >= 3712, -sign * 2.0 ** 25, 1 + u))
    S = np.zeros((p, p))
    np.fill_diagonal(S, 2.0 ** 60)
    S[j, j] = 2048.0
    S[:3840, j] = S[j, :3840] = 4 * x
    S[3900, j] = S[j, 3900] = -4 * 2000 * u
    assert x.sum() - 2000 * u == 3584 + 1584 * u
    D = np.array([0.25, -0.25])                          # two rows, mirrored
    W = np.zeros((2, p))
    W[:, :3840] = D[:, None]
    W[:, 3900] = D
    W[:, j] = -D                                         # t = 4.5 + 1584 u / 2048, 1.5 - 1584 u / 2048
    W[:, 4000], W[:, 4001] = -3.0, 4.0
    for codes in _two_sweeps(W, S):
        assert codes[:, j].tolist() == [5, 1]
        assert np.all(codes[:, :3840] == ZERO)


@pytest.mark.parametrize("dj", [13421780.0, 13421788.0, 13421796.0, 13421804.0])
def test_recompute_divides_in_binary64(dj):
    """beta~ / s + z = 2.5 + 2^-24 / Sigma_jj, about 2^-48 above a midpoint whose even side is
    below.  (A binary32 quotient corrected once from its remainder gives 2.5 at these Sigma_jj.)"""
    p, j = 64, 40
    S = np.zeros((p, p))
    np.fill_diagonal(S, 2.0 ** 60)
    S[j, j] = dj
    S[10, j] = S[j, 10] = 2 * dj
    S[11, j] = S[j, 11] = 2.0 ** -22
    W = np.zeros((1, p))                                 # no negative weight: zero-point 0
    W[:, 1] = 7.0
    W[:, 10] = W[:, 11] = 1.25
    W[:, j] = 2.0
    for codes in _two_sweeps(W, S):
        assert codes[0, j] == 3
        assert codes[0, 10] == codes[0, 11] == 1
