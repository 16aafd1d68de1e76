// Tensor-core GEMM of libqe: D[M x N] = sum_t A_{pa(t)} . B_{pb(t)}^T over K, on
// tcgen05 (bf16 x bf16 -> fp32 accumulators in TMEM), operands fed by TMA in
// 128-byte-swizzled K-major tiles (MN-major for token-major X).  One kernel serves
// four contractions of the method, selected by the epilogue:
//   Sigma = X X^T                         (Lemma 1; upper tiles + mirror)
//   P = W (I + Sigma_bar)                 (Algorithm 3, "P = W Sigma^norm")
//   R = (P - s (C - z) Sigma_bar) / s + z  (Algorithm 3, "P_hat = What Sigma^norm"), grid steps
//   partial_k = Delta' Sigma_bar[0:b0, block]  (Eq. cd-update-closed-2, the
//                                          dW_{:,1:j} Sigma^norm_{1:j,j} term,
//                                          deferred per column block, split-K)
// fp32 accuracy for the Sigma_bar products comes from splitting an fp32 operand
// into three bf16 planes (hi + mid + lo, 24 significant bits) and summing the
// cross products down to 2^-16 relative order in the same accumulator (planes
// are stacked along rows in one tensor map).
//
// Two CTAs of a cluster (the two SMs of a TPC) work on one 256 x BN tile: each holds 128
// rows of A and half of B's rows in its shared memory, the leader (rank 0) issues the
// MMAs for both (cta_group::2, M = 256), and each keeps its 128 rows of the result in its
// own TMEM.  A CTA per 128 x 256 tile that loads all of B itself is bound by shared memory:
// 48 KB written and 48 KB read per k-step of 512 MMA cycles, 128 bytes a cycle, made 721
// (780 us for 4096 features x 65536 tokens; 745 with the loads left out, and the same with the
// folds left out).  The pair moves 32 KB each way: 568 us on zeros (1936 TFLOP/s), 664 on
// random data (1656 TFLOP/s).  Longer runs on random data meet the power cap: 1405 TFLOP/s over the
// 3.1 ms of 4096 features x 262144 tokens, 1390 over the 160 ms of 59392 x 65536.
//
// Warp roles: warp 0 issues TMA for its CTA's operands, warp 1 of the leader issues the MMAs
// (warp 1 owns the TMEM allocation: two accumulation buffers), the others (16; 8 for BN = 64)
// fold the chunk partial sums into fp32 registers and run the epilogue (warp w reads TMEM
// lanes 32 (w mod 4) .. +31 = output rows, and its share of the columns).  Barriers: `full`
// and `acc_empty` count in the leader (both CTAs' bytes and epilogue warps), `empty` and
// `acc_full` in each CTA (the leader's commits arrive in both).  What limits the pair is the
// round trip of an accumulation buffer (commit, fold, arrivals, next chunk), which has the
// 2048 cycles of the other buffer's chunk: hence the light arrivals (mbar_arrive_cluster).
#include <cudaTypedefs.h>

#include "qe_common.cuh"
#include "qe_internal.h"

namespace qe {

template <int BN>
struct GemmCfg {
    static constexpr int BM = 128;                      // rows per CTA (256 per pair)
    static constexpr int BK = 64;                       // 64 bf16 = one 128-byte swizzle row
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = BN / 2 * BK * 2;     // this CTA's half of B's rows
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = (BN == 256) ? 7 : 8;
    static constexpr int TMEM_COLS = 2 * BN;           // two accumulation buffers
    // A chunk's buffer is free again once both CTAs have folded it, and the MMAs of the next
    // chunk cover only 2048 cycles of that: 16 warps of 64 columns halve the fold's part of it
    // against 8 of 128 (and 576 threads leave them enough registers).
    static constexpr int EPI_WARPS = (BN == 64) ? 8 : 16;
    static constexpr int HALF = BN / (EPI_WARPS / 4);  // columns per epilogue thread
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;   // producer, MMA, epilogue
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
    static_assert(BN == 64 || BN == 128 || BN == 256, "BN");
    static_assert(SMEM_BYTES <= 232448, "smem");
    static_assert(EPI_WARPS * 32 * HALF * 4 <= STAGES * STAGE_BYTES, "epilogue staging fits the ring");
};

// Virtual K steps (k-block x operand-plane product) accumulated in one TMEM
// buffer before the epilogue warps fold it into fp32 registers.  The tensor-core
// accumulator loses up to about one unit in the last place per accumulate, with
// a bias toward zero (measured: ~1e-5 relative after 256 accumulates), so long K
// is summed as short chunks (4 MMA per step -> 16 accumulates per chunk, a
// relative bias of ~1e-6) whose partial sums are added with round-to-nearest
// fp32 on the CUDA cores.  Folding every 8 steps would gain a few percent for twice the
// bias; every 2, the buffers' round trip would no longer fit.
constexpr int kChunkSteps = 4;

// Sigma's tile order.  Only the tiles on or above the diagonal run (the mirror
// writes the rest).  They are taken in groups of kSigmaGroupM consecutive tile
// rows; inside a group the tile row runs fastest, then the tile column, from the
// first column that reaches the group's diagonal.  A wave of CTAs then covers a
// compact patch of tiles: at a given k-step it reads a few hundred kilobytes of
// distinct rows of X, where row-by-row order (one tile row against 152 tile
// columns) read several megabytes per k-step and left the GEMM waiting on DRAM
// for wide layers.
constexpr int kSigmaGroupM = 4;   // tile rows of 256

// Tiles of group gi (tile rows [gi * kSigmaGroupM, ...)), counting from the
// first tile column whose BN columns reach the group's first row.
__host__ __device__ __forceinline__ int64_t sigma_group_tiles(int gi, int mt, int nt, int BN) {
    const int mlo = gi * kSigmaGroupM;
    const int gm = (mt - mlo) < kSigmaGroupM ? (mt - mlo) : kSigmaGroupM;
    const int ns = static_cast<int>((static_cast<int64_t>(mlo) * 256) / BN);
    return static_cast<int64_t>(gm) * (nt - ns);
}

__host__ __device__ __forceinline__ int64_t sigma_tiles(int mt, int nt, int BN) {
    int64_t t = 0;
    for (int gi = 0; gi * kSigmaGroupM < mt; ++gi) t += sigma_group_tiles(gi, mt, nt, BN);
    return t;
}

// Linear tile id -> (tile row, tile column) in the grouped order.
__host__ __device__ __forceinline__ void sigma_tile(int64_t id, int mt, int nt, int BN, int &m, int &n) {
    int gi = 0;
    for (;;) {
        const int64_t t = sigma_group_tiles(gi, mt, nt, BN);
        if (id < t || (gi + 1) * kSigmaGroupM >= mt) break;
        id -= t;
        ++gi;
    }
    const int mlo = gi * kSigmaGroupM;
    const int gm = (mt - mlo) < kSigmaGroupM ? (mt - mlo) : kSigmaGroupM;
    const int ns = static_cast<int>((static_cast<int64_t>(mlo) * 256) / BN);
    m = mlo + static_cast<int>(id % gm);
    n = ns + static_cast<int>(id / gm);
}

__device__ __forceinline__ float load_w(const GemmArgs &g, int64_t r, int64_t c) {
    if (g.w_is_bf16)
        return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(g.W)[r * g.ldw + c]);
    return reinterpret_cast<const float *>(g.W)[r * g.ldw + c];
}

template <int N>
__device__ __forceinline__ void ld_fv(const float *p, float *v) {
    if constexpr (N == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (N == 2) {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x; v[1] = t.y;
    } else {
        v[0] = *p;
    }
}

template <int N>
__device__ __forceinline__ void st_fv(float *p, const float *v) {
    if constexpr (N == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (N == 2) *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    else *p = v[0];
}

// Staging of an epilogue warp's 32 rows x HALF columns in shared memory: row r keeps its
// 4-column pieces permuted by r mod 8, so that the three access patterns of the
// epilogue (a thread writing along its row, the lanes reading across a row, the lanes
// reading 4 columns of 32 rows) each touch all 32 banks evenly without padding.
template <int HALF>
__device__ __forceinline__ float *stg_at(float *stg, int r, int c) {
    return stg + r * HALF + 4 * ((c >> 2) ^ (r & 7)) + (c & 3);
}

// Columns [cl, cl + N) of row p, those at or past `n` left out (zero).
template <int N>
__device__ __forceinline__ void ld_cols(const float *p, int64_t cl, int n, bool vec, float *v) {
    if (vec) {
        ld_fv<N>(p + cl, v);
    } else {
#pragma unroll
        for (int e = 0; e < N; ++e) v[e] = (cl + e < n) ? p[cl + e] : 0.0f;
    }
}
template <int N>
__device__ __forceinline__ void st_cols(float *p, int64_t cl, int n, bool vec, const float *v) {
    if (vec) {
        st_fv<N>(p + cl, v);
    } else {
#pragma unroll
        for (int e = 0; e < N; ++e)
            if (cl + e < n) p[cl + e] = v[e];
    }
}

// Epilogue of one warp: 32 output rows r0 .. r0 + 31, columns [c0, c0 + HALF).  Each
// thread holds one row of the tile, so writing from registers would touch 32 rows per
// warp access; the warp's values go through shared memory (the operand ring is idle
// once the last chunk has been folded) and are then processed row by row with the
// lanes across the columns: every global access is one contiguous piece of a row.
// What bounds it is the latency of the loads a row needs (P, W, codes, the old Sigma),
// so the rows go in batches of kRowBatch whose loads are all issued before the first
// is used.  (Written from the threads' own rows, an accumulating Sigma of 4096 features
// and 2048 tokens took 116 us, about 90 of them in two waves of this epilogue; now 59.
// The residual refresh of a 4096 x 4096 layer: 336 -> 287 us.)  `objacc` collects the fused objective of EPI_RFULL (when requested).
constexpr int kRowBatch = 8;

template <int HALF>
__device__ __forceinline__ void epilogue_rows(const GemmArgs &g, float *stg, int r0, int c0, int lane,
                                              const float (&acc)[HALF], int split, double &objacc) {
    constexpr int VEC = HALF / 32;        // columns per lane
    constexpr int U = kRowBatch;
    const int cl = c0 + VEC * lane, N = g.N;
    float cs[VEC];                        // the B operand's row scaling, undone
#pragma unroll
    for (int e = 0; e < VEC; ++e) cs[e] = (g.colscale && cl + e < N) ? g.colscale[cl + e] * g.ascale : 1.0f;
#pragma unroll
    for (int i = 0; i < HALF; i += 4)
        *reinterpret_cast<float4 *>(stg_at<HALF>(stg, lane, i)) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
    __syncwarp();
    const bool full = cl + VEC <= N;
    auto aligned = [](const void *p, int64_t ld) {   // rows of VEC-float pieces
        return (ld % VEC) == 0 && (reinterpret_cast<uintptr_t>(p) & (4u * VEC - 1u)) == 0;
    };
    const bool vo = full && aligned(g.out, g.ldo);
    if (g.mode == EPI_TRAIL) {
        float *out = g.out + static_cast<int64_t>(split) * g.split_stride;
        const bool vt = vo && (g.split_stride % VEC) == 0;
#pragma unroll 4
        for (int rr = 0; rr < 32; ++rr) {
            if (r0 + rr >= g.M) break;
            float v[VEC];
            ld_fv<VEC>(stg_at<HALF>(stg, rr, VEC * lane), v);
#pragma unroll
            for (int e = 0; e < VEC; ++e) v[e] *= cs[e];
            st_cols<VEC>(out + (r0 + rr) * g.ldo, cl, N, vt, v);
        }
    } else if (g.mode == EPI_PINIT) {
        const bool w16 = g.w_is_bf16 != 0;
        const bool vw = full && (g.ldw % VEC) == 0 &&
                        (reinterpret_cast<uintptr_t>(g.W) & ((w16 ? 2u : 4u) * VEC - 1u)) == 0;
        for (int rb = 0; rb < 32; rb += U) {
            if (r0 + rb >= g.M) break;
            float w[U][VEC];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t r = r0 + rb + u;
                if (r < g.M && vw && w16 && VEC == 2) {   // (BN = 256, the P GEMM's tile)
                    const uint32_t x = *reinterpret_cast<const uint32_t *>(static_cast<const __nv_bfloat16 *>(g.W) + r * g.ldw + cl);
                    w[u][0] = __uint_as_float(x << 16);
                    w[u][1 % VEC] = __uint_as_float(x & 0xffff0000u);
                } else if (r < g.M && vw && !w16) {
                    ld_fv<VEC>(static_cast<const float *>(g.W) + r * g.ldw + cl, w[u]);
                } else {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) w[u][e] = (r < g.M && cl + e < N) ? load_w(g, r, cl + e) : 0.0f;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t r = r0 + rb + u;
                if (r >= g.M) break;
                const float rs = g.rowscale ? g.rowscale[r] : 1.0f;
                float v[VEC];
                ld_fv<VEC>(stg_at<HALF>(stg, rb + u, VEC * lane), v);
#pragma unroll
                for (int e = 0; e < VEC; ++e) v[e] = w[u][e] + v[e] * cs[e] * rs;
                st_cols<VEC>(g.out + r * g.ldo, cl, N, vo, v);
            }
        }
    } else if (g.mode == EPI_SIGMA) {
        // rows (upper triangle), the new values back to the staging for the mirror
        for (int rb = 0; rb < 32; rb += U) {
            if (r0 + rb >= g.M) break;
            float old[U][VEC];
            if (g.accumulate) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t r = r0 + rb + u;
#pragma unroll
                    for (int e = 0; e < VEC; ++e) old[u][e] = 0.0f;
                    if (r < g.M && cl + VEC > r) ld_cols<VEC>(g.out + r * g.ldo, cl, N, vo, old[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t r = r0 + rb + u;
                if (r >= g.M) break;
                float v[VEC];
                float *sp = stg_at<HALF>(stg, rb + u, VEC * lane);
                ld_fv<VEC>(sp, v);
                if (g.accumulate) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) v[e] = old[u][e] + v[e];
                    st_fv<VEC>(sp, v);
                }
                if (cl >= r) {
                    st_cols<VEC>(g.out + r * g.ldo, cl, N, vo, v);
                } else {
#pragma unroll
                    for (int e = 0; e < VEC; ++e)
                        if (cl + e >= r && cl + e < N) g.out[r * g.ldo + cl + e] = v[e];
                }
            }
        }
        __syncwarp();
        // the mirror: lane = row, 4 columns at a time; column c's 32 rows are contiguous in
        // row c of the output
        const int64_t r = r0 + lane;
        if (r < g.M) {
#pragma unroll 4
            for (int c = 0; c < HALF; c += 4) {
                if (c0 + c >= N) break;
                float v[4];
                ld_fv<4>(stg_at<HALF>(stg, lane, c), v);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int64_t cc = c0 + c + e;
                    if (cc < N && cc > r) g.out[cc * g.ldo + r] = v[e];
                }
            }
        }
    } else {   // EPI_RFULL: R in grid-step units
        // per-row grids: (P - s (C - z) Sigma_bar) / s + z = P / s - acc + z; grouped grids
        // (absolute): acc = s_g (C - z_g) Sigma_bar, R = (P - acc) / s_g + z_g (a lane's columns
        // lie in one group)
        const int64_t gc = g.ngroups > 1 ? cl / g.gsize : 0, ng = g.ngroups > 1 ? g.ngroups : 1;
        const bool vp = full && aligned(g.P, g.ldp);
        const bool obj = g.obj_part != nullptr;
        for (int rb = 0; rb < 32; rb += U) {
            if (r0 + rb >= g.M) break;
            float pv[U][VEC], sc[U], zz[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t r = (r0 + rb + u < g.M) ? r0 + rb + u : g.M - 1;
                ld_cols<VEC>(g.P + r * g.ldp, cl, N, vp, pv[u]);
                const int64_t gi = cl < N ? r * ng + gc : r * ng;
                sc[u] = g.scale[gi];
                zz[u] = g.zero[gi];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t r = r0 + rb + u;
                if (r >= g.M) break;
                float v[VEC], o[VEC];
                float *sp = stg_at<HALF>(stg, rb + u, VEC * lane);
                ld_fv<VEC>(sp, v);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    v[e] *= cs[e];
                    o[e] = g.absolute ? __fdiv_rn(pv[u][e] - v[e], sc[u]) + zz[u]
                                      : (__fdiv_rn(pv[u][e], sc[u]) - v[e]) + zz[u];
                }
                st_cols<VEC>(g.out + r * g.ldo, cl, N, vo, o);
                if (obj) st_fv<VEC>(sp, o);   // the fused objective reads R from the staging
            }
        }
        if (!obj) return;
        // (D Sigma)_ij = d_j (R_ij - What_ij) = d_j s (R'_ij - C_ij) with R' = R / s + z:
        // f = sum D_ij d_j s (R'_ij - C_ij), D = W - What (- H).  Thread = row; 32 columns are
        // summed in binary32, their sums in binary64.
        __syncwarp();
        const int64_t r = r0 + lane;
        if (r >= g.M) return;
        const bool al16 = (reinterpret_cast<uintptr_t>(g.W) & 15u) == 0 && (reinterpret_cast<uintptr_t>(g.codes) & 15u) == 0 &&
                          (g.ldc % 16) == 0 && (g.ldw % 8) == 0 &&
                          (g.Hd == nullptr || ((g.ldh % 4) == 0 && (reinterpret_cast<uintptr_t>(g.Hd) & 15u) == 0));
#pragma unroll 1
        for (int q = 0; q < HALF; q += 32) {
            const int cq = c0 + q;
            if (cq >= N) break;
            const int64_t gi = r * ng + (g.ngroups > 1 ? cq / g.gsize : 0);   // the 32 columns lie in one group
            const float sc = g.scale[gi], z = g.zero[gi];
            float part = 0.0f;
            if (al16 && g.w_is_bf16 && cq + 32 <= N) {
                const uint4 *wp = reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(g.W) + r * g.ldw + cq);
                const uint4 *cp = reinterpret_cast<const uint4 *>(g.codes + r * g.ldc + cq);
                const uint4 c0v = cp[0], c1v = cp[1];
                uint4 wv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) wv[u] = wp[u];
                const uint32_t cw[8] = {c0v.x, c0v.y, c0v.z, c0v.w, c1v.x, c1v.y, c1v.z, c1v.w};
#pragma unroll
                for (int k = 0; k < 8; ++k) {   // 4 columns at a time
                    float o[4], dv[4], h[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    ld_fv<4>(stg_at<HALF>(stg, lane, q + 4 * k), o);
                    ld_fv<4>(g.dvec + cq + 4 * k, dv);
                    if (g.Hd) ld_fv<4>(g.Hd + r * g.ldh + cq + 4 * k, h);
                    const uint32_t w01 = (k & 1) ? wv[k >> 1].z : wv[k >> 1].x, w23 = (k & 1) ? wv[k >> 1].w : wv[k >> 1].y;
                    const float w[4] = {__uint_as_float(w01 << 16), __uint_as_float(w01 & 0xffff0000u),
                                        __uint_as_float(w23 << 16), __uint_as_float(w23 & 0xffff0000u)};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float cj = static_cast<float>((cw[k] >> (8 * e)) & 0xffu);
                        const float wh = sc * (cj - z);
                        const float t = (w[e] - wh) - h[e];
                        const float dj = dv[e] > 0.0f ? dv[e] : 0.0f;
                        part += t * dj * (sc * (o[e] - cj));
                    }
                }
            } else {
                // fp32 W or unaligned rows: 8 columns' loads at a time (16-byte ones of fp32 W where
                // its rows allow; one column at a time this took 3/4 of a 768-wide layer's refresh)
                const bool w4 = !g.w_is_bf16 && (g.ldw % 4) == 0 && (reinterpret_cast<uintptr_t>(g.W) & 15u) == 0;
#pragma unroll
                for (int e0 = 0; e0 < 32; e0 += 8) {
                    float w[8], cj[8], dj[8], h[8];
                    if (w4 && cq + e0 + 8 <= N) {
                        const float *wr = static_cast<const float *>(g.W) + r * g.ldw + cq + e0;
                        ld_fv<4>(wr, w);
                        ld_fv<4>(wr + 4, w + 4);
                    } else {
#pragma unroll
                        for (int e = 0; e < 8; ++e) w[e] = cq + e0 + e < N ? load_w(g, r, cq + e0 + e) : 0.0f;
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int c = cq + e0 + e;
                        const bool in = c < N;
                        dj[e] = in ? g.dvec[c] : 0.0f;
                        cj[e] = in ? static_cast<float>(g.codes[r * g.ldc + c]) : 0.0f;
                        h[e] = g.Hd && in ? g.Hd[r * g.ldh + c] : 0.0f;
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float wh = sc * (cj[e] - z);
                        float t = w[e] - wh;
                        if (g.Hd) t -= h[e];
                        if (dj[e] > 0.0f) part += t * dj[e] * (sc * (*stg_at<HALF>(stg, lane, q + e0 + e) - cj[e]));
                    }
                }
            }
            objacc += static_cast<double>(part);
        }
    }
}

template <int BN>
__global__ void __launch_bounds__(GemmCfg<BN>::THREADS, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
              const GemmArgs g) {
    using C = GemmCfg<BN>;
    if (g.gate) {
        after_previous();
        if (*g.gate != g.gate_run) return;   // uniform: the other form of the sweep runs
    }
    extern __shared__ uint8_t smem_raw[];
    const uint32_t pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
    uint8_t *smem = smem_raw + pad;   // the same offset in both CTAs of the pair
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::STAGES * C::STAGE_BYTES);
    uint64_t *empty = full + C::STAGES;
    uint64_t *acc_full = empty + C::STAGES;   // [2]: chunk accumulated in buffer b
    uint64_t *acc_empty = acc_full + 2;       // [2]: buffer b drained by both CTAs' epilogues
    uint64_t *drain = acc_empty + 2;          // every MMA the pair issued has completed
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;
    // The grid's x counts CTAs, two per tile.  Consecutive tiles walk down M, so a
    // wave shares a few B column slices (each read once from DRAM) instead of sweeping all
    // of B.  Sigma: the tiles on or above the diagonal in groups of kSigmaGroupM tile rows
    // (sigma_tile).
    int m0, n0;
    const int tile = static_cast<int>(blockIdx.x >> 1);
    if (g.mode == EPI_SIGMA) {
        int mt_, nt_;
        sigma_tile(tile, static_cast<int>(ceil_div(g.M, 2 * C::BM)), static_cast<int>(ceil_div(g.N, BN)), BN, mt_, nt_);
        m0 = mt_ * 2 * C::BM;
        n0 = nt_ * BN;
    } else {
        m0 = tile * 2 * C::BM;
        n0 = blockIdx.y * BN;
    }
    // Sigma: a tile whose every element lies strictly below the diagonal is
    // produced by the mirror of its transpose (both CTAs leave, before any barrier).
    if (g.mode == EPI_SIGMA && n0 + BN <= m0) return;
    m0 += static_cast<int>(rank) * C::BM;   // this CTA's rows

    const int split = blockIdx.z;
    const int splits = gridDim.z;
    const int kb_lo = g.kb_begin + static_cast<int>((static_cast<long long>(g.kb_count) * split) / splits);
    const int kb_hi =
        g.kb_begin + static_cast<int>((static_cast<long long>(g.kb_count) * (split + 1)) / splits);
    const int nsteps = (kb_hi - kb_lo) * g.n_prod;
    const int nchunks = (nsteps + kChunkSteps - 1) / kChunkSteps;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 2 * C::EPI_WARPS);   // of both CTAs
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tensormap(&ta);
        prefetch_tensormap(&tb);
    }
    if (warp == 1) tmem_alloc(tmem_slot, C::TMEM_COLS);
    __syncwarp();
    tc_fence_before();
    cluster_sync();   // both CTAs' barriers are ready
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    after_previous();   // the set-up above ran while the grid before this one finished
    allow_next();

    // The producer and the MMA warp run their loops as whole warps and elect one lane at the
    // instructions: loop control, stages and descriptors can then live in uniform registers,
    // which TMA and MMA take.
    if (warp == 0) {
        // ---- TMA producer: this CTA's rows of A and half of B's rows ----
        int s = 0, done = 0;
        uint32_t ph = 1u;   // the parity of the stage's release that is waited for
        bool ok = true;
        const int brow = g.b_row0 + n0 + static_cast<int>(rank) * (BN / 2);
        for (int kb = kb_lo; kb < kb_hi && ok; ++kb) {
            for (int t = 0; t < g.n_prod; ++t) {
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(&empty[s], ph, abort_flag));
                if (!ok) break;
                if (elect_one()) {
                    uint8_t *sa = smem + s * C::STAGE_BYTES;
                    const uint32_t bar = cluster_addr(&full[s], 0);
                    if (leader) mbar_arrive_expect_tx(&full[s], 2 * C::STAGE_BYTES);   // both CTAs' bytes
                    if (g.mn_major) {   // token-major X: boxes of 64 features x 64 tokens
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            tma_load_2d_pair(&ta, sa + h * 8192, bar, m0 + 64 * h, kb * C::BK);
                            if (64 * h < BN / 2)
                                tma_load_2d_pair(&tb, sa + C::A_BYTES + h * 8192, bar, brow + 64 * h, kb * C::BK);
                        }
                    } else {
                        tma_load_2d_pair(&ta, sa, bar, kb * C::BK, g.a_row0 + m0 + g.prod_a[t] * g.a_plane_rows);
                        tma_load_2d_pair(&tb, sa + C::A_BYTES, bar, kb * C::BK, brow + g.prod_b[t] * g.b_plane_rows);
                    }
                }
                __syncwarp();
                ++done;
                if (++s == C::STAGES) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        if (!ok) {
            *abort_flag = 1;
            if (lane == 0) set_error(g.err, ERR_TIMEOUT);
        }
        // The leader's commits for the last stages have arrived here before this CTA may
        // leave (they write its barriers); so the stages' loads have landed as well.
        const int last = done > C::STAGES ? done - C::STAGES : 0;
        bool released = true;
        for (int k = last; k < done && released; ++k)
            released = mbar_wait_bounded(&empty[k % C::STAGES], (k / C::STAGES) & 1u, abort_flag);
        // After a wait that gave up, loads may be unconsumed: the leader, where both CTAs'
        // loads count, keeps the pair until the last load into each stage has landed.
        if (!released && leader)
            for (int k = last; k < done; ++k)
                mbar_wait_bounded(&full[k % C::STAGES], (k / C::STAGES) & 1u, nullptr);
    } else if (warp == 1) {
        if (leader) {
            // ---- MMA issuer: chunk c accumulates into TMEM buffer c & 1 ----
            const uint32_t idesc = (g.f16 ? idesc_f16_f32(2 * C::BM, BN) : idesc_bf16_f32(2 * C::BM, BN)) |
                                   (g.mn_major ? kIdescMnMajor : 0u);
            const uint64_t desc0 = g.mn_major ? smem_desc_mn128(smem_u32(smem)) : smem_desc_k128(smem_u32(smem));
            const uint32_t kadv = g.mn_major ? 128u : 2u;   // 16 along K
            int st = 0, s = 0;
            uint32_t ph = 0u;
            bool ok = true;
            for (int c = 0; c < nchunks && ok; ++c) {
                const int buf = c & 1;
                if (c >= 2) {
                    ok = __all_sync(0xffffffffu, mbar_wait_bounded(&acc_empty[buf], ((c >> 1) - 1) & 1u, abort_flag));
                    if (!ok) break;
                }
                tc_fence_after();
                const uint32_t dst = tmem + static_cast<uint32_t>(buf * BN);
                const int st_end = (st + kChunkSteps < nsteps) ? st + kChunkSteps : nsteps;
                for (uint32_t acc = 0u; st < st_end; ++st, acc = 1u) {
                    ok = __all_sync(0xffffffffu, mbar_wait_bounded(&full[s], ph, abort_flag));
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t da = desc0 + static_cast<uint32_t>(s) * (C::STAGE_BYTES >> 4);
                    const uint64_t db = da + (C::A_BYTES >> 4);
                    if (elect_one()) {
                        mma_bf16_ss(dst, da, db, idesc, acc);
#pragma unroll
                        for (int k = 1; k < C::BK / 16; ++k) mma_bf16_ss(dst, da + kadv * k, db + kadv * k, idesc, 1u);
                        mma_commit(&empty[s]);
                    }
                    __syncwarp();
                    if (++s == C::STAGES) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                if (elect_one()) mma_commit(&acc_full[buf]);   // arrives when this chunk's MMAs complete
                __syncwarp();
            }
            if (!ok) {
                *abort_flag = 1;
                if (lane == 0) set_error(g.err, ERR_TIMEOUT);
            }
            // Drain: every MMA issued so far has completed before TMEM is released (on
            // the normal path they have by the time the epilogue folds the last chunk).
            if (elect_one()) mma_commit_own(drain);
            __syncwarp();
            mbar_wait_bounded(drain, 0u, nullptr);
        }
    } else {
        // ---- epilogue warps: fold chunks into fp32 registers, then store ----
        const int quad = warp & 3;                    // TMEM lanes 32*quad .. +31
        const int half = (warp - 2) >> 2;             // columns [half * HALF, + HALF)
        const uint32_t tl = tmem + (static_cast<uint32_t>(quad * 32) << 16) +
                            static_cast<uint32_t>(half * C::HALF);
        const uint32_t drained = cluster_addr(&acc_empty[0], 0);
        float acc[C::HALF];
#pragma unroll
        for (int i = 0; i < C::HALF; ++i) acc[i] = 0.0f;
        bool ok = true;
        for (int c = 0; c < nchunks; ++c) {
            const int buf = c & 1;
            if (!mbar_wait_bounded(&acc_full[buf], (c >> 1) & 1u, abort_flag)) {
                ok = false;
                if (lane == 0) set_error(g.err, ERR_TIMEOUT);
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int q = 0; q < C::HALF / 32; ++q) {
                float v[32];
                tmem_ld_32x32b_x32(tl + static_cast<uint32_t>(buf * BN + q * 32), v);
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[q * 32 + i] += v[i];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(drained + 8u * buf);
        }
        double objacc = 0.0;
        if (ok && *abort_flag == 0) {
            // every MMA has completed (the last chunk was folded), so the operand
            // ring is free: EPI_WARPS x 32 rows x HALF floats fit in it
            float *stg = reinterpret_cast<float *>(smem) + (warp - 2) * 32 * C::HALF;
            epilogue_rows<C::HALF>(g, stg, m0 + quad * 32, n0 + half * C::HALF, lane, acc, split, objacc);
        }
        if (g.obj_part) {   // one fp64 partial per epilogue warp, reduced later in a fixed order
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) objacc += __shfl_xor_sync(0xffffffffu, objacc, o);
            if (lane == 0)
                g.obj_part[(static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x) * C::EPI_WARPS + (warp - 2)] = objacc;
        }
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync();   // neither CTA leaves while the other's copies, commits or arrivals may reach it
    if (warp == 1) tmem_dealloc(tmem, C::TMEM_COLS);
}

// ---- host side ---------------------------------------------------------------
static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

static bool get_encode() {
    if (g_encode) return true;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || fn == nullptr)
        return false;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return true;
}

bool make_tmap_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld,
                    uint32_t box_rows) {
    if (!get_encode()) return false;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0 || ((ld * 2) & 15u) != 0) return false;
    if (rows == 0 || cols == 0 || box_rows == 0 || box_rows > 256) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {ld * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    const CUresult r =
        g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides,
                 box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_tmap_f16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld,
                   uint32_t box_rows) {
    if (!get_encode()) return false;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0 || ((ld * 2) & 15u) != 0) return false;
    if (rows == 0 || cols == 0 || box_rows == 0 || box_rows > 256) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {ld * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    const CUresult r =
        g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(base), dims, strides,
                 box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

template <int BN>
static cudaError_t launch_bn(const CUtensorMap &ta, const CUtensorMap &tb, const GemmArgs &g,
                             int splits, cudaStream_t s) {
    using C = GemmCfg<BN>;
    cudaError_t e = cudaFuncSetAttribute(k_tc_gemm<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    const unsigned nt = static_cast<unsigned>(ceil_div(g.N, BN)), mt = static_cast<unsigned>(ceil_div(g.M, 2 * C::BM));
    dim3 grid(2 * mt, nt, static_cast<unsigned>(splits));
    if (g.mode == EPI_SIGMA) {
        const int64_t tiles = sigma_tiles(static_cast<int>(mt), static_cast<int>(nt), BN);
        if (tiles > 0x3fffffffll) return cudaErrorInvalidValue;
        grid = dim3(static_cast<unsigned>(2 * tiles), 1, static_cast<unsigned>(splits));
    }
    return launch_after(k_tc_gemm<BN>, grid, dim3(C::THREADS), C::SMEM_BYTES, s, 2u, ta, tb, g);
}

cudaError_t launch_tc_gemm(int BN, const CUtensorMap &ta, const CUtensorMap &tb, const GemmArgs &g,
                           int splits, cudaStream_t s) {
    if (g.mn_major && (g.mode != EPI_SIGMA || BN != 256)) return cudaErrorInvalidValue;
    if (g.M <= 0 || g.N <= 0 || splits < 1 || g.n_prod < 1 || g.n_prod > 6)
        return cudaErrorInvalidValue;
    if (g.mode != EPI_SIGMA && ceil_div(g.N, BN) > 65535) return cudaErrorInvalidValue;
    if (splits > 65535) return cudaErrorInvalidValue;
    switch (BN) {
        case 64: return launch_bn<64>(ta, tb, g, splits, s);
        case 128: return launch_bn<128>(ta, tb, g, splits, s);
        case 256: return launch_bn<256>(ta, tb, g, splits, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_sigma_direct(const void *X, bool token_major, int64_t n, int64_t p, int64_t ld, int64_t chunk,
                                int accumulate, GemmArgs g, cudaStream_t s, bool *taken) {
    // a map's boxes are addressed by 32-bit coordinates (one beyond them faults): a map per 2^30 tokens
    const int64_t most = int64_t{1} << 30, span = token_major ? most / chunk * chunk : most;
    const int64_t pass = token_major ? chunk : span;
    *taken = false;
    g.mn_major = token_major ? 1 : 0;
    for (int64_t m0 = 0; m0 < n; m0 += span) {
        const int64_t len = (n - m0) < span ? n - m0 : span;
        const __nv_bfloat16 *base = static_cast<const __nv_bfloat16 *>(X) + (token_major ? m0 * ld : m0);
        CUtensorMap t;   // token-major: columns = features, a box is 64 of them x 64 tokens
        if (token_major ? !make_tmap_bf16(&t, base, len, p, ld, 64) : !make_tmap_bf16(&t, base, p, len, ld, 128))
            return *taken ? cudaErrorInvalidValue : cudaSuccess;
        *taken = true;
        for (int64_t n0 = 0; n0 < len; n0 += pass) {
            g.kb_begin = static_cast<int>(n0 / 64);
            g.kb_count = static_cast<int>(ceil_div((len - n0) < pass ? len - n0 : pass, 64));
            g.accumulate = m0 + n0 > 0 ? 1 : accumulate;
            const cudaError_t e = launch_tc_gemm(256, t, t, g, 1, s);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace qe
