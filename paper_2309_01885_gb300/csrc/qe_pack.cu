// Bit-packed codes: the storage form of a quantized layer (the paper leaves the
// format open; Sec. 2.1 only fixes the codes as integers 0 .. 2^b - 1).  Row i
// is a little-endian bit stream: code j occupies bits [j b, (j + 1) b) of the
// row's bytes, least significant bit first.
//
// Both kernels are HBM-bound by their work (q p bytes of codes, q p b / 8 of stream), so
// what counts is that every global access is wide and whole: a CTA takes up to 4096
// codes of a row; bytes go between global and shared memory in aligned 16-byte pieces
// whatever the row's alignment (the shared copy starts at the same offset modulo 16),
// and a thread converts 16 codes, which are exactly 2 b bytes of the stream.  Rows of
// whole 32-code groups, 16-byte aligned codes and 4-byte aligned streams (every layer whose
// width is a multiple of 32, in the layout of the Python calls) need no shared memory: a
// thread's 32 codes are b whole words, and without barriers every thread's loads are in
// flight at once.
// (11008 x 4096 codes, 3 bits, pack and unpack: 230 us with a byte load per code and
// output word, 66 through shared memory, see below for the direct form.)
#include "../../include/qe.h"
#include "qe_common.cuh"
#include "qe_internal.h"

namespace qe {
namespace {

constexpr int kPackThreads = 256;
constexpr int kPackShared = 32 * kPackThreads;   // 16 codes and a row's offset per thread

// A CTA's threads: x along a row (16 codes each), y over rows: one row of whole warps, or
// several of at most a warp, which then need no barrier of the CTA.  (One narrow row to a CTA
// left most of its threads idle: unpacking 200000 x 16 codes took 73 us with the call, now 26.)
__device__ __forceinline__ void row_sync() {
    if (blockDim.x <= 32) __syncwarp();
    else __syncthreads();
}

// Copies nbytes between global memory and shared memory, whose addresses agree modulo 16.
template <bool TO_SHARED>
__device__ __forceinline__ void copy_bytes(uint8_t *sm, uint8_t *gl, int nbytes) {
    const int head0 = static_cast<int>((16u - (reinterpret_cast<uintptr_t>(gl) & 15u)) & 15u);
    const int head = head0 < nbytes ? head0 : nbytes;
    const int body = (nbytes - head) / 16, tail = nbytes - head - 16 * body;
    for (int k = threadIdx.x; k < body; k += blockDim.x) {
        if (TO_SHARED)
            *reinterpret_cast<uint4 *>(sm + head + 16 * k) = *reinterpret_cast<const uint4 *>(gl + head + 16 * k);
        else
            *reinterpret_cast<uint4 *>(gl + head + 16 * k) = *reinterpret_cast<const uint4 *>(sm + head + 16 * k);
    }
    for (int e = threadIdx.x; e < head + tail; e += blockDim.x) {
        const int k = e < head ? e : nbytes - tail + e - head;
        if (TO_SHARED) sm[k] = gl[k];
        else gl[k] = sm[k];
    }
}

__device__ __forceinline__ uint8_t *same_offset(uint8_t *sm, const void *gl) {
    return sm + (reinterpret_cast<uintptr_t>(gl) & 15u);
}

__global__ void __launch_bounds__(kPackThreads) k_pack_codes(const uint8_t *codes, int64_t q, int64_t p, int64_t ldc,
                                                             int bits, uint8_t *out, int64_t ldo) {
    __shared__ __align__(16) uint8_t s_in[kPackShared], s_out[kPackShared];
    const int64_t step = 16 * static_cast<int64_t>(blockDim.x);
    const int64_t j0 = blockIdx.x * step;
    const int width = static_cast<int>((p - j0) < step ? (p - j0) : step);
    const int row = threadIdx.y * (16 * blockDim.x + 16);   // of the shared arrays
    const uint32_t mask = (1u << bits) - 1u;
    for (int64_t i0 = static_cast<int64_t>(blockIdx.y) * blockDim.y; i0 < q; i0 += static_cast<int64_t>(gridDim.y) * blockDim.y) {
        const int64_t i = i0 + threadIdx.y;
        const int n = i < q ? width : 0;
        uint8_t *src = const_cast<uint8_t *>(codes + i * ldc + j0), *dst = out + i * ldo + j0 / 8 * bits;
        uint8_t *si = same_offset(s_in + row, src), *so = same_offset(s_out + row, dst);
        copy_bytes<true>(si, src, n);
        row_sync();
        const int c0 = 16 * threadIdx.x;
        if (c0 < n) {   // 16 codes -> 2 bits bytes (codes past the row's end are zero)
            uint64_t half[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint64_t w = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int c = c0 + 8 * h + k;
                    const uint32_t v = c < n ? si[c] & mask : 0u;
                    w |= static_cast<uint64_t>(v) << (k * bits);
                }
                half[h] = w;   // 8 codes: `bits` bytes
            }
            uint8_t *o = so + 2 * bits * threadIdx.x;
            for (int k = 0; k < bits; ++k) {
                o[k] = static_cast<uint8_t>(half[0] >> (8 * k));
                o[bits + k] = static_cast<uint8_t>(half[1] >> (8 * k));
            }
        }
        row_sync();
        copy_bytes<false>(so, dst, (n * bits + 7) / 8);
        row_sync();
    }
}

__global__ void __launch_bounds__(kPackThreads) k_unpack_codes(const uint8_t *packed, int64_t q, int64_t p, int64_t ldp,
                                                               int bits, uint8_t *codes, int64_t ldc) {
    __shared__ __align__(16) uint8_t s_in[kPackShared], s_out[kPackShared];
    const int64_t step = 16 * static_cast<int64_t>(blockDim.x);
    const int64_t j0 = blockIdx.x * step;
    const int width = static_cast<int>((p - j0) < step ? (p - j0) : step);
    const int row = threadIdx.y * (16 * blockDim.x + 16);   // of the shared arrays
    const uint32_t mask = (1u << bits) - 1u;
    for (int64_t i0 = static_cast<int64_t>(blockIdx.y) * blockDim.y; i0 < q; i0 += static_cast<int64_t>(gridDim.y) * blockDim.y) {
        const int64_t i = i0 + threadIdx.y;
        const int n = i < q ? width : 0;
        uint8_t *src = const_cast<uint8_t *>(packed + i * ldp + j0 / 8 * bits), *dst = codes + i * ldc + j0;
        uint8_t *si = same_offset(s_in + row, src), *so = same_offset(s_out + row, dst);
        const int nb = (n * bits + 7) / 8;
        copy_bytes<true>(si, src, nb);
        row_sync();
        const int c0 = 16 * threadIdx.x;
        if (c0 < n) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k0 = 2 * bits * static_cast<int>(threadIdx.x) + bits * h;
                uint64_t w = 0;
                for (int k = 0; k < bits; ++k)
                    if (k0 + k < nb) w |= static_cast<uint64_t>(si[k0 + k]) << (8 * k);
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (c0 + 8 * h + k < n) so[c0 + 8 * h + k] = static_cast<uint8_t>((w >> (k * bits)) & mask);
            }
        }
        row_sync();
        copy_bytes<false>(so, dst, n);
        row_sync();
    }
}

// 4 codes in the bytes of x <-> 4 b-bit fields in the low 4 b bits.
template <int B>
__device__ __forceinline__ uint32_t squeeze4(uint32_t x) {
    constexpr uint32_t m = (1u << B) - 1u, m2 = (1u << (2 * B)) - 1u;
    x = (x & (m * 0x00010001u)) | ((x >> (8 - B)) & ((m << B) * 0x00010001u));
    return (x & m2) | ((x >> (16 - 2 * B)) & static_cast<uint32_t>(static_cast<uint64_t>(m2) << (2 * B)));
}
template <int B>
__device__ __forceinline__ uint32_t spread4(uint32_t x) {
    constexpr uint32_t m = (1u << B) - 1u, m2 = (1u << (2 * B)) - 1u;
    x = (x & m2) | (((x >> (2 * B)) & m2) << 16);
    return (x & (m * 0x00010001u)) | ((x << (8 - B)) & (m * 0x01000100u));
}

// The direct form: thread g takes group g mod G of row g / G (G groups of 32 codes a row).
template <int B>
__global__ void __launch_bounds__(256) k_pack_direct(const uint8_t *codes, int64_t total, uint32_t G, int64_t ldc, uint8_t *out,
                                                     int64_t ldo) {
    const int64_t g = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (g >= total) return;
    const int64_t i = g / G;
    const uint32_t k = static_cast<uint32_t>(g - i * G);
    const uint4 *src = reinterpret_cast<const uint4 *>(codes + i * ldc + 32 * static_cast<int64_t>(k));
    const uint4 a = __ldcs(src), b = __ldcs(src + 1);
    const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t w[B];
#pragma unroll
    for (int e = 0; e < B; ++e) w[e] = 0u;
#pragma unroll
    for (int e = 0; e < 8; ++e) {   // field e: bits [4 B e, 4 B (e + 1)) of the group
        const uint32_t f = squeeze4<B>(x[e]);
        constexpr int W = 4 * B;
        const int lo = W * e / 32, sh = W * e % 32;
        w[lo] |= f << sh;
        if (sh + W > 32) w[lo + 1] |= f >> (32 - sh);
    }
    uint32_t *dst = reinterpret_cast<uint32_t *>(out + i * ldo) + B * static_cast<int64_t>(k);
#pragma unroll
    for (int e = 0; e < B; ++e) dst[e] = w[e];
}

template <int B>
__global__ void __launch_bounds__(256) k_unpack_direct(const uint8_t *packed, int64_t total, uint32_t G, int64_t ldp,
                                                       uint8_t *codes, int64_t ldc) {
    const int64_t g = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (g >= total) return;
    const int64_t i = g / G;
    const uint32_t k = static_cast<uint32_t>(g - i * G);
    const uint32_t *src = reinterpret_cast<const uint32_t *>(packed + i * ldp) + B * static_cast<int64_t>(k);
    uint32_t w[B], x[8];
#pragma unroll
    for (int e = 0; e < B; ++e) w[e] = src[e];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        constexpr int W = 4 * B;
        const int lo = W * e / 32, sh = W * e % 32;
        uint32_t f = w[lo] >> sh;
        if (sh + W > 32) f |= w[lo + 1] << (32 - sh);
        x[e] = spread4<B>(f);
    }
    uint4 *dst = reinterpret_cast<uint4 *>(codes + i * ldc + 32 * static_cast<int64_t>(k));
    __stcs(dst, make_uint4(x[0], x[1], x[2], x[3]));
    __stcs(dst + 1, make_uint4(x[4], x[5], x[6], x[7]));
}

template <int B>
void launch_direct(bool pack, const uint8_t *in, int64_t q, int64_t p, int64_t ldi, uint8_t *out, int64_t ldo, cudaStream_t s) {
    const int64_t G = p / 32, total = q * G;
    const unsigned blocks = static_cast<unsigned>(ceil_div(total, 256));
    if (pack) k_pack_direct<B><<<blocks, 256, 0, s>>>(in, total, static_cast<uint32_t>(G), ldi, out, ldo);
    else k_unpack_direct<B><<<blocks, 256, 0, s>>>(in, total, static_cast<uint32_t>(G), ldi, out, ldo);
}

// The direct form when it applies (codes, their leading dimension and the stream aligned).
bool run_direct(bool pack, int bits, const uint8_t *in, int64_t q, int64_t p, int64_t ldi, uint8_t *out, int64_t ldo,
                cudaStream_t s) {
    const uint8_t *codes = pack ? in : out, *stream = pack ? out : in;
    const int64_t ldc = pack ? ldi : ldo, lds = pack ? ldo : ldi;
    if (p % 32 != 0 || ldc % 16 != 0 || lds % 4 != 0 || (reinterpret_cast<uintptr_t>(codes) & 15u) != 0 ||
        (reinterpret_cast<uintptr_t>(stream) & 3u) != 0 || p / 32 > 0xffffffffll || ceil_div(q * (p / 32), 256) > 0x7fffffffll)
        return false;
    switch (bits) {
        case 1: launch_direct<1>(pack, in, q, p, ldi, out, ldo, s); break;
        case 2: launch_direct<2>(pack, in, q, p, ldi, out, ldo, s); break;
        case 3: launch_direct<3>(pack, in, q, p, ldi, out, ldo, s); break;
        case 4: launch_direct<4>(pack, in, q, p, ldi, out, ldo, s); break;
        case 5: launch_direct<5>(pack, in, q, p, ldi, out, ldo, s); break;
        case 6: launch_direct<6>(pack, in, q, p, ldi, out, ldo, s); break;
        case 7: launch_direct<7>(pack, in, q, p, ldi, out, ldo, s); break;
        default: launch_direct<8>(pack, in, q, p, ldi, out, ldo, s); break;
    }
    return true;
}

// A row's threads (16 codes each: whole warps, or a power of two of a warp's lanes), the rows of
// a CTA, and the grid over row pieces and rows.
void pack_grid(int64_t q, int64_t p, dim3 &grid, dim3 &block) {
    int64_t t = ceil_div(p, 16);
    if (t > 32) {
        t = round_up(t, 32) < kPackThreads ? round_up(t, 32) : kPackThreads;
        block = dim3(static_cast<unsigned>(t), 1);
    } else {
        unsigned lanes = 1;
        while (lanes < t) lanes *= 2;
        block = dim3(lanes, kPackThreads / lanes);
    }
    const int64_t rows = ceil_div(q, block.y);
    grid = dim3(static_cast<unsigned>(ceil_div(p, 16 * static_cast<int64_t>(block.x))),
                static_cast<unsigned>(rows < 65535 ? rows : 65535));
}

}  // namespace
}  // namespace qe

using namespace qe;

extern "C" {

qe_status qe_pack_codes(const uint8_t *codes, int64_t q, int64_t p, int64_t ldc, int bits, uint8_t *out,
                        int64_t ldo, qe_stream_t stream) {
    if (!codes || !out || q < 1 || p < 1 || bits < 1 || bits > 8 || ldc < p) return QE_ERR_INVALID_ARG;
    const int64_t nbytes = (p * bits + 7) / 8;
    if (ldo < nbytes) return QE_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (!run_direct(true, bits, codes, q, p, ldc, out, ldo, s)) {
        dim3 grid, block;
        pack_grid(q, p, grid, block);
        k_pack_codes<<<grid, block, 0, s>>>(codes, q, p, ldc, bits, out, ldo);
    }
    if (cudaGetLastError() != cudaSuccess) return QE_ERR_CUDA;
    return QE_OK;
}

qe_status qe_unpack_codes(const uint8_t *packed, int64_t q, int64_t p, int64_t ldp, int bits, uint8_t *codes,
                          int64_t ldc, qe_stream_t stream) {
    if (!packed || !codes || q < 1 || p < 1 || bits < 1 || bits > 8 || ldc < p) return QE_ERR_INVALID_ARG;
    const int64_t nbytes = (p * bits + 7) / 8;
    if (ldp < nbytes) return QE_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (!run_direct(false, bits, packed, q, p, ldp, codes, ldc, s)) {
        dim3 grid, block;
        pack_grid(q, p, grid, block);
        k_unpack_codes<<<grid, block, 0, s>>>(packed, q, p, ldp, bits, codes, ldc);
    }
    if (cudaGetLastError() != cudaSuccess) return QE_ERR_CUDA;
    return QE_OK;
}

}  // extern "C"
