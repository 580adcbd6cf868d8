// umma.cuh -- a BF16 GEMM on the fifth-generation tensor cores (tcgen05) for the surrogate's
// training and batched forward passes:
//     C[M x N] = A[M x K] * B[N x K]^T   (+ bias[n], tanh, BF16 copy of C)
// A and B are BF16 matrices in global memory (row stride lda / ldb elements, a multiple of 8),
// K-major ([M][K], [N][K]) or MN-major ([K][M], [K][N]; then bn is a multiple of 64), C is
// row-major FP32; a split of K over blockIdx.z writes its partial product to its own slice of C.
// One CTA of eight warps computes a 128 x bn tile (bn = N rounded up to a multiple of 16, at most
// 256; wider N takes several tiles):
//   - TMA (cp.async.bulk.tensor, 128-byte swizzle) brings 64-column K slices of the A tile
//     (128 x 64) and the B tile (bn x 64) into a shared-memory ring of four stages (two when bn is
//     above 128), completing on an mbarrier with the transaction byte count;
//   - one thread issues four tcgen05.mma (M 128, N bn, K 16) per slice with the FP32 accumulator
//     in tensor memory, and tcgen05.commit releases the slice's stage (and, after the last
//     slice, the accumulator) through an mbarrier;
//   - the warps read the accumulator with tcgen05.ld and apply the epilogue (store_tile).
// Out-of-range rows and columns of a tile are zero-filled by TMA and not stored.  Every mbarrier
// wait is bounded: on timeout the kernel writes a nonzero code to *err, stops issuing, waits
// (bounded) for the copies and products it started, frees its tensor memory and returns.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "internal.cuh"

namespace rtbte {
namespace umma {

constexpr int kTM = 128;        // tile rows (accumulator lanes)
constexpr int kTK = 64;         // K per stage: 64 BF16 = 128 bytes = one swizzle span
constexpr int kThreads = 256;  // two warps per 32 accumulator rows, 32 of 64 columns each
constexpr int kWaitLimit = 1 << 24;  // polls of an mbarrier before giving up
// MN-major tiles with 128-byte swizzle: blocks of 64 M (or N) elements x kTK K rows; the leading
// byte offset is the distance between such blocks, the stride byte offset the distance between
// 8-row K groups inside one (checked against a host reference)
constexpr uint32_t kMnLbo = kTK * 128, kMnSbo = 1024;

struct Args {
    int M, N, K, bn;
    int ldc, act;
    const float *back;    // [M][ldc] activations a: C = acc (1 - a^2) (the gradient through tanh), or null
    const float *bias;
    float *C;
    __nv_bfloat16 *Cb;
    int *err;
    int polls;            // of an mbarrier before a wait gives up (0: at once)
    int a_mn, b_mn;       // operand stored MN-major (M or N contiguous) instead of K-major
    int k_base;           // first K of this CTA's range (split-K over blockIdx.z: K range k_base + z * K)
    long long c_split;    // element stride of C between split-K slices
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
// true when the phase with `parity` completed within the poll limit (of the current phase and the one
// before it: an older phase is not told from the current one).  The first poll is always made: a limit
// known at run time and tested before it cost a training step 1.3 us of 238.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int polls = kWaitLimit) {
    for (int i = 1;; ++i) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (i >= polls) return false;
    }
}

// 64-bit shared-memory matrix descriptor of a K-major tile with 128-byte swizzle: rows of 128
// bytes, 8-row atoms of 1024 bytes (stride byte offset), version 1, swizzle mode 2.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr, uint32_t lbo = 16u, uint32_t sbo = 1024u) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);         // start address
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;    // leading byte offset
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;    // stride byte offset
    d |= (uint64_t)1 << 46;                         // descriptor version
    d |= (uint64_t)2 << 61;                         // 128-byte swizzle
    return d;
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, M x N; a_mn / b_mn select
// the MN-major (transposed) layout of an operand
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn = 0, int b_mn = 0) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
            dst),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Epilogue of a 128-row accumulator, 64 columns at a time.  A warp reads rows of its quadrant of
// tensor memory (one row a lane), so storing from there would touch 32 cache lines per
// instruction (the input-gradient convolution spent half its 21 us so: 17 us since); the columns pass through a
// shared-memory tile instead and leave as whole rows, sixteen lanes each.
constexpr int kEpiLd = 64 + 4;  // floats per tile row: 16-byte accesses spread over all banks
constexpr int kEpiBytes = kTM * kEpiLd * 4;

// this warp's half of 64 accumulator columns from tmem column c0 (32 of its row) into r
__device__ __forceinline__ void read_acc32(uint32_t tmem, int c0, float *r) {
    const int warp = threadIdx.x >> 5;
    const uint32_t at = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(c0 + 32 * (warp >> 2));
#pragma unroll
    for (int h = 0; h < 32; h += 16) {
        uint32_t u[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
            "[%16];\n"
            : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
              "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
            : "r"(at + (uint32_t)h));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int j = 0; j < 16; ++j) r[h + j] = __uint_as_float(u[j]);
    }
}
__device__ __forceinline__ void put_tile(float *tile, const float *r) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *t = tile + (32 * (warp & 3) + lane) * kEpiLd + 32 * (warp >> 2);
#pragma unroll
    for (int j = 0; j < 32; j += 4) *reinterpret_cast<float4 *>(t + j) = make_float4(r[j], r[j + 1], r[j + 2], r[j + 3]);
}
// columns [col0, col0 + 64) of rows [m0, m0 + 128), clipped to M x N: + bias, tanh, times 1 - back^2,
// FP32 to C and BF16 to Cb (each may be null except C)
__device__ __forceinline__ void store_tile(const float *tile, int m0, int col0, int M, int N, int ldc, const float *bias,
                                           bool act, const float *back, float *C, __nv_bfloat16 *Cb) {
    constexpr int RS = kThreads / 16, NR = kTM / RS, NB = 4;  // a thread's rows are RS apart, all at the same columns
    const int r0 = threadIdx.x >> 4, j = (threadIdx.x & 15) * 4, col = col0 + j;
    if (col >= N) return;
    const int n = min(4, N - col);
    const bool vec = n == 4 && (ldc & 3) == 0;
    const auto acc = [&](int k) { return *reinterpret_cast<const float4 *>(tile + (r0 + k * RS) * kEpiLd + j); };
    const auto put = [&](long long at, const float4 &v) {
        *reinterpret_cast<float4 *>(C + at) = v;
        if (!Cb) return;
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t *>(&h0);
        u.y = *reinterpret_cast<const uint32_t *>(&h1);
        *reinterpret_cast<uint2 *>(Cb + at) = u;
    };
    if (back && vec && !bias && !act) {
        // Four rows' `back` values are requested before the first is stored: C may alias them as far as
        // the compiler knows, so in the loop below each load would wait for the store before it (input
        // gradient of a 64-channel layer at batch 8 of 60 x 60: 16.2 us with one row at a time, 13.4 so).
        for (int k0 = 0; k0 < NR; k0 += NB) {
            float4 h[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const int row = m0 + r0 + (k0 + k) * RS;
                if (row < M) h[k] = *reinterpret_cast<const float4 *>(back + (long long)row * ldc + col);
            }
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const int row = m0 + r0 + (k0 + k) * RS;
                if (row >= M) break;
                const float4 t = acc(k0 + k);
                put((long long)row * ldc + col, make_float4(t.x * (1.f - h[k].x * h[k].x), t.y * (1.f - h[k].y * h[k].y),
                                                            t.z * (1.f - h[k].z * h[k].z), t.w * (1.f - h[k].w * h[k].w)));
            }
        }
        return;
    }
#pragma unroll 1
    for (int k = 0; k < NR; ++k) {
        const int row = m0 + r0 + k * RS;
        if (row >= M) break;
        const float4 t = acc(k);
        float v[4] = {t.x, t.y, t.z, t.w};
        const long long at = (long long)row * ldc + col;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i >= n) break;
            if (bias) v[i] += bias[col + i];
            if (act) v[i] = tanhf(v[i]);
            if (back) {
                const float h = back[at + i];
                v[i] = v[i] * (1.f - h * h);
            }
        }
        if (vec) {
            put(at, make_float4(v[0], v[1], v[2], v[3]));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i >= n) break;
                C[at + i] = v[i];
                if (Cb) Cb[at + i] = __float2bfloat16(v[i]);
            }
        }
    }
}

// NS-stage ring (NS = 2 or 4) of A and B slices; stage s holds A at base + s*a_bytes and B at
// base + NS*a_bytes + s*b_bytes, then the mbarriers full[NS], empty[NS], done and the TMEM slot.
template <int NCOLS, int NS>
__global__ void __launch_bounds__(kThreads) gemm_tc(const __grid_constant__ CUtensorMap tA,
                                                   const __grid_constant__ CUtensorMap tB, Args a) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // 128-byte swizzled tiles sit on 1024-byte boundaries
    const int bn = a.bn;
    const uint32_t a_bytes = kTM * kTK * 2, b_bytes = (uint32_t)bn * kTK * 2;
    uint32_t sA[NS], sB[NS], full[NS], empty[NS];
    const uint32_t bars = base + NS * (a_bytes + b_bytes);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        sA[i] = base + i * a_bytes;
        sB[i] = base + NS * a_bytes + i * b_bytes;
        full[i] = bars + 8 * i;
        empty[i] = bars + 8 * (NS + i);
    }
    const uint32_t done = bars + 16 * NS, tslot = done + 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * kTM, n0 = blockIdx.y * bn;
    const int nk = (a.K + kTK - 1) / kTK;
    const int kb = a.k_base + blockIdx.z * a.K;  // this CTA's first K
    // one stage's copies: a K-major tile is one box {64 K, rows}; an MN-major tile is boxes of
    // {64 M or N, 64 K}, one per 64 rows, kTK * 128 bytes apart
    auto load_stage = [&](int s, int kt) {
        const int k0 = kb + kt * kTK;
        mbar_expect_tx(full[s], a_bytes + b_bytes);
        if (a.a_mn) {
            for (int h = 0; h < kTM / 64; ++h) tma_load_2d(sA[s] + h * (kTK * 128), &tA, m0 + 64 * h, k0, full[s]);
        } else {
            tma_load_2d(sA[s], &tA, k0, m0, full[s]);
        }
        if (a.b_mn) {
            for (int h = 0; h < bn / 64; ++h) tma_load_2d(sB[s] + h * (kTK * 128), &tB, n0 + 64 * h, k0, full[s]);
        } else {
            tma_load_2d(sB[s], &tB, k0, n0, full[s]);
        }
    };

    if (threadIdx.x == 0) {
        for (int i = 0; i < NS; ++i) {
            mbar_init(full[i], 1);
            mbar_init(empty[i], 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {  // tensor memory for the accumulator: NCOLS columns x 128 lanes
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tslot), "r"(NCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem;
    asm volatile("ld.shared.b32 %0, [%1];\n" : "=r"(tmem) : "r"(tslot) : "memory");

    pdl_begin();  // (after the allocation: the next kernel's cannot come between this grid's)
    pdl_wait();
    __shared__ int s_fail;
    if (threadIdx.x == 0) {
        s_fail = 0;
        const uint32_t idesc = idesc_bf16(kTM, bn, a.a_mn, a.b_mn);
        int issued = 0;  // slices whose TMA was started
        int products = 0;  // slices whose copies have landed and whose MMAs were committed
        for (int s = 0; s < NS && s < nk; ++s) {
            load_stage(s, s);
            ++issued;
        }
        bool ok = a.polls > 0;
        for (int kt = 0; kt < nk && ok; ++kt) {
            const int s = kt % NS;
            const uint32_t par = (uint32_t)((kt / NS) & 1);
            if (!(ok = mbar_wait(full[s], par, a.polls))) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
            for (int k16 = 0; k16 < kTK / 16; ++k16) {
                // K step of 16: 32 bytes along a K-major row, or two 8-row K groups of an MN-major block
                const uint64_t da = a.a_mn ? sw128_desc(sA[s] + 2048u * k16, kMnLbo, kMnSbo)
                                           : sw128_desc(sA[s] + 32u * k16);
                const uint64_t db = a.b_mn ? sw128_desc(sB[s] + 2048u * k16, kMnLbo, kMnSbo)
                                           : sw128_desc(sB[s] + 32u * k16);
                const uint32_t acc = (kt > 0 || k16 > 0) ? 1u : 0u;
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                    "l"(da), "l"(db), "r"(idesc), "r"(acc)
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(empty[s])
                         : "memory");
            ++products;
            if (kt + NS < nk) {  // refill this stage once its MMAs have read it
                if (!(ok = mbar_wait(empty[s], par, a.polls))) break;
                load_stage(s, kt + NS);
                ++issued;
            }
        }
        if (ok) {
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(done)
                         : "memory");
        } else {  // give up: record it, let the copies and products already started end before the CTA leaves
            s_fail = 1;
            atomicExch(a.err, 1);
            for (int kt = products; kt < issued; ++kt) mbar_wait(full[kt % NS], (uint32_t)((kt / NS) & 1));
            if (products > 0) mbar_wait(empty[(products - 1) % NS], (uint32_t)(((products - 1) / NS) & 1));
        }
    }
    __syncthreads();
    bool bad = s_fail != 0;
    if (!bad && !mbar_wait(done, 0, a.polls)) {
        bad = true;
        if (lane == 0) atomicExch(a.err, 2);
    }
    if (__syncthreads_or(bad)) {
        if (threadIdx.x == 0 && !s_fail) mbar_wait(done, 0);
    } else {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        // the ring is free: every slice was read before `done`
        float *tile = reinterpret_cast<float *>(smem_raw + (base - raw));
        for (int c0 = 0; c0 < bn; c0 += 64) {
            float r[32];
            if (c0 + 32 * (warp >> 2) < NCOLS) {
                read_acc32(tmem, c0, r);
                put_tile(tile, r);
            }
            __syncthreads();
            // (bn is N rounded up to 16: columns past N hold zeros or the next tile's share and are clipped)
            store_tile(tile, m0, n0 + c0, a.M, min(a.N, n0 + bn), a.ldc, a.bias, a.act != 0, a.back,
                       a.C + (long long)blockIdx.z * a.c_split, a.Cb);
            __syncthreads();
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(NCOLS) : "memory");
}

// ---- periodic 3x3 convolutions of 64 channels as implicit GEMMs ---------------------------------
// The K slices of a convolution's GEMM over (tap, channel) are its taps: a slice of the A operand
// is the 128 points' neighbours of one tap, 128 bytes of channels each.  These kernels gather the
// slices from the activations themselves (cp.async, 16 bytes a thread, eight threads a row, written
// in the 128-byte swizzle that TMA would write) instead of from an im2col matrix nine times their
// size, so a layer reads 3.7 MB instead of writing and reading 33 MB (batch 8 of 60 x 60), and the
// input gradient adds its nine taps in registers instead of through a 66 MB column matrix.  The
// slices, their order and every rounding are those of the GEMMs over im2col columns.  Bound by the
// latency of a slice's round trip (L2 gather, proxy fence, MMA, commit) at six or twelve warps per
// SM; per layer at batch 8 of 60 x 60: forward 98 + 17 -> 11.5 us, input gradient 40 + 21 + 7 ->
// 13.4 us, weight gradient 17 -> 10.5 us (from one launch's end to the next's).
constexpr int kConvC = 64;      // channels in and out
constexpr int kConvStages = 4;  // ring of A (16 KB) and B (8 KB) slices: two CTAs per SM
constexpr int kConvA = kTM * kTK * 2, kConvB = kConvC * kTK * 2;

struct ConvArgs {
    const __nv_bfloat16 *src;  // [P][64] gathered operand
    int P, ny, nx;             // points of the batch, sample grid
    int kchunk;                // weight gradient: points per split
    const float *bias;         // forward
    const float *back;         // input gradient: [P][64] activations a, out = sum (1 - a^2)
    float *out;                // [P][64], or the weight gradient's partials [split][576][64]
    __nv_bfloat16 *outb;       // [P][64] BF16 copy of out
    int *err;
    int polls;                 // of an mbarrier before a wait gives up (0: at once)
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// A point of the batch as (first point of its sample, y, x).
struct Point {
    int b0, y, x;
    __device__ __forceinline__ void set(int p, int ny, int nx) {
        const int per = ny * nx, b = p / per, yx = p - b * per;
        b0 = b * per;
        y = yx / nx;
        x = yx - y * nx;
    }
    // its neighbour across tap (dy + 1) * 3 + dx + 1 (periodic)
    __device__ __forceinline__ int at(int dy, int dx, int ny, int nx) const {
        int ys = y + dy, xs = x + dx;
        ys += ys < 0 ? ny : 0;
        ys -= ys >= ny ? ny : 0;
        xs += xs < 0 ? nx : 0;
        xs -= xs >= nx ? nx : 0;
        return b0 + ys * nx + xs;
    }
};

enum { CONV_FORWARD = 0, CONV_BACK = 1, CONV_WEIGHT = 2 };

// CONV_FORWARD  out[p][n] = tanh(sum_tap sum_c src[p + tap][c] W[tap, c][n] + bias[n]), tB: W^T [64][576]
// CONV_BACK     out[p][c] = (sum_tap sum_n src[p - tap][n] W[tap, c][n]) (1 - a[p][c]^2), tB: W [576][64];
//               each tap's product is rounded to FP32 and the nine are added in tap order
// CONV_WEIGHT   part[z][(tap, c)][n] = sum over the split's points of src[p + tap][c] g[p][n],
//               tB: g [P][64]; both operands MN-major, two taps a tile
// Every barrier wait is bounded; after one that gave up nothing more is issued and *err is set.
template <int MODE>
__global__ void __launch_bounds__(kThreads, 2) conv_tc(const __grid_constant__ CUtensorMap tB, ConvArgs a) {
    extern __shared__ unsigned char smem_raw[];
    constexpr int NS = kConvStages;
    constexpr uint32_t kCols = MODE == CONV_BACK ? 256u : 64u;  // CONV_BACK: four accumulators in turn
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bars = base + NS * (kConvA + kConvB);  // full[NS] (B slices), used[NS] (MMAs done), TMEM slot
    auto sA = [&](int s) { return base + (uint32_t)s * kConvA; };
    auto sB = [&](int s) { return base + NS * kConvA + (uint32_t)s * kConvB; };
    auto full = [&](int s) { return bars + 8u * s; };
    auto used = [&](int s) { return bars + 8u * (NS + s); };
    const uint32_t tslot = bars + 16 * NS;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int m0 = blockIdx.x * kTM;  // first point, or first (tap, channel) row
    const int k0 = MODE == CONV_WEIGHT ? blockIdx.y * a.kchunk : 0;
    const int nk = MODE == CONV_WEIGHT ? a.kchunk / kTK : 9;
    bool bad = false;  // this thread saw a wait give up

    if (tid == 0) {
        for (int i = 0; i < NS; ++i) {
            mbar_init(full(i), 1);
            mbar_init(used(i), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(tslot), "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem;
    asm volatile("ld.shared.b32 %0, [%1];\n" : "=r"(tmem) : "r"(tslot) : "memory");

    pdl_begin();  // (after the allocation: the next kernel's cannot come between this grid's)
    // gather role: chunk c of rows r0 + 32 i; all of a thread's rows have the same row mod 8
    const int c = tid & 7, r0 = tid >> 3;
    const uint32_t gdst = (uint32_t)r0 * 128u + ((uint32_t)(c ^ (r0 & 7)) << 4);
    Point pt[4];  // the tile's points (forward and input gradient)
    if (MODE != CONV_WEIGHT) {
#pragma unroll
        for (int i = 0; i < 4; ++i) pt[i].set(min(m0 + r0 + 32 * i, a.P - 1), a.ny, a.nx);
    }
    // start slice kt's copies into stage s: thread 0 the B slice, every thread its rows of the A slice
    auto load = [&](int s, int kt) {
        if (tid == 0) {
            mbar_expect_tx(full(s), kConvB);
            if (MODE == CONV_FORWARD) tma_load_2d(sB(s), &tB, kt * kTK, 0, full(s));
            if (MODE == CONV_BACK) tma_load_2d(sB(s), &tB, 0, kt * kConvC, full(s));
            if (MODE == CONV_WEIGHT) tma_load_2d(sB(s), &tB, 0, k0 + kt * kTK, full(s));
        }
        if (MODE != CONV_WEIGHT) {
            const int dy = MODE == CONV_BACK ? 1 - kt / 3 : kt / 3 - 1, dx = MODE == CONV_BACK ? 1 - kt % 3 : kt % 3 - 1;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                cp_async16(sA(s) + gdst + 4096u * i, a.src + (long long)pt[i].at(dy, dx, a.ny, a.nx) * kConvC + 8 * c,
                           m0 + r0 + 32 * i < a.P);
        } else {
            const int t0 = m0 / kConvC;  // two taps: blocks of 64 points x 128 bytes
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int p = k0 + kt * kTK + r0 + 32 * i;
                Point q;
                q.set(min(p, a.P - 1), a.ny, a.nx);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int tap = min(t0 + h, 8);  // (rows of a tenth tap are not stored)
                    cp_async16(sA(s) + (uint32_t)h * 8192u + gdst + 4096u * i,
                               a.src + (long long)q.at(tap / 3 - 1, tap % 3 - 1, a.ny, a.nx) * kConvC + 8 * c, p < a.P);
                }
            }
        }
    };
    auto give_up = [&](int code) {
        bad = true;
        atomicExch(a.err, code);
    };
    float sum[32];  // this warp's half of an accumulator row
    auto add_tap = [&](int kt) {
        float v[32];
        read_acc32(tmem, MODE == CONV_BACK ? 64 * (kt & 3) : 0, v);
#pragma unroll
        for (int j = 0; j < 32; ++j) sum[j] = MODE == CONV_BACK && kt > 0 ? sum[j] + v[j] : v[j];
    };

    pdl_wait();
    int loaded = 0;  // slices whose copies were started
    int products = 0;  // (thread 0) slices whose copies have landed and whose MMAs were committed
    for (; loaded < NS - 1 && loaded < nk; ++loaded) {
        load(loaded, loaded);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    for (int i = loaded; i < NS - 1; ++i) asm volatile("cp.async.commit_group;\n" ::: "memory");
    const uint32_t idesc = idesc_bf16(kTM, kConvC, MODE == CONV_WEIGHT, MODE == CONV_WEIGHT);
    if (a.polls <= 0) give_up(3);
    for (int kt = 0; kt < nk; ++kt) {
        const int s = kt % NS;
        // slice kt is the oldest of the NS - 1 groups in flight; its bytes become visible to the
        // tensor core through the proxy fence of the threads that wrote them
        asm volatile("cp.async.wait_group %0;\n" ::"n"(NS - 2) : "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        if (__syncthreads_or(bad)) break;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            if (!mbar_wait(full(s), (uint32_t)((kt / NS) & 1), a.polls)) give_up(3);
            else {
                const uint32_t d = tmem + (MODE == CONV_BACK ? 64u * (kt & 3) : 0u);
#pragma unroll
                for (int k16 = 0; k16 < kTK / 16; ++k16) {
                    const uint64_t da = MODE == CONV_WEIGHT ? sw128_desc(sA(s) + 2048u * k16, kMnLbo, kMnSbo)
                                                            : sw128_desc(sA(s) + 32u * k16);
                    const uint64_t db = MODE == CONV_WEIGHT ? sw128_desc(sB(s) + 2048u * k16, kMnLbo, kMnSbo)
                                                            : sw128_desc(sB(s) + 32u * k16);
                    const uint32_t acc = ((MODE != CONV_BACK && kt > 0) || k16 > 0) ? 1u : 0u;
                    asm volatile(
                        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                        "l"(da), "l"(db), "r"(idesc), "r"(acc)
                        : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                                 used(s))
                             : "memory");
                ++products;
            }
        }
        // the previous slice's MMAs: their stage is free, and (CONV_BACK) their product complete
        if (kt > 0) {
            if (!mbar_wait(used((kt - 1) % NS), (uint32_t)(((kt - 1) / NS) & 1), a.polls)) give_up(4);
            if (MODE == CONV_BACK) {
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                __syncwarp();
                add_tap(kt - 1);
            }
        }
        if (loaded < nk && !bad) {  // into the stage slice kt - 1 used (slice NS - 1: unused so far)
            load(loaded % NS, loaded);
            ++loaded;
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    bool any = __syncthreads_or(bad);
    if (!any) {
        if (!mbar_wait(used((nk - 1) % NS), (uint32_t)(((nk - 1) / NS) & 1), a.polls)) give_up(5);
        any = __syncthreads_or(bad);
    }
    if (any) {  // copies of B slices not waited for yet, and products, end before the CTA leaves
        if (tid == 0) {
            for (int kt = products; kt < loaded; ++kt) mbar_wait(full(kt % NS), (uint32_t)((kt / NS) & 1));
            if (products > 0) mbar_wait(used((products - 1) % NS), (uint32_t)(((products - 1) / NS) & 1));
        }
        __syncthreads();
    } else {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        add_tap(nk - 1);
        float *tile = reinterpret_cast<float *>(smem_raw + (base - smem_u32(smem_raw)));  // the ring is free
        put_tile(tile, sum);
        __syncthreads();
        if (MODE == CONV_WEIGHT)
            store_tile(tile, m0, 0, 9 * kConvC, kConvC, kConvC, nullptr, false, nullptr,
                       a.out + (long long)blockIdx.y * (9 * kConvC) * kConvC, nullptr);
        else
            store_tile(tile, m0, 0, a.P, kConvC, kConvC, a.bias, MODE == CONV_FORWARD,
                       MODE == CONV_BACK ? a.back : nullptr, a.out, a.outb);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols) : "memory");
}

inline size_t conv_smem_bytes() { return 1024 + (size_t)kConvStages * (kConvA + kConvB) + 16 * kConvStages + 16; }

// Stages of the ring: four while they fit beside each other in 128 KB, else two.
inline int stages_for(int bn) { return 4 * ((size_t)(kTM * kTK * 2) + (size_t)bn * kTK * 2) <= 131072 ? 4 : 2; }
// Dynamic shared memory of one CTA: the ring's A and B tiles, barriers, alignment slack.
inline size_t smem_bytes(int bn) {
    const int ns = stages_for(bn);
    return 1024 + (size_t)ns * ((size_t)(kTM * kTK * 2) + (size_t)bn * kTK * 2) + 16 * (size_t)ns + 64;
}

}  // namespace umma
}  // namespace rtbte
