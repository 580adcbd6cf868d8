// small.cu -- RHS evaluations and adaptive attempts of small instances in one launch each.
//
// The launch sequence of a small instance is latency: three launches for an RHS, fourteen for an
// attempted Zonneveld step, each a few microseconds for work that would take one.  Where the
// populations of the single instance of a context fit in shared memory together (f, every mode's
// N and the sub-lattice N), each CTA can own a set of state rows: it holds a copy of all
// populations, runs every work item of its rows -- whatever their part and mode -- and sums them
// itself, so no partial leaves the SM and the only exchange between CTAs is the new populations.
//   - rhs_small: one launch per RHS, populations straight from y, rows straight to ydot;
//   - attempts_small: up to `cap` attempted steps per launch on a cooperative grid of at most half the
//     SMs (see kSmallQuarter): S grid barriers an attempt to exchange populations (the last one the
//     squared errors too, one more where the norm's chunks exceed 8 rows); every CTA runs the
//     controller on its own copy, beside the first stage of the next attempt.  The state the launch
//     started from is kept beside the one it writes, so that a barrier wait that gives up leaves a
//     whole state to go back to.  Where they fit, the CTA's items and entries stay in shared memory
//     for the launch: a barrier's acquire drops L1, so each stage would fetch them from L2 again
//     (with a CTA on every SM, toy 12 x 12 FP64 31.1 -> 30.2 us an attempt, graphene 36 FP32 64 -> 62).
// Items, their lanes and entry order, the order of a row's items, the norm's chunks and the
// controller are those of the launch sequence (collide.cuh, rows.cuh, step.cuh), so both give the
// same results bit for bit.  The 12 x 12 toy model in FP64 (15 174 entries), launch sequence and one
// launch: RHS 12.1 and 4.8 us a call, Bogacki-Shampine attempts 58.8 and 29.2 us.  What is left of an
// attempt is latency (measured with a CTA on every SM: of a stage's 7.5 us 2.4 in the barrier, 2 in
// the items, 2 in the rows' chains of FP64 operations, 0.6 in the populations' copy).  Messages in
// place of the barriers (values with a sequence number beside them, polled by every CTA) took 38 us
// an attempt: the polling of all CTAs on the same few lines costs more than the barrier saves.
#include <algorithm>
#include <cstring>
#include <memory>

#include "collide.cuh"
#include "internal.cuh"
#include "rows.cuh"
#include "step.cuh"

namespace rtbte {

namespace {

// A run of items of one group that a CTA owns: items [a, b) of the plan's own item array, whose
// slots index the CTA's partials, with what the item loop needs of the group.
struct __align__(16) SmallRun {
    const uint32_t *idx;
    const void *W;
    int a, b;
    short part, sb, pb, lg;
    int N_at, pad[3];  // e-ph: the mode's first population in the CTA's N
};
// A state row that a CTA owns: its partials (ph-e before mid, ph-ph from mid; an electron's all
// before mid) and where its value goes in the population copies.
struct __align__(16) SmallRow {
    int row, p0, mid, p1;
    int f, N, P, pad;  // index in f / N / the sub-lattice N, or -1
};
// Rows and their items come in shares, one per SM.  A CTA of the RHS takes one, a CTA of the attempt
// loop `fold` neighbouring ones, whose items are kept together by group.
struct SmallPlan {
    const SmallRun *runs;  // [CTA][max_runs] (empty runs fill up)
    const SmallRow *rows;
    const int2 *off;       // [shares + 1] first row and first partial slot (for a CTA its first item too)
    int shares, fold;
    int max_runs, max_items, max_rows;  // largest CTA's
    int n_f, n_N, n_P;     // populations held: f, all modes' N (mode stride N_q_pad), sub-lattice N
    const int *pp_full;    // [M] phonon of each sub-lattice state
    const int *item_at;    // [items] entries of the items before this one
    int max_entries;       // largest CTA's entries; 0: the attempts' lists are not held
    __device__ __forceinline__ int2 begin() const { return __ldg(off + blockIdx.x * fold); }
    __device__ __forceinline__ int2 end() const { return __ldg(off + min((int)(blockIdx.x + 1) * fold, shares)); }
};

template <class R> struct SmallMem {  // shared memory of a CTA
    R *f, *N, *P;
    R *partials;  // indexed by slot: the CTA's first one's is slot0
    SmallRun *runs;
    // attempts only:
    SmallRow *rows;
    double *y;  // [2][max_rows] state of the owned rows: current and attempted, in turn
    double *K;  // [stages][max_rows]
    ItemRec *items;  // [max_items], if the lists are held
    R *W;            // [max_entries]
    uint32_t *idx;
    __device__ __forceinline__ SmallMem(unsigned char *raw, const SmallPlan &S, int slot0) {
        runs = reinterpret_cast<SmallRun *>(raw);
        f = reinterpret_cast<R *>(runs + S.max_runs);
        N = f + S.n_f;
        P = N + S.n_N;
        partials = P + S.n_P - slot0;
        rows = reinterpret_cast<SmallRow *>(P + S.n_P + S.max_items);
        y = reinterpret_cast<double *>(rows + S.max_rows);
        K = y + 2 * S.max_rows;
        items = reinterpret_cast<ItemRec *>(K + kMaxStages * S.max_rows);
        W = reinterpret_cast<R *>(items + S.max_items);
        idx = reinterpret_cast<uint32_t *>(W + S.max_entries);
    }
};
size_t small_smem(size_t R, const SmallPlan &S, bool attempts) {  // every array a multiple of 16 bytes
    return sizeof(SmallRun) * S.max_runs + R * (size_t)(S.n_f + S.n_N + S.n_P + S.max_items) +
           (attempts ? (sizeof(SmallRow) + sizeof(double) * (2 + kMaxStages)) * S.max_rows : 0) +
           (attempts && S.max_entries > 0 ? sizeof(ItemRec) * S.max_items + (4 + R) * (size_t)S.max_entries : 0);
}

template <class T> __device__ __forceinline__ void copy_in(T *dst, const T *src, int n) {  // 16-byte units
    const int m = n * (int)(sizeof(T) / 16);
    for (int i = threadIdx.x; i < m; i += blockDim.x)
        reinterpret_cast<int4 *>(dst)[i] = __ldg(reinterpret_cast<const int4 *>(src) + i);
}

// Every item of this CTA's rows whose part is in the mask, by `nwarps` warps of which this is
// number `warp`.  Warps take packets in turn across the runs, so short runs do not all fall to the
// first warps.
template <class R, int LOAD>
__device__ __forceinline__ void own_items(const KParams &P, const SmallPlan &S, const SmallMem<R> &M, unsigned parts,
                                          int warp, int nwarps) {
    const int lane = threadIdx.x & 31;
    KParams L = P;
    L.partials = M.partials;
    if (LOAD == LOAD_SHARED) L.items = M.items;
    for (int u = 0; u < S.max_runs; ++u) {
        const SmallRun &run = M.runs[u];
        const int a = run.a, b = run.b;
        if (a >= b || !(parts & (1u << run.part))) continue;
        GroupView<R> V;
        V.idx = run.idx;
        V.W = reinterpret_cast<const R *>(run.W);
        V.part = run.part;
        V.sb = run.sb;
        V.pb = run.pb;
        V.lg = run.lg;
        V.s0 = V.part == PART_PP ? M.P : M.f;
        V.s1 = M.N + run.N_at;
        V.Nglob = M.N;
        run_range<R, false, LOAD>(L, V, a, b, warp, nwarps, lane);
        const int packets = (b - a + (32 >> V.lg) - 1) >> (5 - V.lg);
        warp -= packets;
        while (warp < 0) warp += nwarps;
    }
}

// RHS value of an owned row from the CTA's partials (row_value of rows.cuh).
template <class R>
__device__ __forceinline__ double own_row(const R *partials, const SmallRow &row, unsigned parts) {
    RowAcc<R> A;
    auto sum = [&](int i0, int i1) {
        if constexpr (sizeof(R) == 8) {
            for (int i = i0; i < i1; ++i) A.add(partials[i]);
        } else {  // eight loads at a time (graphene 36: 9.8 -> 9.5 us an RHS; in FP64 the toy's 4.9 -> 5.3)
            for (int i = i0; i < i1; i += 8) {
                R v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = i + j < i1 ? partials[i + j] : R(0);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (i + j < i1) A.add(v[j]);
            }
        }
    };
    if (row.f >= 0) {
        if (!(parts & RTBTE_EPH)) return 0.0;
        sum(row.p0, row.p1);
        return -A.value();
    }
    if (parts & RTBTE_PHE) sum(row.p0, row.mid);
    if (parts & RTBTE_PHPH) sum(row.mid, row.p1);
    return -A.value();
}

// One RHS of the state y (FP64): populations converted into shared memory, own items, own rows.
template <class R, int NT>
__global__ void __launch_bounds__(NT) rhs_small(KParams P, SmallPlan S, const InstDev *inst, unsigned parts,
                                                const double *y, double *ydot) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int2 from = S.begin();
    const SmallMem<R> M(smem_raw, S, from.y);
    copy_in(M.runs, S.runs + (long long)blockIdx.x * S.max_runs, S.max_runs);
    const int r0 = from.x + threadIdx.x, r1 = S.end().x;
    const InstDev I = *inst;
    pdl_begin();
    pdl_wait();
    for (int i = threadIdx.x; i < I.n_c; i += NT) M.f[i] = (R)y[i];
    const double *yN = y + I.n_c;
    if (I.N_q == I.N_q_pad) {
        for (int p = threadIdx.x; p < I.n_ph; p += NT) M.N[p] = (R)yN[p];
    } else {
        for (int p = threadIdx.x; p < I.n_ph; p += NT) {
            const int nu = p / I.N_q;
            M.N[nu * I.N_q_pad + (p - nu * I.N_q)] = (R)yN[p];
        }
    }
    if (parts & RTBTE_PHPH)
        for (int a = threadIdx.x; a < I.M; a += NT) M.P[a] = (R)yN[__ldg(S.pp_full + a)];
    __syncthreads();
    own_items<R, LOAD_STREAM>(P, S, M, parts, threadIdx.x >> 5, NT / 32);
    __syncthreads();
    for (int r = r0; r < r1; r += NT) {
        const SmallRow row = S.rows[r];
        ydot[row.row] = own_row<R>(M.partials, row, parts);
    }
}

// ---- attempt loop ---------------------------------------------------------------------------------
struct SmallSync {
    unsigned arrived;          // barrier arrivals so far
    int failed;                // a barrier wait gave up
    unsigned long long range;  // rows out of range in all attempts so far
    Ctl start;                 // the controller the launch started from
};

// Grid barrier (arrivals reach `target`); false in every thread if it was not seen in `polls` polls.
__device__ __forceinline__ bool grid_barrier(SmallSync *sync, unsigned target, int polls) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 0;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(&sync->arrived) : "memory");
        for (int i = 0; i < polls; ++i) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(&sync->arrived) : "memory");
            if ((int)(v - target) >= 0) {
                ok = 1;
                break;
            }
        }
        if (!ok) atomicExch(&sync->failed, 1);
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Population copies of three states: the current one (kept while attempts from it are rejected)
// and two that the stages alternate between.
struct SmallPops {
    void *f[3], *N[3], *P[3];
};

// Sum of the squared weighted errors of all rows, in the order of wrms_chunks and the controller:
// 128 chunks of L rows, each by the butterfly of its first warp, then the butterfly of 128.  For
// L <= 8, by the first four warps, one chunk a thread: of a chunk's 256 strided terms only the
// first L are not 0, and adding zeros is exact, so its butterfly is a tree over 8 values.  The
// first warp returns the sum.
__device__ __forceinline__ double small_wrms(const double *wsq, long long ni, int L) {
    __shared__ double ws[4];
    const int t = threadIdx.x;
    if (t < kWrmsChunks) {
        double v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const long long r = (long long)t * L + j;
            v[j] = j < L && r < ni ? __ldcg(wsq + r) : 0.0;
        }
        double s = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 31) == 0) ws[t >> 5] = s;
    }
    __syncthreads();
    return t < 32 ? ((ws[0] + ws[1]) + ws[2]) + ws[3] : 0.0;
}

// Copies the CTA's items and their entries into shared memory and points its runs at them.
template <class R, int NT>
__device__ __forceinline__ void hold_lists(const KParams &P, const SmallPlan &S, const SmallMem<R> &M, int item0) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int u = 0; u < S.max_runs; ++u) {
        const SmallRun &run = M.runs[u];
        for (int k = run.a + warp; k < run.b; k += NT / 32) {
            const int4 d = __ldg(reinterpret_cast<const int4 *>(P.items) + k);
            const Item it = item_from(d);
            const int at = __ldg(S.item_at + k) - __ldg(S.item_at + item0), vw = (int)(it.len * sizeof(R) / 16);
            const uint4 *ip = reinterpret_cast<const uint4 *>(run.idx + it.begin);
            const uint4 *wp = reinterpret_cast<const uint4 *>(reinterpret_cast<const R *>(run.W) + it.begin);
            for (int v = lane; v < it.len >> 2; v += 32) reinterpret_cast<uint4 *>(M.idx + at)[v] = __ldg(ip + v);
            for (int v = lane; v < vw; v += 32) reinterpret_cast<uint4 *>(M.W + at)[v] = __ldg(wp + v);
            if (lane == 0) reinterpret_cast<int4 *>(M.items)[k - item0] = make_int4(at, d.y, d.z, d.w & 0xffffff);
        }
    }
    __syncthreads();
    for (int u = threadIdx.x; u < S.max_runs; u += NT) {
        SmallRun &run = M.runs[u];
        if (run.a < run.b) {
            run.a -= item0;
            run.b -= item0;
        }
        run.idx = M.idx;
        run.W = M.W;
    }
}

// LOAD: LOAD_SHARED where the CTAs' lists fit in shared memory, else LOAD_CACHED.
template <class R, int NT, int LOAD>
__global__ void __launch_bounds__(NT) attempts_small(KParams P, SmallPlan S, SmallPops B, StageArgs a, double *chunks,
                                                     int cap, int polls, SmallSync *sync) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Ctl C;
    __shared__ int s_accept;
    const int2 from = S.begin();
    const int slot0 = from.y, row0 = from.x, nrows = S.end().x - row0;
    const SmallMem<R> M(smem_raw, S, slot0);
    if (threadIdx.x == 0) C = a.ctl[0];
    copy_in(M.runs, S.runs + (long long)blockIdx.x * S.max_runs, S.max_runs);
    copy_in(M.rows, S.rows + row0, nrows);
    __syncthreads();
    if (C.done) return;  // (alike in every CTA)
    const int cur0 = C.cur;
    if (blockIdx.x == 0 && threadIdx.x == 0) sync->start = C;
    if (LOAD == LOAD_SHARED) hold_lists<R, NT>(P, S, M, slot0);
    const long long ni = a.n;
    const int L = (int)((ni + kWrmsChunks - 1) / kWrmsChunks);  // rows of a chunk
    const int warp = threadIdx.x >> 5;
    unsigned barriers = 0;
    unsigned long long range_seen = 0;
    int cur = 0, n = 0;  // population set of the current state, attempts run
    int yc = 0;          // which of M.y is the current state
    bool ok = true;
    auto put = [&](int set, const SmallRow &row, R v) {  // into a set of population copies
        if (row.f >= 0) {
            reinterpret_cast<R *>(B.f[set])[row.f] = v;
        } else {
            reinterpret_cast<R *>(B.N[set])[row.N] = v;
            if (row.P >= 0) reinterpret_cast<R *>(B.P[set])[row.P] = v;
        }
    };
    {
        const double *y = cur0 ? a.Y1 : a.Y0;
        for (int r = threadIdx.x; r < nrows; r += NT) {
            const double v = y[M.rows[r].row];
            M.y[r] = v;
            put(0, M.rows[r], (R)v);
        }
        ok = grid_barrier(sync, ++barriers * gridDim.x, polls);
    }
    bool pending = false;  // the last attempt's controller runs beside the first stage of the next
    double sum = 0.0;
    while (ok) {
        int in = cur;
        for (int i = 0; i < a.T.S && ok; ++i) {
            // This stage's populations (written by every CTA before the last barrier: L2 copies) and
            // items.  With a controller pending the first warp runs it meanwhile -- its logarithms
            // and exponential in FP64 take longer than these small sums -- and the others do both.
            const bool split = i == 0 && pending;
            if (split && warp == 0) {
                unsigned long long r = 0;
                if (threadIdx.x == 0) r = __ldcg(&sync->range);
                control(&C, a.cp, sum, ni, r - range_seen);
                if (threadIdx.x == 0) range_seen = r;
            } else {
                const int t0 = split ? 32 : 0;
                stage_part<R>(M.f, reinterpret_cast<const R *>(B.f[in]), S.n_f, t0);
                stage_part<R>(M.N, reinterpret_cast<const R *>(B.N[in]), S.n_N, t0);
                if (a.parts & RTBTE_PHPH) stage_part<R>(M.P, reinterpret_cast<const R *>(B.P[in]), S.n_P, t0);
                asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
                if (split) asm volatile("bar.sync 1, %0;\n" ::"n"(NT - 32) : "memory");
                else __syncthreads();
                own_items<R, LOAD>(P, S, M, a.parts, warp - t0 / 32, (NT - t0) / 32);
            }
            __syncthreads();
            if (split) {
                pending = false;
                if (C.done || n == cap) {  // that attempt was the last one
                    ok = false;
                    break;
                }
            }
            const double h = C.h_try;
            int out = 0;  // a set neither current nor being read
            while (out == cur || out == in) ++out;
            for (int r = threadIdx.x; r < nrows; r += NT) {
                const SmallRow row = M.rows[r];
                double k = own_row<R>(M.partials, row, a.parts);
                if (a.forcing) k += __ldg(a.forcing + row.row);
                M.K[i * S.max_rows + r] = k;
                auto K = [&](int j) { return M.K[j * S.max_rows + r]; };
                const double y = M.y[yc * S.max_rows + r];
                double z;
                if (i < a.T.S - 1) {
                    z = stage_next(a.T, i, h, y, K);
                } else {
                    double x2;
                    bool beyond;
                    z = stage_last(a, row.f >= 0, h, y, K, &x2, &beyond);
                    M.y[(yc ^ 1) * S.max_rows + r] = z;
                    a.wsq[row.row] = x2;
                    if (beyond) atomicAdd(&sync->range, 1ULL);
                }
                put(out, row, (R)z);
            }
            in = out;
            ok = grid_barrier(sync, ++barriers * gridDim.x, polls);
        }
        if (!ok) break;
        if (L <= 8) {
            sum = small_wrms(a.wsq, ni, L);
        } else {
            for (int ch = blockIdx.x; ch < kWrmsChunks; ch += gridDim.x) {
                const long long b = (long long)ch * L, e = b + L < ni ? b + L : ni;
                const double s = block_sum<true>(a.wsq, b, e > b ? e - b : 0);
                if (threadIdx.x == 0) chunks[ch] = s;
            }
            if (!(ok = grid_barrier(sync, ++barriers * gridDim.x, polls))) break;
            sum = small_wrms(chunks, kWrmsChunks, 1);
        }
        // accepted or not decides which state the next attempt starts from; the rest of the
        // controller follows beside its first stage
        if (warp == 0) {
            const double eps = sqrt(sum / (double)ni);
            if (threadIdx.x == 0) s_accept = isfinite(eps) && (C.fixed || eps <= 1.0);
        }
        __syncthreads();
        if (s_accept) {
            cur = in;
            yc ^= 1;
        }
        pending = true;
        ++n;
    }
    __syncthreads();
    // The result goes into the other buffer, whichever the attempts' count would name: where some CTA's
    // wait gave up, CTAs have left at different attempts (and others not at all), and the host goes back to
    // the state and controller at the start (small_give_up).
    double *y = cur0 ? a.Y0 : a.Y1;
    for (int r = threadIdx.x; r < nrows; r += NT) y[M.rows[r].row] = M.y[yc * S.max_rows + r];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        C.cur = cur0 ^ 1;
        a.ctl[0] = C;
    }
}

constexpr int kSmallThreads = 768, kSmallThreads64 = 512;  // RHS; attempts: kSmallThreads64

KParams small_params(rtbte_ctx *ctx) {
    KParams P;
    std::memset(&P, 0, sizeof(P));
    P.items = reinterpret_cast<const ItemRec *>(ctx->small_tab.as<char>() + ctx->small_at[0]);
    return P;
}

SmallPlan small_plan(rtbte_ctx *ctx, bool attempts) {
    SmallPlan S;
    const SmallCtaMax &Z = ctx->small_max[attempts];
    const InstHost &I = ctx->inst[0];
    const char *tab = ctx->small_tab.as<char>();
    S.runs = reinterpret_cast<const SmallRun *>(tab + ctx->small_at[1]) +
             (attempts ? (size_t)ctx->small_grid * ctx->n_groups : 0);
    S.rows = reinterpret_cast<const SmallRow *>(tab + ctx->small_at[2]);
    S.off = reinterpret_cast<const int2 *>(tab + ctx->small_at[3]);
    S.shares = ctx->small_grid;
    S.fold = attempts ? ctx->small_fold : 1;
    S.max_runs = ctx->n_groups;
    S.max_items = Z.items;
    S.max_rows = Z.rows;
    S.n_f = I.n_c_pad;
    S.n_N = I.d.nmodes * I.N_q_pad;
    S.n_P = I.M_pad;
    S.pp_full = I.t_ppfull.as<int>();
    S.item_at = reinterpret_cast<const int *>(tab + ctx->small_at[4]);
    S.max_entries = Z.entries;
    return S;
}

const void *rhs_fn(const rtbte_ctx *ctx) {
    return ctx->precision == RTBTE_PREC_FP64 ? (const void *)rhs_small<double, kSmallThreads64>
                                             : (const void *)rhs_small<float, kSmallThreads>;
}
const void *attempts_fn(const rtbte_ctx *ctx) {
    if (ctx->small_max[1].entries > 0)
        return ctx->precision == RTBTE_PREC_FP64 ? (const void *)attempts_small<double, kSmallThreads64, LOAD_SHARED>
                                                 : (const void *)attempts_small<float, kSmallThreads64, LOAD_SHARED>;
    return ctx->precision == RTBTE_PREC_FP64 ? (const void *)attempts_small<double, kSmallThreads64, LOAD_CACHED>
                                             : (const void *)attempts_small<float, kSmallThreads64, LOAD_CACHED>;
}
int small_threads(const rtbte_ctx *ctx) {
    return ctx->precision == RTBTE_PREC_FP64 ? kSmallThreads64 : kSmallThreads;
}

}  // namespace

// Entry slots up to which a single instance takes the one-launch kernels.  In FP32 about where the 3 us
// that they save an RHS take some hundred of them to cover building their plan; in FP64, where the
// arithmetic dominates sooner, where they save nothing any more.  us per RHS, one launch / launch sequence:
//   FP32  graphene 24, 0.23M entries  7.0 / 10.8    graphene 48, 2.65M  13.6 / 15.1 (plan 0.7 ms)
//         graphene 36, 0.96M          9.5 / 11.2    graphene 54, 4.17M  17.2 / 17.2
//         graphene 42, 1.71M         10.9 / 14.1    graphene 60, 6.00M  20.9 / 20.1
//         (plan 0.5 ms beside 0.5)                  silicon 12, 4.70M   10.9 / 15.2
//   FP64  graphene 24, 0.23M         12.5 / 15.0    graphene 42, 1.71M  29.5 / 28.3
//         graphene 36, 0.96M         19.0 / 21.7    graphene 48, 2.65M  39.0 / 36.9
//         graphene 39, 1.28M         23.3 / 25.9    silicon 10, 1.77M   22.1 / 26.4
constexpr double kSmallSlots = 2e6, kSmallSlots64 = 1.5e6;

// The attempt loop holds whole SMs (its registers fill one) for as many as 64 attempts, about 2 ms, so it
// takes half of them at most and leaves the rest to other streams; a quarter for the smallest lists, which
// are as fast there.  Beside a 12 x 12 FP64 integration a 108 us RHS of graphene 120 takes 171 us and a copy
// of 1 GB 174 instead of 162 us (1290 us with every SM taken; 167 and 167 by the launch sequence it was
// before).  us per attempt of all contexts, 1 / 4 / 8 of them on their own streams:
//                             launch sequence        every SM             half (toy 12: a quarter)
//   toy 12 FP64               58.8 / 21.4 / 16.2     29.9 / 29.8 / 30.0   29.2 /  7.4 /  7.5
//   toy 20 FP64               64.8 / 24.5 / 19.7     37.2 / 36.9 / 36.9   46.0 / 23.2 / 23.2
//   graphene 24, 0.23M        76.0 / 30.0 / 21.2     53.9 / 46.4 / 45.0   52.8 / 24.0 / 23.3
//   graphene 36, 0.96M        78.1 / 36.0 / 26.5     57.1 / 51.7 / 51.0   63.4 / 29.5 / 29.4
//   graphene 42, 1.71M        89.9 / 41.6 / 35.3     -                    87.0 / 41.8 / 40.8
//   graphene 24 FP64, 0.23M   93.7 / 40.0 / 29.5     -                    97.0 / 45.9 / 45.1
// so FP64 attempts, bound by the FP64 pipes of their SMs, take the launch sequence from 0.2M slots on.
constexpr double kSmallQuarter = 6e4, kSmallAttempts64 = 2e5;

// Row ownership of a single small instance, or none (ctx->small_grid = 0).  `items` in launch
// order with their row-major slots, `rowoff` / `rowmid` the rows' slots.
int make_small_plan(rtbte_ctx *ctx, const ItemRec *items, int n, const std::vector<Group> &groups,
                    const std::vector<int> &rowoff, const std::vector<int> &rowmid) {
    ctx->small_grid = ctx->small_fold = 0;
    if (ctx->inst.size() != 1 || ctx->sliced || n == 0) return RTBTE_OK;
    const InstHost &I = ctx->inst[0];
    const size_t R = ctx->real_size;
    const size_t pops = R * ((size_t)I.n_c_pad + (size_t)I.d.nmodes * I.N_q_pad + I.M_pad);
    const double slots = (double)(ctx->part_slots[0] + ctx->part_slots[1] + ctx->part_slots[2]);
    if (pops > 160 * 1024 || slots > (R == 8 ? kSmallSlots64 : kSmallSlots) || groups.size() > 64) return RTBTE_OK;
    std::unique_ptr<int[]> by_slot(new int[n]);
    std::unique_ptr<short[]> group_of(new short[n]);
    for (int g = 0; g < (int)groups.size(); ++g)
        for (int k = groups[g].item_begin; k < groups[g].item_end; ++k) {
            by_slot[items[k].slot] = k;
            group_of[k] = (short)g;
        }
    // Rows dealt to the shares family by family (electrons, sub-lattice phonons, other phonons: so
    // every parts mask is spread evenly), back and forth; dearest first where a share gets only a few
    // (many rows average out, and sorting them would cost more than it evens).
    const int ny = (int)ctx->n_y, nc = I.d.n_c, Nq = (int)I.N_q, ng = (int)groups.size();
    const int G = (int)std::max(1.0, std::min((double)ctx->num_sms, std::ceil(slots / 64.0)));
    const ItemCost *cost = ctx->item_cost_h.get();
    std::vector<std::pair<long long, int>> rows_of[3];  // (-cost, row)
    for (int c = 0; c < ny; ++c) {
        const int f = c < nc ? 0 : (I.M > 0 && I.compact[c - nc] >= 0 ? 1 : 2);
        long long w = 0;
        if (ny < 8 * G)
            for (int s = rowoff[c]; s < rowoff[c + 1]; ++s) w -= cost[by_slot[s]].slots;
        rows_of[f].push_back({w, c});
    }
    std::vector<std::vector<int>> own(G);
    for (auto &o : own) o.reserve(ny / G + 3);
    int at = 0, dir = 1;
    for (auto &rows : rows_of) {
        if (ny < 8 * G) std::sort(rows.begin(), rows.end());
        for (const auto &r : rows) {
            own[at].push_back(r.second);
            at += dir;
            if (at == G || at < 0) {
                dir = -dir;
                at += dir;
            }
        }
    }
    // shares per CTA of the attempt loop (0: attempts take the launch sequence), and where each share's
    // rows and slots start; the slots of its rows follow each other
    ctx->small_fold = R == 8 && slots > kSmallAttempts64 ? 0 : slots <= kSmallQuarter ? 4 : 2;
    const int F = std::max(ctx->small_fold, 1), nb = (G + F - 1) / F;
    std::vector<int2> off(G + 1, make_int2(0, 0));
    for (int b = 0; b < G; ++b) {
        int m = 0;
        for (int c : own[b]) m += rowoff[c + 1] - rowoff[c];
        off[b + 1] = make_int2(off[b].x + (int)own[b].size(), off[b].y + m);
    }
    // one buffer, copied at once: items, runs of the RHS and of the attempt loop, rows, the shares' offsets, places
    // of the items' entries
    const size_t len[5] = {sizeof(ItemRec) * n, sizeof(SmallRun) * (size_t)(G + nb) * ng, sizeof(SmallRow) * ny,
                           sizeof(int2) * (G + 1), sizeof(int) * n};
    size_t bytes = 0;
    for (int k = 0; k < 5; ++k) {
        ctx->small_at[k] = bytes;
        bytes += (len[k] + 15) / 16 * 16;
    }
    std::unique_ptr<char[]> tab(new char[bytes]);
    ItemRec *out = reinterpret_cast<ItemRec *>(tab.get() + ctx->small_at[0]);
    SmallRun *runs = reinterpret_cast<SmallRun *>(tab.get() + ctx->small_at[1]);
    SmallRow *rows = reinterpret_cast<SmallRow *>(tab.get() + ctx->small_at[2]);
    int *item_at = reinterpret_cast<int *>(tab.get() + ctx->small_at[4]);
    std::memcpy(tab.get() + ctx->small_at[3], off.data(), len[3]);
    std::memset(runs, 0, len[1]);
    // Items of F shares by group, within a group by share and, within a share, alike ones together (the
    // packets of order_packets in rhs.cu): counting sort over (group, share, process, vectors per lane)
    std::unique_ptr<int[]> count(new int[(size_t)8 * F * ng + 1]), key(new int[n]);
    for (int b0 = 0; b0 < G; b0 += F) {
        const int b1 = std::min(b0 + F, G), i0 = off[b0].y;
        std::fill(count.get(), count.get() + (size_t)8 * F * ng + 1, 0);
        int m = i0;  // slot
        for (int b = b0; b < b1; ++b) {
            SmallRow *r = rows + off[b].x;
            for (int c : own[b]) {
                r->row = c;
                r->p0 = m;
                r->mid = m + rowmid[c] - rowoff[c];
                for (int s = rowoff[c]; s < rowoff[c + 1]; ++s, ++m) {
                    const int k = by_slot[s];
                    key[m] = 8 * (F * group_of[k] + b - b0) + 4 * (items[k].proc != 0) + 4 -
                             cost[k].slots / (4 * cost[k].lanes);
                    ++count[key[m] + 1];
                }
                r->p1 = m;
                const int p = c - nc;
                r->f = c < nc ? c : -1;
                r->N = c < nc ? -1 : p / Nq * I.N_q_pad + p % Nq;
                r->P = c < nc || I.M == 0 ? -1 : I.compact[p];
                r->pad = 0;
                ++r;
            }
        }
        for (int k = 0; k < 8 * F * ng; ++k) count[k + 1] += count[k];
        auto add_run = [&](SmallRun *&q, int g, int a, int b) {
            if (a == b) return;
            const Group &Q = groups[g];
            q->idx = Q.idx;
            q->W = Q.W;
            q->a = i0 + a;
            q->b = i0 + b;
            q->part = (short)Q.part;
            q->sb = (short)Q.s_bits;
            q->pb = (short)Q.pp_bits;
            q->lg = (short)Q.lanes_log2;
            q->N_at = Q.nu * Q.n_q_pad;
            ++q;
        };
        for (int b = b0; b < b1; ++b) {
            SmallRun *q = runs + (size_t)b * ng;
            for (int g = 0; g < ng; ++g) add_run(q, g, count[8 * (F * g + b - b0)], count[8 * (F * g + b - b0 + 1)]);
        }
        SmallRun *q = runs + (size_t)(G + b0 / F) * ng;
        for (int g = 0; g < ng; ++g) add_run(q, g, count[8 * F * g], count[8 * F * (g + 1)]);
        m = i0;
        for (int b = b0; b < b1; ++b)
            for (int c : own[b])
                for (int s = rowoff[c]; s < rowoff[c + 1]; ++s, ++m) {
                    ItemRec &it = out[i0 + count[key[m]]++];
                    it = items[by_slot[s]];
                    it.slot = (unsigned)m;
                }
    }
    for (int k = 0, e = 0; k < n; e += out[k++].len) item_at[k] = e;
    auto largest = [&](int fold) {  // CTA of `fold` shares
        SmallCtaMax Z;
        for (int b0 = 0; b0 < G; b0 += fold) {
            const int b1 = std::min(b0 + fold, G), i0 = off[b0].y, i1 = off[b1].y;
            Z.items = std::max(Z.items, (int)round_up(i1 - i0, 4));
            Z.rows = std::max(Z.rows, (int)round_up(off[b1].x - off[b0].x, 2));
            if (fold == F && i1 > i0) Z.entries = std::max(Z.entries, item_at[i1 - 1] + out[i1 - 1].len - item_at[i0]);
        }
        return Z;
    };
    ctx->small_max[0] = largest(1);
    ctx->small_max[1] = largest(F);
    if (ctx->small_tab.bytes < bytes) {
        ctx->small_tab.release();
        RT_CUDA(ctx, cudaMalloc(&ctx->small_tab.p, bytes));
        ctx->small_tab.bytes = bytes;
    }
    RT_CUDA(ctx, cudaMemcpyAsync(ctx->small_tab.p, tab.get(), bytes, cudaMemcpyHostToDevice, ctx->stream));
    ctx->small_grid = G;
    const auto fits = [&](bool attempts) {
        return small_smem(R, small_plan(ctx, attempts), attempts) + 2048 <= ctx->smem_optin;
    };
    if (ctx->small_fold > 0 && !fits(true)) {
        ctx->small_max[1].entries = 0;
        if (!fits(true)) ctx->small_fold = 0;
    }
    if (!fits(false)) {
        ctx->small_grid = ctx->small_fold = 0;
        return RTBTE_OK;
    }
    for (const void *f : {rhs_fn(ctx), attempts_fn(ctx)}) RT_CUDA(ctx, allow_max_dynamic_smem(f));
    ctx->small_pops.release();  // (of another plan)
    RT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return RTBTE_OK;
}

int launch_small_rhs(rtbte_ctx *ctx, unsigned parts, const double *y, double *ydot, cudaStream_t s) {
    KParams P = small_params(ctx);
    SmallPlan S = small_plan(ctx, false);
    const InstDev *inst = ctx->instdev.as<InstDev>();
    void *args[] = {&P, &S, &inst, &parts, &y, &ydot};
    std::pair<cudaEvent_t, cudaEvent_t> ev;
    int rc;
    if ((rc = timing_begin(ctx, s, &ev))) return rc;
    RT_CUDA(ctx, launch_pdl_fn(rhs_fn(ctx), dim3(ctx->small_grid), dim3(small_threads(ctx)),
                               small_smem(ctx->real_size, S, false), s, args));
    ctx->launches++;
    return timing_end(ctx, s, ev);
}

int read_small(rtbte_ctx *ctx) {
    RT_CUDA(ctx, cudaMemcpyAsync(ctx->small_sync_host, ctx->small_sync.p, sizeof(SmallSync), cudaMemcpyDeviceToHost,
                                 ctx->stream));
    return RTBTE_OK;
}
bool small_give_up(const rtbte_ctx *ctx, Ctl *c) {
    const SmallSync *sync = reinterpret_cast<const SmallSync *>(ctx->small_sync_host);
    if (!sync->failed) return false;
    *c = sync->start;
    c->status = RTBTE_E_TIMEOUT;
    c->done = 1;
    return true;
}

namespace {
// Buffers of the attempt loop, made on its first use.
int ensure_attempts(rtbte_ctx *ctx) {
    if (ctx->small_pops.p) return RTBTE_OK;
    const size_t R = ctx->real_size;
    // two more sets of population copies beside popf / popN / popP, and the barrier
    const size_t bf = R * (size_t)(ctx->popf_len + 4), bN = R * (size_t)(ctx->popN_len + 4), bP = R * (size_t)(ctx->popP_len + 4);
    const size_t al = 256, set = (bf + al - 1) / al * al + (bN + al - 1) / al * al + (bP + al - 1) / al * al;
    RT_CUDA(ctx, cudaMalloc(&ctx->small_pops.p, 2 * set));
    ctx->small_pops.bytes = 2 * set;
    RT_CUDA(ctx, cudaMemsetAsync(ctx->small_pops.p, 0, 2 * set, ctx->stream));
    if (!ctx->small_sync.p) {
        RT_CUDA(ctx, cudaMalloc(&ctx->small_sync.p, sizeof(SmallSync)));
        ctx->small_sync.bytes = sizeof(SmallSync);
    }
    if (!ctx->small_sync_host) RT_CUDA(ctx, cudaMallocHost(&ctx->small_sync_host, sizeof(SmallSync)));
    return RTBTE_OK;
}
}  // namespace

int launch_small_attempts(rtbte_ctx *ctx, const void *stage_args, int cap, cudaStream_t s) {
    int rc;
    if ((rc = ensure_attempts(ctx))) return rc;
    KParams P = small_params(ctx);
    SmallPlan S = small_plan(ctx, true);
    StageArgs a = *reinterpret_cast<const StageArgs *>(stage_args);
    const size_t R = ctx->real_size, al = 256;
    SmallPops B;
    B.f[0] = ctx->popf.p;
    B.N[0] = ctx->popN.p;
    B.P[0] = ctx->popP.p;
    char *p = ctx->small_pops.as<char>();
    for (int k = 1; k < 3; ++k) {
        B.f[k] = p;
        p += (R * (size_t)(ctx->popf_len + 4) + al - 1) / al * al;
        B.N[k] = p;
        p += (R * (size_t)(ctx->popN_len + 4) + al - 1) / al * al;
        B.P[k] = p;
        p += (R * (size_t)(ctx->popP_len + 4) + al - 1) / al * al;
    }
    double *chunks = ctx->wrms_part.as<double>() + 2 * ctx->n_y;
    SmallSync *sync = ctx->small_sync.as<SmallSync>();
    RT_CUDA(ctx, cudaMemsetAsync(sync, 0, sizeof(SmallSync), s));
    int polls = ctx->wait_polls < 0 ? kBarrierPolls : ctx->wait_polls;
    void *args[] = {&P, &S, &B, &a, &chunks, &cap, &polls, &sync};
    RT_CUDA(ctx, cudaLaunchCooperativeKernel(attempts_fn(ctx), dim3((S.shares + S.fold - 1) / S.fold), dim3(kSmallThreads64), args,
                                             small_smem(R, S, true), s));
    ctx->launches++;
    return RTBTE_OK;
}

}  // namespace rtbte
