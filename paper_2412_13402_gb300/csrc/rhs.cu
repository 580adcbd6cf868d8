// rhs.cu -- the collision-integral kernels (Eq. e-ph, Eq. ph-ph) and their execution plan.
//
// One persistent launch evaluates the selected parts of the RHS for every instance.  The
// stored channel entries are streamed from HBM exactly once per evaluation (16-byte
// cache-streaming loads, 4 entries per lane), while the populations they gather are
// staged per CTA in shared memory: the instance's electron occupations f plus, for e-ph
// work, the occupations N of one phonon mode, or of one wavevector block of it where the
// whole mode does not fit (the e-ph lists are blocked by mode and block for this reason); for
// ph-e work only f; for ph-ph work the sub-lattice N.  A work item is a piece
// of a single destination segment; groups of long segments give each warp one item of up to
// 512 entries, groups of short ones give each sub-warp of 4, 8 or 16 lanes one item of up to 64,
// 128 or 256 entries.  Lanes accumulate their entries with
// compensated (two-sum) additions in FP32, plain ones in FP64, and add the lanes with a shuffle
// tree; the partial is
// written per item to the item's slot -- the slots of one row's items are consecutive -- and
// the row kernels add a row's partials in slot order (deterministic).  CTAs
// first run a static share of the items (split by estimated cost), then take the rest in
// chunks from a counter; warps may prefetch upcoming items' entries into L2.  FP32 runs at 24 warps
// per SM, FP64 at 16.
//
// Per-entry arithmetic uses the exact algebraic reductions of the paper's factors
// (Methods A):  F_em = f(1-f') + N(f-f'),  F_abs = N(f-f') - f'(1-f),
//               G_em = N(N'+N''+1) - N'N'',  G_abs = N(N''-N') - N'(N''+1).
#include <algorithm>
#include <cstring>
#include <numeric>

#include "collide.cuh"
#include "internal.cuh"
#include "rows.cuh"

namespace rtbte {

namespace {

// Point V at group g's populations, staging them in shared memory unless this CTA already
// holds them (`staged` is the group currently in shared memory).  Called by all threads.
template <class R, bool STAGED>
__device__ __forceinline__ void enter_group(const KParams &P, int g, R *sm, int &staged, GroupView<R> &V) {
    const Group &G = P.groups[g];
    V.idx = G.idx;
    V.W = reinterpret_cast<const R *>(G.W);
    V.part = G.part;
    V.sb = G.s_bits;
    V.pb = G.pp_bits;
    V.lg = G.lanes_log2;
    V.Nglob = reinterpret_cast<const R *>(P.popN) + G.N_inst;
    const R *src0 = reinterpret_cast<const R *>(G.part == PART_PP ? P.popP : P.popf) + G.stage0_src;
    const R *src1 = reinterpret_cast<const R *>(P.popN) + G.stage1_src;
    if (STAGED) {
        const int l0 = G.stage0_len, l1 = G.stage1_len;
        if (staged != g) {
            __syncthreads();  // the previous group's readers are done with the buffer
            stage_copy<R>(sm, src0, l0);
            if (l1 > 0) stage_copy<R>(sm + l0, src1, l1);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            __syncthreads();
            staged = g;
        }
        V.s0 = sm;
        V.s1 = sm + l0 - G.stage1_q0;  // indexed by the full q index of the mode
    } else {
        V.s0 = src0;
        V.s1 = src1 - G.stage1_q0;
    }
}

// Persistent collision kernel.  Each CTA first runs its static unit (ranges of equal estimated
// cost), then takes dynamic units of the remaining items from a shared counter until none is
// left, so that SMs that finish early absorb the tail of the work.  Every item writes its own
// partial, so the result does not depend on which CTA ran it.
template <class R, bool STAGED, bool WIDE, bool CACHED, int MINB, int NT>
__global__ void __launch_bounds__(NT, MINB) rhs_kernel(KParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_unit;
    R *sm = reinterpret_cast<R *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    int staged = -1;
    // (no pdl_begin: blocks of the row kernel behind this one, waiting on SMs that finish early, slow the
    // others down -- graphene 180 345 -> 361 us, 64 instances 991 -> 1090)
    if (!P.n_tail_d) {  // (a device re-split writes the bounds just before)
        // the first packets' entries on their way to L2 while the populations are still computed
        const int4 from = P.bound[blockIdx.x];
        const Group &G = P.groups[from.y];
        const int lg = WIDE ? 5 : G.lanes_log2;
        const int k = from.x + warp * (32 >> lg) + (lane >> lg);
        if ((lane & ((1 << lg) - 1)) == 0 && k < min(P.bound[blockIdx.x + 1].x, G.item_end)) {
            GroupView<R> V;
            V.idx = G.idx;
            V.W = reinterpret_cast<const R *>(G.W);
            prefetch_item(V, __ldg(reinterpret_cast<const int4 *>(P.items) + k));
        }
    }
    pdl_wait();
    const int n_tail = P.n_tail_d ? *P.n_tail_d : P.n_tail;
    for (int u = blockIdx.x;;) {
        const int4 from = P.bound[u];
        const int end = P.bound[u + 1].x;
        for (int a = from.x, g = from.y, at = from.z; a < end;) {
            const Group &G = P.groups[g];
            const int b = min(end, G.item_end);
            if (a < b && !(P.ctl && P.ctl[G.inst].done)) {  // (done: the instance is at its t_out)
                GroupView<R> V;
                enter_group<R, STAGED>(P, g, sm, staged, V);
                run_range<R, WIDE, CACHED ? LOAD_CACHED : LOAD_STREAM>(P, V, a, b, warp, nwarps, lane);
            }
            if (end <= G.item_end) break;
            g = P.act[++at];
            if (g < 0) break;
            a = P.groups[g].item_begin;
        }
        if (n_tail == 0) return;
        __syncthreads();  // every warp is done with the previous unit and with s_unit
        if (threadIdx.x == 0) s_unit = atomicAdd(P.tail_ctr, 1);
        __syncthreads();
        if (s_unit >= n_tail) break;
        u = gridDim.x + s_unit;
    }
    if (threadIdx.x == 0) {  // the last CTA out resets the counters
        __threadfence();
        if (atomicAdd(P.tail_ctr + 1, 1) == (int)gridDim.x - 1) {
            P.tail_ctr[0] = 0;
            P.tail_ctr[1] = 0;
            __threadfence();
        }
    }
}

// Work split over the groups still active (instance not done, part in the mask), recomputed
// on the device before the collision launches of an attempt of a batched integration.  One block:
//   - the active groups are listed in order in act[] (terminated by -1);
//   - the units' bounds cut the active weight into `grid` static ranges holding 1 - tail_share of
//     it and, when a CTA's share is above tail_min, kTailUnits x grid equal dynamic units; a
//     bound's item is found by interpolating linearly within the active group holding its weight
//     (items of one group carry similar weights; the split affects balance only, never results).
// Finished instances cost a collision launch nothing.
constexpr int kTailUnits = 4;  // dynamic units per CTA of a re-split
constexpr double kResplitTail = 0.2;               // weight left to them
constexpr long long kResplitTailMin = 2048LL * 300000;  // ... where a CTA's share is at least this
__global__ void split_kernel(const Group *groups, int n_groups, const long long *gw, const Ctl *ctl, unsigned mask,
                             int grid, double tail_share, long long tail_min, int4 *bound, int *act, int *n_tail,
                             int *memo, int n_inst) {
    __shared__ long long A[1025];   // inclusive prefix of active weight over groups (A[0] = 0)
    __shared__ int Cn[1025];        // active groups before group g
    __shared__ long long wsum[32];
    __shared__ int csum[32];
    __shared__ int s_same;
    const int T = blockDim.x;  // 256 threads, n_groups <= 1024 (checked on the host)
    pdl_begin();
    pdl_wait();
    // the tables of the last split still hold when the same instances are active for the same
    // parts (memo: the done flags and mask it was made for, and a flag the host clears whenever
    // the item weights change)
    if (threadIdx.x == 0) s_same = memo[n_inst + 1] == 1 && memo[n_inst] == (int)mask;
    __syncthreads();
    for (int i = threadIdx.x; i < n_inst; i += T)
        if (memo[i] != ctl[i].done) s_same = 0;
    __syncthreads();
    if (s_same) return;
    const int C = (n_groups + T - 1) / T;
    const int g0 = threadIdx.x * C;
    long long run = 0;
    int nrun = 0;
    for (int g = g0; g < g0 + C && g < n_groups; ++g) {
        const Group &G = groups[g];
        const bool on = (mask & (1u << G.part)) && !ctl[G.inst].done && G.item_end > G.item_begin;
        run += on ? gw[g] : 0;
        nrun += on ? 1 : 0;
        A[g + 1] = run;
        Cn[g + 1] = nrun;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long incl = run;
    int nincl = nrun;
    for (int o = 1; o < 32; o <<= 1) {
        const long long v = __shfl_up_sync(0xffffffffu, incl, o);
        const int nv = __shfl_up_sync(0xffffffffu, nincl, o);
        if (lane >= o) {
            incl += v;
            nincl += nv;
        }
    }
    if (lane == 31) {
        wsum[wid] = incl;
        csum[wid] = nincl;
    }
    if (threadIdx.x == 0) {
        A[0] = 0;
        Cn[0] = 0;
    }
    __syncthreads();
    if (wid == 0) {
        long long w = lane < (T >> 5) ? wsum[lane] : 0;
        int nw = lane < (T >> 5) ? csum[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const long long v = __shfl_up_sync(0xffffffffu, w, o);
            const int nv = __shfl_up_sync(0xffffffffu, nw, o);
            if (lane >= o) {
                w += v;
                nw += nv;
            }
        }
        if (lane < (T >> 5)) {
            wsum[lane] = w;
            csum[lane] = nw;
        }
    }
    __syncthreads();
    const long long before = incl - run + (wid > 0 ? wsum[wid - 1] : 0);
    const int nbefore = nincl - nrun + (wid > 0 ? csum[wid - 1] : 0);
    for (int g = g0; g < g0 + C && g < n_groups; ++g) {
        A[g + 1] += before;
        Cn[g + 1] += nbefore;
    }
    __syncthreads();
    const long long total = A[n_groups];
    const int n_act = Cn[n_groups];
    for (int g = threadIdx.x; g < n_groups; g += T)  // compact list of the active groups
        if (Cn[g + 1] > Cn[g]) act[Cn[g]] = g;
    if (threadIdx.x == 0) act[n_act] = -1;
    const bool tail = total / grid >= tail_min;
    const int nt = tail ? kTailUnits * grid : 0;
    const long long stat = tail ? total - (long long)(tail_share * (double)total) : total;
    if (threadIdx.x == 0) *n_tail = nt;
    for (int c = threadIdx.x; c <= grid + nt; c += T) {
        if (total == 0) {
            bound[c] = make_int4(0, 0, 0, 0);
            continue;
        }
        if (c == grid + nt) {  // end of the last active group's items
            int last = n_groups - 1;
            while (last > 0 && Cn[last + 1] == Cn[last]) --last;
            bound[c] = make_int4(groups[last].item_end, last, n_act - 1, 0);
            continue;
        }
        const long long t = c < grid ? stat / grid * c + stat % grid * c / grid
                                     : stat + (total - stat) / nt * (c - grid) + (total - stat) % nt * (c - grid) / nt;
        int lo = 0, hi = n_groups - 1;  // group g with A[g] <= t < A[g+1]
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (A[mid] <= t) lo = mid; else hi = mid - 1;
        }
        while (lo < n_groups - 1 && A[lo + 1] == A[lo]) ++lo;  // skip inactive groups
        const Group &G = groups[lo];
        const long long wg = A[lo + 1] - A[lo];
        const long long ni = G.item_end - G.item_begin;
        bound[c] = make_int4(G.item_begin + (int)((double)(t - A[lo]) * (double)ni / (double)(wg > 0 ? wg : 1)), lo,
                             Cn[lo], 0);
    }
    for (int i = threadIdx.x; i < n_inst; i += T) memo[i] = ctl[i].done;
    if (threadIdx.x == 0) {
        memo[n_inst] = (int)mask;
        memo[n_inst + 1] = 1;
    }
}

// y (FP64) -> population copies in the compute precision
template <class R>
__global__ void __launch_bounds__(256) prep_kernel(RowParams Q, const double *y, long long n) {
    pdl_begin();
    pdl_wait();
    for_rows(Q, n, [&](int, const InstDev &I, long long c) { write_pops<R>(Q, I, c - I.y_off, (R)y[c]); });
}

template <class R>
__global__ void __launch_bounds__(256) rows_kernel(RowParams Q, unsigned parts, double *out, const double *forcing,
                                                   long long n) {
    pdl_begin();
    pdl_wait();
    for_rows(Q, n, [&](int, const InstDev &I, long long c) {
        double v = row_value<R>(Q, I, c - I.y_off, parts);
        if (forcing) v += forcing[c];
        out[c] = v;
    });
}

int upload_raw(rtbte_ctx *ctx, DevBuf &b, const void *h, size_t n) {
    b.release();
    const size_t bytes = std::max<size_t>(n, 16);
    RT_CUDA(ctx, cudaMalloc(&b.p, bytes));
    b.bytes = bytes;
    if (n) RT_CUDA(ctx, cudaMemcpyAsync(b.p, h, n, cudaMemcpyHostToDevice, ctx->stream));
    return RTBTE_OK;
}
template <class T> int upload_vec(rtbte_ctx *ctx, DevBuf &b, const std::vector<T> &h) {
    return upload_raw(ctx, b, h.data(), h.size() * sizeof(T));
}

// Tables of the device re-split in ctx->dyn_tab: unit bounds, active groups, number of dynamic
// units, and the memo of the last split ([n_inst] done flags it saw, its parts mask, a valid flag).
struct DynTab {
    int4 *bound;  // [(1 + kTailUnits) x grid + 1]
    int *act;     // [n_groups + 1]
    int *n_tail;  // [1]
    int *memo;    // [n_inst + 2]
};
size_t dyn_tab_bytes(const rtbte_ctx *ctx) {
    return sizeof(int4) * ((1 + kTailUnits) * (size_t)ctx->grid + 1) +
           sizeof(int) * ((size_t)ctx->n_groups + 1 + 1 + ctx->inst.size() + 2);
}
DynTab dyn_tab(const rtbte_ctx *ctx) {
    DynTab T;
    T.bound = ctx->dyn_tab.as<int4>();
    T.act = reinterpret_cast<int *>(T.bound + (1 + kTailUnits) * (size_t)ctx->grid + 1);
    T.n_tail = T.act + ctx->n_groups + 1;
    T.memo = T.n_tail + 1;
    return T;
}

}  // namespace

RowParams row_params(rtbte_ctx *ctx) {
    RowParams Q;
    Q.inst = ctx->instdev.as<InstDev>();
    Q.n_inst = (int)ctx->inst.size();
    Q.rowoff = ctx->rowoff.as<int>();
    Q.rowmid = ctx->rowmid.as<int>();
    Q.compact = ctx->compact.as<int>();
    Q.blocks = ctx->row_blocks.as<int2>();
    Q.n_blocks = ctx->n_rblk;
    Q.partials = ctx->partials.p;
    Q.popf = ctx->popf.p;
    Q.popN = ctx->popN.p;
    Q.popP = ctx->popP.p;
    return Q;
}

// Per-mask work units of the persistent grid, from item weights: (entry slots + w x the item's
// share of a warp) x the part's cost per entry, with each mask's own w and part costs.  The slots
// count the vectors its lanes step through together, used or not (a warp's packet takes as long
// as its longest lane), and w is the cost of a packet beyond its entries.  The first share sf of a
// mask's weight is split into equal static ranges, one per CTA; the rest is cut into dynamic
// units of decreasing weight (half the remaining weight per grid, at least 1/40 of a CTA's share,
// never across a group boundary), taken by CTAs in order at run time.
int split_tables(rtbte_ctx *ctx) {
    const int G = ctx->grid, n = ctx->n_items;
    const int ng = (int)ctx->group_begin_h.size();
    const ItemCost *cost = ctx->item_cost_h.get();
    auto group_end = [&](int g) { return g + 1 < ng ? ctx->group_begin_h[g + 1] : n; };
    // sums of the unscaled weights (32 x slots + w x lanes) of blocks of 64 items, per distinct w
    auto raw = [&](int w, int k) { return 32LL * cost[k].slots + (long long)w * cost[k].lanes; };
    std::map<int, std::vector<long long>> block_sums;
    auto blocks_of = [&](int w) -> const std::vector<long long> & {
        std::vector<long long> &p = block_sums[w];
        if (p.empty()) {
            p.resize(n / 64 + 1);
            parallel_for((n / 64 + 1023) / 1024, n > 500000, [&](int c) {
                for (int b = 1024 * c; b < std::min(1024 * (c + 1), n / 64); ++b) {
                    long long s = 0;
                    for (int k = 64 * b; k < 64 * (b + 1); ++k) s += raw(w, k);
                    p[b] = s;
                }
            });
        }
        return p;
    };
    auto sum_of = [&](int w, int k0, int k1) {  // items [k0, k1)
        const std::vector<long long> &p = blocks_of(w);
        long long s = 0;
        while (k0 < k1) {
            if ((k0 & 63) == 0 && k0 + 64 <= k1) {
                s += p[k0 >> 6];
                k0 += 64;
            } else {
                s += raw(w, k0++);
            }
        }
        return s;
    };
    auto scale = [](const LaunchTuning &L, int part) { return (long long)(64.0 * L.ps[part] + 0.5); };
    std::map<int, std::vector<long long>> group_sums;  // raw weight of each group, per w
    auto groups_of = [&](int w) -> const std::vector<long long> & {
        std::vector<long long> &p = group_sums[w];
        if (p.empty()) {
            p.resize(std::max(ng, 1));
            for (int g = 0; g < ng; ++g) p[g] = sum_of(w, ctx->group_begin_h[g], group_end(g));
        }
        return p;
    };
    std::vector<int4> bound;
    std::vector<int> act;
    std::vector<long long> start;  // weight of the mask's items before each of its groups, and the total
    for (unsigned mask = 1; mask <= 7; ++mask) {
        const LaunchTuning &L = ctx->lt[mask];
        const std::vector<long long> &blocks = blocks_of(L.w), &gsum = groups_of(L.w);
        ctx->bound_off[mask] = (int)bound.size();
        ctx->act_off[mask] = (int)act.size();
        const int act0 = (int)act.size();
        start.assign(1, 0);
        for (int g = 0; g < ng; ++g) {
            const int part = ctx->group_part_h[g];
            if (!(mask & (1u << part)) || group_end(g) == ctx->group_begin_h[g]) continue;
            act.push_back(g);
            start.push_back(start.back() + scale(L, part) * gsum[g]);
        }
        const int na = (int)act.size() - act0;
        act.push_back(-1);
        const long long total = start.back();
        // a position among the mask's items that moves forward only: item `at` of its group number
        // `ai`, with weight `before` in front of it (ai == na: past the last item)
        int ai = 0, at = 0;
        long long before = 0;
        auto enter = [&](int k) {
            ai = k;
            before = start[k];
            at = k < na ? ctx->group_begin_h[act[act0 + k]] : group_end(act[act0 + na - 1]);
        };
        auto move_to = [&](long long t) {  // the first item with weight t or more in front
            if (ai < na && start[ai + 1] <= t) {
                int k = ai + 1;
                while (k < na && start[k + 1] <= t) ++k;
                enter(k);
            }
            if (ai == na) return;
            const int g = act[act0 + ai], end = group_end(g);
            const long long sc = scale(L, ctx->group_part_h[g]);
            while (at < end && before < t) {
                if ((at & 63) == 0 && at + 64 <= end && before + sc * blocks[at >> 6] <= t) {
                    before += sc * blocks[at >> 6];
                    at += 64;
                } else {
                    before += sc * raw(L.w, at++);
                }
            }
            if (at == end) enter(ai + 1);
        };
        auto add = [&] {
            const int k = std::min(ai, na - 1);
            bound.push_back(make_int4(at, act[act0 + k], k, 0));
        };
        int n_tail = 0;
        if (na == 0) {
            for (int c = 0; c <= G; ++c) bound.push_back(make_int4(0, 0, 0, 0));
        } else {
            const long long split = L.sf >= 1.0 ? total : (long long)(L.sf * (double)total);
            enter(0);
            for (int c = 0; c < G; ++c) {
                move_to(split / G * c + split % G * c / G);
                add();
            }
            move_to(split);
            const long long wmin = std::max<long long>(1, total / (40LL * G));
            while (ai < na) {
                add();
                ++n_tail;
                const int k = ai;
                move_to(before + std::max(wmin, (total - before) / (2LL * G)));
                if (ai > k) enter(k + 1);  // units end with their group
            }
            add();
        }
        ctx->tail_n[mask] = n_tail;
    }
    // per-group weights for the device re-split of batched integrations (full-RHS parameters)
    std::vector<long long> gwt(ng);
    for (int g = 0; g < ng; ++g) gwt[g] = scale(ctx->lt[7], ctx->group_part_h[g]) * groups_of(ctx->lt[7].w)[g];
    int rc;
    if ((rc = upload_vec(ctx, ctx->gwt, gwt))) return rc;
    // the device re-split's memo no longer matches the weights: clear its valid flag
    if (ctx->dyn_tab.p) {
        const DynTab T = dyn_tab(ctx);
        RT_CUDA(ctx, cudaMemsetAsync(T.memo + ctx->inst.size() + 1, 0, sizeof(int), ctx->stream));
    }
    if ((rc = upload_vec(ctx, ctx->act_tab, act))) return rc;
    return upload_vec(ctx, ctx->bound_tab, bound);
}

// The collision kernel of a plan and its threads per SM (per CTA in the form that reads
// populations from global memory: two CTAs per SM in FP32; one in FP64, where two at 64 registers
// spill -- silicon at 80^3 / 40^3, 2.1e9 entries: 16.1 ms with two, 15.4 with one).
template <bool CACHED> const void *collision_kernel_of(const rtbte_ctx *ctx) {
    const bool fp64 = ctx->precision == RTBTE_PREC_FP64;
    if (!ctx->staged)
        return fp64 ? (const void *)rhs_kernel<double, false, false, CACHED, 1, kRhsThreads64>
                    : (const void *)rhs_kernel<float, false, false, CACHED, 2, kRhsThreads64>;
    if (fp64)
        return ctx->wide ? (const void *)rhs_kernel<double, true, true, CACHED, 1, kRhsThreads64>
                         : (const void *)rhs_kernel<double, true, false, CACHED, 1, kRhsThreads64>;
    return ctx->wide ? (const void *)rhs_kernel<float, true, true, CACHED, 1, kRhsThreads>
                     : (const void *)rhs_kernel<float, true, false, CACHED, 1, kRhsThreads>;
}
// Ordinary or streaming loads of the lists.  Inside an integration the same lists are read again
// at once: below kKeepBytes, two thirds of L2's 129 MB, they stay there with ordinary loads (57 MB: 156 ->
// 138 us an attempt, 79 MB: 27.0 -> 25.0 us a launch; but 105 MB: 205 -> 226 us an attempt), and several
// instances take ordinary loads whatever their size, since
// what is read shrinks as they finish (16-instance window: 32.2 -> 31.1 ms of collision time).
// Otherwise streaming loads, whose lines are evicted first, keep a part of the stream for the next
// reading where ordinary ones would evict all of it (streaming / ordinary loads, us an RHS: 105 MB
// 34.6 / 36.5, 154 MB 41.9 / 44.7, 345 MB 73.7 / 74.3, 546 MB 108.8 / 110.6, 827 MB 146.9 / 148.8; three
// contexts of 57 MB in turn 31.1 / 32.2), up to sizes where no part matters and ordinary loads are as
// fast or 1-2% faster (1.20 GB 201.4 / 200.6, 1.68 GB 270.5 / 268.6, 2.27 GB 348.6 / 345.0, 2.78 GB 413 /
// 406).
constexpr double kKeepBytes = 85e6, kStreamBytes = 1e9;
const void *collision_kernel(const rtbte_ctx *ctx, unsigned parts, bool integrating) {
    double bytes = 0;
    for (int part = 0; part < 3; ++part)
        if (parts & (1u << part)) bytes += (double)ctx->part_slots[part] * (4 + ctx->real_size);
    const bool ordinary = bytes >= kStreamBytes || (integrating && (ctx->inst.size() > 1 || bytes <= kKeepBytes));
    return ordinary ? collision_kernel_of<true>(ctx) : collision_kernel_of<false>(ctx);
}
int collision_threads(const rtbte_ctx *ctx) {
    return ctx->staged && ctx->precision != RTBTE_PREC_FP64 ? kRhsThreads : kRhsThreads64;
}

// Launch parameters of the masks the autotuner has not set.  A prefetch distance of one packet is
// the fastest or within 2% of it at every FP32 size measured (graphene 36-180, silicon 16-32, 2-64
// instances: none costs 15-30%, two packets up to 4%); FP64, bound by its arithmetic, is 2% faster
// without (graphene 120: 728 against 745 us).  Packet weight and part costs come from static launches
// (sf 1) over w 64-384 and costs 0.9-1.3: graphene 75 32.6 -> 31.4 us, graphene 90 49.7 -> 47.4, three
// instances 98 -> 92, FP64 graphene 63 79.9 -> 75.9, against w 192 and equal costs.  The share split statically: dynamic
// units even out what the weights do not model, at ~1 us and a staging copy each, which pays in
// launches above ~250 us (FP32: 0.9 against 1.0, graphene 180 365 / 384 us, silicon 32 421 / 437 us,
// but graphene 150 202 / 198 us; FP64, bound by its arithmetic, already at 90 us: graphene 63 93 / 99
// us) and with several instances, whose groups differ most (0.5: 64 instances 990 / 1175 us, 16
// instances 389 / 440 us; fewer groups than ~100, 0.8: 6 instances 167 / 186 us).
void default_tuning(rtbte_ctx *ctx) {
    const bool fp64 = ctx->precision == RTBTE_PREC_FP64;
    for (unsigned m = 0; m < 8; ++m) {
        if (ctx->lt_tuned) continue;  // a tuned mask's parameters serve the others
        LaunchTuning L;
        if (fp64) {
            L.w = 64;
            L.pf = 0;
        } else {  // a ph-e entry takes two gathers of f and one operation more, a ph-ph entry two of N
            L.ps[PART_PHE] = 1.1;
            L.ps[PART_PP] = 1.05;
        }
        double tot = 0;
        for (int part = 0; part < 3; ++part) tot += (m & (1u << part)) ? (double)ctx->part_slots[part] : 0.0;
        if (ctx->inst.size() > 1) L.sf = tot < 4e6 ? 1.0 : ctx->n_groups >= 100 ? 0.5 : 0.8;
        else L.sf = tot > (fp64 ? 4e6 : 2e8) ? 0.9 : 1.0;
        ctx->lt[m] = L;
    }
}

// Vectors a lane steps through for an item of `len` entries on 1 << lg lanes (1..4).
int item_rounds(int len, int lg) { return std::max(1, ((len >> 2) + (1 << lg) - 1) >> lg); }

// Order of the items of groups with several items to a warp: a packet's sub-warps run in step, so
// a packet costs its longest item and, for ph-ph, one pass per process present in it.  Within
// windows of kSortWindow items (which keep the entry stream local) the items are ordered by
// process and by vectors per lane, longest first, so that packets hold alike items.  The partials'
// slots are already set: sums do not depend on the order.
constexpr int kSortWindow = 1024;
void order_packets(ItemRec *items, const Group &G) {
    if (G.lanes_log2 == 5) return;
    ItemRec tmp[kSortWindow];
    for (int w0 = G.item_begin; w0 < G.item_end; w0 += kSortWindow) {
        const int n = std::min(kSortWindow, G.item_end - w0);
        int at[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        auto key = [&](const ItemRec &it) { return 4 * (it.proc != 0) + 4 - item_rounds(it.len, G.lanes_log2); };
        for (int i = 0; i < n; ++i) ++at[key(items[w0 + i]) + 1];
        for (int b = 0; b < 8; ++b) at[b + 1] += at[b];
        for (int i = 0; i < n; ++i) tmp[at[key(items[w0 + i])]++] = items[w0 + i];
        std::copy(tmp, tmp + n, items + w0);
    }
}

// Build the work items, staging groups, per-row partial slots and per-CTA work ranges.
int make_plan(rtbte_ctx *ctx) {
    const size_t R = ctx->real_size;
    const size_t NI = ctx->inst.size();
    std::vector<Group> groups;
    std::vector<InstDev> idev(NI);
    size_t max_stage = 0;
    // Staging groups in item order: e-ph (instance, mode, q-block), ph-e (instance), ph-ph (instance).
    // Each comes with its destinations' segments: destination r holds segments [r * nproc, ...) of
    // off (from segment seg0), the first of them of process proc0; dest_of maps r to the items' dest.
    struct Source {
        const std::vector<long long> *off, *plen;
        long long seg0, rows;
        int nproc, proc0, N_q, N_q_pad;  // ph-e: destinations are stored by mode with a padded stride
        long long at;                    // first entry of this group's row offsets in row_items
        long long slots;                 // entry slots of its items
    };
    std::vector<Source> src;
    std::vector<long long> eoff_base(NI), poff_base(NI), ppoff_base(NI);
    long long n_row_items = 0;
    auto add_group = [&](Group &G, const InstHost &I, Source S) {
        G.f_inst = I.f_off;
        G.N_inst = I.N_off;
        G.P_inst = I.P_off;
        S.at = n_row_items;
        n_row_items += S.rows + 1;
        groups.push_back(G);
        src.push_back(S);
        max_stage = std::max(max_stage, (size_t)(G.stage0_len + G.stage1_len) * R);
    };
    int part_group[4] = {0, 0, 0, 0};  // first group of each part
    for (size_t i = 0; i < NI; ++i) {
        const InstHost &I = ctx->inst[i];
        eoff_base[i] = n_row_items;
        const int nqb = std::max(I.eph_nqb, 1);
        const int qblk = I.eph_qblk > 0 ? I.eph_qblk : I.N_q_pad;
        for (int blk = 0; blk < I.d.nmodes * nqb; ++blk) {  // (mode, q-block)
            const int nu = blk / nqb, qb = blk % nqb;
            const int q_lo = qb * qblk, q_len = std::min(qblk, I.N_q_pad - q_lo);
            Group G{};
            G.idx = I.eph_idx.as<uint32_t>();
            G.W = I.eph_W.p;
            G.part = PART_EPH;
            G.inst = (int)i;
            G.nu = nu;
            G.s_bits = I.s_bits;
            G.n_q_pad = I.N_q_pad;
            G.stage0_len = I.n_c_pad;
            G.stage0_src = I.f_off;
            G.stage1_len = q_len;
            G.stage1_src = I.N_off + (long long)nu * I.N_q_pad + q_lo;
            G.stage1_q0 = q_lo;
            add_group(G, I, {&I.eph_off, &I.eph_plen, 2LL * blk * I.d.n_c, I.d.n_c, 2, 0, 0, 0, 0, 0});
        }
    }
    part_group[PART_PHE] = (int)groups.size();
    for (size_t i = 0; i < NI; ++i) {
        const InstHost &I = ctx->inst[i];
        poff_base[i] = n_row_items;
        Group G{};
        G.idx = I.phe_idx.as<uint32_t>();
        G.W = I.phe_W.p;
        G.part = PART_PHE;
        G.inst = (int)i;
        G.s_bits = I.s_bits;
        G.n_q_pad = I.N_q_pad;
        G.stage0_len = I.n_c_pad;
        G.stage0_src = I.f_off;
        add_group(G, I, {&I.phe_off, &I.phe_plen, 0, I.n_ph, 1, 1, (int)I.N_q, I.N_q_pad, 0, 0});
    }
    part_group[PART_PP] = (int)groups.size();
    for (size_t i = 0; i < NI; ++i) {
        const InstHost &I = ctx->inst[i];
        ppoff_base[i] = n_row_items;
        if (I.M == 0) continue;
        Group G{};
        G.idx = I.pp_idx.as<uint32_t>();
        G.W = I.pp_W.p;
        G.part = PART_PP;
        G.inst = (int)i;
        G.pp_bits = I.pp_bits;
        G.stage0_len = I.M_pad;
        G.stage0_src = I.P_off;
        add_group(G, I, {&I.pp_off, &I.pp_plen, 0, I.M, 2, 0, 0, 0, 0, 0});
    }
    part_group[3] = (int)groups.size();
    // Lanes per item of each group -- from the mean padded length of its non-empty segments, counted
    // over every row (also those outside a row slice, so that a sliced context cuts its items as a
    // full one does), so that a sub-warp's item holds about one segment -- and its items per row.
    std::vector<int> row_items(n_row_items);  // first item of each row of each group, from its own 0
    std::vector<long long> group_items(groups.size());
    const bool threads = n_row_items > 100000;
    parallel_for((int)groups.size(), threads, [&](int g) {
        const Source &S = src[g];
        long long tot = 0, n = 0;
        for (long long s = S.seg0; s < S.seg0 + S.rows * S.nproc; ++s)
            if ((*S.plen)[s] > 0) {
                tot += (*S.plen)[s];
                ++n;
            }
        const double mean = n ? (double)tot / (double)n : 0.0;
        const int lg = mean <= 64.0 ? 2 : mean <= 128.0 ? 3 : mean <= 256.0 ? 4 : 5, sh = lg + 4;
        groups[g].lanes_log2 = lg;
        const long long *off = S.off->data() + S.seg0;
        long long k = 0;
        for (long long r = 0; r < S.rows; ++r) {
            row_items[S.at + r] = (int)k;
            for (int p = 0; p < S.nproc; ++p, ++off) k += (off[1] - off[0] + (1 << sh) - 1) >> sh;
        }
        row_items[S.at + S.rows] = (int)k;
        group_items[g] = k;
    });
    long long total_items = 0;
    for (size_t g = 0; g < groups.size(); ++g) {
        const long long k = group_items[g];
        if (total_items + k >= (long long)INT32_MAX) return fail(ctx, RTBTE_E_UNSUPPORTED, "too many work items");
        groups[g].item_begin = (int)total_items;
        total_items += k;
        groups[g].item_end = (int)total_items;
    }
    const int n_items = (int)total_items;
    for (const Source &S : src)
        if ((*S.off)[S.seg0 + S.rows * S.nproc] > (1LL << 40))
            return fail(ctx, RTBTE_E_UNSUPPORTED, "channel list longer than 2^40 entries");
    for (int part = 0; part < 3; ++part) {
        const int g0 = part_group[part], g1 = part_group[part + 1];
        ctx->part_first[part] = g0 < (int)groups.size() ? groups[g0].item_begin : n_items;
        ctx->part_items[part] = g1 > g0 ? groups[g1 - 1].item_end - groups[g0].item_begin : 0;
    }
    // the items themselves (arrays left uninitialised: every element is written below)
    std::unique_ptr<ItemRec[]> items_h(new ItemRec[std::max(n_items, 1)]);
    ItemRec *items = items_h.get();
    parallel_for((int)groups.size(), threads, [&](int g) {
        const Source &S = src[g];
        const int cut = 16 << groups[g].lanes_log2;  // entries per item at most
        ItemRec *it = items + groups[g].item_begin;
        const long long *off = S.off->data() + S.seg0;
        for (long long r = 0; r < S.rows; ++r) {
            const int dest = S.N_q > 0 ? (int)((int)r / S.N_q * S.N_q_pad + (int)r % S.N_q) : (int)r;
            for (int p = 0; p < S.nproc; ++p, ++off)
                for (long long x = off[0]; x < off[1]; x += cut, ++it) {
                    it->begin_lo = (unsigned)(x & 0xffffffffLL);
                    it->begin_hi = (unsigned char)((x >> 32) & 0xff);
                    it->slot = 0;  // set below
                    it->dest = dest;
                    it->len = (unsigned short)std::min<long long>(cut, off[1] - x);
                    it->proc = (unsigned char)(S.proc0 + p);
                }
        }
        for (long long r = 0; r <= S.rows; ++r) row_items[S.at + r] += groups[g].item_begin;
    });
    // partial slots, row-major: every row's items get consecutive slots in the order the row
    // adds them (an electron row: its (mode, q-block) blocks in turn, emission then absorption
    // items of each; a phonon row: its ph-e items, then its ph-ph items if it is a sub-lattice
    // phonon), so a row kernel reads one offset pair and one contiguous run of partials
    std::vector<int> rowoff(ctx->n_y + 1, 0), rowmid(std::max<long long>(ctx->n_y, 1), 0);
    std::vector<long long> first_slot(NI + 1, 0);
    for (size_t g = 0; g < groups.size(); ++g) first_slot[groups[g].inst + 1] += groups[g].item_end - groups[g].item_begin;
    for (size_t i = 0; i < NI; ++i) first_slot[i + 1] += first_slot[i];
    std::atomic<bool> covered{true};
    parallel_for((int)NI, threads, [&](int i) {
        const InstHost &I = ctx->inst[i];
        const int nc = I.d.n_c, nblk = I.d.nmodes * std::max(I.eph_nqb, 1);
        long long next = first_slot[i];
        auto take = [&](long long o) {
            for (int k = row_items[o]; k < row_items[o + 1]; ++k) items[k].slot = (unsigned)next++;
        };
        for (int d = 0; d < nc; ++d) {
            const long long c = I.y_off + d;
            rowoff[c] = (int)next;
            for (int blk = 0; blk < nblk; ++blk) take(eoff_base[i] + (long long)blk * (nc + 1) + d);
            rowmid[c] = (int)next;
        }
        for (long long p = 0; p < I.n_ph; ++p) {
            const long long c = I.y_off + nc + p;
            rowoff[c] = (int)next;
            take(poff_base[i] + p);
            rowmid[c] = (int)next;
            const int a = I.M > 0 ? I.compact[p] : -1;
            if (a >= 0) take(ppoff_base[i] + a);
        }
        if (next != first_slot[i + 1]) covered = false;
    });
    rowoff[ctx->n_y] = n_items;
    if (!covered) return fail(ctx, RTBTE_E_UNSUPPORTED, "work items not covered by rows");
    // item order within groups of several items to a warp, and what each item costs
    ctx->item_cost_h.reset(new ItemCost[std::max(n_items, 1)]);
    ItemCost *cost = ctx->item_cost_h.get();
    parallel_for((int)groups.size(), threads, [&](int g) {
        const Group &G = groups[g];
        order_packets(items, G);
        long long slots = 0;
        for (int k = G.item_begin; k < G.item_end; ++k) {
            cost[k] = {(unsigned short)(item_rounds(items[k].len, G.lanes_log2) << (G.lanes_log2 + 2)),
                       (unsigned short)(1 << G.lanes_log2)};
            slots += cost[k].slots;
        }
        src[g].slots = slots;
    });
    for (int part = 0; part < 3; ++part) {
        ctx->part_slots[part] = 0;
        for (int g = part_group[part]; g < part_group[part + 1]; ++g) ctx->part_slots[part] += src[g].slots;
    }
    ctx->n_items = n_items;
    ctx->n_groups = (int)groups.size();
    ctx->wide = std::all_of(groups.begin(), groups.end(), [](const Group &G) { return G.lanes_log2 == 5; });
    // instance layout for the row kernels
    std::vector<int> compact;
    for (size_t i = 0; i < ctx->inst.size(); ++i) {
        InstHost &I = ctx->inst[i];
        InstDev &D = idev[i];
        D.y_off = I.y_off;
        D.n_c = I.d.n_c;
        D.n_ph = (int)I.n_ph;
        D.M = (int)I.M;
        D.nmodes = I.d.nmodes;
        D.N_q = (int)I.N_q;
        D.N_q_pad = I.N_q_pad;
        D.f_off = I.f_off;
        D.N_off = I.N_off;
        D.P_off = I.P_off;
        D.compact_base = (long long)compact.size();
        compact.insert(compact.end(), I.compact.begin(), I.compact.end());
    }
    // staging decision and launch shape: 24 (FP32) or 16 (FP64) warps per SM, as 1, 2 or 4 CTAs --
    // several CTAs per SM when their staging fits, so one CTA's group change (barrier + staging copy)
    // overlaps the others' streaming
    ctx->staged = max_stage + 64 <= ctx->smem_optin;  // 64 B left for the kernel's static shared memory
    ctx->smem_bytes = ctx->staged ? std::max<size_t>(max_stage, 16) : 0;
    int per_sm = 1;
    const bool fp64 = ctx->precision == RTBTE_PREC_FP64;
    const void *fns[2] = {collision_kernel_of<false>(ctx), collision_kernel_of<true>(ctx)};
    const int nt = collision_threads(ctx);
    if (ctx->staged) {
        for (const void *fn : fns) {
            RT_CUDA(ctx, allow_max_dynamic_smem(fn));
            RT_CUDA(ctx, cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
        }
        for (int k : {4, 2}) {
            int nb = 0, nb2 = 0;
            RT_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fns[0], nt / k, ctx->smem_bytes));
            RT_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb2, fns[1], nt / k, ctx->smem_bytes));
            if (std::min(nb, nb2) >= k) {
                per_sm = k;
                break;
            }
        }
    }
    ctx->per_sm = per_sm;
    ctx->grid = ctx->num_sms * (ctx->staged ? per_sm : fp64 ? 1 : 2);
    ctx->group_begin_h.resize(groups.size());
    ctx->group_part_h.resize(groups.size());
    for (size_t g = 0; g < groups.size(); ++g) {
        ctx->group_begin_h[g] = groups[g].item_begin;
        ctx->group_part_h[g] = groups[g].part;
    }
    default_tuning(ctx);
    int rc;
    if (!ctx->tail_ctr.p) {
        RT_CUDA(ctx, cudaMalloc(&ctx->tail_ctr.p, 16));
        ctx->tail_ctr.bytes = 16;
        RT_CUDA(ctx, cudaMemsetAsync(ctx->tail_ctr.p, 0, 16, ctx->stream));
    }
    if ((rc = upload_raw(ctx, ctx->items, items, sizeof(ItemRec) * (size_t)n_items))) return rc;
    if ((rc = upload_vec(ctx, ctx->groups, groups))) return rc;
    if ((rc = upload_vec(ctx, ctx->rowoff, rowoff))) return rc;
    if ((rc = upload_vec(ctx, ctx->rowmid, rowmid))) return rc;
    if ((rc = upload_vec(ctx, ctx->instdev, idev))) return rc;
    if ((rc = upload_vec(ctx, ctx->compact, compact))) return rc;
    if (ctx->n_y >= (long long)INT32_MAX) return fail(ctx, RTBTE_E_UNSUPPORTED, "state vector too long");
    if (ctx->inst.size() > (size_t)kMaxBatch) return fail(ctx, RTBTE_E_UNSUPPORTED, "more than 1024 instances");
    std::vector<int2> rblk;  // several instances: blocks of 256 rows of one instance
    if (NI > 1)
        for (size_t i = 0; i < NI; ++i)
            for (long long r = 0; r < ctx->inst[i].d.n_c + ctx->inst[i].n_ph; r += 256) rblk.push_back(make_int2((int)i, (int)r));
    ctx->n_rblk = (int)rblk.size();
    if ((rc = upload_vec(ctx, ctx->row_blocks, rblk))) return rc;
    ctx->dyn_tab.release();  // reallocated below for this plan's sizes
    if ((rc = split_tables(ctx))) return rc;
    if (ctx->n_groups > 1024) return fail(ctx, RTBTE_E_UNSUPPORTED, "more than 1024 staging groups");
    ctx->dyn_tab.release();
    ctx->dyn_tab.bytes = dyn_tab_bytes(ctx);
    RT_CUDA(ctx, cudaMalloc(&ctx->dyn_tab.p, ctx->dyn_tab.bytes));
    RT_CUDA(ctx, cudaMemsetAsync(ctx->dyn_tab.p, 0, ctx->dyn_tab.bytes, ctx->stream));
    ctx->partials.release();
    size_t pb = std::max<size_t>(R * (size_t)std::max(ctx->n_items, 1), 16);
    RT_CUDA(ctx, cudaMalloc(&ctx->partials.p, pb));
    ctx->partials.bytes = pb;
    RT_CUDA(ctx, cudaMemsetAsync(ctx->partials.p, 0, pb, ctx->stream));
    RT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if ((rc = init_stage_grid(ctx))) return rc;
    if ((rc = make_small_plan(ctx, items, n_items, groups, rowoff, rowmid))) return rc;
    ctx->plan_valid = true;
    return RTBTE_OK;
}

// Blocks of the row kernels: at most 8 per SM, one pass each otherwise.
static int row_grid(const rtbte_ctx *ctx) {
    const long long want = ctx->inst.size() > 1 ? ctx->n_rblk : (ctx->n_y + 255) / 256;
    return (int)std::max<long long>(1, std::min<long long>(want, 8LL * ctx->num_sms));
}

int launch_prep_from_y(rtbte_ctx *ctx, const double *y, cudaStream_t s) {
    RowParams Q = row_params(ctx);
    const int threads = 256;
    const int blocks = row_grid(ctx);
    RT_CUDA(ctx, launch_pdl(ctx->precision == RTBTE_PREC_FP64 ? prep_kernel<double> : prep_kernel<float>, dim3(blocks),
                            dim3(threads), 0, s, Q, y, ctx->n_y));
    ctx->launches++;
    return RTBTE_OK;
}

// Units of the collision launches of one attempt of a batched integration (the set of instances
// still integrating changes only after it).
int launch_resplit(rtbte_ctx *ctx, unsigned parts, const Ctl *ctl, cudaStream_t s) {
    if (ctx->inst.size() <= 1) return RTBTE_OK;
    const DynTab T = dyn_tab(ctx);
    RT_CUDA(ctx, launch_pdl(split_kernel, dim3(1), dim3(256), 0, s, ctx->groups.as<Group>(), ctx->n_groups,
                            ctx->gwt.as<long long>(), ctl, parts, ctx->grid, kResplitTail, kResplitTailMin, T.bound, T.act,
                            T.n_tail, T.memo, (int)ctx->inst.size()));
    ctx->launches++;
    return RTBTE_OK;
}

// Events around a standalone collision launch (rtbte_set_kernel_timing; none while capturing).
int timing_begin(rtbte_ctx *ctx, cudaStream_t s, std::pair<cudaEvent_t, cudaEvent_t> *ev) {
    *ev = {nullptr, nullptr};
    if (!ctx->timing) return RTBTE_OK;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    RT_CUDA(ctx, cudaStreamIsCapturing(s, &cs));
    if (cs != cudaStreamCaptureStatusNone) return RTBTE_OK;
    for (cudaEvent_t *e : {&ev->first, &ev->second}) {
        if (ctx->ev_pool.empty()) {
            cudaEvent_t ne;
            RT_CUDA(ctx, cudaEventCreate(&ne));
            ctx->ev_pool.push_back(ne);
        }
        *e = ctx->ev_pool.back();
        ctx->ev_pool.pop_back();
    }
    RT_CUDA(ctx, cudaEventRecord(ev->first, s));
    return RTBTE_OK;
}
int timing_end(rtbte_ctx *ctx, cudaStream_t s, const std::pair<cudaEvent_t, cudaEvent_t> &ev) {
    if (!ev.first) return RTBTE_OK;
    RT_CUDA(ctx, cudaEventRecord(ev.second, s));
    ctx->ev_pending.push_back(ev);
    return RTBTE_OK;
}

template <class R>
static int launch_core_t(rtbte_ctx *ctx, unsigned parts, const Ctl *ctl, cudaStream_t s) {
    KParams P;
    std::memset(&P, 0, sizeof(P));
    P.items = ctx->items.as<ItemRec>();
    P.groups = ctx->groups.as<Group>();
    P.pf_dist = ctx->lt[parts].pf;
    P.tail_ctr = ctx->tail_ctr.as<int>();
    if (ctl && ctx->inst.size() > 1) {  // batched integration: units over the active instances (launch_resplit)
        const DynTab T = dyn_tab(ctx);
        P.bound = T.bound;
        P.act = T.act;
        P.n_tail_d = T.n_tail;
    } else {
        P.bound = ctx->bound_tab.as<int4>() + ctx->bound_off[parts];
        P.act = ctx->act_tab.as<int>() + ctx->act_off[parts];
        P.n_tail = ctx->tail_n[parts];
    }
    P.partials = ctx->partials.p;
    P.popf = ctx->popf.p;
    P.popN = ctx->popN.p;
    P.popP = ctx->popP.p;
    P.ctl = ctl;
    std::pair<cudaEvent_t, cudaEvent_t> ev;
    int rc;
    if ((rc = timing_begin(ctx, s, &ev))) return rc;
    void *args[] = {&P};
    RT_CUDA(ctx, launch_pdl_fn(collision_kernel(ctx, parts, ctl != nullptr), dim3(ctx->grid),
                               dim3(collision_threads(ctx) / (ctx->staged ? ctx->per_sm : 1)),
                               ctx->staged ? ctx->smem_bytes : 0, s, args));
    RT_CUDA(ctx, cudaGetLastError());
    ctx->launches++;
    return timing_end(ctx, s, ev);
}

int launch_rhs_core(rtbte_ctx *ctx, unsigned parts, const Ctl *ctl, cudaStream_t s) {
    if (parts == 0 || parts > 7) return fail(ctx, RTBTE_E_INVALID_ARG, "parts must be a non-empty subset of RTBTE_ALL");
    return ctx->precision == RTBTE_PREC_FP64 ? launch_core_t<double>(ctx, parts, ctl, s)
                                             : launch_core_t<float>(ctx, parts, ctl, s);
}

namespace {

// Time `reps` collision launches for `parts` after one untimed launch.
int time_launches(rtbte_ctx *ctx, unsigned parts, cudaEvent_t e0, cudaEvent_t e1, int reps, float *ms) {
    int rc;
    if ((rc = launch_rhs_core(ctx, parts, nullptr, ctx->stream))) return rc;
    RT_CUDA(ctx, cudaEventRecord(e0, ctx->stream));
    for (int r = 0; r < reps; ++r)
        if ((rc = launch_rhs_core(ctx, parts, nullptr, ctx->stream))) return rc;
    RT_CUDA(ctx, cudaEventRecord(e1, ctx->stream));
    RT_CUDA(ctx, cudaEventSynchronize(e1));
    RT_CUDA(ctx, cudaEventElapsedTime(ms, e0, e1));
    return RTBTE_OK;
}

// Tuning of mask `parts`'s work split: packet weight, per-part
// entry costs, L2 prefetch distance and static share, each timed over 3 launches and the
// fastest kept.
int tune_split(rtbte_ctx *ctx, unsigned parts, cudaEvent_t e0, cudaEvent_t e1) {
    static const int cand[] = {32, 96, 192, 320, 512, 1024};
    LaunchTuning &L = ctx->lt[parts];
    int best = L.w, rc = RTBTE_OK;
    float best_ms = 1e30f;
    for (int w : cand) {
        float ms = 0.f;
        L.w = w;
        if ((rc = split_tables(ctx)) || (rc = time_launches(ctx, parts, e0, e1, 3, &ms))) return rc;
        if (ms < best_ms) {
            best_ms = ms;
            best = w;
        }
    }
    L.w = best;
    if ((rc = split_tables(ctx))) return rc;
    // calibrate the relative cost of an entry in each part from single-part launches (run with
    // this mask's parameters), keep it if this mask's launch gets faster
    const double scale0[3] = {L.ps[0], L.ps[1], L.ps[2]};
    double t[3] = {0, 0, 0}, wsum[3] = {0, 0, 0};
    int used = 0;
    for (int part = 0; part < 3; ++part) {
        if (!(parts & (1u << part)) || ctx->part_items[part] == 0 || (parts == (1u << part))) continue;
        for (int k = ctx->part_first[part]; k < ctx->part_first[part] + ctx->part_items[part]; ++k)
            wsum[part] += ctx->item_cost_h[k].slots + best * ctx->item_cost_h[k].lanes / 32.0;
        const unsigned pm = 1u << part;
        const LaunchTuning keep = ctx->lt[pm];
        ctx->lt[pm] = L;
        float ms = 0.f;
        rc = split_tables(ctx);
        if (!rc) rc = time_launches(ctx, pm, e0, e1, 3, &ms);
        ctx->lt[pm] = keep;
        if (rc) return rc;
        t[part] = ms;
        used |= pm;
    }
    if (used) {
        double ref = 0.0;
        int nref = 0;
        for (int part = 0; part < 3; ++part)
            if (used & (1u << part)) {
                ref += t[part] / wsum[part];
                ++nref;
            }
        ref /= nref;
        for (int part = 0; part < 3; ++part)
            if (used & (1u << part)) L.ps[part] = (t[part] / wsum[part]) / ref;
        float ms = 0.f;
        if ((rc = split_tables(ctx)) || (rc = time_launches(ctx, parts, e0, e1, 3, &ms))) return rc;
        if (ms > best_ms) {  // calibration did not help: back to the previous costs
            for (int part = 0; part < 3; ++part) L.ps[part] = scale0[part];
            if ((rc = split_tables(ctx))) return rc;
        }
    }
    // L2 prefetch distance, then the share of the work split statically (the rest is taken
    // dynamically by CTAs that finish early)
    static const int dists[] = {0, 1, 2, 3, 4};
    int best_d = L.pf;
    float best_d_ms = 1e30f;
    for (int d : dists) {
        L.pf = d;
        float ms = 0.f;
        if ((rc = time_launches(ctx, parts, e0, e1, 3, &ms))) return rc;
        if (ms < best_d_ms) {
            best_d_ms = ms;
            best_d = d;
        }
    }
    L.pf = best_d;
    static const double fracs[] = {1.0, 0.9, 0.8, 0.6, 0.4};
    double best_f = 1.0;
    float best_f_ms = 1e30f;
    for (double f : fracs) {
        L.sf = f;
        float ms = 0.f;
        if ((rc = split_tables(ctx)) || (rc = time_launches(ctx, parts, e0, e1, 3, &ms))) return rc;
        if (ms < best_f_ms) {
            best_f_ms = ms;
            best_f = f;
        }
    }
    L.sf = best_f;
    return split_tables(ctx);
}

}  // namespace

// Autotuner of the collision launch of one parts mask.  The result belongs to this mask; masks
// never tuned themselves take it as their own.
int autotune(rtbte_ctx *ctx, unsigned parts, int *chosen) {
    cudaEvent_t e0, e1;
    RT_CUDA(ctx, cudaEventCreate(&e0));
    RT_CUDA(ctx, cudaEventCreate(&e1));
    const LaunchTuning start = ctx->lt[parts];
    const int rc = tune_split(ctx, parts, e0, e1);
    if (rc) ctx->lt[parts] = start;
    if (!rc) {
        ctx->lt_tuned |= 1u << parts;
        for (unsigned m = 1; m <= 7; ++m)
            if (!(ctx->lt_tuned & (1u << m))) ctx->lt[m] = ctx->lt[parts];
    }
    const int rc2 = split_tables(ctx);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    if (rc2) return rc2;
    if (chosen) *chosen = ctx->lt[parts].w;
    return RTBTE_OK;
}

// Linearised ph-ph rates: one warp per sub-lattice destination a of one instance,
//   Gamma_a = -dI^{ph-ph}_a/dN_a = sum_em W (N' + N'' + 1) + sum_abs W (N'' - N')
// (Eq. ph-ph with G_em, G_abs differentiated in the destination population; W as stored,
// pair and absorption factors included), from the compute-precision sub-lattice copy popP,
// summed in FP64 per lane then a fixed butterfly; written to rates[y_off + n_c + full(a)].
// The FP64 pipe bounds it (2 or 3 operations per entry: 0.35 ms for graphene 180's 8.8e7 entries;
// the list streams in 0.16 ms).  STAGED: one CTA per SM holds the populations in shared memory,
// widened to FP64 (S) where they fit so; lanes read four entries with a 16-byte load, four such
// vectors in flight, and the next destination's entries are prefetched into L2 (graphene 180, FP64
// lists: 1043 us with one entry per lane and load and gathers from global memory, 489 us so; FP32
// lists, whose weights are widened one by one: 1586 us before, 508 us so).
constexpr int kRateThreads = 512;
// x in FP64 where it is zero or a normal number, by integer operations: the bias of the exponent grows
// by 1023 - 127, the fraction moves up by 29 bits.  (The conversion instruction shares the FP64 pipe;
// with it the FP32 lists of graphene 180 take 686 us.)
__device__ __forceinline__ bool zero_or_normal(float x) {
    const unsigned u = __float_as_uint(x);
    return (u << 1) == 0u || (u & 0x7f800000u) - 0x00800000u < 0x7f000000u;
}
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x);
    const unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20));
    return __hiloint2double((int)((u << 1) == 0u ? u : hi), (int)(u << 29));
}
// the four weights of a vector, exactly
__device__ __forceinline__ void weights4(const Batch<float, 4> &B, int j, double (&w)[4]) {
    if (zero_or_normal(B.w(j, 0)) && zero_or_normal(B.w(j, 1)) && zero_or_normal(B.w(j, 2)) && zero_or_normal(B.w(j, 3))) {
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = widen(B.w(j, k));
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = (double)B.w(j, k);
    }
}
__device__ __forceinline__ void weights4(const Batch<double, 4> &B, int j, double (&w)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = B.w(j, k);
}
template <class R, class S, bool STAGED>
__global__ void __launch_bounds__(kRateThreads) pp_rates_kernel(const uint32_t *idx, const R *W, const long long *off,
                                                                const R *popP, int n_stage, const int *pp_full,
                                                                int pp_bits, int M, long long row0, double *rates) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const S *P = reinterpret_cast<const S *>(popP);
    if constexpr (STAGED) {
        S *sm = reinterpret_cast<S *>(smem_raw);
        if constexpr (sizeof(S) == sizeof(R)) {
            stage_copy<R>(sm, popP, n_stage);
            asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
        } else {
            for (int i = threadIdx.x; i < n_stage; i += kRateThreads) sm[i] = (S)popP[i];
        }
        __syncthreads();
        P = sm;
    }
    const int lane = threadIdx.x & 31;
    const unsigned pmask = (1u << pp_bits) - 1u;
    // destinations dealt over the CTAs first: neighbouring segments have alike lengths
    const int step = gridDim.x * (kRateThreads >> 5);
    for (int a = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; a < M; a += step) {
        const long long o0 = off[2 * a], o1 = off[2 * a + 1], o2 = off[2 * a + 2];
        if (a < M - step && lane == 0) {
            const long long p0 = off[2 * (a + step)], p1 = off[2 * (a + step) + 2];
            if (p1 > p0) {
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(idx + p0),
                             "r"((unsigned)((p1 - p0) * 4)) : "memory");
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(W + p0),
                             "r"((unsigned)((p1 - p0) * sizeof(R))) : "memory");
            }
        }
        double acc = 0.0;
        // adds W (N' + N'' + 1), or W (N'' - N'), over a segment, in FP64 whatever the lists' precision
        auto segment = [&](long long b, long long e, auto emission) {
            constexpr bool EM = decltype(emission)::value;
            const int nv = (int)((e - b) >> 2);  // segments are padded to whole vectors
            GroupView<R> V;
            V.idx = idx;
            V.W = W;
            V.part = PART_PP;
            Item it;
            it.len = 0;
            for (int v0 = 0; v0 < nv; v0 += 128) {
                it.begin = b + 4LL * v0;
                it.len = (unsigned short)(4 * min(nv - v0, 128));
                Batch<R, 4> B;
                B.issue(V, it, lane, 5);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (lane + 32 * j >= (it.len >> 2)) break;
                    double w[4];
                    weights4(B, j, w);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned x = comp4(B.iv[j], k);
                        const double Nb = (double)P[x & pmask], Nc = (double)P[x >> pp_bits];
                        acc = fma(w[k], EM ? Nb + Nc + 1.0 : Nc - Nb, acc);
                    }
                }
            }
        };
        segment(o0, o1, std::true_type{});
        segment(o1, o2, std::false_type{});
#pragma unroll
        for (int m = 16; m; m >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
        if (lane == 0) rates[row0 + pp_full[a]] = acc;
    }
}

template <class R, class S, bool STAGED>
static int launch_pp_rates_t(rtbte_ctx *ctx, InstHost &I, double *rates, cudaStream_t s) {
    const int grid = (int)std::min<long long>((I.M + 7) / 8, (long long)ctx->num_sms);
    const auto fn = pp_rates_kernel<R, S, STAGED>;
    if (STAGED) RT_CUDA(ctx, allow_max_dynamic_smem((const void *)fn));
    fn<<<grid, kRateThreads, STAGED ? sizeof(S) * (size_t)I.M_pad : 0, s>>>(
        I.pp_idx.as<uint32_t>(), I.pp_W.as<R>(), I.pp_off_dev.as<long long>(),
        reinterpret_cast<const R *>(ctx->popP.p) + I.P_off, STAGED ? I.M_pad : 0, I.t_ppfull.as<int>(), I.pp_bits,
        (int)I.M, I.y_off + I.d.n_c, rates);
    RT_CUDA(ctx, cudaGetLastError());
    ctx->launches++;
    return RTBTE_OK;
}

int launch_pp_rates(rtbte_ctx *ctx, int inst, double *rates, cudaStream_t s) {
    InstHost &I = ctx->inst[inst];
    if (I.M == 0) return RTBTE_OK;
    if (!I.pp_off_dev.p) {
        RT_CUDA(ctx, cudaMalloc(&I.pp_off_dev.p, sizeof(long long) * I.pp_off.size()));
        I.pp_off_dev.bytes = sizeof(long long) * I.pp_off.size();
        RT_CUDA(ctx, cudaMemcpyAsync(I.pp_off_dev.p, I.pp_off.data(), I.pp_off_dev.bytes, cudaMemcpyHostToDevice, s));
    }
    const auto fits = [&](size_t size) { return size * (size_t)I.M_pad + 64 <= ctx->smem_optin; };
    if (ctx->precision == RTBTE_PREC_FP64)
        return fits(8) ? launch_pp_rates_t<double, double, true>(ctx, I, rates, s)
                       : launch_pp_rates_t<double, double, false>(ctx, I, rates, s);
    return fits(8)   ? launch_pp_rates_t<float, double, true>(ctx, I, rates, s)
           : fits(4) ? launch_pp_rates_t<float, float, true>(ctx, I, rates, s)
                     : launch_pp_rates_t<float, float, false>(ctx, I, rates, s);
}

int launch_rows(rtbte_ctx *ctx, unsigned parts, double *out, const double *forcing, cudaStream_t s) {
    RowParams Q = row_params(ctx);
    const int threads = 256;
    const int blocks = row_grid(ctx);
    RT_CUDA(ctx, launch_pdl(ctx->precision == RTBTE_PREC_FP64 ? rows_kernel<double> : rows_kernel<float>, dim3(blocks),
                            dim3(threads), 0, s, Q, parts, out, forcing, ctx->n_y));
    ctx->launches++;
    return RTBTE_OK;
}

}  // namespace rtbte
