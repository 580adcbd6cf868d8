// collide.cuh -- device code of the collision sums: factors, entry loads, item sums and the loop
// of a warp over its share of a group's items.  Used by the persistent collision kernel (rhs.cu)
// and by the row-owning kernels of small instances (small.cu).
#pragma once

#include "internal.cuh"

namespace rtbte {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// s + c += x with the rounding error of the addition kept in c (Knuth two-sum).
template <class R> __device__ __forceinline__ void two_sum(R &s, R &c, R x) {
    R t = s + x;
    R bp = t - s;
    R e = (s - (t - bp)) + (x - bp);
    s = t;
    c += e;
}

struct KParams {
    const ItemRec *items;
    const Group *groups;
    // Work units: unit u is the items from bound[u] up to bound[u + 1] of the groups listed in act,
    // in order (parts not evaluated and finished instances are not in the list).  Units 0..grid-1
    // are the CTAs' static ranges, units grid.. are taken from a counter.
    const int4 *bound;    // {first item, its group, that group's index in act, 0}
    const int *act;       // groups to evaluate, ascending (-1 ends)
    int n_tail;           // dynamic units
    const int *n_tail_d;  // batched integration: their number, set by split_kernel (else null)
    void *partials;
    const void *popf, *popN, *popP;
    const Ctl *ctl;  // per-instance controllers: launches inside an integrator skip finished instances
    int *tail_ctr;     // [0] next dynamic unit, [1] CTAs finished (reset by the last one)
    int pf_dist;       // L2 prefetch distance in packets of a warp's sequence (0: off)
};

// n elements (a multiple of 16 bytes) from global to shared memory, asynchronously, by the threads
// of the block from t0 on.
template <class R>
__device__ __forceinline__ void stage_part(R *dst, const R *src, int n, int t0) {
    const int nvec = (int)((long long)n * sizeof(R) / 16);
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(dst);
    for (int i = (int)threadIdx.x - t0; i < nvec; i += blockDim.x - t0) {
        const char *g = reinterpret_cast<const char *>(src) + 16LL * i;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sbase + 16u * i), "l"(g) : "memory");
    }
}
template <class R>
__device__ __forceinline__ void stage_copy(R *dst, const R *src, int n) { stage_part<R>(dst, src, n, 0); }

// Fields of a group that the item loop needs, held in registers.
template <class R> struct GroupView {
    const uint32_t *idx;
    const R *W;
    const R *s0, *s1;  // staged (or global) populations: e-ph f & N of one mode, ph-e f, ph-ph N
    const R *Nglob;    // instance phonon populations (ph-e destinations)
    int part, sb, pb;
    int lg;  // lanes per item = 1 << lg
};

// How items and entries are loaded: streaming or ordinary loads from global memory (items always
// ordinary), or generic ones from shared memory.
enum { LOAD_STREAM = 0, LOAD_CACHED = 1, LOAD_SHARED = 2 };
template <int LOAD, class T> __device__ __forceinline__ T load16(const T *p) {
    return LOAD == LOAD_STREAM ? __ldcs(p) : LOAD == LOAD_CACHED ? __ldg(p) : *p;
}

// Entry loads of one item on a sub-warp of 1 << lg lanes: VPL vectors of 4 entries per lane, 16
// bytes a load; sl is the lane's index in its sub-warp.
template <class R, int VPL> struct Batch;
template <int VPL> struct Batch<float, VPL> {
    uint4 iv[VPL];
    float4 wv[VPL];
    float Np;  // ph-e destination population, loaded with the entries
    template <int LOAD = LOAD_STREAM>
    __device__ __forceinline__ void issue(const GroupView<float> &V, const Item &it, int sl, int lg) {
        const int nv = it.len >> 2;
        if (V.part == PART_PHE) Np = V.Nglob[it.dest];
        const uint4 *ip = reinterpret_cast<const uint4 *>(V.idx + it.begin);
        const float4 *wp = reinterpret_cast<const float4 *>(V.W + it.begin);
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const int v = sl + (j << lg);
            if (v < nv) {
                iv[j] = load16<LOAD>(ip + v);
                wv[j] = load16<LOAD>(wp + v);
            }
        }
    }
    __device__ __forceinline__ float w(int j, int k) const {
        return k == 0 ? wv[j].x : k == 1 ? wv[j].y : k == 2 ? wv[j].z : wv[j].w;
    }
};
template <int VPL> struct Batch<double, VPL> {
    uint4 iv[VPL];
    double2 wa[VPL], wb[VPL];
    double Np;  // ph-e destination population, loaded with the entries
    template <int LOAD = LOAD_STREAM>
    __device__ __forceinline__ void issue(const GroupView<double> &V, const Item &it, int sl, int lg) {
        const int nv = it.len >> 2;
        if (V.part == PART_PHE) Np = V.Nglob[it.dest];
        const uint4 *ip = reinterpret_cast<const uint4 *>(V.idx + it.begin);
        const double2 *wp = reinterpret_cast<const double2 *>(V.W + it.begin);
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const int v = sl + (j << lg);
            if (v < nv) {
                iv[j] = load16<LOAD>(ip + v);
                wa[j] = load16<LOAD>(wp + 2 * v);
                wb[j] = load16<LOAD>(wp + 2 * v + 1);
            }
        }
    }
    __device__ __forceinline__ double w(int j, int k) const {
        return k == 0 ? wa[j].x : k == 1 ? wa[j].y : k == 2 ? wb[j].x : wb[j].y;
    }
};

__device__ __forceinline__ unsigned comp4(const uint4 &e, int k) {
    return k == 0 ? e.x : k == 1 ? e.y : k == 2 ? e.z : e.w;
}

// Per-lane sum of W*F over one item.  FP32: each 4-entry vector is summed with an FMA chain and the
// vector sums are added into (acc, cmp) with two-sum; FP64: one FMA chain.  The warp reduction
// follows in finish_item.  The FP64 pipe (2 lanes per clock per SM) bounds FP64 launches -- 86%
// busy at graphene 120 -- so there the factors take the forms with the fewest operations (4 per
// entry with the weight) and no additions beyond the chain (728 -> 615 us).
// FULL: every lane holds VPL vectors (a whole-warp item of the maximum length), so the vectors
// carry no bounds tests.
template <class R, int VPL, bool FULL, class F>
__device__ __forceinline__ void lane_sum(const Batch<R, VPL> &b, int nv, int sl, int lg, R &acc, R &cmp, F &&factor) {
    acc = R(0);
    cmp = R(0);
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        if (!FULL && sl + (j << lg) >= nv) break;
        R t = sizeof(R) == 8 ? acc : R(0);
#pragma unroll
        for (int k = 0; k < 4; ++k) t = fma(b.w(j, k), factor(comp4(b.iv[j], k)), t);
        if (sizeof(R) == 8 || j == 0) acc = t;
        else two_sum(acc, cmp, t);
    }
}

template <class R, int VPL, bool FULL>
__device__ __forceinline__ void compute_item(const GroupView<R> &V, const Item &it, const Batch<R, VPL> &b, int sl,
                                             int lg, R &acc, R &cmp) {
    const int nv = it.len >> 2;
    if (V.part == PART_EPH) {
        // F_em = f(1-f') + N(f-f') = fma(N, f-f', fma(f', -f, f)),
        // F_abs = N(f-f') - f'(1-f) = fma(N, f-f', fma(f', -(1-f), 0)): one form with the two
        // coefficients chosen per item, so sub-warps on emission and on absorption items of the
        // same warp do not diverge
        const unsigned smask = (1u << V.sb) - 1u;
        const R fd = V.s0[it.dest];
        const R cb = it.proc == 0 ? -fd : -(R(1) - fd), c0 = it.proc == 0 ? fd : R(0);
        lane_sum<R, VPL, FULL>(b, nv, sl, lg, acc, cmp, [&](unsigned e) {
            const R fs = V.s0[e & smask], N = V.s1[e >> V.sb];
            return fma(N, fd - fs, fma(fs, cb, c0));
        });
    } else if (V.part == PART_PHE) {  // F_abs(f_d, f_s, N_p) with N_p per item
        const unsigned smask = (1u << V.sb) - 1u;
        const R Np = b.Np;
        lane_sum<R, VPL, FULL>(b, nv, sl, lg, acc, cmp, [&](unsigned e) {
            const R fd = V.s0[e & smask], fs = V.s0[e >> V.sb];
            if constexpr (sizeof(R) == 8) return fma(Np, fd - fs, fma(fs, fd, -fs));
            else return fma(Np, fd - fs, -fs * (R(1) - fd));
        });
    } else {
        const unsigned pmask = (1u << V.pb) - 1u;
        const R Na = V.s0[it.dest];
        if (it.proc == 0) {  // G_em = N(N'+N''+1) - N'N''
            lane_sum<R, VPL, FULL>(b, nv, sl, lg, acc, cmp, [&](unsigned e) {
                const R Nb = V.s0[e & pmask], Nc = V.s0[e >> V.pb];
                return fma(-Nb, Nc, fma(Na, Nb + Nc, Na));
            });
        } else {  // G_abs = N(N''-N') - N'(N''+1)
            lane_sum<R, VPL, FULL>(b, nv, sl, lg, acc, cmp, [&](unsigned e) {
                const R Nb = V.s0[e & pmask], Nc = V.s0[e >> V.pb];
                if constexpr (sizeof(R) == 8) return fma(Na, Nc - Nb, fma(-Nb, Nc, -Nb));
                else return fma(Na, Nc - Nb, -Nb * (Nc + R(1)));
            });
        }
    }
}

__device__ __forceinline__ Item item_from(const int4 &d) {  // decode an ItemRec
    Item it;
    it.begin = ((long long)((unsigned)d.w >> 24) << 32) | (unsigned)d.x;
    it.slot = (unsigned)d.y;
    it.dest = d.z;
    it.len = (unsigned short)(d.w & 0xffff);
    it.proc = (unsigned char)((d.w >> 16) & 0xff);
    return it;
}

// L2 prefetch of an item's entry arrays (one bulk prefetch per array), so that its streaming
// loads, issued some items later, find the lines in L2.
template <class R> __device__ __forceinline__ void prefetch_item(const GroupView<R> &V, const int4 &d) {
    const Item it = item_from(d);
    if (it.len > 0) {
        const uint32_t *ip = V.idx + it.begin;
        const R *wp = V.W + it.begin;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(ip), "r"((unsigned)it.len * 4u) : "memory");
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(wp), "r"((unsigned)(it.len * sizeof(R)))
                     : "memory");
    }
}

// Item sum in FP32: the lane's compensated sum, rounded once, added over the sub-warp by a
// butterfly in a fixed order (every lane ends with the same bits).  The RHS error is set by the
// conversion of the populations to FP32 (about 5e-8 relative on the parity models), not by this
// tree: the compensated tree measured the same to two digits.
__device__ __forceinline__ void finish_item(const KParams &P, unsigned slot, bool valid, float acc, int sl, int lg) {
#pragma unroll
    for (int o = 16; o; o >>= 1)
        if (o < (1 << lg)) acc += __shfl_xor_sync(kFull, acc, o);
    if (sl == 0 && valid) reinterpret_cast<float *>(P.partials)[slot] = acc;
}

// Item sums in FP64, four packets at a time.  The butterfly of one packet costs lg additions on
// the FP64 pipe, which bounds these launches; four packets share them: at the first level (lanes
// L/2 apart, L the lanes per item) two packets' sums go to the two halves of the sub-warp, at the
// second two such pairs to its quarters, and the rest runs once, 6 additions for 4 packets of 32
// lanes instead of 20 (graphene 120: 615 -> 575 us).  Every item's terms meet in the order of the
// single butterfly, so the sums are the same.
struct ItemSum4 {
    double held0, held1;
    unsigned slot;  // where this lane writes its quarter's sum (kNoSlot: nowhere)
    int n;          // packets held
    static constexpr unsigned kNoSlot = 0xffffffffu;
    __device__ __forceinline__ ItemSum4() : held0(0), held1(0), slot(kNoSlot), n(0) {}
    static __device__ __forceinline__ double merge(double first, double second, int half, int sl) {
        const bool up = sl & half;
        const double mine = up ? second : first, other = up ? first : second;
        return mine + __shfl_xor_sync(kFull, other, half);
    }
    // every lane of the warp; n advances alike in all
    __device__ __forceinline__ void add(const KParams &P, unsigned s, bool valid, double acc, int sl, int lg) {
        const int L2 = 1 << (lg - 1), L4 = L2 >> 1;
        if ((sl & (L4 - 1)) == 0 && ((sl & L2) ? 1 : 0) + ((sl & L4) ? 2 : 0) == n) slot = valid ? s : kNoSlot;
        ++n;
        if (n & 1) {
            held0 = acc;
            return;
        }
        const double m = merge(held0, acc, L2, sl);
        if (n == 2) {
            held1 = m;
            return;
        }
        double r = merge(held1, m, L4, sl);
#pragma unroll
        for (int o = 4; o; o >>= 1)
            if (o < L4) r += __shfl_xor_sync(kFull, r, o);
        if (slot != kNoSlot) reinterpret_cast<double *>(P.partials)[slot] = r;
        slot = kNoSlot;
        n = 0;
    }
    __device__ __forceinline__ void flush(const KParams &P, int sl, int lg) {  // the packets still held
        while (n) add(P, 0, false, 0.0, sl, lg);
    }
};

// A warp's share of items [a, b) of one group.  The warp works on G = 32 >> lg consecutive items
// at a time, one per sub-warp of 1 << lg lanes (the group's items are cut to at most 16 << lg
// entries, so groups of short segments pack two to eight items to a warp), and the warps of the
// CTA take such packets in turn.  WIDE is the variant for plans whose groups all use whole-warp
// items (lg = 5 at compile time).  Every sub-warp loads its own descriptors, one packet ahead of
// their use (uniform 16-byte loads: no shuffles, no index division).  The loop is bound by issue
// slots and latency as much as by HBM, so what an item costs beyond its entries counts: with
// descriptors fetched 32 at a time and broadcast by shuffles (two divisions by the runtime stride
// and eight shuffles an item), bounds tests on full items and separate emission / absorption
// branches, graphene 180 took 395 us (full RHS, 2.27 GB), silicon 32 470 us and a 64-instance
// ensemble 1.76 ms; without them 363, 430 and 1.42 ms.
template <class R, bool WIDE, int LOAD>
__device__ __forceinline__ void run_range(const KParams &P, const GroupView<R> &V, int a, int b, int warp, int nwarps,
                                          int lane) {
    const int lg = WIDE ? 5 : V.lg;
    const int G = 32 >> lg;
    const int step = nwarps * G;
    int kb = a + warp * G;  // first item of the warp's packet
    if (kb >= b) return;
    const int sl = lane & ((1 << lg) - 1);
    int k = kb + (lane >> lg);
    const int4 *items = reinterpret_cast<const int4 *>(P.items);
    // (unsigned: an index past INT_MAX near the end of a very long list is out of range, not negative)
    auto fetch = [&](unsigned i) {
        return i < (unsigned)b ? load16<LOAD == LOAD_SHARED ? LOAD_SHARED : LOAD_CACHED>(items + i) : make_int4(0, 0, 0, 0);
    };
    const int pf = P.pf_dist;  // packets ahead whose entries are prefetched into L2 (0: none)
    const bool lead = LOAD != LOAD_SHARED && sl == 0 && pf > 0;
    int4 d = fetch(k), dn = fetch(k + step), dp = make_int4(0, 0, 0, 0);
    if (lead) {
        for (int j = 1; j < pf; ++j) prefetch_item(V, fetch((unsigned)k + j * step));
        dp = fetch((unsigned)k + pf * step);
    }
    ItemSum4 sums;  // (FP64)
    for (; kb < b; kb += step, k += step) {
        const Item it = item_from(d);
        d = dn;
        dn = fetch((unsigned)k + 2 * step);
        Batch<R, 4> B;
        B.template issue<LOAD>(V, it, sl, lg);
        if (lead) {
            prefetch_item(V, dp);
            dp = fetch((unsigned)k + (pf + 1) * step);
        }
        R acc, cmp;
        if (WIDE && it.len == kItemEntries) compute_item<R, 4, true>(V, it, B, sl, lg, acc, cmp);
        else compute_item<R, 4, false>(V, it, B, sl, lg, acc, cmp);
        if constexpr (sizeof(R) == 8) sums.add(P, it.slot, k < b, acc, sl, lg);
        else finish_item(P, it.slot, k < b, acc + cmp, sl, lg);
    }
    if constexpr (sizeof(R) == 8) sums.flush(P, sl, lg);
}

}  // namespace

}  // namespace rtbte
