// rows.cuh -- per-row device helpers shared by the RHS and integrator kernels.
//
// A "row" is one component of the state vector y = [f; N] (Eq. state_vec).  Its RHS value
// is minus the sum of the compensated partial sums of its work items (the collision
// integrals of Eq. e-ph and Eq. ph-ph carry an overall minus sign), accumulated in FP64 in
// item order, so a row's value does not depend on how items were scheduled.
#pragma once

#include "internal.cuh"

namespace rtbte {

struct RowParams {
    const InstDev *inst;
    int n_inst;
    const int *rowoff;               // [n_y+1] first partial slot of each state row
    const int *rowmid;               // [n_y] phonon rows: first ph-ph slot (ph-e slots before it)
    const int *compact;              // sub-lattice index of each phonon or -1
    const int2 *blocks;              // several instances: {instance, first row} of each block of 256 rows
    int n_blocks;
    const void *partials;            // one sum per item, compute precision
    void *popf, *popN, *popP;        // population copies, compute precision
};

// f(instance, row of y) for every row, by a grid of 256-thread blocks.  Several instances: a block
// takes blocks of 256 rows of one instance (a search over the instances per row took as long as
// the work on it: 64 instances, 1.6M rows, copies to the populations 21.8 us with it and 11.4
// without; the row sums, bound by their partials, 25.4 and 24.8 us).
template <class F> __device__ __forceinline__ void for_rows(const RowParams &Q, long long n, F &&f) {
    if (Q.n_inst > 1) {
        for (int b = blockIdx.x; b < Q.n_blocks; b += gridDim.x) {
            const int2 B = __ldg(Q.blocks + b);
            const InstDev &I = Q.inst[B.x];
            const int r = B.y + (int)threadIdx.x;
            if (r < I.n_c + I.n_ph) f(B.x, I, I.y_off + r);
        }
        return;
    }
    const InstDev &I = Q.inst[0];
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        f(0, I, c);
}

// Accumulator of item partials in item order.  FP64 partials add in FP64.  FP32 partials add as
// an FP32 head/tail pair (two-sum on the heads, tails summed) and are widened once at the end:
// about 48 significant bits, far below the partials' own rounding, with no FP64 arithmetic per
// item (FP64 throughput is low on this GPU).
template <class R> struct RowAcc {
    double acc = 0.0;
    __device__ __forceinline__ void add(R x) { acc += (double)x; }
    __device__ __forceinline__ double value() const { return acc; }
};
template <> struct RowAcc<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        const float bp = t - s;
        c += (s - (t - bp)) + (x - bp);
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

template <class R>
__device__ __forceinline__ void item_sum(const RowParams &Q, int i0, int i1, RowAcc<R> &A) {
    // eight partials' loads in flight, added in order
    const R *P = reinterpret_cast<const R *>(Q.partials);
    for (int it = i0; it < i1; it += 8) {
        R v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = it + j < i1 ? P[it + j] : R(0);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (it + j < i1) A.add(v[j]);
    }
}

// RHS value of row `local` of instance I for the selected parts.  The row's partials sit in
// consecutive slots: an electron row's e-ph items in (mode, q-block) order, a phonon row's ph-e
// items then its ph-ph items (sub-lattice phonons only).
template <class R>
__device__ __forceinline__ double row_value(const RowParams &Q, const InstDev &I, long long local, unsigned parts) {
    const long long c = I.y_off + local;
    const int s0 = Q.rowoff[c], s1 = Q.rowmid[c], s2 = Q.rowoff[c + 1];
    RowAcc<R> A;
    if (local < I.n_c) {
        if (!(parts & RTBTE_EPH)) return 0.0;
        item_sum<R>(Q, s0, s2, A);
        return -A.value();
    }
    if (parts & RTBTE_PHE) item_sum<R>(Q, s0, s1, A);
    if (parts & RTBTE_PHPH) item_sum<R>(Q, s1, s2, A);
    return -A.value();
}

// Store component value v of row `local` into the population copies read by the RHS.
template <class R>
__device__ __forceinline__ void write_pops(const RowParams &Q, const InstDev &I, long long local, R v) {
    if (local < I.n_c) {
        reinterpret_cast<R *>(Q.popf)[I.f_off + local] = v;
        return;
    }
    const int p = (int)local - I.n_c, nu = p / I.N_q;  // (32-bit: n_ph is an int)
    reinterpret_cast<R *>(Q.popN)[I.N_off + (long long)nu * I.N_q_pad + (p - nu * I.N_q)] = v;
    if (I.M > 0) {
        const int a = Q.compact[I.compact_base + p];
        if (a >= 0) reinterpret_cast<R *>(Q.popP)[I.P_off + a] = v;
    }
}

}  // namespace rtbte
