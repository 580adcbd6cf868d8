// step.cuh -- device code of one attempted step of an explicit RK method (Methods B): the stage
// combination of a row, fixed-order block sums and the step-size controller.  Used by the launch
// sequence of integrate.cu and by the one-launch attempt loop of small instances (small.cu), whose
// results are therefore the same.
#pragma once

#include "internal.cuh"
#include "rows.cuh"

namespace rtbte {

namespace {

constexpr int kRedThreads = 256;

struct StageArgs {
    Tableau T;
    CtlParams cp;
    Ctl *ctl;  // one controller per instance
    double *Y0, *Y1, *K;
    const double *forcing;
    double *wsq;  // per-row squared weighted error of the last stage
    unsigned long long *range;  // per instance: rows of the attempted state out of range
    long long n;
    unsigned parts;
    int stage;         // -1: populations <- y; 0..S-1: combine stage `stage`
    int respect_done;  // inside an attempt sequence: skip instances whose integration is done
    int batched;       // several instances: rows visited by row blocks of active instances only
};

__device__ __forceinline__ double atol_of(const CtlParams &cp, const InstDev &I, long long local) {
    return local < I.n_c ? cp.atol_c : cp.atol_ph;
}

// The next stage's value of a row after stage i < S - 1: y + h sum_j A_{i+1,j} k_j, k_j = K(j).
template <class KAt> __device__ __forceinline__ double stage_next(const Tableau &T, int i, double h, double y, KAt K) {
    double acc = 0.0;
    for (int j = 0; j <= i; ++j) acc += T.A[i + 1][j] * K(j);
    return y + h * acc;
}

// The row's new state after the last stage, its squared weighted error (x2; not a number where the
// state is not finite) and whether it lies outside its physical range (f in [0,1], N >= 0) by more
// than the absolute tolerance.
template <class KAt>
__device__ __forceinline__ double stage_last(const StageArgs &a, bool electron, double h, double y, KAt K, double *x2,
                                             bool *out) {
    double s1 = 0.0, s2 = 0.0;
    for (int j = 0; j < a.T.S; ++j) {
        const double kj = K(j);
        s1 += a.T.b[j] * kj;
        s2 += (a.T.b[j] - a.T.bt[j]) * kj;
    }
    const double ynew = y + h * s1;
    *out = electron ? (ynew < -a.cp.atol_c || ynew > 1.0 + a.cp.atol_c) : (ynew < -a.cp.atol_ph);
    *x2 = 0.0;
    if (a.T.has_emb) {  // error weight and weighted error in FP64 (step acceptance reads them)
        const double w = 1.0 / (a.cp.rtol * fabs(y) + (electron ? a.cp.atol_c : a.cp.atol_ph));
        const double x = h * s2 * w;
        *x2 = x * x;
    }
    if (!isfinite(ynew)) *x2 = __longlong_as_double(0x7ff8000000000000LL);
    return ynew;
}

template <class R>
__device__ __forceinline__ void stage_row(const RowParams &Q, const StageArgs &a, int ii, const InstDev &I, long long c) {
    const int i = a.stage;
    const Ctl *C = a.ctl + ii;
    const long long local = c - I.y_off;
    const double *y = C->cur ? a.Y1 : a.Y0;
    if (i < 0) {
        write_pops<R>(Q, I, local, y[c]);
        return;
    }
    double k = row_value<R>(Q, I, local, a.parts);
    if (a.forcing) k += a.forcing[c];
    a.K[(long long)i * a.n + c] = k;
    const double h = C->h_try;
    auto K = [&](int j) { return a.K[(long long)j * a.n + c]; };
    if (i < a.T.S - 1) {
        write_pops<R>(Q, I, local, (R)stage_next(a.T, i, h, y[c], K));
        return;
    }
    double x2;
    bool out;
    (C->cur ? a.Y0 : a.Y1)[c] = stage_last(a, local < I.n_c, h, y[c], K, &x2, &out);
    if (out && a.range) atomicAdd(a.range + ii, 1ULL);  // per attempt; counted if it is accepted
    a.wsq[c] = x2;
}

// Fixed-order sum of v[b .. b+n) by one block of at least kRedThreads threads, of which the first
// kRedThreads add: strided per-thread sums, a butterfly within each warp (both partners of a pair
// add the same two values, so every lane holds the same bits), then the warp sums in warp order.
// Every thread returns the sum.  COHERENT: v was written by other SMs during this kernel.
template <bool COHERENT = false>
__device__ double block_sum(const double *v, long long b, long long n) {
    __shared__ double ws[kRedThreads / 32];
    double acc = 0.0;
    if (threadIdx.x < kRedThreads) {
        for (long long r = threadIdx.x; r < n; r += kRedThreads) acc += COHERENT ? __ldcg(v + b + r) : v[b + r];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
    }
    __syncthreads();
    double r = 0.0;
    for (int w = 0; w < kRedThreads / 32; ++w) r += ws[w];
    __syncthreads();  // ws is free for the next call
    return r;
}

__device__ __forceinline__ void arm(Ctl *c) {
    double hk = c->h;
    c->last = 0;
    if (c->fixed) {  // classical fixed steps: last step ends exactly at t_out
        c->last = (c->steps + 1 >= c->max_steps) ? 1 : 0;
        c->h_try = c->last ? c->t_out - c->t : hk;
        return;
    }
    if (c->t + hk >= c->t_out) {
        hk = c->t_out - c->t;
        c->last = 1;
    }
    c->h_try = hk;
}

// Accept or reject an attempt and propose the next step (Eqs. wrms_norm, pid_controller), from the
// sum of the squared weighted errors of ni rows; nr rows were out of range.  By one whole warp.
__device__ __forceinline__ void control(Ctl *c, const CtlParams &cp, double sum, long long ni, unsigned long long nr) {
    const double eps = sqrt(sum / (double)ni);
    // logarithms of the three PID factors, one per lane, ahead of the scalar logic of thread 0:
    // FP64 transcendental functions are slow in a single thread on this GPU, and the three are
    // independent (lane 0: the floored error norm, lanes 1-2: the two previous ones)
    double lg = 0.0;
    if (threadIdx.x < 3) lg = log(threadIdx.x == 0 ? fmax(eps, 1e-10) : threadIdx.x == 1 ? c->eps1 : c->eps2);
    const double lg1 = __shfl_sync(0xffffffffu, lg, 1), lg2 = __shfl_sync(0xffffffffu, lg, 2);
    if (threadIdx.x != 0) return;
    const double lg0 = lg;
    c->attempts++;
    if (!isfinite(eps)) {
        c->status = RTBTE_E_NONFINITE;
        c->done = 1;
        return;
    }
    if (c->fixed) {
        c->cur ^= 1;
        c->t = c->last ? c->t_out : c->t + c->h_try;
        c->steps++;
        c->range_viol += (long long)nr;
        c->h_last = c->h_try;
        if (c->last) c->done = 1;
        else arm(c);
        return;
    }
    c->eps = eps;
    if (eps <= 1.0) {
        c->cur ^= 1;
        c->t = c->last ? c->t_out : c->t + c->h_try;
        c->steps++;
        c->range_viol += (long long)nr;
        const double e = eps > 1e-10 ? eps : 1e-10;
        // e^(-a1/p) eps1^(+-a2/p) eps2^(-a3/p) as one exponential of the lanes' logarithms
        double eta = exp(cp.x1 * lg0 + cp.x2 * lg1 + cp.x3 * lg2);
        eta *= cp.safety;
        double cap = c->first ? cp.growth_first : cp.growth;
        if (c->nef > 0 && cap > 1.0) cap = 1.0;
        if (eta > cap) eta = cap;
        double h = c->h_try * eta;
        if (cp.hmax > 0 && h > cp.hmax) h = cp.hmax;
        c->h = h;
        c->eps2 = c->eps1;
        c->eps1 = e;
        c->first = 0;
        c->nef = 0;
        c->h_last = c->h_try;
        if (c->t >= c->t_out) {
            c->done = 1;
            return;
        }
        if (!(c->t + h > c->t)) {  // the proposed step no longer advances time
            c->status = RTBTE_E_STEP_UNDERFLOW;
            c->done = 1;
            return;
        }
        if (c->steps - c->steps_base >= c->max_steps) {
            c->status = RTBTE_E_TOO_MANY_STEPS;
            c->done = 1;
            return;
        }
    } else {
        c->fails++;
        c->nef++;
        if (c->nef >= cp.max_nef) {
            c->status = RTBTE_E_ERR_TEST_FAIL;
            c->done = 1;
            return;
        }
        double eta = cp.safety * exp(cp.xf * lg0);  // eps^(-1/p); eps > 1 here, so lg0 = log(eps)
        if (eta < cp.etamin) eta = cp.etamin;
        if (eta > 1.0) eta = 1.0;
        if (c->nef >= cp.small_nef && eta > cp.etamxf) eta = cp.etamxf;
        const double h = c->h_try * eta;
        c->h = h;
        if (h < cp.hmin || !(c->t + h > c->t)) {
            c->status = RTBTE_E_STEP_UNDERFLOW;
            c->done = 1;
            return;
        }
    }
    arm(c);
}

}  // namespace

}  // namespace rtbte
