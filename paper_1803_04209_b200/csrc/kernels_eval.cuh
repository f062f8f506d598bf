// Evaluation of cutoff rules on recorded run-times (Sections 3, 3.1.1 and 4.1; Fig. 2 and Fig. 4):
// per SGD step the observed run-times are sorted, then
//   Omega(c) = c / x~_(c) for every c, its maximum and the cutoff that attains it (known in hindsight only),
//   the throughput of waiting for all workers, N / x~_(N),
//   the throughput and the duration x~_(c) of the step under each of M given cutoffs;
// over a whole trace: the best static cutoff (one c for all steps), and the "order" baseline -- the cutoff
// that maximises c / E[x~_(c)] with Elfving's normal-theory expectations from the running mean and
// deviation of everything observed before the step.
#pragma once
#include <cmath>

#include "common.cuh"
#include "kernels_sort.cuh"

namespace cutoff {

// The larger throughput and its cutoff; equal ones keep the larger cutoff.  Cutoff 0 = nothing.
__device__ __forceinline__ void better_cutoff(double& bv, int& bi, double ov, int oi) {
    if (oi != 0 && (bi == 0 || ov > bv || (ov == bv && oi > bi))) { bv = ov; bi = oi; }
}
__device__ __forceinline__ void warp_best_cutoff(double& bv, int& bi) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, bv, off);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
        better_cutoff(bv, bi, ov, oi);
    }
}

// Where position j of a sorted row sits in shared memory: lanes write E consecutive positions each, which would all fall into
// the same few banks without the gap after every 32.
__device__ __forceinline__ int row_at(int j) { return j + (j >> 5); }

// One sorted row in shared memory -> the step's scores, by WARPS warps of which this is warp `warp`; red_val, red_idx: WARPS
// entries of shared memory.  The divisions of a thread are independent (unrolled): one after the other they took longer than the sort.
template <int WARPS, typename Sync>
__device__ __forceinline__ void eval_sorted_row(const float* __restrict__ sorted, int N, int warp, int lane, Sync sync,
                                                double* red_val, int* red_idx, int64_t t, int64_t T,
                                                const int32_t* __restrict__ cutoffs, int M,
                                                int32_t* __restrict__ best_c, float* __restrict__ best,
                                                float* __restrict__ all, float* __restrict__ achieved,
                                                float* __restrict__ time_at) {
    // hindsight maximum of Omega(c) = c / x~_(c); ties go to the larger c
    const int tid = warp * 32 + lane;
    double bv = -INFINITY;
    int bi = 0;
#pragma unroll 8
    for (int j = tid; j < N; j += 32 * WARPS) {
        const double om = static_cast<double>(j + 1) / static_cast<double>(sorted[row_at(j)]);
        if (om >= bv) { bv = om; bi = j + 1; }
    }
    warp_best_cutoff(bv, bi);
    if (WARPS > 1) {
        if (lane == 0) { red_val[warp] = bv; red_idx[warp] = bi; }
        sync();
    }
    if (tid == 0) {
        for (int k = 1; k < WARPS; ++k) better_cutoff(bv, bi, red_val[k], red_idx[k]);
        best_c[t] = bi;
        best[t] = static_cast<float>(bv);
        all[t] = static_cast<float>(static_cast<double>(N) / static_cast<double>(sorted[row_at(N - 1)]));
    }
    for (int m = tid; m < M; m += 32 * WARPS) {
        int c = cutoffs[static_cast<int64_t>(m) * T + t];
        c = c < 1 ? 1 : (c > N ? N : c);
        const float x_c = sorted[row_at(c - 1)];
        achieved[static_cast<int64_t>(m) * T + t] = static_cast<float>(static_cast<double>(c) / static_cast<double>(x_c));
        time_at[static_cast<int64_t>(m) * T + t] = x_c;
    }
    sync();
}

// N <= 1024: one warp per step, E = P / 32 keys per lane.  Few warps per CTA: a trace has some hundred steps, and a step's
// sort is latency, so they are spread over the SMs (500 steps: 125 CTAs).
constexpr int kEvalWarps = 4;

template <int E>
__global__ void __launch_bounds__(kEvalWarps * 32) k_eval_trace_warp(const float* __restrict__ trace, int64_t T, int N, int ld,
                                                                      const int32_t* __restrict__ cutoffs, int M,
                                                                      int32_t* __restrict__ best_c, float* __restrict__ best,
                                                                      float* __restrict__ all, float* __restrict__ achieved,
                                                                      float* __restrict__ time_at,
                                                                      float* __restrict__ sorted_out) {
    __shared__ float rows[kEvalWarps][33 * E];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    launch_dependents();
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * kEvalWarps + warp; t < T; t += static_cast<int64_t>(gridDim.x) * kEvalWarps) {
        const float* src = trace + t * ld;
        float v[E];
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int e = r * 32 + lane;
            v[r] = e < N ? src[e] : INFINITY;
        }
        warp_bitonic_sort<float, E>(v, lane);
#pragma unroll
        for (int r = 0; r < E; ++r) rows[warp][row_at(lane * E + r)] = v[r];
        __syncwarp();
        if (sorted_out)
            for (int j = lane; j < N; j += 32) sorted_out[t * N + j] = rows[warp][row_at(j)];
        eval_sorted_row<1>(rows[warp], N, 0, lane, [] { __syncwarp(); }, nullptr, nullptr, t, T, cutoffs, M,
                        best_c, best, all, achieved, time_at);
    }
}

// 1024 < N <= 4096: a CTA of WPR warps per step.
template <int WPR>
__global__ void __launch_bounds__(WPR * 32) k_eval_trace_cta(const float* __restrict__ trace, int64_t T, int N, int ld,
                                                              const int32_t* __restrict__ cutoffs, int M,
                                                              int32_t* __restrict__ best_c, float* __restrict__ best,
                                                              float* __restrict__ all, float* __restrict__ achieved,
                                                              float* __restrict__ time_at, float* __restrict__ sorted_out) {
    __shared__ float xch[WPR * 33 * 32];
    __shared__ double red_val[WPR];
    __shared__ int red_idx[WPR];
    constexpr int E = 32, T_ = WPR * 32;
    launch_dependents();
    for (int64_t t = blockIdx.x; t < T; t += gridDim.x) {
        const float* src = trace + t * ld;
        float v[E];
#pragma unroll
        for (int r = 0; r < E; ++r) {
            const int e = r * T_ + threadIdx.x;
            v[r] = e < N ? src[e] : INFINITY;
        }
        cta_bitonic_sort<float, WPR>(v, xch);
        __syncthreads();                                   // the exchange buffer is free: it now holds the sorted row
#pragma unroll
        for (int r = 0; r < E; ++r) xch[row_at(threadIdx.x * E + r)] = v[r];
        __syncthreads();
        if (sorted_out)
            for (int j = threadIdx.x; j < N; j += T_) sorted_out[t * N + j] = xch[row_at(j)];
        eval_sorted_row<WPR>(xch, N, threadIdx.x >> 5, threadIdx.x & 31, [] { __syncthreads(); }, red_val, red_idx, t, T, cutoffs, M,
                        best_c, best, all, achieved, time_at);
    }
}

// Best static cutoff: argmax_c sum_t c / x~_(c)(t) over the sorted rows of a trace (ties -> larger c).  32 columns per CTA,
// 32 slices of steps each (slice s adds steps s, s + 32, ..), the slices then added in order; a second kernel of one CTA takes
// the argmax.  (One CTA for all columns, a thread adding 500 quotients one after the other, took 0.3 ms.)
constexpr int kStaticSlices = 32;

__global__ void __launch_bounds__(32 * kStaticSlices) k_static_totals(const float* __restrict__ sorted, int64_t T, int N,
                                                                      double* __restrict__ totals) {
    __shared__ double red[kStaticSlices][32];
    dependency_wait();
    launch_dependents();
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (j < N) {
#pragma unroll 4
        for (int64_t t = slice; t < T; t += kStaticSlices) s += static_cast<double>(j + 1) / static_cast<double>(sorted[t * N + j]);
    }
    red[slice][lane] = s;
    __syncthreads();
    if (slice == 0 && j < N) {
        double total = 0.0;
#pragma unroll
        for (int k = 0; k < kStaticSlices; ++k) total += red[k][lane];
        totals[j] = total;
    }
}
__global__ void __launch_bounds__(1024) k_best_static(const double* __restrict__ totals, int N, int32_t* __restrict__ static_c) {
    __shared__ double val[32];
    __shared__ int idx[32];
    dependency_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double bv = -INFINITY;
    int bi = 0;
    for (int j = threadIdx.x; j < N; j += 1024) better_cutoff(bv, bi, totals[j], j + 1);
    warp_best_cutoff(bv, bi);
    if (lane == 0) { val[warp] = bv; idx[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
        bv = val[lane];
        bi = idx[lane];
        warp_best_cutoff(bv, bi);
        if (lane == 0) *static_c = bi;
    }
}

// ---- the "order" baseline (Fig. 4; Elfving's formula, Section 3.1.1) ----------------------------------------
// Per-step sums of x and x^2 in double, fixed order: a warp per step.  The CTAs behind those of the steps form the normal
// quantiles q_j = Phi^-1((j - pi/8) / (n - pi/4 + 1)), j = 1..n (the standard form of the fraction).
constexpr int kMomentWarps = 8;

__global__ void __launch_bounds__(kMomentWarps * 32) k_step_moments(const float* __restrict__ trace, int64_t T, int N, int ld,
                                                                    double* __restrict__ sum1, double* __restrict__ sum2,
                                                                    double* __restrict__ q, unsigned step_ctas) {
    launch_dependents();
    if (blockIdx.x >= step_ctas) {
        const int j = (blockIdx.x - step_ctas) * kMomentWarps * 32 + threadIdx.x;
        if (j >= N) return;
        const double pi = 3.14159265358979323846;
        q[j] = normcdfinv((static_cast<double>(j + 1) - pi / 8.0) / (static_cast<double>(N) - pi / 4.0 + 1.0));
        return;
    }
    const int lane = threadIdx.x & 31;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kMomentWarps + (threadIdx.x >> 5);
    if (t >= T) return;
    double a = 0.0, b = 0.0;
#pragma unroll 8
    for (int j = lane; j < N; j += 32) {
        const double v = static_cast<double>(trace[t * ld + j]);
        a += v;
        b += v * v;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (lane == 0) { sum1[t] = a; sum2[t] = b; }
}

// In place: sums of step t -> mean and deviation of everything observed in steps 0 .. t-1 (exclusive running sums).  One
// CTA, 1024 steps at a time: a scan within each warp, then over the warps, then the running total of the steps before.
__global__ void __launch_bounds__(1024) k_running_moments(int64_t T, int N, double* __restrict__ sum1, double* __restrict__ sum2) {
    __shared__ double w1[32], w2[32];
    dependency_wait();
    launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double before1 = 0.0, before2 = 0.0;
    for (int64_t t0 = 0; t0 < T; t0 += 1024) {
        const int64_t t = t0 + threadIdx.x;
        double a = t < T ? sum1[t] : 0.0, b = t < T ? sum2[t] : 0.0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const double oa = __shfl_up_sync(0xffffffffu, a, off), ob = __shfl_up_sync(0xffffffffu, b, off);
            if (lane >= off) { a += oa; b += ob; }
        }
        if (lane == 31) { w1[warp] = a; w2[warp] = b; }
        // what the lanes before this one have, and not its own sum minus its own value: that would leave the rounding of a far
        // outlier in the moments of the very step that is to be decided without it
        a = __shfl_up_sync(0xffffffffu, a, 1);
        b = __shfl_up_sync(0xffffffffu, b, 1);
        if (lane == 0) a = b = 0.0;
        __syncthreads();
        double pa = before1, pb = before2, all1 = before1, all2 = before2;
        for (int k = 0; k < 32; ++k) {
            if (k < warp) { pa += w1[k]; pb += w2[k]; }
            all1 += w1[k];
            all2 += w2[k];
        }
        if (t < T) {
            const double count = static_cast<double>(t) * static_cast<double>(N);
            const double sum_a = pa + a, sum_b = pb + b;
            const double mu = t > 0 ? sum_a / count : 0.0;
            const double var = t > 0 ? sum_b / count - mu * mu : 0.0;
            sum1[t] = mu;
            sum2[t] = sqrt(var > 0.0 ? var : 0.0);
        }
        before1 = all1;
        before2 = all2;
        __syncthreads();
    }
}

// Cutoff of step t: argmax_c c / (mu_t + sigma_t q_c) over the c with a positive expectation; ties -> larger c;
// c = N for step 0 (nothing observed yet) and when no c is admissible.  One warp per step.
__global__ void __launch_bounds__(256) k_order_cutoffs(int64_t T, int N, const double* __restrict__ mu,
                                                        const double* __restrict__ sigma, const double* __restrict__ q,
                                                        int32_t* __restrict__ cutoffs) {
    dependency_wait();
    const int lane = threadIdx.x & 31;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
    if (t >= T) return;
    double bv = -INFINITY;
    int bi = 0;
    if (t > 0) {
        const double m = mu[t], s = sigma[t];
#pragma unroll 8
        for (int j = lane; j < N; j += 32) {
            const double e = m + s * q[j];
            if (e > 0.0) {
                const double om = static_cast<double>(j + 1) / e;
                if (om >= bv) { bv = om; bi = j + 1; }
            }
        }
    }
    warp_best_cutoff(bv, bi);
    if (lane == 0) cutoffs[t] = bi == 0 ? N : bi;
}

}  // namespace cutoff
