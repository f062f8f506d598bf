// Observation handling, the guide q_phi, the transition and the first emission layer, and the
// fp32 FMA version of the emission output layer.
#pragma once
#include "common.cuh"
#include "half_operand.cuh"
#include "rng.cuh"
#include "tile_product.cuh"

namespace cutoff {

// ---------------------------------------------------------------------------------------------
// push: obs <- obs U r_w for one whole step (Algorithm 1), plus the normaliser of Section 3.1.3
// (twice the mean of the first fixed-lag window).  One CTA; the sum is a fixed-order tree.
// ---------------------------------------------------------------------------------------------
constexpr int kPushThreads = 1024, kPushPer = 4;             // N <= 4096: every run-time is read once, into a register

// src may be pinned host memory (read over the bus: one round trip, less than a copy and the launch behind it).  host_state: null = do
// not report.
__global__ void __launch_bounds__(kPushThreads) k_push(const float* __restrict__ src, float* __restrict__ ring,
                                                       DevState* st, int N, int W, DevState* host_state) {
    __shared__ double red[kPushThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    dependency_wait();
    launch_dependents();
    float v[kPushPer];
#pragma unroll
    for (int i = 0; i < kPushPer; ++i) v[i] = tid + i * kPushThreads < N ? src[tid + i * kPushThreads] : 1.0f;
    const uint32_t pushes = st->push_count;
    int bad = 0;
#pragma unroll
    for (int i = 0; i < kPushPer; ++i)
        if (!(v[i] > 0.0f) || !isfinite(v[i])) bad = 1;
    if (tid == 0 && (st->error_flags & kErrNoFinisher)) bad = 1;   // raised by the imputation that precedes this push
    bad = __syncthreads_or(bad);
    if (bad) {
        if (tid == 0) {
            st->error_flags |= kErrBadValue;
            publish_state(st, host_state);
        }
        return;
    }
    float* dst = ring + static_cast<size_t>(pushes % W) * N;
#pragma unroll
    for (int i = 0; i < kPushPer; ++i)
        if (tid + i * kPushThreads < N) dst[tid + i * kPushThreads] = v[i];
    if (pushes < static_cast<uint32_t>(W)) {           // the normaliser is still being formed
        double s = 0.0;
#pragma unroll
        for (int i = 0; i < kPushPer; ++i)
            if (tid + i * kPushThreads < N) s += static_cast<double>(v[i]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) red[warp] = s;
        __syncthreads();
        if (warp == 0) {
            s = red[lane];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (lane == 0) {
                const double total = st->norm_sum + s;
                st->norm_sum = total;
                if (pushes + 1 == static_cast<uint32_t>(W)) {
                    const double scale = 2.0 * total / (static_cast<double>(N) * W);
                    st->scale = static_cast<float>(scale);
                    st->inv_scale = static_cast<float>(1.0 / scale);
                }
            }
        }
    }
    if (tid == 0) {
        st->push_count = pushes + 1;
        publish_state(st, host_state);
    }
}

// ---------------------------------------------------------------------------------------------
// Censored run-times (Section 4.2): a worker that was killed at the cutoff gets a draw from its own
// predictive distribution of this step, left-truncated at the cutoff time (the largest run-time
// that was observed).  The predictive distribution is the Monte-Carlo one: column j of the sample
// matrix of the last decision.  The draws are iid, so the first one above the threshold, scanning
// cyclically from a start that does not depend on their values (Philox word 0 of counter
// (worker, 0, 0x300, decision number) modulo S), is an exact draw from the truncated distribution;
// if there is none the threshold itself is used.
// A warp per censored worker, the workers j = b, b + CTAs, .. in CTA b.  A warp's load touches 32 rows, so what bounds one CTA is
// its SM's load unit: N=158, S=2048 took 32 us in one CTA, 14 us in 16.  More CTAs would each read the run-times and the
// mask over the bus for little (20 KB at N=4096).
// ---------------------------------------------------------------------------------------------
constexpr int kImputeThreads = 512, kImputeCtas = 16;
constexpr uint32_t kStreamImpute = 0x300u;

// src and censored may be pinned host memory; stage receives the completed vector.  Draws above the threshold are rare, so a
// column is mostly read to its end: kImputeAhead blocks of 32 draws are in flight at a time.
constexpr int kImputeAhead = 8;

__global__ void __launch_bounds__(kImputeThreads) k_impute(const float* __restrict__ src, const uint8_t* __restrict__ censored,
                                                            float* __restrict__ stage, const float* __restrict__ x, int ldx, int S, int N,
                                                            DevState* __restrict__ st, NoiseKey key) {
    __shared__ float red[kImputeThreads / 32];
    __shared__ uint16_t mine[4096];                     // this CTA's censored workers, in any order
    __shared__ int n_mine;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) n_mine = 0;
    __syncthreads();
    float m = -INFINITY;
    for (int j = threadIdx.x; j < N; j += kImputeThreads) {
        const uint8_t c = censored[j];
        const float v = src[j];
        if (!c) m = fmaxf(m, v);
        if (j % gridDim.x != blockIdx.x) continue;
        if (c) mine[atomicAdd(&n_mine, 1)] = static_cast<uint16_t>(j);
        else stage[j] = v;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if (lane == 0) red[warp] = m;
    __syncthreads();
    m = red[lane % (kImputeThreads / 32)];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    const float threshold = m;
    if (!(threshold > -INFINITY)) {
        // nobody finished, so there is no cutoff time to truncate at: flag the vector; the push kernel that
        // follows sees the flag and leaves the window untouched
        if (blockIdx.x == 0 && threadIdx.x == 0) st->error_flags |= kErrNoFinisher;
        return;
    }
    const float scale = st->scale;
    const uint32_t step = st->step;
    for (int t = warp; t < n_mine; t += kImputeThreads / 32) {
        const int j = mine[t];
        const uint32_t start = philox4x32_10(static_cast<uint32_t>(j), 0u, kStreamImpute, step, key.seed_lo, key.seed_hi).x %
                               static_cast<uint32_t>(S);
        float value = threshold;
        bool found = false;
        for (int base = 0; base < S && !found; base += 32 * kImputeAhead) {
            float v[kImputeAhead];
#pragma unroll
            for (int u = 0; u < kImputeAhead; ++u) {
                const int i = base + 32 * u + lane;
                v[u] = -INFINITY;
                if (i < S) {
                    uint32_t k = start + static_cast<uint32_t>(i);
                    if (k >= static_cast<uint32_t>(S)) k -= static_cast<uint32_t>(S);
                    v[u] = x[static_cast<size_t>(k) * ldx + j] * scale;
                }
            }
#pragma unroll
            for (int u = 0; u < kImputeAhead; ++u) {
                const uint32_t hit = __ballot_sync(0xffffffffu, v[u] > threshold);
                if (hit && !found) {
                    value = __shfl_sync(0xffffffffu, v[u], __ffs(hit) - 1);
                    found = true;
                }
            }
        }
        if (lane == 0) stage[j] = value;
    }
}

// ---------------------------------------------------------------------------------------------
// Encoder, part 1: input projections of both RNNs, cached per ring slot,
//   R[dir][slot][i] = sum_j Wx_dir[i][j] * x_slot[j]          (raw seconds: the normaliser is applied by part 2,
//                                                              so a slot's projection never has to be redone)
// Four warps per hidden unit, a quarter of the workers each; the weight row is read once for all slots of the launch, into
// registers, before the kernel waits for the push in front of it.  (One warp per row with its loads behind the wait: 20 us for
// N = 2175, whose rows are not aligned, and for N = 4096, H = 512; 5 us for N = 1024.)
// newest_only = 1: only the slot of the vector pushed last (launched after every push);
// newest_only = 0: every slot (after the ring or the weights were replaced).  Both run the same
// arithmetic per slot, so a cached projection equals a recomputed one bit for bit.
// ---------------------------------------------------------------------------------------------
constexpr int kProjRows = 2, kProjSplit = 4, kProjThreads = kProjRows * kProjSplit * 32;
constexpr int kProjPer = 4096 / kProjSplit / 32;              // columns per lane at most

template <bool VEC>          // VEC: N is a multiple of 4, rows and ring slots start on 16 bytes
__device__ __forceinline__ void load_quarter(const float* __restrict__ row, int c0, int c1, int lane, float (&v)[kProjPer]) {
    if (VEC) {
#pragma unroll
        for (int i = 0; i < kProjPer; i += 4) {
            const int c = c0 + i * 32 + 4 * lane;
            const float4 q = c < c1 ? *reinterpret_cast<const float4*>(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[i] = q.x; v[i + 1] = q.y; v[i + 2] = q.z; v[i + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kProjPer; ++i) {
            const int c = c0 + i * 32 + lane;
            v[i] = c < c1 ? row[c] : 0.f;
        }
    }
}

template <bool VEC>
__global__ void __launch_bounds__(kProjThreads) k_enc_proj(ModelDev m, const float* __restrict__ ring,
                                                            const DevState* __restrict__ st, int newest_only,
                                                            float* __restrict__ proj /*[2][W slots][H]*/) {
    __shared__ float red[kProjRows][kProjSplit];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = warp % kProjSplit, r = warp / kProjSplit;
    const int i = blockIdx.x * kProjRows + r, dir = blockIdx.y;
    const int len = (m.N + 4 * kProjSplit - 1) / (4 * kProjSplit) * 4, c0 = part * len, c1 = min(c0 + len, m.N);
    float w[kProjPer], x[kProjPer];
    load_quarter<VEC>((dir ? m.Wxb : m.Wxf) + static_cast<size_t>(min(i, m.H - 1)) * m.N, c0, c1, lane, w);
    dependency_wait();
    launch_dependents();
    const int slot_first = newest_only ? static_cast<int>((st->push_count + m.W - 1) % m.W) : 0;
    const int n_slots = newest_only ? 1 : m.W;
    for (int s = 0; s < n_slots; ++s) {
        load_quarter<VEC>(ring + static_cast<size_t>(slot_first + s) * m.N, c0, c1, lane, x);
        float acc[4] = {};
#pragma unroll
        for (int k = 0; k < kProjPer; ++k) acc[k & 3] = fmaf(w[k], x[k], acc[k & 3]);
        float v = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) red[r][part] = v;
        __syncthreads();
        if (part == 0 && lane == 0 && i < m.H)
            proj[(static_cast<size_t>(dir) * m.W + slot_first + s) * m.H + i] = (red[r][0] + red[r][1]) + (red[r][2] + red[r][3]);
        __syncthreads();
    }
}

// Input projection of window position t (0 = oldest) for hidden unit i: the cached raw projection of the ring slot
// that holds position t, scaled by 1 / s (Section 3.1.3: observations are divided by twice the mean of the first
// window), plus the bias.
__device__ __forceinline__ float window_projection(const ModelDev& m, const float* __restrict__ proj, int dir, int t, int i,
                                                   uint32_t pushes, float inv_scale) {
    const int slot = static_cast<int>((pushes + static_cast<uint32_t>(t)) % static_cast<uint32_t>(m.W));
    return fmaf(proj[(static_cast<size_t>(dir) * m.W + slot) * m.H + i], inv_scale, (dir ? m.bb : m.bf)[i]);
}

// ---------------------------------------------------------------------------------------------
// Encoder, part 2: the two recurrences (h_left forward, h_right backward; Section 3.1.3).
//   a_t = relu(P[0][t] + Whf a_{t-1}),  b_t = relu(P[1][t] + Whb b_{t+1}).
// One CTA per direction; the state lives in shared memory.  hlr[dir][t][i] is written.
// ---------------------------------------------------------------------------------------------
constexpr int kRnnThreads = 1024;

__global__ void __launch_bounds__(kRnnThreads) k_enc_rnn(ModelDev m, const float* __restrict__ proj,
                                                          const DevState* __restrict__ st,
                                                          float* __restrict__ hlr /*[2][W][H]*/) {
    extern __shared__ float sm_rnn[];
    float* state = sm_rnn;
    float* next = sm_rnn + m.H;
    const int dir = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* Wh = dir ? m.Whb : m.Whf;
    const float* init = dir ? m.b0 : m.a0;
    dependency_wait();
    launch_dependents();
    const uint32_t pushes = st->push_count;
    const float inv_scale = st->inv_scale;
    for (int i = threadIdx.x; i < m.H; i += kRnnThreads) state[i] = init[i];
    __syncthreads();
    for (int s = 0; s < m.W; ++s) {
        const int t = dir ? (m.W - 1 - s) : s;
        for (int i = warp; i < m.H; i += kRnnThreads / 32) {
            const float* wrow = Wh + static_cast<size_t>(i) * m.H;
            float acc = 0.0f;
            for (int j = lane; j < m.H; j += 32) acc = fmaf(wrow[j], state[j], acc);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (lane == 0) next[i] = fmaxf(acc + window_projection(m, proj, dir, t, i, pushes, inv_scale), 0.0f);
        }
        __syncthreads();
        float* out = hlr + (static_cast<size_t>(dir) * m.W + t) * m.H;
        for (int i = threadIdx.x; i < m.H; i += kRnnThreads) {
            const float v = next[i];
            state[i] = v;
            out[i] = v;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------
// Encoder, part 2, latency version for H <= 128: the recurrence matrix never leaves the registers.
// One CTA per direction, 4 threads per hidden unit; thread (i, q) owns columns q*H/4 .. of row i.
// The state is double-buffered in shared memory, so a step costs one __syncthreads.
// ---------------------------------------------------------------------------------------------
template <int HQ>   // HQ = H / 4 <= 32
__global__ void __launch_bounds__(16 * HQ) k_enc_rnn_resident(ModelDev m, const float* __restrict__ wh_threads,
                                                              const float* __restrict__ proj,
                                                              const DevState* __restrict__ dev_state,
                                                              float* __restrict__ hlr /*[2][W][H]*/) {
    static_assert(HQ <= 32, "a thread keeps its HQ weights in registers");
    constexpr int H = 4 * HQ, T = 16 * HQ, PAD = HQ + 4;
    extern __shared__ __align__(16) float sm_rr[];
    float* state = sm_rr;                         // [2][4][PAD]
    float* sproj = state + 2 * 4 * PAD;           // [W][H]
    const int dir = blockIdx.x;
    const int t = threadIdx.x, i = t >> 2, q = t & 3;
    // wh_threads holds both recurrence matrices regrouped per thread, [dir][j4][thread][4]: the j4-th group of
    // four weights of thread (i, q) is Wh[i][q*HQ + 4*j4 ..], so that consecutive threads read consecutive 16 bytes
    const float4* Wh = reinterpret_cast<const float4*>(wh_threads) + static_cast<size_t>(dir) * (HQ / 4) * T;
    const float* init = dir ? m.b0 : m.a0;
    float w[HQ];
#pragma unroll
    for (int j4 = 0; j4 < HQ / 4; ++j4) {
        const float4 v = Wh[static_cast<size_t>(j4) * T + t];
        w[4 * j4 + 0] = v.x; w[4 * j4 + 1] = v.y; w[4 * j4 + 2] = v.z; w[4 * j4 + 3] = v.w;
    }
    if (t < H) state[(t / HQ) * PAD + (t % HQ)] = init[t];
    dependency_wait();            // up to here: weights.  The projections and the device state are earlier kernels'
    launch_dependents();
    {
        const uint32_t pushes = dev_state->push_count;
        const float inv_scale = dev_state->inv_scale;
        for (int idx = t; idx < m.W * H; idx += T) sproj[idx] = window_projection(m, proj, dir, idx / H, idx % H, pushes, inv_scale);
    }
    __syncthreads();
    int cur = 0;
    for (int s = 0; s < m.W; ++s) {
        const int tt = dir ? (m.W - 1 - s) : s;
        const float* st = state + cur * 4 * PAD + q * PAD;
        float acc = 0.0f;
#pragma unroll
        for (int j4 = 0; j4 < HQ / 4; ++j4) {
            const float4 v = *reinterpret_cast<const float4*>(st + 4 * j4);
            acc = fmaf(w[4 * j4 + 0], v.x, acc); acc = fmaf(w[4 * j4 + 1], v.y, acc);
            acc = fmaf(w[4 * j4 + 2], v.z, acc); acc = fmaf(w[4 * j4 + 3], v.w, acc);
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (q == 0) {
            const float v = fmaxf(acc + sproj[tt * H + i], 0.0f);
            state[(cur ^ 1) * 4 * PAD + (i / HQ) * PAD + (i % HQ)] = v;
            hlr[(static_cast<size_t>(dir) * m.W + tt) * H + i] = v;
        }
        __syncthreads();
        cur ^= 1;
    }
}

inline size_t enc_rnn_resident_smem_floats(int H, int W) {
    return 2 * 4 * (H / 4 + 4) + static_cast<size_t>(W) * H;
}

// ---------------------------------------------------------------------------------------------
// Encoder, part 2, for multiples of 32 up to 608 that k_enc_rnn_resident does not serve: the recurrence matrix of a direction is split over the shared
// memories of a cluster of 8 CTAs (H/8 rows each), so it is read from global memory once.  Every CTA
// keeps the whole state (double-buffered); after a step each row's new value is written into the next
// state buffer of all 8 CTAs through distributed shared memory, and one cluster barrier (a hardware
// barrier: no thread leaves before the last step) separates the steps.
// 8 threads per row: thread p of a row takes the 16-byte column chunks p, p+8, ...; rows are padded by
// 8 floats so that the four rows of a warp fall into different banks.  Grid: 16 CTAs (2 clusters).
// ---------------------------------------------------------------------------------------------
constexpr int kRnnClusterSize = 8;

inline size_t enc_rnn_cluster_smem_floats(int H, int W) {
    const int R = H / kRnnClusterSize;
    return static_cast<size_t>(R) * (H + 8) + 2 * static_cast<size_t>(H) + static_cast<size_t>(W) * R;
}

__global__ void __cluster_dims__(kRnnClusterSize, 1, 1) __launch_bounds__(1024)
k_enc_rnn_cluster(ModelDev m, const float* __restrict__ proj, const DevState* __restrict__ dev_state,
                  float* __restrict__ hlr /*[2][W][H]*/) {
    extern __shared__ __align__(16) float sm_rc[];
    const int H = m.H, W = m.W, R = H / kRnnClusterSize, ldw = H + 8;
    float* sW = sm_rc;                         // [R][ldw]  rows rank*R .. of the recurrence matrix
    float* state = sW + static_cast<size_t>(R) * ldw;      // [2][H]
    float* sproj = state + 2 * H;              // [W][R]
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int dir = blockIdx.x / kRnnClusterSize;
    const int row = threadIdx.x >> 3, part = threadIdx.x & 7;          // blockDim.x = 8 R
    const int i = static_cast<int>(rank) * R + row;                    // hidden unit of this thread's row
    const float* Wh = (dir ? m.Whb : m.Whf) + static_cast<size_t>(rank) * R * H;
    const float* init = dir ? m.b0 : m.a0;
    // R * H / 4 = blockDim.x * H / 32 chunks of 16 bytes: every thread moves H / 32 of them, eight loads in flight
    for (int base = 0; base < R * (H / 4); base += 8 * blockDim.x) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int idx = base + u * blockDim.x + threadIdx.x;
            if (idx < R * (H / 4)) v[u] = *reinterpret_cast<const float4*>(Wh + static_cast<size_t>(idx / (H / 4)) * H + 4 * (idx % (H / 4)));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int idx = base + u * blockDim.x + threadIdx.x;
            if (idx < R * (H / 4)) *reinterpret_cast<float4*>(sW + static_cast<size_t>(idx / (H / 4)) * ldw + 4 * (idx % (H / 4))) = v[u];
        }
    }
    for (int k = threadIdx.x; k < H; k += blockDim.x) state[k] = init[k];
    dependency_wait();            // up to here: weights.  The projections and the device state are earlier kernels'
    launch_dependents();          // the chain kernel may set itself up on the SMs this kernel leaves free
    {
        const uint32_t pushes = dev_state->push_count;
        const float inv_scale = dev_state->inv_scale;
        for (int idx = threadIdx.x; idx < W * R; idx += blockDim.x)
            sproj[idx] = window_projection(m, proj, dir, idx / R, static_cast<int>(rank) * R + idx % R, pushes, inv_scale);
    }
    // every CTA of the cluster has started and initialised its buffers before anyone writes into them
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    const float* wrow = sW + static_cast<size_t>(row) * ldw;
    int cur = 0;
    for (int s = 0; s < W; ++s) {
        const int t = dir ? (W - 1 - s) : s;
        const float* st = state + cur * H;
        float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;      // four chains: the sum's order is fixed all the same
        for (int c = part; c < H / 4; c += 8) {
            const float4 w = *reinterpret_cast<const float4*>(wrow + 4 * c);
            const float4 v = *reinterpret_cast<const float4*>(st + 4 * c);
            a0 = fmaf(w.x, v.x, a0); a1 = fmaf(w.y, v.y, a1);
            a2 = fmaf(w.z, v.z, a2); a3 = fmaf(w.w, v.w, a3);
        }
        float acc = (a0 + a1) + (a2 + a3);
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        acc += __shfl_xor_sync(0xffffffffu, acc, 4);
        const float v = fmaxf(acc + sproj[t * R + row], 0.0f);
        // thread `part` of the row delivers the new value to CTA `part` of the cluster
        {
            const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(state + (cur ^ 1) * H + i));
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(static_cast<uint32_t>(part)));
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
        }
        if (part == 0) hlr[(static_cast<size_t>(dir) * W + t) * H + i] = v;
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        cur ^= 1;
    }
}

// ---------------------------------------------------------------------------------------------
// Per-sample chain: guide steps over the window, transition, first emission layer.
//
// SPL samples are worked on by a group of G = D/4 adjacent lanes.  Lane g of the group owns, of
// every hidden layer, the units i = 4(g + G m) .. 4(g + G m) + 3 (m = 0, 1, ...) and the four
// latent dimensions 4g..4g+3 (exactly one Philox call per noise stream and sample).  Every lane
// keeps the whole latent vector of its samples in registers.  A layer pair
//      hidden = act(A z + a),   out += B hidden
// is evaluated four hidden units at a time as two small outer-product updates: A is staged
// transposed ([D][H]) and B as it is ([out][H]), so that the four weights a lane needs for one
// input or output dimension are one 16-byte shared-memory load, which the G lanes of a group read
// from consecutive addresses and all groups of a warp read as a broadcast.  Partial outputs are
// summed over the group with xor-shuffles.  Each weight read serves all SPL samples of the lane.
// ---------------------------------------------------------------------------------------------
template <int D> struct ChainShape {
    static constexpr int G = D / 4;                   // lanes per group
    static constexpr int SPL = D <= 16 ? 2 : 1;       // samples per lane
    // threads of the phase-staged kernel: its shared memory allows one CTA per SM at D = 32, so that CTA is wide
    static constexpr int kThreads = D <= 16 ? 128 : 384;
    static constexpr int kSamplesPerCta = kThreads / G * SPL;
};

__device__ __forceinline__ float softplusf(float x) { return x > 20.0f ? x : log1pf(expf(x)); }

// tanh(x) = 1 - 2 / (exp(2x) + 1) with the hardware exp2 and reciprocal: absolute error below 3e-7.
__device__ __forceinline__ float tanh_fast(float x) {
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * 2.8853900817779268f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(e + 1.0f));
    return fmaf(-2.0f, r, 1.0f);
}

__device__ __forceinline__ float round_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

__device__ __forceinline__ void stage_vector(float* dst, const float* __restrict__ src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// hidden[s][c] = sum_k A^T[k][i0 + c] * z[s][k] + bias[i0 + c]       (A^T staged as [D][H])
template <int D, int SPL>
__device__ __forceinline__ void hidden_block(const float* sAT, const float* sbias, int H, int i0,
                                             const float (&z)[SPL][D], float (&hid)[SPL][4]) {
    const float4 b = lds4(sbias + i0);
#pragma unroll
    for (int s = 0; s < SPL; ++s) { hid[s][0] = b.x; hid[s][1] = b.y; hid[s][2] = b.z; hid[s][3] = b.w; }
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float4 w = lds4(sAT + k * H + i0);
#pragma unroll
        for (int s = 0; s < SPL; ++s) {
            hid[s][0] = fmaf(w.x, z[s][k], hid[s][0]);
            hid[s][1] = fmaf(w.y, z[s][k], hid[s][1]);
            hid[s][2] = fmaf(w.z, z[s][k], hid[s][2]);
            hid[s][3] = fmaf(w.w, z[s][k], hid[s][3]);
        }
    }
}

// out[s][o] += sum_c B[o][i0 + c] * hid[s][c]                        (B staged as [M][H])
template <int M, int SPL>
__device__ __forceinline__ void output_block(const float* sB, int H, int i0, const float (&hid)[SPL][4],
                                             float (&out)[SPL][M]) {
#pragma unroll
    for (int o = 0; o < M; ++o) {
        const float4 w = lds4(sB + o * H + i0);
#pragma unroll
        for (int s = 0; s < SPL; ++s)
            out[s][o] = fmaf(w.w, hid[s][3], fmaf(w.z, hid[s][2], fmaf(w.y, hid[s][1], fmaf(w.x, hid[s][0], out[s][o]))));
    }
}

// Sum y over the G lanes of a group; every lane ends with the total.
template <int G, int M>
__device__ __forceinline__ void group_allreduce(float (&y)[M]) {
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1)
#pragma unroll
        for (int d = 0; d < M; ++d) y[d] += __shfl_xor_sync(0xffffffffu, y[d], off);
}

// own[c] = y[base + 4g + c] without dynamic register indexing.
template <int G, int M>
__device__ __forceinline__ void select_own(const float (&y)[M], int base, int g, float (&own)[4]) {
#pragma unroll
    for (int gg = 0; gg < G; ++gg)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (gg == g) own[c] = y[base + 4 * gg + c];
}

// z[4gg + c] = own[c] of lane gg of the group.
template <int G, int D>
__device__ __forceinline__ void group_allgather(const float (&own)[4], float (&z)[D]) {
#pragma unroll
    for (int gg = 0; gg < G; ++gg)
#pragma unroll
        for (int c = 0; c < 4; ++c) z[4 * gg + c] = __shfl_sync(0xffffffffu, own[c], gg, G);
}

// Shared memory needed by k_chain, in floats.
inline size_t chain_smem_floats(int D, int H, int W) {
    const size_t guide = 2 * static_cast<size_t>(H) * D + H + static_cast<size_t>(W) * H + static_cast<size_t>(D) * D;
    const size_t trans = 3 * static_cast<size_t>(H) * D + H;
    return guide > trans ? guide : trans;
}

__device__ __forceinline__ void stage_vector4(float* dst, const float* __restrict__ src, int n) {   // n % 4 == 0
    const float4* s4 = reinterpret_cast<const float4*>(src);
    float4* d4 = reinterpret_cast<float4*>(dst);
    for (int i = threadIdx.x; i < n / 4; i += blockDim.x) d4[i] = s4[i];
}

struct ChainNoise {
    NoiseKey key;
    uint32_t step;
    uint32_t sample0;          // global index of the lane's first sample
};

// Guide: z_t = mu + sigma * eps for t = 0..W-1 (Section 3.1.3).  z holds z_{T-l-1} on entry, z_T on exit.
template <int D>
__device__ __forceinline__ void chain_guide(const ModelDev& m, const float* sWzT, const float* sWmu, const float* sWsig,
                                            const float* sbz, const float* shl, int g, const ChainNoise& nz,
                                            float (&z)[ChainShape<D>::SPL][D]) {
    constexpr int G = ChainShape<D>::G, SPL = ChainShape<D>::SPL;
    const int H = m.H, W = m.W;
    for (int t = 0; t < W; ++t) {
        float mu[SPL][D];
#pragma unroll
        for (int s = 0; s < SPL; ++s)
#pragma unroll
            for (int d = 0; d < D; ++d) mu[s][d] = 0.0f;
        const float* hl = shl + t * H;
        for (int i0 = 4 * g; i0 < H; i0 += 4 * G) {
            float hid[SPL][4];
            hidden_block<D, SPL>(sWzT, sbz, H, i0, z, hid);
            const float4 lr = lds4(hl + i0);
            const float lrv[4] = {lr.x, lr.y, lr.z, lr.w};
#pragma unroll
            for (int s = 0; s < SPL; ++s)
#pragma unroll
                for (int c = 0; c < 4; ++c) hid[s][c] = (tanh_fast(hid[s][c]) + lrv[c]) * (1.0f / 3.0f);
            output_block<D, SPL>(sWmu, H, i0, hid, mu);
        }
#pragma unroll
        for (int s = 0; s < SPL; ++s) {
            group_allreduce<G, D>(mu[s]);
#pragma unroll
            for (int d = 0; d < D; ++d) mu[s][d] += m.bmu[d];
        }
#pragma unroll
        for (int s = 0; s < SPL; ++s) {
            float eps[4], mu_own[4], z_own[4];
            normal4(static_cast<uint32_t>(g), nz.sample0 + s, static_cast<uint32_t>(t), nz.step, nz.key.seed_lo,
                    nz.key.seed_hi, eps);
            select_own<G, D>(mu[s], 0, g, mu_own);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float pre = m.bsig[4 * g + c];
                const float* wrow = sWsig + (4 * g + c) * D;
#pragma unroll
                for (int e4 = 0; e4 < D / 4; ++e4) {
                    const float4 w = lds4(wrow + 4 * e4);
                    pre = fmaf(w.x, mu[s][4 * e4 + 0], pre);
                    pre = fmaf(w.y, mu[s][4 * e4 + 1], pre);
                    pre = fmaf(w.z, mu[s][4 * e4 + 2], pre);
                    pre = fmaf(w.w, mu[s][4 * e4 + 3], pre);
                }
                z_own[c] = fmaf(softplusf(pre), eps[c], mu_own[c]);
            }
            group_allgather<G, D>(z_own, z[s]);
        }
    }
}

// Transition: z_{T+1} = mean + exp(logvar / 2) * eps with [mean | logvar] = W2 relu(W1 z + b1) + b2.
template <int D>
__device__ __forceinline__ void chain_transition(const ModelDev& m, const float* sW1T, const float* sW2, const float* sb1,
                                                 int g, const ChainNoise& nz, float (&z)[ChainShape<D>::SPL][D]) {
    constexpr int G = ChainShape<D>::G, SPL = ChainShape<D>::SPL;
    const int H = m.H;
    float head[SPL][2 * D];
#pragma unroll
    for (int s = 0; s < SPL; ++s)
#pragma unroll
        for (int o = 0; o < 2 * D; ++o) head[s][o] = 0.0f;
    for (int i0 = 4 * g; i0 < H; i0 += 4 * G) {
        float hid[SPL][4];
        hidden_block<D, SPL>(sW1T, sb1, H, i0, z, hid);
#pragma unroll
        for (int s = 0; s < SPL; ++s)
#pragma unroll
            for (int c = 0; c < 4; ++c) hid[s][c] = fmaxf(hid[s][c], 0.0f);
        output_block<2 * D, SPL>(sW2, H, i0, hid, head);
    }
#pragma unroll
    for (int s = 0; s < SPL; ++s) {
        group_allreduce<G, 2 * D>(head[s]);
        float eps[4], mean_own[4], logvar_own[4], z_own[4];
        normal4(static_cast<uint32_t>(g), nz.sample0 + s, kStreamTransition, nz.step, nz.key.seed_lo, nz.key.seed_hi, eps);
        select_own<G, 2 * D>(head[s], 0, g, mean_own);
        select_own<G, 2 * D>(head[s], D, g, logvar_own);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float mean = mean_own[c] + m.b2[4 * g + c];
            const float logvar = logvar_own[c] + m.b2[D + 4 * g + c];
            z_own[c] = fmaf(expf(0.5f * logvar), eps[c], mean);
        }
        group_allgather<G, D>(z_own, z[s]);
    }
}

// Where the chain's last layer goes: floats (fp32 emission), or halves scaled per sample (tensor-core emission).
struct ChainOut {
    float* v;               // [count][H], or null
    HalfRows half;          // used when v is null: values are rounded to tf32 first
};

// Four entries i0 .. i0 + 3 of a sample's row, and (lane 0 of the group) the row's inverse scale.
template <int D>
__device__ __forceinline__ void store_hidden(const ChainOut& out, int k, int H, int i0, const float (&h)[4], float scale) {
    if (out.v) {
        *reinterpret_cast<float4*>(out.v + static_cast<size_t>(k) * H + i0) = make_float4(h[0], h[1], h[2], h[3]);
    } else {
        *reinterpret_cast<uint2*>(out.half.p + static_cast<size_t>(k) * out.half.ld + i0) =
            make_uint2(pack_half2(round_tf32(h[0]) * scale, round_tf32(h[1]) * scale), pack_half2(round_tf32(h[2]) * scale, round_tf32(h[3]) * scale));
    }
}
template <int D>
__device__ __forceinline__ float hidden_scale(const ChainOut& out, int k, bool exists, int g, const float (&z)[D]) {
    if (out.v) return 1.0f;
    float zm = 0.0f, scale, inv;
#pragma unroll
    for (int d = 0; d < D; ++d) zm = fmaxf(zm, fabsf(z[d]));
    half_scale(out.half, zm, scale, inv);
    if (g == 0 && exists) out.half.inv_scale[k] = inv;
    return scale;
}

// Last layer, act(A z + b) with the ReLU of the emission's hidden layer or none (literal: u), for the samples k0 .. k0+SPL-1
// that exist.
template <int D, bool RELU>
__device__ __forceinline__ void chain_last_layer(const float* sAT, const float* sbias, int H, int g,
                                                 const float (&z)[ChainShape<D>::SPL][D], int k0, int count, const ChainOut& out) {
    constexpr int G = ChainShape<D>::G, SPL = ChainShape<D>::SPL;
    float scale[SPL];
#pragma unroll
    for (int s = 0; s < SPL; ++s) scale[s] = hidden_scale<D>(out, k0 + s, k0 + s < count, g, z[s]);
    for (int i0 = 4 * g; i0 < H; i0 += 4 * G) {
        float hid[SPL][4];
        hidden_block<D, SPL>(sAT, sbias, H, i0, z, hid);
#pragma unroll
        for (int s = 0; s < SPL; ++s) {
            if (RELU) {
#pragma unroll
                for (int c = 0; c < 4; ++c) hid[s][c] = fmaxf(hid[s][c], 0.0f);
            }
            if (k0 + s < count) store_hidden<D>(out, k0 + s, H, i0, hid[s], scale[s]);
        }
    }
}

// Variant 1: weights staged phase by phase (any model size whose largest phase fits in shared memory).
template <int D>
__global__ void __launch_bounds__(ChainShape<D>::kThreads) k_chain(ModelDev m, const float* __restrict__ hlr,
                                                          const DevState* __restrict__ st, NoiseKey key,
                                                          uint32_t sample_base, int count, ChainOut out) {
    constexpr int G = ChainShape<D>::G, SPL = ChainShape<D>::SPL;
    extern __shared__ __align__(16) float sm[];
    const int H = m.H, W = m.W;
    const int g = threadIdx.x % G;
    const int k0 = (blockIdx.x * (ChainShape<D>::kThreads / G) + threadIdx.x / G) * SPL;      // first sample of the lane

    float* sWzT = sm;                   // [D][H]
    float* sWmu = sWzT + H * D;         // [D][H]
    float* sWsig = sWmu + H * D;        // [D][D]
    float* sbz = sWsig + D * D;         // [H]
    float* shl = sbz + H;               // [W][H]  h_left + h_right
    stage_vector4(sWzT, m.WzT, H * D);
    stage_vector4(sWmu, m.Wmu, H * D);
    stage_vector4(sWsig, m.Wsig, D * D);
    stage_vector4(sbz, m.bz, H);
    dependency_wait();            // up to here: weights
    launch_dependents();
    const ChainNoise nz{key, st->step, sample_base + static_cast<uint32_t>(k0)};
    for (int i = threadIdx.x; i < W * H; i += blockDim.x) shl[i] = hlr[i] + hlr[W * H + i];
    __syncthreads();
    float z[SPL][D];
#pragma unroll
    for (int s = 0; s < SPL; ++s)
#pragma unroll
        for (int d = 0; d < D; ++d) z[s][d] = m.z0[d];
    chain_guide<D>(m, sWzT, sWmu, sWsig, sbz, shl, g, nz, z);
    __syncthreads();

    float* sW1T = sm;                   // [D][H]
    float* sW2 = sW1T + H * D;          // [2D][H]
    float* sb1 = sW2 + 2 * H * D;       // [H]
    stage_vector4(sW1T, m.W1T, H * D);
    stage_vector4(sW2, m.W2, 2 * H * D);
    stage_vector4(sb1, m.b1, H);
    __syncthreads();
    chain_transition<D>(m, sW1T, sW2, sb1, g, nz, z);
    __syncthreads();

    float* sW3T = sm;                   // [D][H]
    float* sb3 = sW3T + H * D;          // [H]
    stage_vector4(sW3T, m.W3T, H * D);
    stage_vector4(sb3, m.b3, H);
    __syncthreads();
    chain_last_layer<D, true>(sW3T, sb3, H, g, z, k0, count, out);
}

// Variant 2: every weight of the chain resident in shared memory, one persistent CTA per SM.
// The weights are staged once; after that the warps never synchronise: warp w of the grid takes
// the sample batches blockIdx + gridDim * w, + (warps in the grid), ... (a batch = the samples one warp covers).
constexpr int kChainResidentThreads = 512;

inline size_t chain_resident_smem_floats(int D, int H, int W) {
    return 6 * static_cast<size_t>(H) * D + static_cast<size_t>(D) * D + 3 * static_cast<size_t>(H) +
           static_cast<size_t>(W) * H;
}

template <int D>
__global__ void __launch_bounds__(kChainResidentThreads, 1)
k_chain_resident(ModelDev m, const float* __restrict__ hlr, const DevState* __restrict__ st, NoiseKey key,
                 uint32_t sample_base, int count, ChainOut out) {
    constexpr int G = ChainShape<D>::G, SPL = ChainShape<D>::SPL;
    constexpr int kBatch = 32 / G * SPL;                // samples per warp and pass
    extern __shared__ __align__(16) float sm[];
    const int H = m.H, W = m.W;
    float* sWzT = sm;                   // [D][H]
    float* sWmu = sWzT + H * D;         // [D][H]
    float* sW1T = sWmu + H * D;         // [D][H]
    float* sW2 = sW1T + H * D;          // [2D][H]
    float* sW3T = sW2 + 2 * H * D;      // [D][H]
    float* sWsig = sW3T + H * D;        // [D][D]
    float* sbz = sWsig + D * D;         // [H]
    float* sb1 = sbz + H;               // [H]
    float* sb3 = sb1 + H;               // [H]
    float* shl = sb3 + H;               // [W][H]
    stage_vector4(sWzT, m.WzT, H * D);
    stage_vector4(sWmu, m.Wmu, H * D);
    stage_vector4(sW1T, m.W1T, H * D);
    stage_vector4(sW2, m.W2, 2 * H * D);
    stage_vector4(sW3T, m.W3T, H * D);
    stage_vector4(sWsig, m.Wsig, D * D);
    stage_vector4(sbz, m.bz, H);
    stage_vector4(sb1, m.b1, H);
    stage_vector4(sb3, m.b3, H);
    dependency_wait();            // up to here: weights
    launch_dependents();
    for (int i = threadIdx.x; i < W * H; i += kChainResidentThreads) shl[i] = hlr[i] + hlr[W * H + i];
    __syncthreads();

    const int lane = threadIdx.x & 31, g = lane % G;
    const int warps_in_grid = gridDim.x * (kChainResidentThreads / 32);
    const int n_batches = ceil_div(count, kBatch);
    const uint32_t step = st->step;
    // consecutive batches go to different CTAs, so that a small decision still spreads over all SMs
    for (int b = blockIdx.x + gridDim.x * (threadIdx.x >> 5); b < n_batches; b += warps_in_grid) {
        const int k0 = b * kBatch + (lane / G) * SPL;
        const ChainNoise nz{key, step, sample_base + static_cast<uint32_t>(k0)};
        float z[SPL][D];
#pragma unroll
        for (int s = 0; s < SPL; ++s)
#pragma unroll
            for (int d = 0; d < D; ++d) z[s][d] = m.z0[d];
        chain_guide<D>(m, sWzT, sWmu, sWsig, sbz, shl, g, nz, z);
        chain_transition<D>(m, sW1T, sW2, sb1, g, nz, z);
        chain_last_layer<D, true>(sW3T, sb3, H, g, z, k0, count, out);
    }
}

// Variant 3: D lanes per sample, one latent component each, for decisions with too few samples to occupy the GPU otherwise.
// What bounds a small decision is the chain of a step -- D multiply-adds per hidden unit, H / (4 D) groups of hidden units per lane, the
// sums over the lanes -- with about one warp per scheduler to hide it: with D / 4 lanes and two samples per lane an SM had one warp at
// N=158, S=2048.  N=158, lag 20: 76 -> 23 us; N=16: 13 -> 7 us; N=2175, lag 20, S=1024 against the tensor-core chain on 8 SMs: 76 -> 32 us.
// With more samples it is the reads of the weights from shared memory, one per lane and sample; SPL = 2 samples per lane
// share them (N=128, S=16384: 31 us with one, 24 with two, 28.5 by the kernel above).
// Drawing the noise of 16 steps at once into shared memory, off the chain, changed nothing (23 us).
constexpr int kChainWideThreads = 512;

// y[0 .. D-1] summed over the D lanes of a group: lane g ends with the total of component g (recursive halving, D - 1 shuffles).
template <int D>
__device__ __forceinline__ float group_reduce_scatter(float (&y)[D], int g) {
#pragma unroll
    for (int off = D / 2; off > 0; off >>= 1)
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const float keep = (g & off) ? y[i + off] : y[i], give = (g & off) ? y[i] : y[i + off];
            y[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    return y[0];
}
template <int D>
__device__ __forceinline__ void group_broadcast(float own, float (&z)[D]) {
#pragma unroll
    for (int d = 0; d < D; ++d) z[d] = __shfl_sync(0xffffffffu, own, d, D);
}
// Element g of a sample's normals: its half of one Box-Muller pair.
__device__ __forceinline__ float normal_element(int g, uint32_t sample, uint32_t stream, uint32_t step, const NoiseKey& key) {
    const Philox4 r = philox4x32_10(static_cast<uint32_t>(g >> 2), sample, stream, step, key.seed_lo, key.seed_hi);
    float c, s;
    box_muller((g & 2) ? r.z : r.x, (g & 2) ? r.w : r.y, c, s);
    return (g & 1) ? s : c;
}

template <int D, int SPL>
__global__ void __launch_bounds__(kChainWideThreads, 1)
k_chain_wide(ModelDev m, const float* __restrict__ hlr, const DevState* __restrict__ st, NoiseKey key,
             uint32_t sample_base, int count, ChainOut out) {
    extern __shared__ __align__(16) float sm[];          // chain_resident_smem_floats
    const int H = m.H, W = m.W;
    float* sWzT = sm;                   // [D][H]
    float* sWmu = sWzT + H * D;         // [D][H]
    float* sW1T = sWmu + H * D;         // [D][H]
    float* sW2 = sW1T + H * D;          // [2D][H]
    float* sW3T = sW2 + 2 * H * D;      // [D][H]
    float* sbz = sW3T + H * D;          // [H]
    float* sb1 = sbz + H;               // [H]
    float* sb3 = sb1 + H;               // [H]
    float* shl = sb3 + H;               // [W][H]
    float* sWsigT = shl + W * H;        // [D][D], transposed: a lane reads its row a column at a time
    stage_vector4(sWzT, m.WzT, H * D);
    stage_vector4(sWmu, m.Wmu, H * D);
    stage_vector4(sW1T, m.W1T, H * D);
    stage_vector4(sW2, m.W2, 2 * H * D);
    stage_vector4(sW3T, m.W3T, H * D);
    stage_vector4(sbz, m.bz, H);
    stage_vector4(sb1, m.b1, H);
    stage_vector4(sb3, m.b3, H);
    for (int i = threadIdx.x; i < D * D; i += kChainWideThreads) sWsigT[(i % D) * D + i / D] = m.Wsig[i];
    const int lane = threadIdx.x & 31, g = lane % D;
    const float bmu = m.bmu[g], bsig = m.bsig[g], b2_mean = m.b2[g], b2_logvar = m.b2[D + g], z0 = m.z0[g];
    dependency_wait();            // up to here: weights
    launch_dependents();
    for (int i = threadIdx.x; i < W * H; i += kChainWideThreads) shl[i] = hlr[i] + hlr[W * H + i];
    __syncthreads();

    constexpr int kBatch = 32 / D * SPL;                 // samples per warp and pass
    const int n_batches = ceil_div(count, kBatch);
    const uint32_t step = st->step;
    // consecutive batches go to different CTAs, so that a small decision still spreads over all SMs
    for (int b = blockIdx.x + gridDim.x * (threadIdx.x >> 5); b < n_batches; b += gridDim.x * (kChainWideThreads / 32)) {
        const int k = b * kBatch + lane / D * SPL;       // the lane's first sample
        const uint32_t sample = sample_base + static_cast<uint32_t>(k);
        float z[SPL][D];
#pragma unroll
        for (int s = 0; s < SPL; ++s) group_broadcast<D>(z0, z[s]);
        for (int t = 0; t < W; ++t) {
            float eps[SPL], mu[SPL][D] = {};
#pragma unroll
            for (int s = 0; s < SPL; ++s) eps[s] = normal_element(g, sample + s, static_cast<uint32_t>(t), step, key);     // off the chain: nothing below feeds it
            const float* hl = shl + t * H;
            for (int i0 = 4 * g; i0 < H; i0 += 4 * D) {
                float hid[SPL][4];
                hidden_block<D, SPL>(sWzT, sbz, H, i0, z, hid);
                const float4 lr = lds4(hl + i0);
                const float lrv[4] = {lr.x, lr.y, lr.z, lr.w};
#pragma unroll
                for (int s = 0; s < SPL; ++s)
#pragma unroll
                    for (int c = 0; c < 4; ++c) hid[s][c] = (tanh_fast(hid[s][c]) + lrv[c]) * (1.0f / 3.0f);
                output_block<D, SPL>(sWmu, H, i0, hid, mu);
            }
#pragma unroll
            for (int s = 0; s < SPL; ++s) {
                const float mu_own = group_reduce_scatter<D>(mu[s], g) + bmu;
                group_broadcast<D>(mu_own, mu[s]);
                float pre = bsig;
#pragma unroll
                for (int e = 0; e < D; ++e) pre = fmaf(sWsigT[e * D + g], mu[s][e], pre);
                group_broadcast<D>(fmaf(softplusf(pre), eps[s], mu_own), z[s]);
            }
        }
        float eps[SPL], mean[SPL][D] = {}, logvar[SPL][D] = {};
#pragma unroll
        for (int s = 0; s < SPL; ++s) eps[s] = normal_element(g, sample + s, kStreamTransition, step, key);
        for (int i0 = 4 * g; i0 < H; i0 += 4 * D) {
            float hid[SPL][4];
            hidden_block<D, SPL>(sW1T, sb1, H, i0, z, hid);
#pragma unroll
            for (int s = 0; s < SPL; ++s)
#pragma unroll
                for (int c = 0; c < 4; ++c) hid[s][c] = fmaxf(hid[s][c], 0.0f);
            output_block<D, SPL>(sW2, H, i0, hid, mean);
            output_block<D, SPL>(sW2 + D * H, H, i0, hid, logvar);
        }
        float scale[SPL];
#pragma unroll
        for (int s = 0; s < SPL; ++s) {
            const float mean_own = group_reduce_scatter<D>(mean[s], g) + b2_mean, logvar_own = group_reduce_scatter<D>(logvar[s], g) + b2_logvar;
            group_broadcast<D>(fmaf(expf(0.5f * logvar_own), eps[s], mean_own), z[s]);
            scale[s] = hidden_scale<D>(out, k + s, k + s < count, g, z[s]);
        }
        for (int i0 = 4 * g; i0 < H; i0 += 4 * D) {
            float hid[SPL][4];
            hidden_block<D, SPL>(sW3T, sb3, H, i0, z, hid);
#pragma unroll
            for (int s = 0; s < SPL; ++s) {
#pragma unroll
                for (int c = 0; c < 4; ++c) hid[s][c] = fmaxf(hid[s][c], 0.0f);
                if (k + s < count) store_hidden<D>(out, k + s, H, i0, hid[s], scale[s]);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Emission output layer in fp32 FMA, with the noise drawn in the epilogue:
//   [mean | logvar] = W4 v + b4,   x_j = mean_j + exp(logvar_j / 2) * eps_j.
// 4 RM samples x 64 workers per CTA of 64 threads; a thread has RM samples x 4 consecutive workers, both heads, so that one
// generator call serves its four draws.  What bounds it is the issue of instructions: 64 multiply-adds per thread and k went through
// with 62 % of the slots taken.  Hence two columns per instruction (their sums are the same two chains), operands by asynchronous
// copies, and the weights with their columns contiguous (k_transpose_heads), so that a pair of columns is a pair of registers.
// N=128, H=128, S=16384: 50 us with 4 x 4 x 2 results per thread of 256 and copies through registers, 52 us with 8 x 8 and single
// multiply-adds, 41 us as it is (multiply-adds alone, at the measured rate: 19 us; the draws' log, sin, cos and exp most of the rest).
// RM = 8 where that makes two CTAs per SM, else RM = 2: N=16, S=1024: 7.0 -> 4.5 us.  The decisions: N=128 105 -> 101 us, N=16 39.5 -> 37.4 us.
// ---------------------------------------------------------------------------------------------
constexpr int kEmitThreads = 64, kEmitTN = 64, kEmitTK = 8, kEmitSlabs = 5;
constexpr int kEmitPitchA = kEmitTK + 4, kEmitPitchB = 2 * kEmitTN + 4;

// W4 [2N][H] as [H][2][ldn], so that the columns of a slab are contiguous (when weights are loaded).
__global__ void k_transpose_heads(const float* __restrict__ W4, int N, int H, int ldn, float* __restrict__ out) {
    __shared__ float tile[32][33];
    const int j0 = blockIdx.x * 32, k0 = blockIdx.y * 32, head = blockIdx.z;
    for (int r = threadIdx.y; r < 32; r += 8)
        tile[r][threadIdx.x] = j0 + r < N && k0 + threadIdx.x < H ? W4[(static_cast<size_t>(head) * N + j0 + r) * H + k0 + threadIdx.x] : 0.f;
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += 8)
        if (k0 + r < H && j0 + threadIdx.x < ldn)
            out[(static_cast<size_t>(k0 + r) * 2 + head) * ldn + j0 + threadIdx.x] = tile[threadIdx.x][r];
}

// ---------------------------------------------------------------------------------------------
// The same layer with the weights of a CTA's workers resident in shared memory: one persistent CTA per SM, 4 TX workers per CTA,
// (32 / TX) RM samples at a time per warp, and no warp waits for another.  A thread has RM samples x 4 workers, both heads.
// Per k a thread issues 4 RM paired multiply-adds (two columns each), RM / 2 loads of two hidden values and two of weights.  What bounds it: the
// reads of shared memory first (N=64, H=128, S=60000: wavefronts 69 % busy, issue slots 52 %, multiply-adds 49 %; N=16: 52, 44 and 40 %).  A
// hidden value is stored twice in a row, so that a load brings the pair that an instruction multiplies two
// columns with; made in registers, the pairs took as many moves as there are multiply-adds to four columns.  The warps of a
// CTA lie evenly on the four schedulers, and CTAs of this size cannot crowd on the SMs that the chain leaves free: the CTAs of 64 threads of
// the kernel below did both (N=16, S=1024: 128 of them on 19 SMs).  Emission stage before and after: N=16 S=60000 33.6 and 15.1 us,
// N=30 S=30000 23.6 and 15.4, N=50 S=8000 23.6 and 15.1, N=16 S=1024 9.1 and 7.2;
// N=64 S=60000, H=128 73.7 and 73.1.  With more worker tiles of 32 the reads of the pairs cost more than it gains (four cycles of the shared-memory pipe for 16 bytes a lane): N=100 S=60000 79 and 87, N=250 S=1500 17 and 23.
// ---------------------------------------------------------------------------------------------
constexpr int kEmitRowsWarps = 16, kEmitRowsTK = 16, kEmitRowsPitch = 2 * kEmitRowsTK + 4;

// Shared memory: the weights [H][2][4 TX], and per warp its samples' hidden values of 16 k.  Never less than half an SM's: one CTA per SM.
template <int TX, int RM> __host__ __device__ constexpr int emit_rows_warp_floats() {
    const int hidden = 32 / TX * RM * kEmitRowsPitch, results = RM * 8 * 32;
    return hidden > results ? hidden : results;
}
template <int TX, int RM> constexpr size_t emit_rows_smem_bytes(int H) {
    const size_t bytes = sizeof(float) * (static_cast<size_t>(H) * 8 * TX + kEmitRowsWarps * emit_rows_warp_floats<TX, RM>());
    return bytes < 116 * 1024 ? 116 * 1024 : bytes;
}

template <int TX, int RM>
__global__ void __launch_bounds__(kEmitRowsWarps * 32, 1) k_emit_rows(ModelDev m, const float* __restrict__ v, const float* __restrict__ W4T, int ldn,
                                                            const DevState* __restrict__ st, NoiseKey key,
                                                            uint32_t sample_base, int count,
                                                            float* __restrict__ x, int ldx) {
    constexpr int TN = 4 * TX, TY = 32 / TX, TM = TY * RM, TK = kEmitRowsTK, kPitch = kEmitRowsPitch;
    constexpr int kQuads = TM * TK / 4, kLoads = (kQuads + 31) / 32;     // 16-byte pieces of a slab, and how many a lane moves
    extern __shared__ __align__(16) float sm_rows[];
    const int H = m.H, N = m.N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tx = lane % TX, ty = lane / TX;
    const int worker_tiles = ceil_div(N, TN), wt = static_cast<int>(blockIdx.x) % worker_tiles, part = static_cast<int>(blockIdx.x) / worker_tiles;
    const int parts = (static_cast<int>(gridDim.x) - wt + worker_tiles - 1) / worker_tiles;      // CTAs that share these workers
    const int j0 = wt * TN, jbase = j0 + 4 * tx;
    float* const weights = sm_rows;
    float* const hidden = sm_rows + static_cast<size_t>(H) * 2 * TN + warp * emit_rows_warp_floats<TX, RM>();
    const uint32_t weights_s = fma32::smem_addr(weights);
    for (int i = threadIdx.x; i < H * 2 * TX; i += kEmitRowsWarps * 32) {
        const int k2 = i / TX, j = j0 + i % TX * 4;                       // k2: k and head
        fma32::copy4<true>(weights_s + 16 * i, j < ldn ? W4T + static_cast<size_t>(k2) * ldn + j : W4T, ldn - j);
    }
    dependency_wait();            // up to here: weights.  No launch_dependents: the row sort after this kernel has a few CTAs per SM, and placed
                                  // early they crowd on the SMs that happen to have room
    fma32::copies_landed();
    __syncthreads();
    const int tiles = ceil_div(count, TM);
    const uint4 column = philox_column(static_cast<uint32_t>(jbase >> 2), kStreamEmission, st->step, key.seed_lo, key.seed_hi);
    const float* const wp = weights + 4 * tx;
    const float* const hp = hidden + ty * kPitch;
    float2* const own = reinterpret_cast<float2*>(hidden) + lane;
    // consecutive tiles go to different CTAs, so that a small decision still spreads over all SMs
#pragma unroll 1
    for (int tile = part + parts * warp; tile < tiles; tile += parts * kEmitRowsWarps) {
        const int row0 = tile * TM;
        float4 next[kLoads];
        const auto request = [&](int k0) {
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const int q = u * 32 + lane, r = q / (TK / 4), k = k0 + q % (TK / 4) * 4;
                next[u] = q < kQuads && row0 + r < count && k < H ? *reinterpret_cast<const float4*>(v + static_cast<size_t>(row0 + r) * H + k)
                                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        };
        unsigned long long sums[RM][4] = {};                     // means of workers 0, 1 and 2, 3, then their log-variances
        request(0);
#pragma unroll 1
        for (int k0 = 0; k0 < H; k0 += TK) {
            __syncwarp();                                        // everyone has finished with the values before these
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const int q = u * 32 + lane, r = q / (TK / 4), c = q % (TK / 4) * 4;
                if (q < kQuads) {
                    float4* const dst = reinterpret_cast<float4*>(hidden + r * kPitch + 2 * c);
                    dst[0] = make_float4(next[u].x, next[u].x, next[u].y, next[u].y);
                    dst[1] = make_float4(next[u].z, next[u].z, next[u].w, next[u].w);
                }
            }
            __syncwarp();
            if (k0 + TK < H) request(k0 + TK);
            const float* w = wp + static_cast<size_t>(k0) * 2 * TN;
#pragma unroll
            for (int k = 0; k < TK; k += 4) {
                if (k0 + k >= H) break;                          // H is a multiple of 4
#pragma unroll
                for (int p = 0; p < 4; p += 2) {
                    ulonglong2 a[RM];
#pragma unroll
                    for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(hp + i * TY * kPitch + 2 * (k + p));
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const ulonglong2 mean = *reinterpret_cast<const ulonglong2*>(w + (k + p + q) * 2 * TN);
                        const ulonglong2 logvar = *reinterpret_cast<const ulonglong2*>(w + (k + p + q) * 2 * TN + TN);
#pragma unroll
                        for (int i = 0; i < RM; ++i) {
                            const unsigned long long s2 = q == 0 ? a[i].x : a[i].y;
                            fma2(sums[i][0], s2, mean.x);
                            fma2(sums[i][1], s2, mean.y);
                            fma2(sums[i][2], s2, logvar.x);
                            fma2(sums[i][3], s2, logvar.y);
                        }
                    }
                }
            }
        }
        // The draws one sample at a time, results through shared memory (each lane its own): unrolled, the generator, its logarithms and
        // sines would be RM copies of their code, which a call that finds the caches cold fetches from memory.
        float b_mean[4], b_logvar[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            b_mean[c] = jbase + c < N ? m.b4[jbase + c] : 0.f;
            b_logvar[c] = jbase + c < N ? m.b4[N + jbase + c] : 0.f;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float2 pair;
                unpack2(sums[i][c], pair.x, pair.y);
                own[(4 * i + c) * 32] = pair;
            }
#pragma unroll 1
        for (int i = 0; i < RM; ++i) {
            const int k = row0 + ty + TY * i;
            if (k >= count || jbase >= N) break;
            float eps[4], mean[4], logvar[4], out[4];
            normal4_row_column(philox_row(sample_base + static_cast<uint32_t>(k), kStreamEmission, key.seed_lo), column, key.seed_lo, key.seed_hi, eps);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float2 mp = own[(4 * i + c) * 32], lp = own[(4 * i + 2 + c) * 32];
                mean[2 * c] = mp.x; mean[2 * c + 1] = mp.y;
                logvar[2 * c] = lp.x; logvar[2 * c + 1] = lp.y;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) out[c] = fmaf(expf(0.5f * (logvar[c] + b_logvar[c])), eps[c], mean[c] + b_mean[c]);
            float* dst = x + static_cast<size_t>(k) * ldx + jbase;           // the row pitch is a multiple of 8 floats
            if (jbase + 3 < N) {
                *reinterpret_cast<float4*>(dst) = make_float4(out[0], out[1], out[2], out[3]);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (jbase + c < N) dst[c] = out[c];
            }
        }
    }
}

template <int RM>
__global__ void __launch_bounds__(kEmitThreads, RM == 8 ? 7 : 8) k_emit_fma(ModelDev m, const float* __restrict__ v, const float* __restrict__ W4T, int ldn,
                                                            const DevState* __restrict__ st, NoiseKey key,
                                                            uint32_t sample_base, int count,
                                                            float* __restrict__ x, int ldx) {
    constexpr int TM = 4 * RM, kFloats = TM * kEmitPitchA + kEmitTK * kEmitPitchB;
    __shared__ __align__(16) float sm[kEmitSlabs * kFloats];
    const int H = m.H, N = m.N, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int row_tiles = ceil_div(count, TM), row0 = static_cast<int>(blockIdx.x) % row_tiles * TM;
    const int j0 = static_cast<int>(blockIdx.x) / row_tiles * kEmitTN, jbase = j0 + 4 * tx;
    const uint32_t smem = fma32::smem_addr(sm);
    // No launch_dependents here: the row sort after this kernel has a few CTAs per SM, and placed early they crowd on the SMs
    // that happen to have room (N=128, S=16384: the decision 119 us with it, 101 us without).
    dependency_wait();
    const int slabs = ceil_div(H, kEmitTK);
    int k_req = 0, buf_req = 0;
    const auto request = [&] {
        if (k_req < H) {
            const uint32_t dst = smem + 4 * buf_req * kFloats;
#pragma unroll
            for (int u = tid; u < TM * kEmitTK / 4; u += kEmitThreads) {
                const int r = u / (kEmitTK / 4), k = k_req + u % (kEmitTK / 4) * 4, valid = row0 + r < count ? H - k : 0;
                fma32::copy4<true>(dst + 4 * (r * kEmitPitchA + u % (kEmitTK / 4) * 4), valid > 0 ? v + static_cast<size_t>(row0 + r) * H + k : v, valid);
            }
#pragma unroll
            for (int u = tid; u < kEmitTK * kEmitTN / 2; u += kEmitThreads) {
                const int kk = u / (kEmitTN / 2), c = u % (kEmitTN / 2) * 4, k = k_req + kk, j = j0 + c % kEmitTN, valid = k < H ? ldn - j : 0;
                fma32::copy4<true>(dst + 4 * (TM * kEmitPitchA + kk * kEmitPitchB + c),
                                   valid > 0 ? W4T + (static_cast<size_t>(k) * 2 + c / kEmitTN) * ldn + j : W4T, valid);
            }
            k_req += kEmitTK;
            if (++buf_req == kEmitSlabs) buf_req = 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < kEmitSlabs - 1; ++i) request();
    unsigned long long sums[RM][4] = {};                     // means of workers 0, 1 and 2, 3, then their log-variances
    int buf = 0;
    for (int it = 0; it < slabs; ++it) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kEmitSlabs - 2) : "memory");
        __syncthreads();                                     // the slab is there for everyone, and everyone has finished with the one before it
        request();
        const float* sa = sm + buf * kFloats + ty * kEmitPitchA;
        const float* sb = sm + buf * kFloats + TM * kEmitPitchA + 4 * tx;
#pragma unroll
        for (int k = 0; k < kEmitTK; k += 4) {
            float4 a[RM];
#pragma unroll
            for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const float4*>(sa + 4 * i * kEmitPitchA + k);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const ulonglong2 mean = *reinterpret_cast<const ulonglong2*>(sb + (k + q) * kEmitPitchB);
                const ulonglong2 logvar = *reinterpret_cast<const ulonglong2*>(sb + (k + q) * kEmitPitchB + kEmitTN);
#pragma unroll
                for (int i = 0; i < RM; ++i) {
                    const float s = q == 0 ? a[i].x : q == 1 ? a[i].y : q == 2 ? a[i].z : a[i].w;
                    const unsigned long long s2 = pack2(s, s);
                    fma2(sums[i][0], s2, mean.x);
                    fma2(sums[i][1], s2, mean.y);
                    fma2(sums[i][2], s2, logvar.x);
                    fma2(sums[i][3], s2, logvar.y);
                }
            }
        }
        if (++buf == kEmitSlabs) buf = 0;
    }
    // The draws one row at a time, through shared memory (each thread its own results): unrolled, the generator and its
    // logarithms and sines would be 30 KB of instructions, which a call that finds the caches cold fetches from memory.
    __syncthreads();
    ulonglong2* own = reinterpret_cast<ulonglong2*>(sm) + tid;
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        own[(2 * i) * kEmitThreads] = make_ulonglong2(sums[i][0], sums[i][1]);
        own[(2 * i + 1) * kEmitThreads] = make_ulonglong2(sums[i][2], sums[i][3]);
    }
    static_assert(2 * RM * kEmitThreads * 4 <= kEmitSlabs * kFloats, "results fit where the slabs were");
    if (jbase >= N) return;
    const uint4 column = philox_column(static_cast<uint32_t>(jbase >> 2), kStreamEmission, st->step, key.seed_lo, key.seed_hi);
    float b_mean[4], b_logvar[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        b_mean[c] = jbase + c < N ? m.b4[jbase + c] : 0.f;
        b_logvar[c] = jbase + c < N ? m.b4[N + jbase + c] : 0.f;
    }
#pragma unroll 1
    for (int i = 0; i < RM; ++i) {
        const int k = row0 + ty + 4 * i;
        if (k >= count) break;
        float eps[4], mean[4], logvar[4], out[4];
        normal4_row_column(philox_row(sample_base + static_cast<uint32_t>(k), kStreamEmission, key.seed_lo), column, key.seed_lo, key.seed_hi, eps);
        *reinterpret_cast<float4*>(mean) = *reinterpret_cast<const float4*>(own + (2 * i) * kEmitThreads);
        *reinterpret_cast<float4*>(logvar) = *reinterpret_cast<const float4*>(own + (2 * i + 1) * kEmitThreads);
#pragma unroll
        for (int c = 0; c < 4; ++c) out[c] = fmaf(expf(0.5f * (logvar[c] + b_logvar[c])), eps[c], mean[c] + b_mean[c]);
        float* dst = x + static_cast<size_t>(k) * ldx + jbase;               // the row pitch is a multiple of 8 floats
        if (jbase + 3 < N) {
            *reinterpret_cast<float4*>(dst) = make_float4(out[0], out[1], out[2], out[3]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (jbase + c < N) dst[c] = out[c];
        }
    }
}

}  // namespace cutoff
