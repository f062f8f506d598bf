// Learning the model on the GPU: the one-sample, reparameterised ELBO of Section 3.1.3 for a batch of windows,
// its gradient with respect to every weight tensor (reverse mode, layer by layer), and Adam with clipping by the
// global norm (Section 4.1), for the compact networks, in fp32.
//
//   ELBO_b = sum_t  log p(x_t | z_t) + log p(z_t | z_{t-1}) - log q(z_t | z_{t-1}, x),     z_t = mu_t + sigma_t eps_t,
//   log N(y; m, exp(lv)) = -1/2 [log 2 pi + lv + (y - m)^2 exp(-lv)],   log q = sum_d -1/2 log 2 pi - log sigma_d - eps_d^2 / 2.
//
// What bounds a step is the number of dependent launches and the length of its chains, not its arithmetic (64 windows of
// the n1024 model: 1.0 G multiply-adds, 28 us at the FMA rate), so the step is laid out by what depends on what.  Only the
// recurrences depend on the previous step of a window, and only within the window: one CTA walks through all of a
// window's steps, a cluster through those of a few windows' RNN, in one launch (the forward RNNs of wide networks and large
// batches: a product per step).  Everything else is one product over all
// B*W (window, step) rows: the input projections, the emission head with its density in the epilogue, the input gradient
// of that head, and the weight gradients as a list of products in one launch.
//
// Rows are window-major: row r = b*W + t.  Every sum has the order of the plain layer-by-layer evaluation: one chain of
// fused multiply-adds over ascending k per product; a weight gradient adds the chains of the steps one after the other,
// the step the reverse pass reaches first coming first.  No product is split over k and nothing depends on tiles,
// clusters or the other windows, so a step is reproducible bit for bit and a change of its schedule does not change it --
// which matters because training is not continuous: Adam turns the sign of a vanishing gradient into a full step, and a
// ReLU whose input is within rounding of zero switches a whole row of a gradient on or off.
//
// A kernel lets its successor start early (launch_dependents) only where the successor has at most one CTA per SM to place: the
// CTAs of the emission head, of its input gradient and of the weight gradients would crowd on the SMs that the path and RNN
// kernels leave free (64 windows, N=1024: 361 us per step with them started early, 314 us without; without any early start
// 333 us, and N=128 122 us against 103).
#pragma once
#include <cmath>

#include "common.cuh"
#include "tile_product.cuh"

namespace cutoff {
namespace fit {

constexpr float kLog2Pi = 1.8378770664093453f;

__device__ __forceinline__ float softplus_f(float v) { return v > 20.f ? v : log1pf(expf(v)); }
__device__ __forceinline__ float sigmoid_f(float v) { return 1.f / (1.f + expf(-v)); }

// ---- tiled products (tile_product.cuh) ------------------------------------------------------------------------------
// Three tiles: 64 x 64 with 8 x 4 results per thread where there are several of them per SM, 32 x 64 with 4 x 4 where there would
// be one or two (the emission head of 384 x 256 values, H=128: 12.1 -> 8.6 us; of 320 x 2048, H=256: 25 -> 20 us), and 16 x 32
// with 2 x 2 where even those do not fill the GPU -- then the time is the chain's: 2048 steps of it take 41 us whatever the tile
// (2 x 4 results per thread 51 us, 1 x 2 48 us, the next four k in registers ahead of time 43 us).
using namespace fma32;
using LargeTile = Tile<64, 64, 8, 4, 16>;        // 128 threads
using MediumTile = Tile<32, 64, 4, 4, 16>;       // 128 threads
using SmallTile = Tile<16, 32, 2, 2, 32>;        // 128 threads

struct Product {
    Operand a, b;
    float* c;
    long long ldc;
    float* a_sums;       // sums over k and the segments of an m-major A (bias gradient), from the first column of tiles; or null
    int K, n_seg;
    int tile0, tiles_n;  // first tile of this product in the launch, tiles per tile row
};

constexpr int kMaxProducts = 16;
struct ProductList {
    Product p[kMaxProducts];
    int n;
};

template <typename T, bool A_KMAJOR, bool B_KMAJOR, bool VEC, bool SEGMENTS>
__device__ __forceinline__ void run_product(Slabs<T, A_KMAJOR, B_KMAJOR>& sm, const Product& q, int tile) {
    const int m0 = tile / q.tiles_n * T::TM, n0 = tile % q.tiles_n * T::TN;
    float a_sum = 0.f;
    if (q.b.rows == 0) {                       // sums only
        if (threadIdx.x < T::TM && m0 + static_cast<int>(threadIdx.x) < q.a.rows) {
#pragma unroll 8
            for (int k = 0; k < q.K; ++k) a_sum += q.a.p[k * q.a.ld + m0 + threadIdx.x];
            q.a_sums[m0 + threadIdx.x] = a_sum;
        }
        return;
    }
    float acc[T::RM][T::RN] = {};
    const auto copy_b = [&](uint32_t dst, int k0, int s) {
        copy_slab<T, T::TN, B_KMAJOR, VEC>(dst, q.b.p + (SEGMENTS ? s * q.b.seg : 0), q.b.ld, q.b.rows, n0, k0, q.K);
    };
    if (SEGMENTS && q.a_sums && n0 == 0) {
        tile_product<T, A_KMAJOR, B_KMAJOR, VEC, true, SEGMENTS>(sm, q.a, m0, q.K, q.n_seg, copy_b, acc, a_sum);
        if (threadIdx.x < T::TM && m0 + static_cast<int>(threadIdx.x) < q.a.rows) q.a_sums[m0 + threadIdx.x] = a_sum;
    } else {
        tile_product<T, A_KMAJOR, B_KMAJOR, VEC, false, SEGMENTS>(sm, q.a, m0, q.K, q.n_seg, copy_b, acc, a_sum);
    }
    const int tx = threadIdx.x % T::TX, ty = threadIdx.x / T::TX;
#pragma unroll
    for (int i = 0; i < T::RM; ++i) {
        const int m = m0 + result_at<T::RM, T::TY, A_KMAJOR>(ty, i);
        if (m >= q.a.rows) continue;
#pragma unroll
        for (int j = 0; j < T::RN; ++j) {
            const int n = n0 + result_at<T::RN, T::TX, B_KMAJOR>(tx, j);
            if (n < q.b.rows) q.c[m * q.ldc + n] = acc[i][j];
        }
    }
}

template <typename T, bool A_KMAJOR, bool B_KMAJOR, bool VEC, bool SEGMENTS>
__global__ void __launch_bounds__(T::kThreads) k_products(const __grid_constant__ ProductList list) {
    __shared__ __align__(16) Slabs<T, A_KMAJOR, B_KMAJOR> sm;
    dependency_wait();
    launch_dependents();
    int which = 0;
    while (which + 1 < list.n && static_cast<int>(blockIdx.x) >= list.p[which + 1].tile0) ++which;
    run_product<T, A_KMAJOR, B_KMAJOR, VEC, SEGMENTS>(sm, list.p[which], blockIdx.x - list.p[which].tile0);
}

// ---- emission head and its density ---------------------------------------------------------------------------------
// head = v W4^T + b4 for T::TM rows x 32 workers: the tile's columns are the means of its workers, then their log-variances,
// so a thread (columns tx, tx + 16, tx + 32, tx + 48) holds both halves of two workers, and at once
//   log N(x; m, exp(lv)) summed over the tile's workers -> part[tile column][row],
//   d_head = [r inv | -1/2 + r^2 inv / 2],  r = x - m, inv = exp(-lv)                    (d_head: null = forward only).
constexpr int kHeadWorkers = LargeTile::TN / 2;

template <typename T, bool VEC>
__global__ void __launch_bounds__(T::kThreads) k_emission_density(const float* __restrict__ v, const float* __restrict__ W4,
                                                                             const float* __restrict__ b4, const float* __restrict__ x,
                                                                             int R, int N, int H, float* __restrict__ d_head,
                                                                             float* __restrict__ part) {
    __shared__ __align__(16) Slabs<T, true, true> sm;
    dependency_wait();
    const int head_tiles = (N + kHeadWorkers - 1) / kHeadWorkers;            // one-dimensional grid: rows reach 2^24
    const int m0 = blockIdx.x / head_tiles * T::TM, head_tile = blockIdx.x % head_tiles, j0 = head_tile * kHeadWorkers;
    const Operand a{v, H, 0, R};
    const auto copy_b = [&](uint32_t dst, int k0, int) {
#pragma unroll
        for (int u = threadIdx.x; u < T::TN * T::TK / 4; u += T::kThreads) {
            const int col = u / (T::TK / 4), k = k0 + u % (T::TK / 4) * 4;
            const int worker = j0 + col % kHeadWorkers, head = col / kHeadWorkers, valid = worker < N ? H - k : 0;
            copy4<VEC>(dst + 4 * (col * T::pitch(T::TN, true) + u % (T::TK / 4) * 4),
                       valid > 0 ? W4 + (static_cast<long long>(head) * N + worker) * H + k : W4, valid);
        }
    };
    float acc[T::RM][T::RN] = {};
    float unused = 0.f;
    tile_product<T, true, true, VEC, false, false>(sm, a, m0, H, 1, copy_b, acc, unused);
    static_assert(T::RN == 4 && 2 * T::TX == kHeadWorkers && T::TX == 16, "columns 0, 1 of a thread are means, 2, 3 their log-variances");
    const int tx = threadIdx.x % T::TX, ty = threadIdx.x / T::TX;
#pragma unroll
    for (int i = 0; i < T::RM; ++i) {
        const int r = m0 + result_at<T::RM, T::TY, true>(ty, i);
        float s = 0.f;
        if (r < R) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int j = j0 + tx + T::TX * c;
                if (j >= N) continue;
                const float mean = acc[i][c] + b4[j], lv = acc[i][2 + c] + b4[N + j];
                const float d = x[static_cast<long long>(r) * N + j] - mean, inv = expf(-lv);
                s += -0.5f * (kLog2Pi + lv + d * d * inv);
                if (d_head) {
                    d_head[static_cast<long long>(r) * 2 * N + j] = d * inv;
                    d_head[static_cast<long long>(r) * 2 * N + N + j] = -0.5f + 0.5f * d * d * inv;
                }
            }
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (tx == 0 && r < R) part[static_cast<long long>(head_tile) * R + r] = s;
    }
}

// elbo[b] = what the guide and the transition contributed + the emission densities of the window's rows (one warp)
__device__ __forceinline__ void window_elbo(const float* __restrict__ part, int n_part, int R, int W, int b,
                                            const float* __restrict__ path, float* __restrict__ elbo, int lane) {
    float s = 0.f;
    for (int i = lane; i < n_part * W; i += 32) s += part[static_cast<long long>(i / W) * R + b * W + i % W];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) elbo[b] = path[b] + s;
}
__global__ void __launch_bounds__(128) k_elbo_finish(const float* __restrict__ part, int n_part, int R, int W, int B,
                                                     const float* __restrict__ path, float* __restrict__ elbo) {
    dependency_wait();
    launch_dependents();
    const int b = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (b < B) window_elbo(part, n_part, R, W, b, path, elbo, threadIdx.x & 31);
}

// ---- the two RNNs --------------------------------------------------------------------------------------------------
// h_t = relu(P_t + Wh h_{t -+ 1}) for RW windows and one direction per cluster, all steps.  A CTA of the cluster owns
// ceil(H / cluster) hidden units: their share of Wh sits in its shared memory for all steps (or, if not even eight CTAs can hold
// it, passes through it in chunks of k at every step), one thread per unit runs the chains of the RW windows, and every
// new value is written into the next-state buffers of all CTAs of the cluster; one cluster barrier per step.  What
// bounds a step is shared-memory wavefronts: one per k and warp for the weights, RW / 4 for the states (H = 256: 2 CTAs, 128
// threads each, about 1500 clocks with RW = 2).
// States: [B][W + 1][H]; forward: slot 0 = a0, slot t + 1 = a_t;  backward: slot t = b_t, slot W = b0 -- so "the state
// before" of row t is slot t (forward) or slot t + 1 (backward).
struct RnnArgs {
    const float* proj;              // [R][2H]: input projections, forward then backward
    const float *Wh[2], *bias[2], *init[2];
    float* state[2];
    // backward pass
    const float* g;                 // [R][H]: d ELBO / d h_t from the combiner, the same for both directions
    float* d_pre[2];                // [R][H]
    float* carry_out[2];            // [B][H]: gradient of the initial state, per window
    int B, W, H;
    int cluster, units;             // CTAs per cluster, units per CTA
    int chunk;                      // k rows of the weights in shared memory at a time (H: all of them, loaded once)
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void store_all(float* p, float v, int cluster) {
    const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    for (int c = 0; c < cluster; ++c) {
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(c));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
    }
}

// Pitch of a window's state vector and of a weight row: both read without bank conflicts (rows of 16-byte chunks; the
// transposing copy writes consecutive k, so the pitch of a weight row is odd).
__host__ __device__ inline int rnn_state_pitch(int H) { return (H + 3) / 4 * 4; }
__host__ __device__ inline int rnn_weight_pitch(int units) { return units | 1; }
inline size_t rnn_smem_bytes(int H, int units, int chunk, int rw) {
    return sizeof(float) * (2 * static_cast<size_t>(rw) * rnn_state_pitch(H) + static_cast<size_t>(chunk) * rnn_weight_pitch(units));
}

// acc[w] += sum_k sW[k][unit] x[w][k0 + k] for k < n, ascending: one chain per window
template <int RW>
__device__ __forceinline__ void rnn_chains(const float* sW, int pitch, const float* x, int xp, int n, float (&acc)[RW]) {
    int k = 0;
#pragma unroll 2
    for (; k + 4 <= n; k += 4) {
        float4 xv[RW];
#pragma unroll
        for (int w = 0; w < RW; ++w) xv[w] = *reinterpret_cast<const float4*>(x + w * xp + k);
        const float w0 = sW[k * pitch], w1 = sW[(k + 1) * pitch], w2 = sW[(k + 2) * pitch], w3 = sW[(k + 3) * pitch];
#pragma unroll
        for (int w = 0; w < RW; ++w) acc[w] = fmaf(w3, xv[w].w, fmaf(w2, xv[w].z, fmaf(w1, xv[w].y, fmaf(w0, xv[w].x, acc[w]))));
    }
    for (; k < n; ++k)
#pragma unroll
        for (int w = 0; w < RW; ++w) acc[w] = fmaf(sW[k * pitch], x[w * xp + k], acc[w]);
}

template <int RW>
__global__ void __launch_bounds__(256) k_rnn_forward(RnnArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int H = a.H, W = a.W, xp = rnn_state_pitch(H), wp = rnn_weight_pitch(a.units), T = blockDim.x;
    const int rank = static_cast<int>(cluster_rank()), dir = blockIdx.y, b0 = static_cast<int>(blockIdx.x) / a.cluster * RW;
    const int u0 = rank * a.units, units = min(a.units, H - u0), tid = threadIdx.x;
    float* cur = sm;                                   // [RW][xp]
    float* next = sm + RW * xp;
    float* sW = sm + 2 * RW * xp;                      // [chunk][wp]: sW[k][u] = Wh[u0 + u][k]
    const float* Wh = a.Wh[dir] + static_cast<long long>(u0) * H;
    const auto stage = [&](int k0, int n) {
        copy_matrix_transposed(sW, wp, Wh + k0, H, units, n);
    };
    if (a.chunk >= H) stage(0, H);                     // weights: no kernel of this step writes them
    dependency_wait();
    launch_dependents();
    float* state = a.state[dir];
    for (int i = tid; i < RW * H; i += T) {
        const int w = i / H, h = i % H;
        const float s = a.init[dir][h];
        cur[w * xp + h] = s;
        if (rank == 0 && b0 + w < a.B) state[(static_cast<long long>(b0 + w) * (W + 1) + (dir ? W : 0)) * H + h] = s;
    }
    copies_landed();
    cluster_sync();                                    // every CTA has started before anyone writes into it
    const int h = u0 + tid;
    const bool mine = tid < units;
    const float bias = mine ? a.bias[dir][h] : 0.f;
    const auto projection = [&](int w, int s) {
        return mine && b0 + w < a.B && s < W ? a.proj[(static_cast<long long>(b0 + w) * W + (dir ? W - 1 - s : s)) * 2 * H + dir * H + h] : 0.f;
    };
    float ahead[RW];                                   // the next step's projections are requested a step early
#pragma unroll
    for (int w = 0; w < RW; ++w) ahead[w] = projection(w, 0);
    for (int s = 0; s < W; ++s) {
        const int t = dir ? W - 1 - s : s;
        float p[RW], acc[RW];
#pragma unroll
        for (int w = 0; w < RW; ++w) {
            acc[w] = 0.f;
            p[w] = ahead[w] + bias;
            ahead[w] = projection(w, s + 1);
        }
        for (int k0 = 0; k0 < H; k0 += a.chunk) {
            const int n = min(a.chunk, H - k0);
            if (a.chunk < H) {
                __syncthreads();
                stage(k0, n);
                copies_landed();
                __syncthreads();
            }
            if (mine) rnn_chains<RW>(sW + tid, wp, cur + k0, xp, n, acc);
        }
        if (mine) {
#pragma unroll
            for (int w = 0; w < RW; ++w) {
                const float v = fmaxf(acc[w] + p[w], 0.f);
                store_all(next + w * xp + h, v, a.cluster);
                if (b0 + w < a.B) state[(static_cast<long long>(b0 + w) * (W + 1) + (dir ? t : t + 1)) * H + h] = v;
            }
        }
        cluster_sync();
        float* swap = cur; cur = next; next = swap;
    }
}

// One step of both recurrences as a product over all windows, for batches so large that the clusters would take turns: a tile of
// windows x units per CTA, a launch per step.  The same chain per result as above.
template <typename T, bool VEC>
__global__ void __launch_bounds__(T::kThreads) k_rnn_step(RnnArgs a, int s) {
    __shared__ __align__(16) Slabs<T, true, true> sm;
    dependency_wait();
    const int H = a.H, W = a.W, dir = blockIdx.y, t = dir ? W - 1 - s : s, unit_tiles = (H + T::TN - 1) / T::TN;
    const int m0 = static_cast<int>(blockIdx.x) / unit_tiles * T::TM, n0 = static_cast<int>(blockIdx.x) % unit_tiles * T::TN;
    const long long pitch = static_cast<long long>(W + 1) * H;             // from one window's states to the next's
    float* const state = a.state[dir];
    float* const before = state + static_cast<long long>(dir ? t + 1 : t) * H;
    float* const after = state + static_cast<long long>(dir ? t : t + 1) * H;
    // the initial state is the same for every window
    const Operand x{s == 0 ? a.init[dir] : before, s == 0 ? 0 : pitch, 0, a.B};
    const auto copy_b = [&](uint32_t dst, int k0, int) { copy_slab<T, T::TN, true, VEC>(dst, a.Wh[dir], H, H, n0, k0, H); };
    float acc[T::RM][T::RN] = {};
    float unused = 0.f;
    tile_product<T, true, true, VEC, false, false>(sm, x, m0, H, 1, copy_b, acc, unused);
    const int tx = threadIdx.x % T::TX, ty = threadIdx.x / T::TX;
#pragma unroll
    for (int i = 0; i < T::RM; ++i) {
        const int b = m0 + result_at<T::RM, T::TY, true>(ty, i);
        if (b >= a.B) continue;
#pragma unroll
        for (int j = 0; j < T::RN; ++j) {
            const int h = n0 + result_at<T::RN, T::TX, true>(tx, j);
            if (h >= H) continue;
            const float p = a.proj[(static_cast<long long>(b) * W + t) * 2 * H + dir * H + h] + a.bias[dir][h];
            after[b * pitch + h] = fmaxf(acc[i][j] + p, 0.f);
            if (s == 0) state[b * pitch + static_cast<long long>(dir ? W : 0) * H + h] = a.init[dir][h];
        }
    }
}

// Backwards through the same recurrences: d_pre_t = (g_t + carry) (h_t > 0), carry = d_pre_t Wh: a CTA owns columns of Wh.
template <int RW>
__global__ void __launch_bounds__(256) k_rnn_backward(RnnArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int H = a.H, W = a.W, xp = rnn_state_pitch(H), wp = rnn_weight_pitch(a.units);
    const int rank = static_cast<int>(cluster_rank()), dir = blockIdx.y, b0 = static_cast<int>(blockIdx.x) / a.cluster * RW;
    const int u0 = rank * a.units, units = min(a.units, H - u0), tid = threadIdx.x;
    float* cur = sm;                                   // [RW][xp]: d_pre of this step, all units
    float* next = sm + RW * xp;
    float* sW = sm + 2 * RW * xp;                      // [chunk][wp]: sW[i][u] = Wh[i][u0 + u]
    const float* Wh = a.Wh[dir] + u0;
    const auto stage = [&](int k0, int n) {
        copy_matrix(sW, wp, Wh + static_cast<long long>(k0) * H, H, n, units);
    };
    if (a.chunk >= H) stage(0, H);
    dependency_wait();
    copies_landed();
    cluster_sync();
    const int h = u0 + tid;
    const bool mine = tid < units;
    float carry[RW];
#pragma unroll
    for (int w = 0; w < RW; ++w) carry[w] = 0.f;
    float g[RW], act[RW];                              // of the coming step, requested a step early
    const auto fetch = [&](int s) {
        const int t = dir ? s : W - 1 - s;
#pragma unroll
        for (int w = 0; w < RW; ++w) {
            const bool there = mine && b0 + w < a.B && s < W;
            g[w] = there ? a.g[(static_cast<long long>(b0 + w) * W + t) * H + h] : 0.f;
            act[w] = there ? a.state[dir][(static_cast<long long>(b0 + w) * (W + 1) + (dir ? t : t + 1)) * H + h] : 0.f;
        }
    };
    fetch(0);
    for (int s = 0; s < W; ++s) {
        const int t = dir ? s : W - 1 - s;
        if (mine) {
#pragma unroll
            for (int w = 0; w < RW; ++w) {
                const float d = act[w] > 0.f ? g[w] + carry[w] : 0.f;
                if (b0 + w < a.B) a.d_pre[dir][(static_cast<long long>(b0 + w) * W + t) * H + h] = d;
                store_all(cur + w * xp + h, d, a.cluster);
                carry[w] = 0.f;
            }
        }
        cluster_sync();
        fetch(s + 1);
        for (int k0 = 0; k0 < H; k0 += a.chunk) {
            const int n = min(a.chunk, H - k0);
            if (a.chunk < H) {
                __syncthreads();
                stage(k0, n);
                copies_landed();
                __syncthreads();
            }
            if (mine) rnn_chains<RW>(sW + tid, wp, cur + k0, xp, n, carry);
        }
        // the other buffer is written next: its readers passed the cluster barrier of this step
        float* swap = cur; cur = next; next = swap;
    }
    if (mine)
#pragma unroll
        for (int w = 0; w < RW; ++w)
            if (b0 + w < a.B) a.carry_out[dir][static_cast<long long>(b0 + w) * H + h] = carry[w];
    cluster_sync();                                    // nobody leaves while others may still write into its buffers
}

// ---- the sampled path: guide, transition density, hidden layers -------------------------------------------------------
// One CTA per window.  The small matrices sit in shared memory (rows padded to an odd length) when they fit.  A latent
// result is a chain over the H hidden units, one thread each (D to 3D of them): about 5 clocks per unit.
constexpr int kPathThreads = 256;

struct PathArgs {
    // weights
    const float *Wz, *bz, *Wmu, *bmu, *Wsig, *bsig, *z0, *W1, *b1, *W2, *b2, *W3, *b3;
    // saved activations, rows r = b*W + t (z: [B][W + 1][D], slot 0 = z0)
    const float *a, *b;             // RNN states [B][W + 1][H]
    const float* eps;               // [R][D]
    float *comb, *hout, *mu, *presig, *z, *u, *v, *dhz;
    float* dzt;                     // [R][D]: d log p(z_t | z_{t-1}) / d z_t
    float* path;                    // [B]: guide and transition part of the ELBO
    // backward
    const float* part;              // emission densities, see k_emission_density
    int n_part;
    float* elbo;
    const float* dv_raw;            // [R][H]: d_head W4
    float *dv, *du, *dpc, *dh, *dmu, *dps;
    float* gz0;                     // [B][D]
    int B, W, D, H;
};

// sum_i M[row][i] in[i], one chain from zero
__device__ __forceinline__ float row_dot(const float* M, int ld, int row, const float* in, int n) {
    const float* p = M + static_cast<long long>(row) * ld;
    float s = 0.f;
#pragma unroll 16
    for (int i = 0; i < n; ++i) s = fmaf(p[i], in[i], s);
    return s;
}
// sum_i M[i][col] in[i], one chain from zero
__device__ __forceinline__ float col_dot(const float* M, int ld, int col, const float* in, int n) {
    float s = 0.f;
#pragma unroll 16
    for (int i = 0; i < n; ++i) s = fmaf(M[static_cast<long long>(i) * ld + col], in[i], s);
    return s;
}

struct PathWeights {
    const float *Wz, *W1, *W3;      // [H][ldd]
    const float *Wmu, *W2;          // [D][ldh], [2D][ldh]
    int ldd, ldh;
};
inline size_t path_weight_floats(int D, int H) {
    return 3 * static_cast<size_t>(H) * (D | 1) + 3 * static_cast<size_t>(D) * (H | 1);
}
// What a step reads from global memory is copied to shared memory a step early: 4 rows of H, 5 of D, twice.
inline size_t path_scratch_floats(int D, int H) { return 11 * static_cast<size_t>(H) + 18 * static_cast<size_t>(D) + 64; }

__device__ __forceinline__ PathWeights path_weights(const PathArgs& a, float* sm, bool staged) {
    if (!staged) return PathWeights{a.Wz, a.W1, a.W3, a.Wmu, a.W2, a.D, a.H};
    PathWeights w;
    w.ldd = a.D | 1;
    w.ldh = a.H | 1;
    const auto put = [&](const float* src, int rows, int cols, int ld) {
        float* dst = sm;
        copy_matrix(dst, ld, src, cols, rows, cols);
        sm += rows * ld;
        return dst;
    };
    w.Wz = put(a.Wz, a.H, a.D, w.ldd);
    w.W1 = put(a.W1, a.H, a.D, w.ldd);
    w.W3 = put(a.W3, a.H, a.D, w.ldd);
    w.Wmu = put(a.Wmu, a.D, a.H, w.ldh);
    w.W2 = put(a.W2, 2 * a.D, a.H, w.ldh);
    return w;
}

// Where the matrices do not fit, they pass through kPathBuffer floats of shared memory at every step, some rows (some columns of
// W_mu and W_2) at a time.  With a thread per row reading its row from global memory instead, forward passes of five steps, N=64, D=64,
// took: H=256, 300 windows 954 us (this way 541), H=512, 64 windows 770 us (552).
constexpr int kPathBuffer = 16 * 1024;

template <bool STAGED>
__global__ void __launch_bounds__(kPathThreads) k_path_forward(PathArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int D = a.D, H = a.H, W = a.W, b = blockIdx.x, tid = threadIdx.x;
    float* z = sm;                   // [D]
    float* mu = z + D;               // [D]
    float* zp = mu + D;              // [D]
    float* hz = zp + D;              // [2D]
    float* h = sm + 8 * D;           // [2][H] (of 3)
    float* scal = h + 3 * H;         // [64]
    float* ahead = scal + 64;        // [2]: h_left, h_right (H each), eps (D)
    const int ahead_n = 4 * H + 5 * D, ldd = D | 1;
    float* buffer = ahead + 2 * ahead_n;
    PathWeights w{};
    if constexpr (STAGED) {
        w = path_weights(a, buffer, true);
        // addresses of unknown space: in loads that it knows to be from shared memory the compiler puts the chains' loads between their
        // multiply-adds (10 us more per five steps)
        asm volatile("" : "+l"(w.Wz), "+l"(w.W1), "+l"(w.W3), "+l"(w.Wmu), "+l"(w.W2));
    }
    dependency_wait();
    const auto fetch = [&](int t) {
        float* dst = ahead + (t & 1) * ahead_n;
        copy_vector(dst, a.a + (static_cast<long long>(b) * (W + 1) + t + 1) * H, H);
        copy_vector(dst + H, a.b + (static_cast<long long>(b) * (W + 1) + t) * H, H);
        copy_vector(dst + 2 * H, a.eps + (static_cast<long long>(b) * W + t) * D, D);
    };
    fetch(0);
    for (int d = tid; d < D; d += kPathThreads) { z[d] = a.z0[d]; a.z[static_cast<long long>(b) * (W + 1) * D + d] = a.z0[d]; }
    float elbo = 0.f;                // of this thread's latent dimensions
    for (int t = 0; t < W; ++t) {
        const long long r = static_cast<long long>(b) * W + t;
        const float* sa = ahead + (t & 1) * ahead_n;
        const float* sb = sa + H;
        const float* eps = sb + H;
        copies_landed();
        __syncthreads();
        if (t + 1 < W) fetch(t + 1);
        // hidden layers that read z_{t-1}: the combiner and the transition's
        const auto hidden = [&](const float* Wz, const float* W1, int i, int row) {
            const float c = tanhf(row_dot(Wz, ldd, row, z, D) + a.bz[i]);
            const float o = (c + sa[i] + sb[i]) * (1.f / 3.f);
            const float u = fmaxf(row_dot(W1, ldd, row, z, D) + a.b1[i], 0.f);
            a.comb[r * H + i] = c;
            a.hout[r * H + i] = o;
            a.u[r * H + i] = u;
            h[i] = o;
            h[H + i] = u;
        };
        if constexpr (STAGED) {
            for (int i = tid; i < H; i += kPathThreads) hidden(w.Wz, w.W1, i, i);
        } else {
            const int rows = kPathBuffer / (2 * ldd);
            for (int r0 = 0; r0 < H; r0 += rows) {
                const int n = min(rows, H - r0);
                __syncthreads();
                copy_matrix(buffer, ldd, a.Wz + static_cast<long long>(r0) * D, D, n, D);
                copy_matrix(buffer + rows * ldd, ldd, a.W1 + static_cast<long long>(r0) * D, D, n, D);
                copies_landed();
                __syncthreads();
                for (int i = tid; i < n; i += kPathThreads) hidden(buffer, buffer + rows * ldd, r0 + i, i);
            }
        }
        __syncthreads();
        if constexpr (STAGED) {
            for (int o = tid; o < 3 * D; o += kPathThreads) {
                if (o < D) mu[o] = row_dot(w.Wmu, w.ldh, o, h, H) + a.bmu[o];
                else hz[o - D] = row_dot(w.W2, w.ldh, o - D, h + H, H) + a.b2[o - D];
            }
        } else {
            // D <= 64: a result per thread, its chain in pieces
            const int cols = kPathBuffer / (3 * D) - 1, ld = cols | 1;
            const float* in = tid < D ? h : h + H;
            float s = 0.f;
            for (int k0 = 0; k0 < H; k0 += cols) {
                const int n = min(cols, H - k0);
                __syncthreads();
                copy_matrix(buffer, ld, a.Wmu + k0, H, D, n);
                copy_matrix(buffer + D * ld, ld, a.W2 + k0, H, 2 * D, n);
                copies_landed();
                __syncthreads();
                if (tid < 3 * D) {
                    const float* p = buffer + tid * ld;
#pragma unroll 16
                    for (int k = 0; k < n; ++k) s = fmaf(p[k], in[k0 + k], s);
                }
            }
            if (tid < D) mu[tid] = s + a.bmu[tid];
            else if (tid < 3 * D) hz[tid - D] = s + a.b2[tid - D];
        }
        __syncthreads();
        for (int d = tid; d < D; d += kPathThreads) {
            const float pre = row_dot(a.Wsig, D, d, mu, D) + a.bsig[d];
            const float sg = softplus_f(pre), e = eps[d], zt = fmaf(sg, e, mu[d]);
            a.mu[r * D + d] = mu[d];
            a.presig[r * D + d] = pre;
            a.z[(static_cast<long long>(b) * (W + 1) + t + 1) * D + d] = zt;
            zp[d] = zt;
            elbo += 0.5f * kLog2Pi + logf(sg) + 0.5f * e * e;                 // - log q
            const float lv = hz[D + d], rr = zt - hz[d], inv = expf(-lv);
            elbo += -0.5f * (kLog2Pi + lv + rr * rr * inv);                  // log p(z_t | z_{t-1})
            a.dzt[r * D + d] = -rr * inv;
            a.dhz[r * 2 * D + d] = rr * inv;
            a.dhz[r * 2 * D + D + d] = -0.5f + 0.5f * rr * rr * inv;
        }
        __syncthreads();
        const auto emission = [&](const float* W3, int i, int row) {
            a.v[r * H + i] = fmaxf(row_dot(W3, ldd, row, zp, D) + a.b3[i], 0.f);
        };
        if constexpr (STAGED) {
            for (int i = tid; i < H; i += kPathThreads) emission(w.W3, i, i);
        } else {
            const int rows = kPathBuffer / ldd;
            for (int r0 = 0; r0 < H; r0 += rows) {
                const int n = min(rows, H - r0);
                __syncthreads();
                copy_matrix(buffer, ldd, a.W3 + static_cast<long long>(r0) * D, D, n, D);
                copies_landed();
                __syncthreads();
                for (int i = tid; i < n; i += kPathThreads) emission(buffer, r0 + i, i);
            }
        }
        float* swap = z; z = zp; zp = swap;            // h, mu and hz are rewritten behind the next barriers
    }
    // D <= 64: the sums sit in the first two warps
    if (tid < 64) scal[tid] = elbo;
    __syncthreads();
    if (tid == 0) {
        float s = 0.f;
        for (int d = 0; d < D; ++d) s += scal[d];
        a.path[b] = s;
    }
}

__global__ void __launch_bounds__(kPathThreads) k_path_backward(PathArgs a, bool staged) {
    extern __shared__ __align__(16) float sm[];
    const int D = a.D, H = a.H, W = a.W, b = blockIdx.x, tid = threadIdx.x;
    float* gz = sm;                  // [D]   d ELBO / d z_t
    float* gzp = gz + D;             // [D]   d ELBO / d z_{t-1}
    float* dmu = gzp + D;            // [D]
    float* dps = dmu + D;            // [D]
    float* h = sm + 8 * D;           // [3][H]: dv, du, dpc
    float* ahead = h + 3 * H + 64;   // [2]: v, u, d_head W4, comb (H each), d transition head (2D), dzt, presig, eps (D each)
    const int ahead_n = 4 * H + 5 * D;
    const PathWeights w = path_weights(a, ahead + 2 * ahead_n, staged);
    for (int d = tid; d < D; d += kPathThreads) gzp[d] = 0.f;
    dependency_wait();
    launch_dependents();
    const auto fetch = [&](int t) {
        float* dst = ahead + (t & 1) * ahead_n;
        const long long r = static_cast<long long>(b) * W + t;
        copy_vector(dst, a.v + r * H, H);
        copy_vector(dst + H, a.u + r * H, H);
        copy_vector(dst + 2 * H, a.dv_raw + r * H, H);
        copy_vector(dst + 3 * H, a.comb + r * H, H);
        copy_vector(dst + 4 * H, a.dhz + r * 2 * D, 2 * D);
        copy_vector(dst + 4 * H + 2 * D, a.dzt + r * D, D);
        copy_vector(dst + 4 * H + 3 * D, a.presig + r * D, D);
        copy_vector(dst + 4 * H + 4 * D, a.eps + r * D, D);
    };
    fetch(W - 1);
    if (tid >= kPathThreads - 32) window_elbo(a.part, a.n_part, a.B * W, W, b, a.path, a.elbo, tid & 31);
    for (int t = W - 1; t >= 0; --t) {
        const long long r = static_cast<long long>(b) * W + t;
        const float* v = ahead + (t & 1) * ahead_n;
        const float *u = v + H, *dv_raw = u + H, *comb = dv_raw + H, *dhz = comb + H, *dzt = dhz + 2 * D, *presig = dzt + D, *eps = presig + D;
        copies_landed();
        __syncthreads();
        if (t > 0) fetch(t - 1);
        for (int d = tid; d < D; d += kPathThreads) gz[d] = gzp[d] + dzt[d];
        // hidden-layer gradients of the emission and of the transition
        for (int i = tid; i < H; i += kPathThreads) {
            const float dv = v[i] > 0.f ? dv_raw[i] : 0.f;
            const float du = u[i] > 0.f ? col_dot(w.W2, w.ldh, i, dhz, 2 * D) : 0.f;
            a.dv[r * H + i] = dv;
            a.du[r * H + i] = du;
            h[i] = dv;
            h[H + i] = du;
        }
        __syncthreads();
        // the two sums in different warps: each is a chain over H
        for (int d = tid; d < 64 + D; d += kPathThreads) {
            if (d < D) gz[d] = col_dot(w.W3, w.ldd, d, h, H) + gz[d];
            else if (d >= 64) gzp[d - 64] = col_dot(w.W1, w.ldd, d - 64, h + H, H);
        }
        __syncthreads();
        // guide: d_mu = g_z + Wsig^T d_pre_sig,  d_pre_sig = (g_z eps + 1 / sigma) sigmoid(pre_sig)
        for (int d = tid; d < D; d += kPathThreads) {
            const float pre = presig[d];
            const float p = fmaf(gz[d], eps[d], 1.f / softplus_f(pre)) * sigmoid_f(pre);
            dps[d] = p;
            a.dps[r * D + d] = p;
        }
        __syncthreads();
        for (int d = tid; d < D; d += kPathThreads) {
            const float s = col_dot(a.Wsig, D, d, dps, D) + gz[d];
            dmu[d] = s;
            a.dmu[r * D + d] = s;
        }
        __syncthreads();
        for (int i = tid; i < H; i += kPathThreads) {
            const float s = col_dot(w.Wmu, w.ldh, i, dmu, D) * (1.f / 3.f);
            const float c = comb[i];
            a.dh[r * H + i] = s;
            const float p = s * (1.f - c * c);
            a.dpc[r * H + i] = p;
            h[2 * H + i] = p;
        }
        __syncthreads();
        for (int d = tid; d < D; d += kPathThreads) gzp[d] = col_dot(w.Wz, w.ldd, d, h + 2 * H, H) + gzp[d];
        __syncthreads();
    }
    for (int d = tid; d < D; d += kPathThreads) a.gz0[static_cast<long long>(b) * D + d] = gzp[d];
}

// ---- Adam with clipping by the global norm (Kingma & Ba 2015; Section 4.1) ---------------------------------------
// pass 1: partial sums of squares of scale * g, one per CTA (fixed order); pass 2: every CTA adds them in the same order
constexpr int kNormThreads = 256;
constexpr int kNormParts = 256;
__global__ void __launch_bounds__(kNormThreads) k_sumsq_partial(const float* __restrict__ g, long long n, float scale,
                                                                 double* __restrict__ partial) {
    __shared__ double red[kNormThreads];
    double s = 0.0;
    for (long long i = static_cast<long long>(blockIdx.x) * kNormThreads + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * kNormThreads) {
        const double v = static_cast<double>(g[i]) * scale;
        s += v * v;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int half = kNormThreads / 2; half > 0; half >>= 1) {
        if (threadIdx.x < half) red[threadIdx.x] += red[threadIdx.x + half];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}
// g' = scale * g, clipped: g' *= clip / norm if norm > clip; then the Adam update of step t (t >= 1).  Every CTA forms
// the norm from the partial sums by the same tree, so no launch of its own is spent on it.
__global__ void __launch_bounds__(kNormThreads) k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                                                       float* __restrict__ v, long long n, float scale,
                                                       const double* __restrict__ partial, int n_part, float* __restrict__ norm_out,
                                                       float clip, float lr, float beta1, float beta2, float eps, float corr1,
                                                       float corr2) {
    __shared__ double red[kNormThreads];
    red[threadIdx.x] = threadIdx.x < n_part ? partial[threadIdx.x] : 0.0;
    __syncthreads();
    for (int half = kNormThreads / 2; half > 0; half >>= 1) {
        if (threadIdx.x < half) red[threadIdx.x] += red[threadIdx.x + half];
        __syncthreads();
    }
    const float nm = static_cast<float>(sqrt(red[0]));
    if (blockIdx.x == 0 && threadIdx.x == 0) *norm_out = nm;
    const float shrink = nm > clip ? clip / nm : 1.f;
    for (long long i = static_cast<long long>(blockIdx.x) * kNormThreads + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * kNormThreads) {
        const float gs = g[i] * scale * shrink;
        const float mi = beta1 * m[i] + (1.f - beta1) * gs;
        const float vi = beta2 * v[i] + (1.f - beta2) * gs * gs;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / corr1) / (sqrtf(vi / corr2) + eps);
    }
}

}  // namespace fit
}  // namespace cutoff
