// Learning the model on the GPU: the one-sample, reparameterised ELBO of Section 3.1.3 for a batch of windows,
// its gradient with respect to every weight tensor (reverse mode, layer by layer), and Adam with clipping by the
// global norm (Section 4.1), for the compact networks, in fp32.
//
//   ELBO_b = sum_t  log p(x_t | z_t) + log p(z_t | z_{t-1}) - log q(z_t | z_{t-1}, x),     z_t = mu_t + sigma_t eps_t,
//   log N(y; m, exp(lv)) = -1/2 [log 2 pi + lv + (y - m)^2 exp(-lv)],   log q = sum_d -1/2 log 2 pi - log sigma_d - eps_d^2 / 2.
//
// What bounds a step is the number of dependent launches, not its arithmetic (64 windows of the n1024 model: 1.0 G
// multiply-adds, 28 us at the FMA rate), so the step is laid out by what depends on what.  Only the recurrences depend
// on the previous step of a window, and only within the window: one CTA walks through all of a window's steps (of a few
// windows' steps for the RNNs) in one launch.  Everything else is one product over all B*W (window, step) rows: the
// input projections, the emission head with its density in the epilogue, the input gradient of the emission head, and
// all weight gradients together in one launch over a list of products.  Nine launches per step.  Measured with Adam, 64
// windows: N = 128, H = 128 replayed as a graph 677 -> 99 us, N = 1024, H = 256 launched one by one 2.95 -> 0.295 ms,
// against one launch per layer, step and orientation (about 150 of them).
//
// Rows are window-major: row r = b*W + t.  Every reduction runs in a fixed order (no floating-point atomics), so a step
// is reproducible bit for bit.
#pragma once
#include <cmath>

#include "common.cuh"

namespace cutoff {
namespace fit {

constexpr float kLog2Pi = 1.8378770664093453f;

__device__ __forceinline__ float softplus_f(float v) { return v > 20.f ? v : log1pf(expf(v)); }
__device__ __forceinline__ float sigmoid_f(float v) { return 1.f / (1.f + expf(-v)); }

// ---- tiled products ----------------------------------------------------------------------------------------------
// C[m][n] = sum_k A(m, k) B(n, k) over 64 x 64 tiles, 16 k at a time, 4 x 4 per thread, the next slab's global loads in
// flight while the current one is multiplied.  An operand is either "k-major" (element (m, k) at m*ld + k) or
// "m-major" (element (m, k) at k*ld + m), so the three orientations a dense layer needs are X W^T, dY W and dY^T X.
constexpr int kTile = 64, kTileK = 16, kGemmThreads = 256, kTilePad = kTile + 4;

struct Operand {
    const float* p;
    long long ld;
    int rows;            // valid m (the other dimension of the product is bounded by its K)
    int skip_every;      // m-major: row k of the product is row k + k / skip_every + skip_first of the array (0: row k)
    int skip_first;
};
struct Product {
    Operand a, b;
    float* c;
    long long ldc;
    float* a_sums;       // column sums of an m-major A (bias gradient), written by the first column of tiles; or null
    int K;
    int tile0, tiles_n;  // first tile of this product in the launch, tiles per tile row
};

// One thread's share of a 64 x 16 slab: 4 values along the operand's contiguous dimension.
template <bool K_MAJOR, bool VEC>
__device__ __forceinline__ float4 load_slab(const Operand& o, int m0, int k0, int K, int tid) {
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (K_MAJOR) {
        const int m = m0 + (tid >> 2), k = k0 + (tid & 3) * 4;
        if (m < o.rows) {
            const float* p = o.p + m * o.ld + k;
            if (VEC && k + 3 < K) return *reinterpret_cast<const float4*>(p);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (k + i < K) v[i] = p[i];
        }
    } else {
        const int k = k0 + (tid >> 4), m = m0 + (tid & 15) * 4;
        if (k < K) {
            const long long row = o.skip_every ? k + k / o.skip_every + o.skip_first : k;
            const float* p = o.p + row * o.ld + m;
            if (VEC && m + 3 < o.rows) return *reinterpret_cast<const float4*>(p);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (m + i < o.rows) v[i] = p[i];
        }
    }
    return make_float4(v[0], v[1], v[2], v[3]);
}
template <bool K_MAJOR>
__device__ __forceinline__ void store_slab(float (*s)[kTilePad], const float4& v, int tid) {
    if (K_MAJOR) {
        const int m = tid >> 2, k = (tid & 3) * 4;
        s[k][m] = v.x; s[k + 1][m] = v.y; s[k + 2][m] = v.z; s[k + 3][m] = v.w;
    } else {
        *reinterpret_cast<float4*>(&s[tid >> 4][(tid & 15) * 4]) = v;
    }
}

struct TileSmem {
    float a[2][kTileK][kTilePad];
    float b[2][kTileK][kTilePad];
};

// acc += A(m0.., k) B(n0.., k) for k in [k_begin, k_end).  load_b(k0) supplies the thread's share of B's slab.
template <bool A_KMAJOR, bool B_KMAJOR, bool VEC, bool SUMS, typename LoadB>
__device__ __forceinline__ void tile_product(TileSmem& sm, const Operand& a, int m0, int k_begin, int k_end, LoadB load_b,
                                             float (&acc)[4][4], float& a_sum) {
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float4 ra = load_slab<A_KMAJOR, VEC>(a, m0, k_begin, k_end, tid), rb = load_b(k_begin);
    int buf = 0;
    for (int k0 = k_begin; k0 < k_end; k0 += kTileK, buf ^= 1) {
        store_slab<A_KMAJOR>(sm.a[buf], ra, tid);
        store_slab<B_KMAJOR>(sm.b[buf], rb, tid);
        __syncthreads();
        if (k0 + kTileK < k_end) {
            ra = load_slab<A_KMAJOR, VEC>(a, m0, k0 + kTileK, k_end, tid);
            rb = load_b(k0 + kTileK);
        }
#pragma unroll
        for (int k = 0; k < kTileK; ++k) {
            const float4 av = *reinterpret_cast<const float4*>(&sm.a[buf][k][4 * ty]);
            const float4 bv = *reinterpret_cast<const float4*>(&sm.b[buf][k][4 * tx]);
            const float x[4] = {av.x, av.y, av.z, av.w}, y[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(x[i], y[j], acc[i][j]);
        }
        if (SUMS && tid < kTile) {
#pragma unroll
            for (int k = 0; k < kTileK; ++k) a_sum += sm.a[buf][k][tid];
        }
        // the other buffer is written next; whoever still reads this one is at most one slab behind (one barrier per slab)
    }
    __syncthreads();
}

__device__ __forceinline__ void store_tile(float* c, long long ldc, int m0, int n0, int M, int N, const float (&acc)[4][4]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, n = n0 + 4 * tx;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + 4 * ty + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (n + j < N) c[m * ldc + n + j] = acc[i][j];
    }
}

// A list of products in one launch, K split over gridDim.y parts: part y goes to c + y * part_stride and whoever uses
// the result adds the parts in order.  Parts are multiples of kTileK.
constexpr int kMaxProducts = 16;
struct ProductList {
    Product p[kMaxProducts];
    int n;
    int k_part;
    long long part_stride;
};

template <bool A_KMAJOR, bool B_KMAJOR, bool VEC>
__global__ void __launch_bounds__(kGemmThreads, 2) k_products(const __grid_constant__ ProductList list) {
    __shared__ __align__(16) TileSmem sm;
    dependency_wait();
    launch_dependents();
    int which = 0;
    while (which + 1 < list.n && static_cast<int>(blockIdx.x) >= list.p[which + 1].tile0) ++which;
    const Product& q = list.p[which];
    const int tile = blockIdx.x - q.tile0, m0 = tile / q.tiles_n * kTile, n0 = tile % q.tiles_n * kTile;
    const int k_begin = blockIdx.y * list.k_part;
    const int k_end = min(q.K, k_begin + list.k_part);
    float acc[4][4] = {};
    float a_sum = 0.f;
    const auto load_b = [&](int k0) { return load_slab<B_KMAJOR, VEC>(q.b, n0, k0, k_end, threadIdx.x); };
    if (q.b.rows == 0) {                       // column sums only: sum_k A(m, k)
        if (threadIdx.x < kTile && m0 + static_cast<int>(threadIdx.x) < q.a.rows) {
            for (int k = k_begin; k < k_end; ++k) a_sum += q.a.p[k * q.a.ld + m0 + threadIdx.x];
            q.a_sums[m0 + threadIdx.x] = a_sum;
        }
        return;
    }
    if (q.a_sums && n0 == 0) {
        tile_product<A_KMAJOR, B_KMAJOR, VEC, true>(sm, q.a, m0, k_begin, k_end, load_b, acc, a_sum);
        if (threadIdx.x < kTile && m0 + static_cast<int>(threadIdx.x) < q.a.rows) q.a_sums[m0 + threadIdx.x] = a_sum;
    } else {
        tile_product<A_KMAJOR, B_KMAJOR, VEC, false>(sm, q.a, m0, k_begin, k_end, load_b, acc, a_sum);
    }
    store_tile(q.c + blockIdx.y * list.part_stride, q.ldc, m0, n0, q.a.rows, q.b.rows, acc);
}

// ---- emission head and its density ---------------------------------------------------------------------------------
// head = v W4^T + b4 for 64 rows x 32 workers (32 means and 32 log-variances: the tile's columns 4t .. 4t+3 are the
// means, then the log-variances, of workers 2t and 2t+1, so a thread holds both halves of its workers), and at once
//   log N(x; m, exp(lv)) summed over the tile's workers -> part[tile column][row],
//   d_head = [r inv | -1/2 + r^2 inv / 2],  r = x - m, inv = exp(-lv)                    (d_head: null = forward only).
constexpr int kHeadWorkers = kTile / 2;

template <bool VEC>
__global__ void __launch_bounds__(kGemmThreads, 2) k_emission_density(const float* __restrict__ v, const float* __restrict__ W4,
                                                                      const float* __restrict__ b4, const float* __restrict__ x,
                                                                      int R, int N, int H, float* __restrict__ d_head,
                                                                      float* __restrict__ part) {
    __shared__ __align__(16) TileSmem sm;
    dependency_wait();
    launch_dependents();
    const int head_tiles = (N + kHeadWorkers - 1) / kHeadWorkers;          // one-dimensional grid: rows reach 2^24
    const int m0 = blockIdx.x / head_tiles * kTile, head_tile = blockIdx.x % head_tiles, j0 = head_tile * kHeadWorkers;
    const Operand a{v, H, R, 0, 0};
    const int tid = threadIdx.x, col = tid >> 2;                             // the column of B this thread loads
    const int worker = j0 + 2 * (col >> 2) + (col & 1), head = (col >> 1) & 1;
    const float* wrow = W4 + (static_cast<long long>(head) * N + (worker < N ? worker : 0)) * H;
    const auto load_b = [&](int k0) {
        const int k = k0 + (tid & 3) * 4;
        if (worker >= N) return make_float4(0.f, 0.f, 0.f, 0.f);
        if (VEC && k + 3 < H) return *reinterpret_cast<const float4*>(wrow + k);
        float t[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] = k + i < H ? wrow[k + i] : 0.f;
        return make_float4(t[0], t[1], t[2], t[3]);
    };
    float acc[4][4] = {};
    float unused = 0.f;
    tile_product<true, true, VEC, false>(sm, a, m0, 0, H, load_b, acc, unused);
    const int tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = m0 + 4 * ty + i;
        float s = 0.f;
        if (r < R) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int j = j0 + 2 * tx + c;
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

// elbo[b] = what the guide and the transition contributed + the emission densities of the window's rows: a warp per window
__global__ void __launch_bounds__(128) k_elbo_finish(const float* __restrict__ part, int n_part, int R, int W, int B,
                                                     const float* __restrict__ path, float* __restrict__ elbo) {
    dependency_wait();
    launch_dependents();
    const int b = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= B) return;
    float s = 0.f;
    for (int i = lane; i < n_part * W; i += 32) s += part[static_cast<long long>(i / W) * R + b * W + i % W];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) elbo[b] = path[b] + s;
}

// ---- the two RNNs --------------------------------------------------------------------------------------------------
// h_t = relu(P_t + Wh h_{t -+ 1}) for kRnnRows windows and one direction per CTA, all steps.  A row of Wh is dotted with
// the states by 8 lanes; every weight read serves the CTA's windows.  Wh sits in shared memory when it fits
// (H <= 200), else it is streamed from L2 at every step (64 bytes per clock and SM: 2 us a step at H = 256, with 4 windows
// about what their multiply-adds take).  States: [B][W + 1][H]; forward: slot 0 = a0, slot t + 1 = a_t;  backward:
// slot t = b_t, slot W = b0 -- so "the state before" of row t is slot t (forward) or slot t + 1 (backward).
constexpr int kRnnRows = 4, kRnnThreads = 512;
constexpr int kRnnSmemH = 200;

struct RnnArgs {
    const float* proj;              // [parts][R][2H]: input projections, forward then backward, to be added over the parts
    int n_parts;
    long long part_stride;
    const float *Wh[2], *bias[2], *init[2];
    float* state[2];
    int B, W, H;
};

inline size_t rnn_smem_bytes(int H, bool staged) {
    return sizeof(float) * (2 * static_cast<size_t>(kRnnRows) * H + (staged ? static_cast<size_t>(H) * (H + 4) : 0));
}

template <bool VEC>
__global__ void __launch_bounds__(kRnnThreads) k_rnn_forward(RnnArgs a, int staged) {
    extern __shared__ __align__(16) float sm[];
    const int H = a.H, W = a.W, dir = blockIdx.y, b0 = blockIdx.x * kRnnRows;
    float* cur = sm;                                   // [kRnnRows][H]
    float* next = sm + kRnnRows * H;
    const float* Wh = a.Wh[dir];
    int ldw = H;
    if (staged) {                                      // rows padded by 4: four consecutive rows fall into different banks
        float* sW = sm + 2 * kRnnRows * H;
        ldw = H + 4;
        for (int i = threadIdx.x; i < H * H; i += kRnnThreads) sW[(i / H) * ldw + i % H] = Wh[i];
        Wh = sW;
    }
    dependency_wait();
    launch_dependents();
    float* state = a.state[dir];
    for (int i = threadIdx.x; i < kRnnRows * H; i += kRnnThreads) {
        const int rb = i / H, h = i % H;
        const float s = a.init[dir][h];
        cur[i] = s;
        if (b0 + rb < a.B) state[(static_cast<long long>(b0 + rb) * (W + 1) + (dir ? W : 0)) * H + h] = s;
    }
    __syncthreads();
    const int part = threadIdx.x & 7, group = threadIdx.x >> 3;
    for (int s = 0; s < W; ++s) {
        const int t = dir ? W - 1 - s : s;
        for (int h0 = group; h0 < ((H + 3) & ~3); h0 += kRnnThreads / 8) {        // a warp's four groups stay together
            const int h = h0 < H ? h0 : H - 1;
            float acc[kRnnRows] = {};
            const float* wrow = Wh + static_cast<long long>(h) * ldw;
            if (VEC) {
#pragma unroll 4
                for (int c = 4 * part; c < H; c += 32) {
                    const float4 w = *reinterpret_cast<const float4*>(wrow + c);
#pragma unroll
                    for (int rb = 0; rb < kRnnRows; ++rb) {
                        const float4 x = *reinterpret_cast<const float4*>(cur + rb * H + c);
                        acc[rb] = fmaf(w.x, x.x, fmaf(w.y, x.y, fmaf(w.z, x.z, fmaf(w.w, x.w, acc[rb]))));
                    }
                }
            } else {
                for (int c = part; c < H; c += 8) {
                    const float w = wrow[c];
#pragma unroll
                    for (int rb = 0; rb < kRnnRows; ++rb) acc[rb] = fmaf(w, cur[rb * H + c], acc[rb]);
                }
            }
#pragma unroll
            for (int rb = 0; rb < kRnnRows; ++rb) {
                acc[rb] += __shfl_xor_sync(0xffffffffu, acc[rb], 1);
                acc[rb] += __shfl_xor_sync(0xffffffffu, acc[rb], 2);
                acc[rb] += __shfl_xor_sync(0xffffffffu, acc[rb], 4);
            }
            // lane `part` finishes window `part`
            float mine = 0.f;
#pragma unroll
            for (int rb = 0; rb < kRnnRows; ++rb)
                if (rb == part) mine = acc[rb];
            if (part < kRnnRows && b0 + part < a.B && h0 < H) {
                const long long r = static_cast<long long>(b0 + part) * W + t;
                float p = a.bias[dir][h];
                for (int k = 0; k < a.n_parts; ++k) p += a.proj[k * a.part_stride + r * 2 * H + dir * H + h];
                const float v = fmaxf(mine + p, 0.f);
                next[part * H + h] = v;
                state[(static_cast<long long>(b0 + part) * (W + 1) + (dir ? t : t + 1)) * H + h] = v;
            }
        }
        __syncthreads();
        float* swap = cur; cur = next; next = swap;
    }
}

// Backwards through the same recurrences: d_pre_t = (g_t + carry) (h_t > 0), carry = d_pre_t Wh.  g_t = d ELBO / d h_t
// from the combiner (the same for both directions).  A thread owns four columns of carry and every kSlices-th row of Wh.
struct RnnBackArgs {
    const float* g;                 // [R][H]
    const float* state[2];
    const float* Wh[2];
    float* d_pre[2];                // [R][H]
    float* carry_out[2];            // [B][H]: gradient of the initial state, per window
    int B, W, H;
};

inline size_t rnn_back_smem_bytes(int H, bool staged) {
    const size_t slices = kRnnThreads / ((H + 3) / 4) > 0 ? kRnnThreads / ((H + 3) / 4) : 1;
    return sizeof(float) * (static_cast<size_t>(kRnnRows) * H * (2 + slices) + (staged ? static_cast<size_t>(H) * H : 0));
}

template <bool VEC>
__global__ void __launch_bounds__(kRnnThreads) k_rnn_backward(RnnBackArgs a, int staged) {
    extern __shared__ __align__(16) float sm[];
    const int H = a.H, W = a.W, dir = blockIdx.y, b0 = blockIdx.x * kRnnRows;
    const int groups = (H + 3) / 4, slices = kRnnThreads / groups > 0 ? kRnnThreads / groups : 1;
    float* dpre = sm;                                  // [H][kRnnRows]: one 16-byte read gives a unit's value in every window
    float* carry = dpre + kRnnRows * H;                // [kRnnRows][H]
    float* red = carry + kRnnRows * H;                 // [slices][kRnnRows][H]
    const float* Wh = a.Wh[dir];
    if (staged) {
        float* sW = red + static_cast<size_t>(slices) * kRnnRows * H;
        for (int i = threadIdx.x; i < H * H; i += kRnnThreads) sW[i] = Wh[i];
        Wh = sW;
    }
    dependency_wait();
    launch_dependents();
    for (int i = threadIdx.x; i < kRnnRows * H; i += kRnnThreads) carry[i] = 0.f;
    __syncthreads();
    for (int s = 0; s < W; ++s) {
        const int t = dir ? s : W - 1 - s;
        for (int i = threadIdx.x; i < kRnnRows * H; i += kRnnThreads) {
            const int rb = i / H, h = i % H;
            float d = 0.f;
            if (b0 + rb < a.B) {
                const long long r = static_cast<long long>(b0 + rb) * W + t;
                const float act = a.state[dir][(static_cast<long long>(b0 + rb) * (W + 1) + (dir ? t : t + 1)) * H + h];
                d = act > 0.f ? a.g[r * H + h] + carry[i] : 0.f;
                a.d_pre[dir][r * H + h] = d;
            }
            dpre[h * kRnnRows + rb] = d;
        }
        __syncthreads();
        for (int w = threadIdx.x; w < groups * slices; w += kRnnThreads) {
            const int c = (w % groups) * 4, slice = w / groups;
            float acc[kRnnRows][4] = {};
#pragma unroll 4
            for (int i = slice; i < H; i += slices) {
                float wv[4];
                const float* p = Wh + static_cast<long long>(i) * H + c;
                if (VEC) {
                    const float4 q = *reinterpret_cast<const float4*>(p);
                    wv[0] = q.x; wv[1] = q.y; wv[2] = q.z; wv[3] = q.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) wv[j] = c + j < H ? p[j] : 0.f;
                }
                const float4 d4 = *reinterpret_cast<const float4*>(dpre + i * kRnnRows);
                const float dv[kRnnRows] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
                for (int rb = 0; rb < kRnnRows; ++rb)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[rb][j] = fmaf(dv[rb], wv[j], acc[rb][j]);
            }
#pragma unroll
            for (int rb = 0; rb < kRnnRows; ++rb)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (c + j < H) red[(slice * kRnnRows + rb) * H + c + j] = acc[rb][j];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kRnnRows * H; i += kRnnThreads) {
            float v = 0.f;
            for (int k = 0; k < slices; ++k) v += red[k * kRnnRows * H + i];
            carry[i] = v;
        }
        // the next step reads only the carry entries this thread has just written, and dpre, red are rewritten behind a barrier
        __syncthreads();
    }
    for (int i = threadIdx.x; i < kRnnRows * H; i += kRnnThreads)
        if (b0 + i / H < a.B) a.carry_out[dir][static_cast<long long>(b0 + i / H) * H + i % H] = carry[i];
}

// ---- the sampled path: guide, transition density, hidden layers -------------------------------------------------------
// One CTA per window.  The small matrices sit in shared memory (rows padded to an odd length) when they fit.
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
    const float* dv_parts;          // [parts][R][H]: d_head W4, to be added over the parts
    int n_parts;
    long long part_stride;
    float *dv, *du, *dpc, *dh, *dmu, *dps;
    float* gz0;                     // [B][D]
    int B, W, D, H;
};

// out[o] = bias[o] + sum_i M[o][i] in[i] for o < O: a warp per output
__device__ __forceinline__ void block_rows_dot(const float* M, int ld, const float* in, int O, int I, const float* bias, float* out) {
    const int lane = threadIdx.x & 31;
    for (int o = threadIdx.x >> 5; o < O; o += kPathThreads / 32) {
        float s = 0.f;
        for (int i = lane; i < I; i += 32) s = fmaf(M[o * ld + i], in[i], s);
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
        if (lane == 0) out[o] = s + (bias ? bias[o] : 0.f);
    }
}
// out[d] += sum_h M[h][d] in[h]: a warp per output
__device__ __forceinline__ void block_cols_dot(const float* M, int ld, const float* in, int D, int H, float* out) {
    const int lane = threadIdx.x & 31;
    for (int d = threadIdx.x >> 5; d < D; d += kPathThreads / 32) {
        float s = 0.f;
        for (int h = lane; h < H; h += 32) s = fmaf(M[h * ld + d], in[h], s);
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
        if (lane == 0) out[d] += s;
    }
}

struct PathWeights {
    const float *Wz, *W1, *W3;      // [H][ldd]
    const float *Wmu, *W2;          // [D][ldh], [2D][ldh]
    int ldd, ldh;
};
inline size_t path_weight_floats(int D, int H) {
    return 3 * static_cast<size_t>(H) * (D | 1) + 3 * static_cast<size_t>(D) * (H | 1);
}
inline size_t path_scratch_floats(int D, int H) { return 3 * static_cast<size_t>(H) + 8 * static_cast<size_t>(D) + 64; }

__device__ __forceinline__ float* stage_padded(float* dst, const float* src, int rows, int cols, int ld) {
    for (int i = threadIdx.x; i < rows * cols; i += kPathThreads) dst[(i / cols) * ld + i % cols] = src[i];
    return dst + rows * ld;
}
__device__ __forceinline__ PathWeights path_weights(const PathArgs& a, float* sm, int staged) {
    if (!staged) return PathWeights{a.Wz, a.W1, a.W3, a.Wmu, a.W2, a.D, a.H};
    PathWeights w;
    w.ldd = a.D | 1;
    w.ldh = a.H | 1;
    w.Wz = sm; sm = stage_padded(sm, a.Wz, a.H, a.D, w.ldd);
    w.W1 = sm; sm = stage_padded(sm, a.W1, a.H, a.D, w.ldd);
    w.W3 = sm; sm = stage_padded(sm, a.W3, a.H, a.D, w.ldd);
    w.Wmu = sm; sm = stage_padded(sm, a.Wmu, a.D, a.H, w.ldh);
    w.W2 = sm; stage_padded(sm, a.W2, 2 * a.D, a.H, w.ldh);
    return w;
}

__device__ __forceinline__ float row_dot(const float* M, int ld, int row, const float* in, int n, float s) {
    const float* p = M + static_cast<long long>(row) * ld;
    for (int i = 0; i < n; ++i) s = fmaf(p[i], in[i], s);
    return s;
}

__global__ void __launch_bounds__(kPathThreads) k_path_forward(PathArgs a, int staged) {
    extern __shared__ __align__(16) float sm[];
    const int D = a.D, H = a.H, W = a.W, b = blockIdx.x, tid = threadIdx.x;
    float* z = sm;                   // [D]
    float* mu = z + D;               // [D]
    float* zp = mu + D;              // [D]
    float* hz = zp + D;              // [2D]
    float* h = sm + 8 * D;           // [H]
    float* scal = h + 3 * H;         // [64]
    const PathWeights w = path_weights(a, scal + 64, staged);
    for (int d = tid; d < D; d += kPathThreads) { z[d] = a.z0[d]; a.z[static_cast<long long>(b) * (W + 1) * D + d] = a.z0[d]; }
    dependency_wait();
    launch_dependents();
    __syncthreads();
    float elbo = 0.f;                // of this thread's latent dimensions
    for (int t = 0; t < W; ++t) {
        const long long r = static_cast<long long>(b) * W + t;
        const float* sa = a.a + (static_cast<long long>(b) * (W + 1) + t + 1) * H;
        const float* sb = a.b + (static_cast<long long>(b) * (W + 1) + t) * H;
        // hidden layers that read z_{t-1}: the combiner and the transition's
        for (int i = tid; i < H; i += kPathThreads) {
            const float c = tanhf(row_dot(w.Wz, w.ldd, i, z, D, a.bz[i]));
            const float o = (c + sa[i] + sb[i]) * (1.f / 3.f);
            const float u = fmaxf(row_dot(w.W1, w.ldd, i, z, D, a.b1[i]), 0.f);
            a.comb[r * H + i] = c;
            a.hout[r * H + i] = o;
            a.u[r * H + i] = u;
            h[i] = o;
            h[H + i] = u;
        }
        __syncthreads();
        block_rows_dot(w.Wmu, w.ldh, h, D, H, a.bmu, mu);
        block_rows_dot(w.W2, w.ldh, h + H, 2 * D, H, a.b2, hz);
        __syncthreads();
        for (int d = tid; d < D; d += kPathThreads) {
            const float pre = row_dot(a.Wsig, D, d, mu, D, a.bsig[d]);
            const float sg = softplus_f(pre), e = a.eps[r * D + d], zt = fmaf(sg, e, mu[d]);
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
        for (int i = tid; i < H; i += kPathThreads)
            a.v[r * H + i] = fmaxf(row_dot(w.W3, w.ldd, i, zp, D, a.b3[i]), 0.f);
        float* swap = z; z = zp; zp = swap;            // h and mu are rewritten behind the next barriers
    }
    // D <= 64: the sums sit in the first two warps
    if (tid < 64) scal[tid] = elbo;
    __syncthreads();
    if (tid == 0) {
        float s = 0.f;
        for (int d = 0; d < (D < 64 ? D : 64); ++d) s += scal[d];
        a.path[b] = s;
    }
}

__global__ void __launch_bounds__(kPathThreads) k_path_backward(PathArgs a, int staged) {
    extern __shared__ __align__(16) float sm[];
    const int D = a.D, H = a.H, W = a.W, b = blockIdx.x, tid = threadIdx.x;
    float* gz = sm;                  // [D]   d ELBO / d z_t
    float* gzp = gz + D;             // [D]   d ELBO / d z_{t-1}
    float* dmu = gzp + D;            // [D]
    float* dps = dmu + D;            // [D]
    float* dhz = dps + D;            // [2D]
    float* h = sm + 8 * D;           // [3][H]: dv, du, dpc
    const PathWeights w = path_weights(a, h + 3 * H + 64, staged);
    for (int d = tid; d < D; d += kPathThreads) gzp[d] = 0.f;
    dependency_wait();
    launch_dependents();
    __syncthreads();
    for (int t = W - 1; t >= 0; --t) {
        const long long r = static_cast<long long>(b) * W + t;
        for (int d = tid; d < D; d += kPathThreads) { gz[d] = gzp[d] + a.dzt[r * D + d]; gzp[d] = 0.f; }
        for (int d = tid; d < 2 * D; d += kPathThreads) dhz[d] = a.dhz[r * 2 * D + d];
        __syncthreads();
        // hidden-layer gradients of the emission (its head's input gradient comes in parts) and of the transition
        for (int i = tid; i < H; i += kPathThreads) {
            float dv = 0.f;
            if (a.v[r * H + i] > 0.f)
                for (int k = 0; k < a.n_parts; ++k) dv += a.dv_parts[k * a.part_stride + r * H + i];
            float du = 0.f;
            if (a.u[r * H + i] > 0.f)
                for (int o = 0; o < 2 * D; ++o) du = fmaf(dhz[o], w.W2[o * w.ldh + i], du);
            a.dv[r * H + i] = dv;
            a.du[r * H + i] = du;
            h[i] = dv;
            h[H + i] = du;
        }
        __syncthreads();
        block_cols_dot(w.W3, w.ldd, h, D, H, gz);
        block_cols_dot(w.W1, w.ldd, h + H, D, H, gzp);
        __syncthreads();
        // guide: d_mu = g_z + Wsig^T d_pre_sig,  d_pre_sig = (g_z eps + 1 / sigma) sigmoid(pre_sig)
        for (int d = tid; d < D; d += kPathThreads) {
            const float pre = a.presig[r * D + d];
            const float p = (gz[d] * a.eps[r * D + d] + 1.f / softplus_f(pre)) * sigmoid_f(pre);
            dps[d] = p;
            a.dps[r * D + d] = p;
        }
        __syncthreads();
        for (int d = tid; d < D; d += kPathThreads) {
            float s = gz[d];
            for (int o = 0; o < D; ++o) s = fmaf(dps[o], a.Wsig[o * D + d], s);
            dmu[d] = s;
            a.dmu[r * D + d] = s;
        }
        __syncthreads();
        for (int i = tid; i < H; i += kPathThreads) {
            float s = 0.f;
            for (int d = 0; d < D; ++d) s = fmaf(dmu[d], w.Wmu[d * w.ldh + i], s);
            s *= 1.f / 3.f;
            const float c = a.comb[r * H + i];
            a.dh[r * H + i] = s;
            const float p = s * (1.f - c * c);
            a.dpc[r * H + i] = p;
            h[2 * H + i] = p;
        }
        __syncthreads();
        block_cols_dot(w.Wz, w.ldd, h + 2 * H, D, H, gzp);
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
