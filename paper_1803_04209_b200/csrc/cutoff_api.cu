// C ABI and host orchestration of the cutoff library (see include/cutoff.h).
#include "../../include/cutoff.h"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "common.cuh"
#include "kernels_model.cuh"
#include "kernels_sort.cuh"
#include "bucket_sort.cuh"
#include "emit_tc.cuh"
#include "emit_tc2.cuh"
#include "chain_tc.cuh"
#include "kernels_literal.cuh"
#include "gemm_tc.cuh"
#include "pipe_rates.cuh"
#include "kernels_eval.cuh"
#include "fit_api.cuh"

using namespace cutoff;

namespace {

constexpr uint32_t kBlobMagic = 0x31465443u;   // "CTF1"
constexpr int kNumStages = 5;
constexpr int kMaxChunks = 64;        // passes per decision (also the number of timing event sets)
constexpr int kPartialRows = 2048;    // partial-sum rows shared by all passes of a decision
const char* const kStageNames[kNumStages] = {"encoder", "chain", "emission", "sort", "decide"};

struct TensorSpec { const char* name; size_t rows, cols; };

}  // namespace

struct cutoff_ctx {
    cutoff_config cfg{};
    int N = 0, D = 0, H = 0, W = 0, S = 0;
    int ldx = 0;            // leading dimension of the sample matrix (N rounded up to 8: rows start on 32 bytes)
    int P = 0;              // sort width: N rounded up to a power of two, at least 32
    int sm_count = 0;
    int chunk_rows = 0;     // samples per pass through chain -> emission -> sort
    int alloc_rows = 0;     // rows the pass buffers were allocated for
    int n_chunks = 0;
    int sort_grid = 0;      // CTAs of the sort kernel per chunk (= partial rows per chunk)
    cudaStream_t stream = nullptr;
    bool owns_stream = false;       // the context created `stream` itself (graph mode with a NULL stream)

    float* d_blob = nullptr;        // tensors as loaded
    float* d_WT = nullptr;          // transposed copies WzT, W1T, W3T: 3 x [D][H]
    float* d_WhR = nullptr;         // recurrence matrices regrouped per thread for k_enc_rnn_resident: 2 x H x H
    ModelDev m{};
    bool weights_loaded = false;

    float* d_ring = nullptr;        // [W][N]
    float* d_stage = nullptr;       // [N] landing buffer for host pushes
    bool draws_valid = false;       // d_x holds every predictive draw of the last decision (needed for imputation)
    DevState* d_state = nullptr;
    float* d_proj = nullptr;        // [2][W slots][H] raw input projections of the ring's vectors, kept up to date by every push
    bool proj_stale = true;         // the ring or the weights were replaced: recompute every slot before the next decision
    float* d_hlr = nullptr;         // [2][W][H]
    float* d_v = nullptr;           // [chunk_rows][H]; fp32 path only
    // tensor-core path: operands of the emission products as halves, row pitch ldh, with inverse scales per row
    int ldh = 0;                    // H rounded up to 8 (rows start on 16 bytes)
    __half* d_v16 = nullptr;        // [alloc_rows][ldh] v (literal: u)
    float* d_v_inv = nullptr;       // [alloc_rows]
    __half* d_w16 = nullptr;        // weights: W4 [2N][ldh]; literal: Wi2 [N], Wj2 [N], M [H] rows
    float* d_w_inv = nullptr;       // their inverse scales
    // [8] bounds of hidden layers' entries, slope * largest |input| + offset each: v (u), from the largest |latent|; literal: r, from the
    // largest |u|; the transition's (literal: the gate's and the proposal's), from the largest |latent|
    float* d_bound = nullptr;
    float* d_x = nullptr;           // [chunk_rows][ldx]
    float* d_partial = nullptr;     // [n_chunks * sort_grid][N]; a second block of kPartialRows rows holds sums of squares
    float* d_std = nullptr;         // [N] spread of each order statistic (when asked for)
    float* d_sq_totals = nullptr;   // [CTA][128 E] for wide rows (when asked for)
    bool want_std = false;
    bool have_std = false;
    double* d_sums = nullptr;       // [N]

    CUtensorMap map_v{};            // TMA view of d_v16 [alloc_rows][H]
    CUtensorMap map_w4{};           // TMA view of d_w16 [2N][H]

    bool literal = false;           // the networks as Section 3.1.3 prints them (CUTOFF_FLAG_LITERAL)
    LiteralDev lit{};
    float* d_I = nullptr;           // [alloc_rows][ldx]  emission mean I (padding columns stay zero); fp32 path only
    float* d_r = nullptr;           // [alloc_rows][H]    hidden layer of the emission scale; fp32 path only
    __half* d_r16 = nullptr;        // [alloc_rows][ldh]  the same as an operand; tensor-core path
    float* d_r_inv = nullptr;       // [alloc_rows]
    float* d_Wj1p = nullptr;        // [H][ldx]           Wj1 with rows padded with zeros to ldx; fp32 path only
    float* d_W4T = nullptr;         // [H][2][ldx]        fp32 compact path: W4 with the columns of both heads contiguous
    float* d_M = nullptr;           // [H][H]             M, before it becomes rows of d_w16
    float* d_Mb = nullptr;          // [H]                b' = Wj1 bi2 + bj1 (tensor-core path: Wj1 I + bj1 = M u + b' with M = Wj1 Wi2)
    CUtensorMap map_r{};            // TMA view of d_r16 [alloc_rows][H]
    CUtensorMap map_wi2{}, map_M{}, map_wj2{};
    bool use_tc = false;            // emission output layer on tensor cores
    int pair_clusters = 0;          // clusters of two CTAs of the two-SM emission kernel that fit the GPU at once
    bool pair_emission = false;     // option "pair_emission": run the output layer on pairs of SMs (slower as measured; off)
    int chain_wide = 0;             // compact chain with D lanes per sample (few samples): samples per lane, 0 = another chain
    bool chain_tc = false;          // per-sample chain on tensor cores as well (D = 16, H in {64, 128, 192, 256}; D = 32, H <= 512)
    uint8_t* d_chain_image = nullptr;   // swizzled operand tiles of the chain

    // pinned host memory that kernels read and write directly (one address on both sides); one block that begins with h_state
    uint8_t* h_mask = nullptr;      // [N] censoring mask of the push in progress
    float* h_stage = nullptr;       // [N] run-times of a host push
    bool stage_in_use = false;      // by a push that may not have been waited for
    DevState* h_state = nullptr;    // the device state as of the last decision, or push that the host waited for
    float* h_E = nullptr;           // [N] expected order statistics of the last decision
    float* h_omega = nullptr;       // [N] throughput per cutoff

    uint32_t pushes = 0;            // host mirror of DevState::push_count
    bool pending = false;           // a decision is enqueued and not yet fetched
    bool pending_warmup = false;
    bool have_result = false;
    bool partial_pending = false;   // the sums of a decision are enqueued, its argmax (and counter step) still to come

    bool timing = false;
    cudaEvent_t ev[kNumStages + 1][kMaxChunks]{};   // per chunk, stage boundaries
    bool ev_created = false;
    float stage_ms[kNumStages]{};
    int timed_chunks = 0;

    cudaGraph_t graph = nullptr;            // captured push + decision (CUTOFF_FLAG_GRAPH)
    cudaGraphExec_t graph_exec = nullptr;
    cudaGraph_t graph_dev = nullptr;        // the same from the device's landing buffer (cutoff_step_device)
    cudaGraphExec_t graph_dev_exec = nullptr;
    int graph_kernels = 0;                  // kernels one replay launches
    bool decided_once = false;              // a decision has run outside capture (function attributes are set)

    int64_t launches = 0;
    std::string last_error;
};

namespace {

#define CU_CHECK(ctx, call)                                                                          \
    do {                                                                                             \
        cudaError_t err__ = (call);                                                                  \
        if (err__ != cudaSuccess) {                                                                  \
            if (ctx) (ctx)->last_error = std::string(#call) + ": " + cudaGetErrorString(err__);      \
            return err__ == cudaErrorMemoryAllocation ? CUTOFF_ERR_NOMEM : CUTOFF_ERR_CUDA;          \
        }                                                                                            \
    } while (0)

// Makes the context's device current for the duration of an entry point and puts the caller's
// current device back on exit.
struct DeviceGuard {
    int prev = -1;
    bool changed = false;
    cudaError_t err = cudaSuccess;
    explicit DeviceGuard(int device) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != device) {
            err = cudaSetDevice(device);
            changed = err == cudaSuccess;
        }
    }
    ~DeviceGuard() {
        if (changed && prev >= 0) cudaSetDevice(prev);
    }
    DeviceGuard(const DeviceGuard&) = delete;
    DeviceGuard& operator=(const DeviceGuard&) = delete;
};

std::vector<TensorSpec> tensor_specs(size_t N, size_t D, size_t H) {
    return {
        {"Wxf", H, N}, {"Whf", H, H}, {"bf", 1, H}, {"a0", 1, H},
        {"Wxb", H, N}, {"Whb", H, H}, {"bb", 1, H}, {"b0", 1, H},
        {"Wz", H, D}, {"bz", 1, H}, {"Wmu", D, H}, {"bmu", 1, D}, {"Wsig", D, D}, {"bsig", 1, D}, {"z0", 1, D},
        {"W1", H, D}, {"b1", 1, H}, {"W2", 2 * D, H}, {"b2", 1, 2 * D},
        {"W3", H, D}, {"b3", 1, H}, {"W4", 2 * N, H}, {"b4", 1, 2 * N},
    };
}

// The literal variant: the guide tensors (the first 15) are the same, then the gated transition and the
// emission networks I and J.
std::vector<TensorSpec> tensor_specs_literal(size_t N, size_t D, size_t H) {
    std::vector<TensorSpec> v = tensor_specs(N, D, H);
    v.resize(15);
    const TensorSpec rest[] = {
        {"Wg1", H, D}, {"bg1", 1, H}, {"Wg2", D, H}, {"bg2", 1, D},
        {"Wh1", H, D}, {"bh1", 1, H}, {"Wh2", D, H}, {"bh2", 1, D},
        {"Wl", D, D}, {"bl", 1, D}, {"Ws", D, D}, {"bs", 1, D},
        {"Wi1", H, D}, {"bi1", 1, H}, {"Wi2", N, H}, {"bi2", 1, N},
        {"Wj1", H, N}, {"bj1", 1, H}, {"Wj2", N, H}, {"bj2", 1, N},
    };
    v.insert(v.end(), std::begin(rest), std::end(rest));
    return v;
}

// Round to tf32 as the tensor cores will see the value (nearest, ties away from zero), kept as an fp32 bit pattern.
float host_tf32(float f) {
    uint32_t u;
    std::memcpy(&u, &f, 4);
    u = (u + 0x1000u) & 0xFFFFE000u;
    std::memcpy(&f, &u, 4);
    return f;
}

// Float index of element (row, col) inside one K-major operand slab of rows x 32 with 128-byte rows whose 16-byte
// chunks are XOR-swizzled with the row index modulo 8 (the layout the tensor cores read from shared memory).
size_t swz(size_t row, size_t col) {
    return (row >> 3) * 256 + (row & 7) * 32 + ((((col >> 2) ^ (row & 7)) << 2) | (col & 3));
}

// A first-layer matrix w [rows][cols] (cols <= 32) into columns col0 .. col0 + cols - 1 of a swizzled tile of
// `rows` rows x 32, rounded to tf32: the B operand of hidden = act(W z + b), K = the latent size.
void put_first_layer(float* tile, const float* w, size_t rows, size_t cols, size_t col0) {
    for (size_t n = 0; n < rows; ++n)
        for (size_t k = 0; k < cols; ++k) tile[swz(n, col0 + k)] = host_tf32(w[n * cols + k]);
}

// A second-layer matrix w [out_rows][H] as K blocks of `block_rows` rows x 64 halves (the other rows stay as they are), swizzled, each
// row multiplied by a power of two as k_half_rows does it; the inverses go to `inv`.  The B operand of out = W hidden, K = H.  `rest`: what the halves leave of the rows.
void put_second_layer_half(uint8_t* tiles, float* inv, const double* w, size_t out_rows, size_t H, size_t row0, size_t block_rows, double* rest = nullptr) {
    for (size_t o = 0; o < out_rows; ++o) {
        float big = 0.0f;
        for (size_t k = 0; k < H; ++k) big = std::fmax(big, static_cast<float>(std::fabs(w[o * H + k])));
        uint32_t bits;
        std::memcpy(&bits, &big, 4);
        const int e = bits ? half_exponent(bits) : 0;
        const double up = std::ldexp(1.0, e), down = std::ldexp(1.0, -e);       // exact factors, as the function itself would be too slow here
        const size_t row = row0 + o;
        for (size_t k = 0; k < H; ++k) {
            const __half h = __float2half_rn(static_cast<float>(w[o * H + k] * up));
            const size_t at = k / 64 * block_rows * 128 + (row >> 3) * 1024 + (row & 7) * 128 + (((k % 64 >> 3) ^ (row & 7)) << 4) + (k & 7) * 2;
            std::memcpy(tiles + at, &h, 2);
            if (rest) rest[o * H + k] = w[o * H + k] - static_cast<double>(__half2float(h)) * down;
        }
        inv[row] = std::ldexp(1.0f, -e);
    }
}
void put_second_layer_half(uint8_t* tiles, float* inv, const float* w, size_t out_rows, size_t H, size_t block_rows) {
    std::vector<double> rounded(out_rows * H);
    for (size_t i = 0; i < rounded.size(); ++i) rounded[i] = host_tf32(w[i]);
    put_second_layer_half(tiles, inv, rounded.data(), out_rows, H, 0, block_rows);
}

// `rows` rows of weights w [rows][H] on the device, already rounded to at most 11 significant bits, into the half-precision
// operand from its row `row0` on.
void half_rows(cutoff_ctx* c, const float* w, int rows, int row0) {
    k_half_rows<<<ceil_div(rows, 8), 256, 0, c->stream>>>(w, rows, c->H, c->ldh, c->d_w16 + static_cast<size_t>(row0) * c->ldh, c->d_w_inv + row0);
}

// A copy from pageable memory, taken from it when this returns, in the order of the context's stream: on the default stream the
// context's kernels would not wait for it.
cudaError_t upload(const cutoff_ctx* c, void* dst, const void* src, size_t bytes) {
    return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, c->stream);
}

// |A x + b| <= slope * max |x| + offset, from the matrix as the tensor cores see it (rounded up a little); of a ReLU layer
// relu(A x + b), where negative biases only lower the result
void layer_bound(const float* w, const float* b, size_t rows, size_t cols, bool relu, float (&bound)[2]) {
    double l1 = 0.0, mb = 0.0;
    for (size_t r = 0; r < rows; ++r) {
        double s = 0.0;
        for (size_t k = 0; k < cols; ++k) s += std::fabs(static_cast<double>(w[r * cols + k]));
        l1 = std::fmax(l1, s);
        mb = std::fmax(mb, relu ? static_cast<double>(b[r]) : std::fabs(static_cast<double>(b[r])));
    }
    bound[0] = static_cast<float>(l1 * 1.001);
    bound[1] = static_cast<float>(mb * 1.001);
}

// Launch `kernel` so that it may begin while the kernel before it in the stream is still running (programmatic
// dependent launch): the kernel itself waits, by dependency_wait(), before it touches that kernel's results.
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

int next_pow2(int n) {
    int p = 1;
    while (p < n) p <<= 1;
    return p;
}

void free_all(cutoff_ctx* c) {
    cudaFree(c->d_I); cudaFree(c->d_r); cudaFree(c->d_Wj1p); cudaFree(c->d_Mb); cudaFree(c->d_M); cudaFree(c->d_W4T);
    cudaFree(c->d_v16); cudaFree(c->d_v_inv); cudaFree(c->d_w16); cudaFree(c->d_w_inv); cudaFree(c->d_bound); cudaFree(c->d_r16); cudaFree(c->d_r_inv);
    cudaFree(c->d_blob); cudaFree(c->d_WT); cudaFree(c->d_WhR); cudaFree(c->d_chain_image);
    cudaFree(c->d_ring); cudaFree(c->d_stage);
    cudaFree(c->d_state); cudaFree(c->d_proj); cudaFree(c->d_hlr); cudaFree(c->d_v); cudaFree(c->d_x);
    cudaFree(c->d_partial); cudaFree(c->d_sq_totals); cudaFree(c->d_std); cudaFree(c->d_sums);
    if (c->h_state) cudaFreeHost(c->h_state);            // the whole pinned block
    if (c->owns_stream && c->stream) cudaStreamDestroy(c->stream);
    if (c->graph_exec) cudaGraphExecDestroy(c->graph_exec);
    if (c->graph) cudaGraphDestroy(c->graph);
    if (c->graph_dev_exec) cudaGraphExecDestroy(c->graph_dev_exec);
    if (c->graph_dev) cudaGraphDestroy(c->graph_dev);
    if (c->ev_created)
        for (auto& row : c->ev)
            for (auto& e : row)
                if (e) cudaEventDestroy(e);
}

// Keys per thread of the bucket sort: N / threads rounded up to a multiple of 4.
int keys_per_thread(int n, int threads) { return ceil_div(ceil_div(n, threads), 4) * 4; }

// Which rows of N <= 1024 keys are sorted by distribution and which by the register network.  Up to 128 keys the network
// is shorter than counting and scanning (128 keys x 65536 rows: 0.033 against 0.035 ms), from 257 on it never is (300 keys x 2048 rows:
// 0.0113 against 0.0091 ms); between, it depends on whether the longer latency of one row is hidden by the rows that
// follow (256 keys: 2048 rows 0.0075 against 0.0086 ms, 65536 rows 0.056 against 0.049 ms; 140 keys x 16384 rows 0.0197 against 0.0172 ms).
bool by_buckets(int n, int64_t rows) { return n > 256 || (n > 128 && rows >= 8192); }

int bucket_wide_ctas(int n) {
    switch (keys_per_thread(n, 128)) {
        case 12: return kBucketWideCtas<12>;
        case 16: return kBucketWideCtas<16>;
        case 20: return kBucketWideCtas<20>;
        case 24: return kBucketWideCtas<24>;
        case 28: return kBucketWideCtas<28>;
        default: return kBucketWideCtas<32>;
    }
}

// Work split: how many samples go through chain -> emission -> sort at a time, and how many
// CTAs the sort kernel uses per pass.
void plan_chunks(cutoff_ctx* c, int chunk_rows_wanted) {
    int rows = chunk_rows_wanted > 0 ? chunk_rows_wanted : c->S;
    if (rows > c->S) rows = c->S;
    if (rows > c->alloc_rows) rows = c->alloc_rows;
    if (ceil_div(c->S, rows) > kMaxChunks) rows = ceil_div(c->S, kMaxChunks);
    c->chunk_rows = rows;
    c->n_chunks = ceil_div(c->S, rows);
    // CTAs of the sort kernel per pass: enough to fill the GPU, within the partial-sum rows available
    int want, cap;
    if (c->N > 1024) { want = rows; cap = c->sm_count * bucket_wide_ctas(c->N); }
    else if (by_buckets(c->N, rows)) { want = rows; cap = c->sm_count; }
    else { want = ceil_div(rows, kSortWarps); cap = c->sm_count * 2; }
    if (cap > kPartialRows / c->n_chunks) cap = kPartialRows / c->n_chunks;
    c->sort_grid = want < cap ? want : cap;
}

template <int E>
void launch_sort_warp(cutoff_ctx* c, int count, float* partial) {
    float* partial_sq = partial + static_cast<size_t>(kPartialRows) * c->N;
    const size_t smem = sort_tma_smem_bytes<E>(c->ldx);
    if (c->want_std) launch_dependent(k_sort_sum_tma<E, true>, dim3(c->sort_grid), dim3(kSortWarps * 32), smem, c->stream, c->d_x, c->ldx, c->N, count, partial, partial_sq, c->d_state);
    else launch_dependent(k_sort_sum_tma<E, false>, dim3(c->sort_grid), dim3(kSortWarps * 32), smem, c->stream, c->d_x, c->ldx, c->N, count, partial, partial_sq, c->d_state);
}

template <int E, bool SQ>
void launch_bucket_warp_sq(cutoff_ctx* c, int count, float* partial) {
    launch_dependent(k_bucket_sum_warp<E, SQ, kBulk>, dim3(c->sort_grid), dim3(kBucketWarps<E> * 32), bucket_smem_bytes<E>(), c->stream,
                     c->d_x, c->ldx, c->N, count, partial, partial + static_cast<size_t>(kPartialRows) * c->N, c->d_state);
}
template <int E>
void launch_bucket_warp(cutoff_ctx* c, int count, float* partial) {
    if (c->want_std) launch_bucket_warp_sq<E, true>(c, count, partial);
    else launch_bucket_warp_sq<E, false>(c, count, partial);
}

template <int E, bool SQ>
void launch_bucket_cta_sq(cutoff_ctx* c, int count, float* partial) {
    launch_dependent(k_bucket_sum_cta<E, SQ>, dim3(c->sort_grid), dim3(128), bucket_wide_smem_bytes<E>(), c->stream,
                     c->d_x, c->ldx, c->N, count, partial, partial + static_cast<size_t>(kPartialRows) * c->N, c->d_sq_totals, c->d_state);
}
template <int E>
void launch_bucket_cta(cutoff_ctx* c, int count, float* partial) {
    if (c->want_std) launch_bucket_cta_sq<E, true>(c, count, partial);
    else launch_bucket_cta_sq<E, false>(c, count, partial);
}

int launch_sort(cutoff_ctx* c, int count, float* partial) {
    if (c->N > 1024) {
        switch (keys_per_thread(c->N, 128)) {
            case 12: launch_bucket_cta<12>(c, count, partial); break;
            case 16: launch_bucket_cta<16>(c, count, partial); break;
            case 20: launch_bucket_cta<20>(c, count, partial); break;
            case 24: launch_bucket_cta<24>(c, count, partial); break;
            case 28: launch_bucket_cta<28>(c, count, partial); break;
            default: launch_bucket_cta<32>(c, count, partial); break;
        }
    } else if (by_buckets(c->N, c->chunk_rows)) {
        switch (keys_per_thread(c->N, 32)) {
            case 8: launch_bucket_warp<8>(c, count, partial); break;
            case 12: launch_bucket_warp<12>(c, count, partial); break;
            case 16: launch_bucket_warp<16>(c, count, partial); break;
            case 20: launch_bucket_warp<20>(c, count, partial); break;
            case 24: launch_bucket_warp<24>(c, count, partial); break;
            case 28: launch_bucket_warp<28>(c, count, partial); break;
            default: launch_bucket_warp<32>(c, count, partial); break;
        }
    } else {
        switch (c->P) {
            case 32: launch_sort_warp<1>(c, count, partial); break;
            case 64: launch_sort_warp<2>(c, count, partial); break;
            case 128: launch_sort_warp<4>(c, count, partial); break;
            default: launch_sort_warp<8>(c, count, partial); break;
        }
    }
    c->launches += 1;
    return CUTOFF_OK;
}

HalfRows half_v(const cutoff_ctx* c) { return HalfRows{c->d_v16, c->d_v_inv, c->ldh, c->d_bound}; }
ChainOut chain_out(const cutoff_ctx* c) { return ChainOut{c->use_tc ? nullptr : c->d_v, half_v(c)}; }

template <int D>
void launch_chain_t(cutoff_ctx* c, uint32_t sample_base, int count, size_t smem) {
    const NoiseKey key{static_cast<uint32_t>(c->cfg.seed), static_cast<uint32_t>(c->cfg.seed >> 32)};
    const size_t resident = chain_resident_smem_floats(c->D, c->H, c->W) * sizeof(float);
    if (c->chain_wide) {
        const auto run = [&](auto* kernel, int spl) {
            const int batches = ceil_div(count, 32 / D * spl);
            launch_dependent(kernel, dim3(batches < c->sm_count ? batches : c->sm_count), dim3(kChainWideThreads), resident, c->stream, c->m, c->d_hlr,
                             c->d_state, key, sample_base, count, chain_out(c));
        };
        bool two = false;
        if constexpr (D <= 16) {
            two = c->chain_wide == 2;
            if (two) run(k_chain_wide<D, 2>, 2);
        }
        if (!two) run(k_chain_wide<D, 1>, 1);
    } else if (resident <= 200 * 1024) {
        // all weights fit: one persistent CTA per SM, as many as there are warp batches to hand out
        const int batch = 32 / ChainShape<D>::G * ChainShape<D>::SPL;
        const int batches = ceil_div(count, batch);
        const int grid = batches < c->sm_count ? batches : c->sm_count;
        launch_dependent(k_chain_resident<D>, dim3(grid), dim3(kChainResidentThreads), resident, c->stream, c->m, c->d_hlr, c->d_state, key,
                         sample_base, count, chain_out(c));
    } else {
        launch_dependent(k_chain<D>, dim3(ceil_div(count, ChainShape<D>::kSamplesPerCta)), dim3(ChainShape<D>::kThreads), smem, c->stream,
                         c->m, c->d_hlr, c->d_state, key, sample_base, count, chain_out(c));
    }
}

// The tensor-core chain of a call of `count` samples, and how many of them are a tile.  Half tiles as long as every one of them has an SM of
// its own (D=16, H=256, S=8192: 27 us, whole tiles on half the SMs 35), then whole tiles, each worked on by all warps of its SM, then, where
// all operands fit, two side by side (S=65536: 68 us; one after the other by all warps 76 to 90).
struct ChainTcChoice {
    void (*kernel)(tc::ChainTcArgs);
    int rows;
};
template <bool LITERAL>
ChainTcChoice chain_tc_choice(const cutoff_ctx* c, int count) {
    const bool wide = c->D == tc::kChain32D;
    if (ceil_div(count, 64) <= c->sm_count) return {wide ? tc::k_chain_tc<32, LITERAL, 16, true> : tc::k_chain_tc<16, LITERAL, 16, true>, 64};
    if (wide) return {tc::k_chain_tc<32, LITERAL, 16, false>, 128};
    return {ceil_div(count, 128) <= c->sm_count ? tc::k_chain_tc<16, LITERAL, 16, false> : tc::k_chain_tc<16, LITERAL, 8, false>, 128};
}
ChainTcChoice chain_tc_choice(const cutoff_ctx* c, int count) { return c->literal ? chain_tc_choice<true>(c, count) : chain_tc_choice<false>(c, count); }

void launch_chain_tc(cutoff_ctx* c, uint32_t sample_base, int count) {
    tc::ChainTcArgs a{};
    const ModelDev& m = c->m;
    a.image = c->d_chain_image;
    a.bz = m.bz; a.b1 = m.b1; a.b3 = m.b3; a.bmu = m.bmu; a.b2 = m.b2; a.z0 = m.z0;
    if (c->literal) {
        const LiteralDev& l = c->lit;
        a.b1 = l.bg1; a.b3 = l.bh1; a.b2 = nullptr;
        a.bi1 = l.bi1; a.bg2 = l.bg2; a.bh2 = l.bh2; a.Wl = l.Wl; a.bl = l.bl; a.bs = l.bs;
    }
    a.hlr = c->d_hlr; a.WzT = m.WzT; a.Wmu = m.Wmu; a.bounds = c->d_bound + 4; a.st = c->d_state;
    a.key = NoiseKey{static_cast<uint32_t>(c->cfg.seed), static_cast<uint32_t>(c->cfg.seed >> 32)};
    a.sample_base = sample_base; a.count = count; a.H = c->H; a.W = c->W; a.v_out = half_v(c);
    const ChainTcChoice choice = chain_tc_choice(c, count);
    const int tiles = ceil_div(count, choice.rows);
    launch_dependent(choice.kernel, dim3(tiles < c->sm_count ? tiles : c->sm_count), dim3(tc::kChainTcThreads),
                     tc::chain_tc_smem_bytes(c->D, c->H, c->W, c->literal), c->stream, a);
    c->launches += 1;
}

template <int D>
void launch_chain_literal_t(cutoff_ctx* c, uint32_t sample_base, int count) {
    const NoiseKey key{static_cast<uint32_t>(c->cfg.seed), static_cast<uint32_t>(c->cfg.seed >> 32)};
    const size_t smem = chain_smem_floats(c->D, c->H, c->W) * sizeof(float);
    launch_dependent(k_chain_literal<D>, dim3(ceil_div(count, ChainShape<D>::kSamplesPerCta)), dim3(ChainShape<D>::kThreads), smem, c->stream,
                     c->m, c->lit, c->d_hlr, c->d_state, key, sample_base, count, chain_out(c));
}

void launch_chain(cutoff_ctx* c, uint32_t sample_base, int count) {
    if (c->chain_tc) { launch_chain_tc(c, sample_base, count); return; }
    if (c->literal) {
        switch (c->D) {
            case 4: launch_chain_literal_t<4>(c, sample_base, count); break;
            case 8: launch_chain_literal_t<8>(c, sample_base, count); break;
            case 16: launch_chain_literal_t<16>(c, sample_base, count); break;
            default: launch_chain_literal_t<32>(c, sample_base, count); break;
        }
        c->launches += 1;
        return;
    }
    const size_t smem = chain_smem_floats(c->D, c->H, c->W) * sizeof(float);
    switch (c->D) {
        case 4: launch_chain_t<4>(c, sample_base, count, smem); break;
        case 8: launch_chain_t<8>(c, sample_base, count, smem); break;
        case 16: launch_chain_t<16>(c, sample_base, count, smem); break;
        default: launch_chain_t<32>(c, sample_base, count, smem); break;
    }
    c->launches += 1;
}

// 2-D tensor map over a row-major [rows][cols] matrix of floats or halves, boxes of 128 rows x 128 bytes
// (one 128-byte-swizzled K-major operand tile).  The driver entry point is looked up at run time.
template <typename T>
int make_tile_map(cutoff_ctx* c, CUtensorMap* map, const T* base, uint64_t rows, uint64_t cols, uint64_t ld = 0) {
    typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static EncodeFn encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        CU_CHECK(c, cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q));
        if (!fn || q != cudaDriverEntryPointSuccess) {
            if (c) c->last_error = "cuTensorMapEncodeTiled is not available from this driver";
            return CUTOFF_ERR_CUDA;
        }
        encode = reinterpret_cast<EncodeFn>(fn);
    }
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {(ld ? ld : cols) * sizeof(T)};
    const cuuint32_t box[2] = {128 / sizeof(T), tc::kBM};
    const cuuint32_t elem[2] = {1, 1};
    const CUresult r = encode(map, sizeof(T) == 2 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<T*>(base), dims, strides, box,
                              elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        if (c) c->last_error = "cuTensorMapEncodeTiled failed with code " + std::to_string(static_cast<int>(r));
        return CUTOFF_ERR_CUDA;
    }
    return CUTOFF_OK;
}

void launch_emission_tc(cutoff_ctx* c, uint32_t sample_base, int count) {
    tc::EmitArgs a;
    a.b4 = c->m.b4; a.v_inv = c->d_v_inv; a.w_inv = c->d_w_inv; a.x = c->d_x; a.st = c->d_state;
    a.key = NoiseKey{static_cast<uint32_t>(c->cfg.seed), static_cast<uint32_t>(c->cfg.seed >> 32)};
    a.sample_base = sample_base; a.count = count; a.N = c->N; a.H = c->H; a.ldx = c->ldx;
    if (c->pair_emission && c->pair_clusters > 0 && count > tc::kBM) {
        // pairs of SMs share a weight tile: 256 samples x 128 workers per cluster and tile
        const int pair_tiles = ceil_div(c->N, tc::kBW) * ceil_div(count, 2 * tc::kBM);
        const int clusters = pair_tiles < c->pair_clusters ? pair_tiles : c->pair_clusters;
        tc::k_emit_tc2<<<2 * clusters, tc::kThreads, tc::kSmem2Bytes, c->stream>>>(c->map_v, c->map_w4, a);
        c->launches += 1;
        return;
    }
    const int tiles = ceil_div(c->N, tc::kBW) * ceil_div(count, tc::kBM);
    const int grid = tiles < c->sm_count ? tiles : c->sm_count;
    launch_dependent(tc::k_emit_tc, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, c->stream, c->map_v, c->map_w4, a);
    c->launches += 1;
}

// Literal emission (Section 3.1.3): I = u Wi2^T + bi2, r = relu(I Wj1^T + bj1), x = I + softplus(r Wj2^T + bj2) * eps.
void launch_gemm_relu_tc(cutoff_ctx* c, const CUtensorMap& map_a, const CUtensorMap& map_b, const tc::GemmTcArgs& a) {
    const int tiles = ceil_div(a.Nout, tc::kGemmBN) * ceil_div(a.M, tc::kBM);
    const int grid = tiles < c->sm_count ? tiles : c->sm_count;
    launch_dependent(tc::k_gemm_relu_tc, dim3(grid), dim3(tc::kThreads), tc::kSmemBytes, c->stream, map_a, map_b, a);
    c->launches += 1;
}

void launch_emission_literal(cutoff_ctx* c, uint32_t sample_base, int count) {
    const NoiseKey key{static_cast<uint32_t>(c->cfg.seed), static_cast<uint32_t>(c->cfg.seed >> 32)};
    const LiteralDev& l = c->lit;
    if (c->use_tc) {
        // r = relu(M u + b') with M = Wj1 Wi2 (I is affine in u), then x = (Wi2 u + bi2) + softplus(Wj2 r + bj2) * eps
        tc::GemmTcArgs a{};
        a.st = c->d_state; a.M = count; a.bias = c->d_Mb; a.a_inv = c->d_v_inv; a.b_inv = c->d_w_inv + 2 * c->N;
        a.out = HalfRows{c->d_r16, c->d_r_inv, c->ldh, c->d_bound + 2};
        a.Nout = c->H; a.K = c->H;
        launch_gemm_relu_tc(c, c->map_v, c->map_M, a);
        tc::EmitDualArgs e;
        e.bias_mean = l.bi2; e.bias_scale = l.bj2; e.u_inv = c->d_v_inv; e.r_inv = c->d_r_inv;
        e.wi_inv = c->d_w_inv; e.wj_inv = c->d_w_inv + c->N; e.x = c->d_x; e.st = c->d_state; e.key = key;
        e.sample_base = sample_base; e.count = count; e.N = c->N; e.H = c->H; e.ldx = c->ldx;
        const int tiles = ceil_div(c->N, tc::kBW) * ceil_div(count, tc::kBM);
        launch_dependent(tc::k_emit_dual_tc, dim3(tiles < c->sm_count ? tiles : c->sm_count), dim3(tc::kThreads), tc::kSmemBytes, c->stream,
                         c->map_v, c->map_r, c->map_wi2, c->map_wj2, e);
        c->launches += 1;
        return;
    }
    GemmFmaArgs a{};
    a.st = c->d_state; a.key = key; a.sample_base = sample_base; a.M = count;
    a.A = c->d_v; a.lda = c->H; a.B = l.Wi2; a.ldb = c->H; a.bias = l.bi2; a.out = c->d_I; a.ld_out = c->ldx;
    a.Nout = c->N; a.K = c->H;
    launch_dependent(k_gemm_fma<kEpiAffine>, dim3(ceil_div(a.Nout, kGemmTN), ceil_div(count, kGemmTM)), dim3(kGemmThreads), 0, c->stream, a);
    a.A = c->d_I; a.lda = c->ldx; a.B = l.Wj1; a.ldb = l.ldn; a.bias = l.bj1; a.out = c->d_r; a.ld_out = c->H;
    a.Nout = c->H; a.K = c->ldx;                                   // the padding columns of both operands are zero
    launch_dependent(k_gemm_fma<kEpiRelu>, dim3(ceil_div(a.Nout, kGemmTN), ceil_div(count, kGemmTM)), dim3(kGemmThreads), 0, c->stream, a);
    a.A = c->d_r; a.lda = c->H; a.B = l.Wj2; a.ldb = c->H; a.bias = l.bj2; a.add = c->d_I; a.out = c->d_x; a.ld_out = c->ldx;
    a.Nout = c->N; a.K = c->H;
    launch_dependent(k_gemm_fma<kEpiScaleNoise>, dim3(ceil_div(a.Nout, kGemmTN), ceil_div(count, kGemmTM)), dim3(kGemmThreads), 0, c->stream, a);
    c->launches += 3;
}

// The fp32 emission keeps its weights in shared memory for up to 64 workers (N=70, S=3000: 19 us either way; N=50, S=8000: 15 against 24;
// N=100, S=60000: 87 against 79), where they fit beside the hidden values (32 workers: H <= 652, 16: every H).
bool emission_rows(const cutoff_ctx* c) {
    return !c->literal && !c->use_tc && c->N <= 64 && (c->N <= 16 ? emit_rows_smem_bytes<4, 4>(c->H) : emit_rows_smem_bytes<8, 4>(c->H)) <= 227 * 1024;
}

// Its kernel for a call of `count` samples, and the shared memory that this takes.  As many samples per lane as still give most warps of the GPU
// a tile: fewer read the weights and hidden values more often.  Not more than four: with eight, tiles twice as large spill and leave
// twice as much of the GPU idle in their last round (N=64, H=320, S=38500: 134 us against 111 with four and 113 without resident
// weights; S=65536: 168 and 162).
struct EmitRowsChoice {
    decltype(&k_emit_rows<4, 4>) kernel;
    size_t smem;
};
template <int TX>
EmitRowsChoice emit_rows_choice(const cutoff_ctx* c, int count) {
    const auto full = [&](int per_lane) { return ceil_div(c->N, 4 * TX) * ceil_div(count, 32 / TX * per_lane) >= 12 * c->sm_count; };
    if (full(4)) return {k_emit_rows<TX, 4>, emit_rows_smem_bytes<TX, 4>(c->H)};
    if (full(2)) return {k_emit_rows<TX, 2>, emit_rows_smem_bytes<TX, 2>(c->H)};
    return {k_emit_rows<TX, 1>, emit_rows_smem_bytes<TX, 1>(c->H)};
}
EmitRowsChoice emit_rows_choice(const cutoff_ctx* c, int count) { return c->N <= 16 ? emit_rows_choice<4>(c, count) : emit_rows_choice<8>(c, count); }

void launch_emission(cutoff_ctx* c, uint32_t sample_base, int count) {
    if (c->literal) { launch_emission_literal(c, sample_base, count); return; }
    if (c->use_tc) { launch_emission_tc(c, sample_base, count); return; }
    const NoiseKey key{static_cast<uint32_t>(c->cfg.seed), static_cast<uint32_t>(c->cfg.seed >> 32)};
    if (emission_rows(c)) {
        const EmitRowsChoice choice = emit_rows_choice(c, count);
        launch_dependent(choice.kernel, dim3(c->sm_count), dim3(kEmitRowsWarps * 32), choice.smem, c->stream, c->m, c->d_v, c->d_W4T, c->ldx,
                         c->d_state, key, sample_base, count, c->d_x, c->ldx);
        c->launches += 1;
        return;
    }
    // 32 samples per CTA read the weights four times less often than 8 do, but need enough samples to occupy the GPU: at N=158, S=2048
    // (192 large tiles) the small ones take 10.3 us
    const int worker_tiles = ceil_div(c->N, kEmitTN), large = worker_tiles * ceil_div(count, 32);
    if (large >= 2 * c->sm_count)
        launch_dependent(k_emit_fma<8>, dim3(large), dim3(kEmitThreads), 0, c->stream, c->m, c->d_v, c->d_W4T, c->ldx, c->d_state, key, sample_base, count,
                         c->d_x, c->ldx);
    else
        launch_dependent(k_emit_fma<2>, dim3(worker_tiles * ceil_div(count, 8)), dim3(kEmitThreads), 0, c->stream, c->m, c->d_v, c->d_W4T, c->ldx, c->d_state,
                         key, sample_base, count, c->d_x, c->ldx);
    c->launches += 1;
}

template <int HQ>
void launch_rnn_resident(cutoff_ctx* c) {
    const size_t smem = enc_rnn_resident_smem_floats(c->H, c->W) * sizeof(float);
    launch_dependent(k_enc_rnn_resident<HQ>, dim3(2), dim3(16 * HQ), smem, c->stream, c->m, c->d_WhR, c->d_proj, c->d_state, c->d_hlr);
}

// Input projections: of the newest vector after a push, of every slot when the ring or the weights changed.
void launch_projection(cutoff_ctx* c, bool newest_only) {
    launch_dependent(c->N % 4 == 0 ? k_enc_proj<true> : k_enc_proj<false>, dim3(ceil_div(c->H, kProjRows), 2), dim3(kProjThreads), 0, c->stream,
                     c->m, c->d_ring, c->d_state, newest_only ? 1 : 0, c->d_proj);
    c->launches += 1;
}

void refresh_projections(cutoff_ctx* c) {
    if (!c->proj_stale) return;
    launch_projection(c, false);
    c->proj_stale = false;
}

// H = 32, 64, 128: one CTA per direction with the recurrence matrix in registers.  Other widths in whole warps, as far as the matrix fits the
// shared memories of a cluster of 8 CTAs (H <= 608, at windows of more than 41 steps less): one of these per direction (H = 256: a thread's share no longer fits its registers, and
// one CTA that keeps part of the matrix in shared memory takes 21 us against 17; H = 192 with one CTA that reads the matrix from
// L2 in every step, lag 6: 62 us, so 17; H = 96, lag 3: 17 and 12).
bool encoder_resident(const cutoff_ctx* c) {
    return (c->H == 32 || c->H == 64 || c->H == 128) && enc_rnn_resident_smem_floats(c->H, c->W) * sizeof(float) <= 200 * 1024;
}
bool encoder_cluster(const cutoff_ctx* c) {
    return !encoder_resident(c) && c->H % 32 == 0 && enc_rnn_cluster_smem_floats(c->H, c->W) * sizeof(float) <= 200 * 1024;
}

void launch_encoder(cutoff_ctx* c) {
    refresh_projections(c);
    if (encoder_resident(c)) {
        if (c->H == 32) launch_rnn_resident<8>(c);
        else if (c->H == 64) launch_rnn_resident<16>(c);
        else launch_rnn_resident<32>(c);
    }
    else if (encoder_cluster(c))
        launch_dependent(k_enc_rnn_cluster, dim3(2 * kRnnClusterSize), dim3(c->H), enc_rnn_cluster_smem_floats(c->H, c->W) * sizeof(float), c->stream,
                         c->m, c->d_proj, c->d_state, c->d_hlr);
    else
        launch_dependent(k_enc_rnn, dim3(2), dim3(kRnnThreads), 2 * c->H * sizeof(float), c->stream, c->m, c->d_proj, c->d_state, c->d_hlr);
    c->launches += 1;
}

int ensure_events(cutoff_ctx* c) {
    if (c->ev_created) return CUTOFF_OK;
    for (auto& row : c->ev)
        for (auto& e : row) CU_CHECK(c, cudaEventCreate(&e));
    c->ev_created = true;
    return CUTOFF_OK;
}

// Enqueue one decision's kernels.  decide = false stops after the per-position sums (a context that holds
// only part of a decision's samples: the argmax follows once the sums of all parts are added).
int enqueue_decision(cutoff_ctx* c, bool decide = true) {
    const bool timed = c->timing;
    if (timed) {
        const int rc = ensure_events(c);
        if (rc) return rc;
        cudaEventRecord(c->ev[0][0], c->stream);
    }
    launch_encoder(c);
    if (timed) cudaEventRecord(c->ev[1][0], c->stream);
    for (int ch = 0; ch < c->n_chunks; ++ch) {
        const int row0 = ch * c->chunk_rows;
        const int count = (c->S - row0) < c->chunk_rows ? (c->S - row0) : c->chunk_rows;
        const uint32_t base = static_cast<uint32_t>(c->cfg.sample_offset) + static_cast<uint32_t>(row0);
        if (timed && ch > 0) cudaEventRecord(c->ev[1][ch], c->stream);
        launch_chain(c, base, count);
        if (timed) cudaEventRecord(c->ev[2][ch], c->stream);
        launch_emission(c, base, count);
        if (timed) cudaEventRecord(c->ev[3][ch], c->stream);
        const int rc = launch_sort(c, count, c->d_partial + static_cast<size_t>(ch) * c->sort_grid * c->N);
        if (rc) return rc;
        if (timed) cudaEventRecord(c->ev[4][ch], c->stream);
    }
    const int64_t total = c->cfg.total_samples > 0 ? c->cfg.total_samples : c->S;
    launch_dependent(k_colsum_decide, dim3(ceil_div(c->N, 32)), dim3(kColsumThreads), 0, c->stream,
                     c->d_partial, c->n_chunks * c->sort_grid, c->N, c->d_sums, 1.0 / static_cast<double>(total), c->d_state,
                     c->h_E, c->h_omega, c->want_std ? c->d_partial + static_cast<size_t>(kPartialRows) * c->N : nullptr,
                     c->d_std, decide ? 1 : 0, c->h_state);
    c->have_std = c->want_std;
    c->launches += 1;
    if (timed) cudaEventRecord(c->ev[5][0], c->stream);
    c->timed_chunks = timed ? c->n_chunks : 0;
    CU_CHECK(c, cudaGetLastError());
    return CUTOFF_OK;
}

int collect_timing(cutoff_ctx* c) {
    for (float& v : c->stage_ms) v = 0.0f;
    if (c->timed_chunks == 0) return CUTOFF_OK;
    float ms = 0.0f;
    CU_CHECK(c, cudaEventElapsedTime(&ms, c->ev[0][0], c->ev[1][0]));
    c->stage_ms[0] = ms;
    for (int ch = 0; ch < c->timed_chunks; ++ch) {
        for (int s = 1; s <= 3; ++s) {
            CU_CHECK(c, cudaEventElapsedTime(&ms, c->ev[s][ch], c->ev[s + 1][ch]));
            c->stage_ms[s] += ms;
        }
    }
    CU_CHECK(c, cudaEventElapsedTime(&ms, c->ev[4][c->timed_chunks - 1], c->ev[5][0]));
    c->stage_ms[4] = ms;
    return CUTOFF_OK;
}

bool valid_latent(int D) { return D == 4 || D == 8 || D == 16 || D == 32; }

// Kernels that need more than 48 KB of dynamic shared memory must be told so once per device, with the context's
// device current (a function attribute belongs to the device's copy of the kernel, not to the process).
template <typename Kernel>
cudaError_t allow_smem(Kernel kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

template <int E>
cudaError_t allow_smem_bucket_warp() {
    cudaError_t e = allow_smem(k_bucket_sum_warp<E, false, kBulk>, bucket_smem_bytes<E>());
    if (e == cudaSuccess) e = allow_smem(k_bucket_sum_warp<E, true, kBulk>, bucket_smem_bytes<E>());
    return e;
}
template <int E>
cudaError_t allow_smem_bucket_cta() {
    cudaError_t e = allow_smem(k_bucket_sum_cta<E, false>, bucket_wide_smem_bytes<E>());
    if (e == cudaSuccess) e = allow_smem(k_bucket_sum_cta<E, true>, bucket_wide_smem_bytes<E>());
    return e;
}
cudaError_t allow_smem_sort(int n) {
    if (n > 1024) {
        switch (keys_per_thread(n, 128)) {
            case 12: return allow_smem_bucket_cta<12>();
            case 16: return allow_smem_bucket_cta<16>();
            case 20: return allow_smem_bucket_cta<20>();
            case 24: return allow_smem_bucket_cta<24>();
            case 28: return allow_smem_bucket_cta<28>();
            default: return allow_smem_bucket_cta<32>();
        }
    }
    switch (n > 128 ? keys_per_thread(n, 32) : 0) {        // the network's rows fit 48 KB
        case 0: return cudaSuccess;
        case 8: return allow_smem_bucket_warp<8>();
        case 12: return allow_smem_bucket_warp<12>();
        case 16: return allow_smem_bucket_warp<16>();
        case 20: return allow_smem_bucket_warp<20>();
        case 24: return allow_smem_bucket_warp<24>();
        case 28: return allow_smem_bucket_warp<28>();
        default: return allow_smem_bucket_warp<32>();
    }
}

// The per-sample chain that the context runs (launch_chain and launch_chain_t choose by the same fields).
template <int D>
cudaError_t allow_smem_chain(const cutoff_ctx* c) {
    if (c->literal) return allow_smem(k_chain_literal<D>, 220 * 1024);
    if constexpr (D <= 16)
        if (c->chain_wide == 2) return allow_smem(k_chain_wide<D, 2>, 220 * 1024);
    if (c->chain_wide) return allow_smem(k_chain_wide<D, 1>, 220 * 1024);
    if (chain_resident_smem_floats(c->D, c->H, c->W) * sizeof(float) <= 200 * 1024) return allow_smem(k_chain_resident<D>, 220 * 1024);
    return allow_smem(k_chain<D>, 220 * 1024);
}

// The kernels that depend on how many samples a call draws: named for the passes of the context's decisions, anew when these change, and for
// the draws that a caller asks for by number.
cudaError_t set_call_attributes(const cutoff_ctx* c, int count) {
    cudaError_t e = cudaSuccess;
    if (c->chain_tc) e = allow_smem(chain_tc_choice(c, count).kernel, 227 * 1024);
    if (e == cudaSuccess && emission_rows(c)) e = allow_smem(emit_rows_choice(c, count).kernel, 227 * 1024);
    return e;
}
cudaError_t set_pass_attributes(const cutoff_ctx* c) {
    const cudaError_t e = set_call_attributes(c, c->chunk_rows);
    return e == cudaSuccess ? set_call_attributes(c, c->S - (c->n_chunks - 1) * c->chunk_rows) : e;      // the last pass may be smaller
}

// Only for the kernels that this context runs, or that an option makes it run: each one is loaded by the driver when it is first named.
cudaError_t set_kernel_attributes(const cutoff_ctx* c) {
    cudaError_t e = allow_smem_sort(c->N);
    if (e == cudaSuccess) e = set_pass_attributes(c);
    if (e == cudaSuccess && !c->chain_tc) {
        switch (c->D) {
            case 4: e = allow_smem_chain<4>(c); break;
            case 8: e = allow_smem_chain<8>(c); break;
            case 16: e = allow_smem_chain<16>(c); break;
            default: e = allow_smem_chain<32>(c); break;
        }
    }
    if (e == cudaSuccess && encoder_resident(c)) {
        switch (c->H) {
            case 32: e = allow_smem(k_enc_rnn_resident<8>, 200 * 1024); break;
            case 64: e = allow_smem(k_enc_rnn_resident<16>, 200 * 1024); break;
            default: e = allow_smem(k_enc_rnn_resident<32>, 200 * 1024); break;
        }
    }
    if (e == cudaSuccess && encoder_cluster(c)) e = allow_smem(k_enc_rnn_cluster, 200 * 1024);
    if (e != cudaSuccess || !c->use_tc) return e;
    if (!c->literal) {
        e = allow_smem(tc::k_emit_tc, tc::kSmemBytes);
        if (e == cudaSuccess) e = allow_smem(tc::k_emit_tc2, tc::kSmem2Bytes);
    } else {
        e = allow_smem(tc::k_gemm_relu_tc, tc::kSmemBytes);
        if (e == cudaSuccess) e = allow_smem(tc::k_emit_dual_tc, tc::kSmemBytes);
    }
    return e;
}

}  // namespace

extern "C" {

const char* cutoff_strerror(int code) {
    switch (code) {
        case CUTOFF_OK: return "ok";
        case CUTOFF_WARMUP: return "warm-up: fewer than lag+1 observations, cutoff = all workers";
        case CUTOFF_DEGENERATE: return "no cutoff has a positive expected time, cutoff = all workers";
        case CUTOFF_ERR_BAD_ARG: return "bad argument";
        case CUTOFF_ERR_BAD_BLOB: return "weight blob does not match the context or is malformed";
        case CUTOFF_ERR_BAD_VALUE: return "run-times must be finite and greater than zero";
        case CUTOFF_ERR_CUDA: return "CUDA error";
        case CUTOFF_ERR_UNSUPPORTED: return "not supported";
        case CUTOFF_ERR_NOMEM: return "out of device memory";
        case CUTOFF_ERR_STATE: return "call out of order";
        case CUTOFF_ERR_TIMEOUT: return "a bounded device-side wait gave up";
        case CUTOFF_ERR_TOO_LARGE: return "request exceeds a fixed built-in capacity (see CUTOFF_STATIC_MAX_N)";
        default: return "unknown code";
    }
}

const char* cutoff_last_error(cutoff_ctx* ctx) { return ctx ? ctx->last_error.c_str() : ""; }

const char* cutoff_stage_name(int i) { return (i >= 0 && i < kNumStages) ? kStageNames[i] : ""; }

int cutoff_create(cutoff_ctx** out, const cutoff_config* cfg) {
    if (!out || !cfg) return CUTOFF_ERR_BAD_ARG;
    if (cfg->n_workers < 1 || cfg->hidden < 4 || cfg->lag < 0 || cfg->n_samples < 1 || cfg->sample_offset < 0 ||
        cfg->total_samples < 0 || cfg->device < 0)
        return CUTOFF_ERR_BAD_ARG;
    if (cfg->precision < CUTOFF_PRECISION_FP32 || cfg->precision > CUTOFF_PRECISION_BF16W) return CUTOFF_ERR_BAD_ARG;
    if (!valid_latent(cfg->latent_dim) || cfg->hidden % cfg->latent_dim != 0) return CUTOFF_ERR_UNSUPPORTED;
    if (cfg->n_workers > 4096 || cfg->hidden > 1024 || cfg->lag > 255) return CUTOFF_ERR_UNSUPPORTED;
    if (cfg->sample_offset + cfg->n_samples > (1ll << 32)) return CUTOFF_ERR_UNSUPPORTED;
    if (cfg->total_samples > 0 && cfg->total_samples < cfg->n_samples) return CUTOFF_ERR_BAD_ARG;

    cutoff_ctx* c = new (std::nothrow) cutoff_ctx();
    if (!c) return CUTOFF_ERR_NOMEM;
    c->cfg = *cfg;
    c->N = cfg->n_workers; c->D = cfg->latent_dim; c->H = cfg->hidden; c->W = cfg->lag + 1; c->S = cfg->n_samples;
    c->ldx = (c->N + 7) & ~7;
    c->ldh = (c->H + 7) & ~7;
    c->P = next_pow2(c->N) < 32 ? 32 : next_pow2(c->N);
    c->stream = static_cast<cudaStream_t>(cfg->stream);
    c->literal = (cfg->flags & CUTOFF_FLAG_LITERAL) != 0;

    auto fail = [&](int rc) { free_all(c); delete c; return rc; };
#define CREATE_CHECK(call)                                                                         \
    do {                                                                                           \
        cudaError_t err__ = (call);                                                                \
        if (err__ != cudaSuccess) return fail(err__ == cudaErrorMemoryAllocation ? CUTOFF_ERR_NOMEM : CUTOFF_ERR_CUDA); \
    } while (0)

    DeviceGuard guard(cfg->device);
    CREATE_CHECK(guard.err);
    if ((cfg->flags & CUTOFF_FLAG_GRAPH) && !c->stream) {
        // the default stream cannot be captured: graph mode without a caller stream runs on its own
        CREATE_CHECK(cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking));
        c->owns_stream = true;
    }
    cudaDeviceProp prop;
    CREATE_CHECK(cudaGetDeviceProperties(&prop, cfg->device));
    c->sm_count = prop.multiProcessorCount;
    if (chain_smem_floats(c->D, c->H, c->W) * sizeof(float) > 220 * 1024) return fail(CUTOFF_ERR_UNSUPPORTED);

    // Pass buffers hold up to 2 GiB of samples; by default one pass covers all S samples.
    {
        // per sample: x and v; literal variant: also r, and I on the fp32 path
        const bool tensor_path = cfg->precision != CUTOFF_PRECISION_FP32;
        const int64_t row_floats = c->ldx + c->H + (c->literal ? c->H + (tensor_path ? 0 : c->ldx) : 0);
        int64_t cap = (2ll << 30) / (row_floats * static_cast<int64_t>(sizeof(float)));
        if (cap < 1024) cap = 1024;
        c->alloc_rows = cap < c->S ? static_cast<int>(cap) : c->S;
    }
    if (ceil_div(c->S, kMaxChunks) > c->alloc_rows) return fail(CUTOFF_ERR_UNSUPPORTED);   // S too large for the pass buffers
    plan_chunks(c, c->alloc_rows);
    c->use_tc = cfg->precision != CUTOFF_PRECISION_FP32;
    c->chain_tc = c->use_tc && tc::chain_tc_window(c->D, c->H, c->W, c->literal) &&
                  ((c->D == tc::kChainD && c->H % 64 == 0 && c->H <= 256) ||
                   (c->D == tc::kChain32D && c->H % 32 == 0 && c->H <= 512));
    // D lanes per sample pay for few samples.  Where the alternative is the resident FMA kernel: one sample per lane up to 12 warps per
    // SM (H=64, lag 20: 4096 samples 28 us against 76; H=128, lag 2: 7000 samples 16.8 against 27), two up to 40 of those warps
    // (9000 samples 16.7 against 19.8 with one and 27; 16384: 24 against 29; 20000: 32 against 39, lag 20: 95 against 110; 36000: 42
    // against 41; D=16, H=128, lag 4: 4700 samples 23 against 27 with one and 39, 10000: 46 against 54; D=32 has no registers for
    // two).  Where it is a tensor-core chain, whose time hardly depends on the samples, up to 16 samples per SM.  Both are equal at (D=16)
    // H=128 2700 samples (lag 4: 23 us) or 3000 (lag 20: 60), H=192 2000 (lag 4: 25) or 2500 (lag 20: 66), H=256 1500 (lag 4: 27), (D=32)
    // H=128 1700 (lag 4: 30) or 2000 (lag 20: 83): one line for all of them.  At its 2368 samples, this one against the tensor-core chain:
    // D=16, lag 4 22 and 23 us at H=128, 27 and 25 at 192, 32 and 27 at 256, lag 20 51 and 60, 64 and 66; D=32, H=128 36 and 30, 91 and 83;
    // in windows of one step 15 and 15, 17 and 15, 19 and 16, at D=32 21 and 17, H=256 30 and 19.
    const int64_t total = cfg->total_samples > 0 ? cfg->total_samples : c->S;       // the same for every shard of a decision, as its draws must be
    const int64_t few = 16 * static_cast<int64_t>(c->sm_count);
    const int64_t warps = total * c->D / 32;
    if (!c->literal && chain_resident_smem_floats(c->D, c->H, c->W) * sizeof(float) <= 200 * 1024)
        c->chain_wide = c->chain_tc ? total <= few : warps <= 3 * few / 4 ? 1 : warps <= 5 * few / 2 && c->D <= 16 ? 2 : warps <= few ? 1 : 0;
    if (c->chain_wide) c->chain_tc = false;

    size_t blob_floats = 0;
    for (const auto& t : c->literal ? tensor_specs_literal(c->N, c->D, c->H) : tensor_specs(c->N, c->D, c->H))
        blob_floats += (t.rows * t.cols + 7) / 8 * 8;            // each tensor starts on a 32-byte boundary
    CREATE_CHECK(cudaMalloc(&c->d_blob, blob_floats * sizeof(float)));
    CREATE_CHECK(cudaMalloc(&c->d_WT, sizeof(float) * 4 * c->H * c->D));
    if (c->literal) {
        if (c->use_tc) {
            CREATE_CHECK(cudaMalloc(&c->d_r16, sizeof(__half) * static_cast<size_t>(c->alloc_rows) * c->ldh));
            CREATE_CHECK(cudaMalloc(&c->d_r_inv, sizeof(float) * c->alloc_rows));
            CREATE_CHECK(cudaMalloc(&c->d_Mb, sizeof(float) * c->H));
            CREATE_CHECK(cudaMalloc(&c->d_M, sizeof(float) * c->H * c->H));
        } else {
            CREATE_CHECK(cudaMalloc(&c->d_r, sizeof(float) * static_cast<size_t>(c->alloc_rows) * c->H));
            CREATE_CHECK(cudaMalloc(&c->d_I, sizeof(float) * static_cast<size_t>(c->alloc_rows) * c->ldx));
            CREATE_CHECK(cudaMalloc(&c->d_Wj1p, sizeof(float) * static_cast<size_t>(c->H) * c->ldx));
            // the padding columns of I are never written and must read as zero
            CREATE_CHECK(cudaMemsetAsync(c->d_I, 0, sizeof(float) * static_cast<size_t>(c->alloc_rows) * c->ldx, c->stream));
        }
    }
    CREATE_CHECK(cudaMalloc(&c->d_WhR, sizeof(float) * 2 * c->H * c->H));
    if (c->chain_tc)
        CREATE_CHECK(cudaMalloc(&c->d_chain_image, tc::chain_tc_image_bytes(c->D, c->H, c->literal) + tc::chain_tc_tail_floats(c->D, c->H) * sizeof(float)));
    CREATE_CHECK(cudaMalloc(&c->d_ring, sizeof(float) * c->W * c->N));
    CREATE_CHECK(cudaMalloc(&c->d_stage, sizeof(float) * c->N));
    CREATE_CHECK(cudaMalloc(&c->d_state, sizeof(DevState)));
    CREATE_CHECK(cudaMalloc(&c->d_proj, sizeof(float) * 2 * c->W * c->H));
    CREATE_CHECK(cudaMalloc(&c->d_hlr, sizeof(float) * 2 * c->W * c->H));
    if (c->use_tc) {
        const size_t w_rows = 2 * static_cast<size_t>(c->N) + (c->literal ? c->H : 0);
        CREATE_CHECK(cudaMalloc(&c->d_v16, sizeof(__half) * static_cast<size_t>(c->alloc_rows) * c->ldh));
        CREATE_CHECK(cudaMalloc(&c->d_v_inv, sizeof(float) * c->alloc_rows));
        CREATE_CHECK(cudaMalloc(&c->d_w16, sizeof(__half) * w_rows * c->ldh));
        CREATE_CHECK(cudaMalloc(&c->d_w_inv, sizeof(float) * w_rows));
        CREATE_CHECK(cudaMalloc(&c->d_bound, 8 * sizeof(float)));
    } else {
        CREATE_CHECK(cudaMalloc(&c->d_v, sizeof(float) * static_cast<size_t>(c->alloc_rows) * c->H));
        if (!c->literal) CREATE_CHECK(cudaMalloc(&c->d_W4T, sizeof(float) * 2 * static_cast<size_t>(c->H) * c->ldx));
    }
    CREATE_CHECK(cudaMalloc(&c->d_x, sizeof(float) * static_cast<size_t>(c->alloc_rows) * c->ldx));
    CREATE_CHECK(cudaMalloc(&c->d_partial, sizeof(float) * 2 * static_cast<size_t>(kPartialRows) * c->N));
    CREATE_CHECK(cudaMalloc(&c->d_std, sizeof(float) * c->N));
    CREATE_CHECK(cudaMalloc(&c->d_sums, sizeof(double) * c->N));
    if (c->use_tc) {
        const uint64_t rows = static_cast<uint64_t>(c->alloc_rows), H = static_cast<uint64_t>(c->H), N = static_cast<uint64_t>(c->N);
        const uint64_t ld = static_cast<uint64_t>(c->ldh);
        int rc = make_tile_map(c, &c->map_v, c->d_v16, rows, H, ld);
        if (!rc && !c->literal) rc = make_tile_map(c, &c->map_w4, c->d_w16, 2 * N, H, ld);
        if (!rc && c->literal) rc = make_tile_map(c, &c->map_r, c->d_r16, rows, H, ld);
        if (!rc && c->literal) rc = make_tile_map(c, &c->map_wi2, c->d_w16, N, H, ld);
        if (!rc && c->literal) rc = make_tile_map(c, &c->map_wj2, c->d_w16 + N * ld, N, H, ld);
        if (!rc && c->literal) rc = make_tile_map(c, &c->map_M, c->d_w16 + 2 * N * ld, H, H, ld);
        if (rc) return fail(rc);
    }
    CREATE_CHECK(set_kernel_attributes(c));
    if (c->use_tc && !c->literal) {
        // how many two-CTA clusters of the two-SM emission kernel the GPU can hold at once
        cudaLaunchConfig_t lc{};
        lc.gridDim = dim3(2 * c->sm_count);
        lc.blockDim = dim3(tc::kThreads);
        lc.dynamicSmemBytes = tc::kSmem2Bytes;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 2; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
        lc.attrs = &at;
        lc.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, tc::k_emit_tc2, &lc) == cudaSuccess && n > 0) c->pair_clusters = n;
        else cudaGetLastError();
    }
    // one pinned block: state | run-times | expected order statistics | throughputs | mask, each on a line of its own
    const size_t line = 128, state_bytes = (sizeof(DevState) + line - 1) / line * line, row_bytes = (sizeof(float) * c->N + line - 1) / line * line;
    CREATE_CHECK(cudaMallocHost(&c->h_state, state_bytes + 3 * row_bytes + c->N));
    char* const pinned = reinterpret_cast<char*>(c->h_state) + state_bytes;
    c->h_stage = reinterpret_cast<float*>(pinned);
    c->h_E = reinterpret_cast<float*>(pinned + row_bytes);
    c->h_omega = reinterpret_cast<float*>(pinned + 2 * row_bytes);
    c->h_mask = reinterpret_cast<uint8_t*>(pinned + 3 * row_bytes);
    CREATE_CHECK(cudaMemsetAsync(c->d_state, 0, sizeof(DevState), c->stream));
    CREATE_CHECK(cudaMemsetAsync(c->d_ring, 0, sizeof(float) * c->W * c->N, c->stream));
    CREATE_CHECK(cudaStreamSynchronize(c->stream));
#undef CREATE_CHECK
    *out = c;
    return CUTOFF_OK;
}

void cutoff_destroy(cutoff_ctx* ctx) {
    if (!ctx) return;
    DeviceGuard guard(ctx->cfg.device);
    cudaStreamSynchronize(ctx->stream);
    free_all(ctx);
    delete ctx;
}

int cutoff_load_weights(cutoff_ctx* c, const void* blob, size_t nbytes) {
    if (!c || !blob) return CUTOFF_ERR_BAD_ARG;
    if (nbytes < 6 * sizeof(uint32_t)) return CUTOFF_ERR_BAD_BLOB;
    uint32_t hdr[6];
    std::memcpy(hdr, blob, sizeof(hdr));
    if (hdr[0] != kBlobMagic || hdr[1] != 1u) return CUTOFF_ERR_BAD_BLOB;
    if (hdr[2] != static_cast<uint32_t>(c->N) || hdr[3] != static_cast<uint32_t>(c->D) ||
        hdr[4] != static_cast<uint32_t>(c->H) || hdr[5] != (c->literal ? 1u : 0u))
        return CUTOFF_ERR_BAD_BLOB;
    const auto specs = c->literal ? tensor_specs_literal(c->N, c->D, c->H) : tensor_specs(c->N, c->D, c->H);
    size_t total = 0;
    for (const auto& t : specs) total += t.rows * t.cols;
    if (nbytes != sizeof(hdr) + total * sizeof(float)) return CUTOFF_ERR_BAD_BLOB;
    const float* src = reinterpret_cast<const float*>(static_cast<const char*>(blob) + sizeof(hdr));
    for (size_t i = 0; i < total; ++i)
        if (!std::isfinite(src[i])) return CUTOFF_ERR_BAD_BLOB;

    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    // device layout: every tensor starts on a 32-byte boundary (16-byte loads and tensor maps need aligned bases)
    std::vector<size_t> off(specs.size());
    size_t o = 0;
    for (size_t i = 0; i < specs.size(); ++i) { off[i] = o; o += (specs[i].rows * specs[i].cols + 7) / 8 * 8; }
    std::vector<float> host(o, 0.0f);
    {
        size_t so = 0;
        for (size_t i = 0; i < specs.size(); ++i) {
            const size_t n = specs[i].rows * specs[i].cols;
            std::memcpy(host.data() + off[i], src + so, n * sizeof(float));
            so += n;
        }
    }
    if (c->use_tc) {
        // Weights of the products that run on the tensor cores, as the tensor cores will see them, kept as
        // fp32 bit patterns: bf16 (nearest even) for the bf16-weight precision, else tf32 (nearest, ties
        // away from zero).  Compact variant: W4; literal variant: Wi2, Wj1, Wj2.
        const std::vector<size_t> rounded = c->literal ? std::vector<size_t>{29, 31, 33} : std::vector<size_t>{21};
        for (size_t t : rounded) {
            float* wt = host.data() + off[t];
            for (size_t i = 0; i < specs[t].rows * specs[t].cols; ++i) {
                uint32_t u;
                std::memcpy(&u, &wt[i], 4);
                if (c->cfg.precision == CUTOFF_PRECISION_BF16W) u = (u + 0x7FFFu + ((u >> 16) & 1u)) & 0xFFFF0000u;
                else u = (u + 0x1000u) & 0xFFFFE000u;
                std::memcpy(&wt[i], &u, 4);
            }
        }
    }
    CU_CHECK(c, upload(c, c->d_blob, host.data(), host.size() * sizeof(float)));
    if (c->use_tc) {
        const int N = c->N, H = c->H, D = c->D;
        if (c->literal) {
            half_rows(c, c->d_blob + off[29], N, 0);                                                     // Wi2
            half_rows(c, c->d_blob + off[33], N, N);                                                     // Wj2
        } else {
            half_rows(c, c->d_blob + off[21], 2 * N, 0);                                                 // W4
        }
        CU_CHECK(c, cudaGetLastError());
        const size_t first = c->literal ? 27 : 19;                                                       // Wi1 or W3, and its bias
        float bound[2];
        layer_bound(host.data() + off[first], host.data() + off[first + 1], H, D, !c->literal, bound);
        CU_CHECK(c, upload(c, c->d_bound, bound, sizeof(bound)));
        for (size_t t = 0; t < (c->literal ? 2u : 1u); ++t) {                                            // W1, or Wg1 and Wh1
            layer_bound(host.data() + off[15 + 4 * t], host.data() + off[16 + 4 * t], H, D, true, bound);
            CU_CHECK(c, upload(c, c->d_bound + 4 + 2 * t, bound, sizeof(bound)));
        }
    }
    if (!c->use_tc && !c->literal) {
        k_transpose_heads<<<dim3(ceil_div(c->ldx, 32), ceil_div(c->H, 32), 2), dim3(32, 8), 0, c->stream>>>(c->d_blob + off[21], c->N, c->H, c->ldx, c->d_W4T);
        CU_CHECK(c, cudaGetLastError());
    }
    // transposed copies [D][H] of the latent-to-hidden matrices for the per-sample chain
    const size_t D = c->D, H = c->H;
    const int n_transposed = c->literal ? 4 : 3;
    std::vector<float> wT(n_transposed * H * D);
    const size_t src_off[4] = {off[8], off[15], off[19], c->literal ? off[27] : 0};   // Wz, W1 | Wg1, W3 | Wh1, - | Wi1
    for (int t = 0; t < n_transposed; ++t) {
        const float* w = host.data() + src_off[t];
        for (size_t i = 0; i < H; ++i)
            for (size_t d = 0; d < D; ++d) wT[t * H * D + d * H + i] = w[i * D + d];
    }
    CU_CHECK(c, upload(c, c->d_WT, wT.data(), wT.size() * sizeof(float)));

    if (H == 32 || H == 64 || H == 128) {
        // recurrence matrices regrouped per thread of k_enc_rnn_resident (the widths that kernel serves; the layout
        // needs H / 4 to be a multiple of 4): [dir][j4][thread = 4*i + q][4]
        const size_t HQ = H / 4, T = 4 * H;
        std::vector<float> whr(2 * H * H);
        const size_t src_off[2] = {off[1], off[5]};                   // Whf, Whb: each [H][H]
        for (int dir = 0; dir < 2; ++dir) {
            const float* w = host.data() + src_off[dir];
            for (size_t i = 0; i < H; ++i)
                for (size_t q = 0; q < 4; ++q)
                    for (size_t j = 0; j < HQ; ++j)
                        whr[dir * H * H + ((j / 4) * T + (4 * i + q)) * 4 + (j % 4)] = w[i * H + q * HQ + j];
        }
        CU_CHECK(c, upload(c, c->d_WhR, whr.data(), whr.size() * sizeof(float)));
    }
    // Operand tiles of the tensor-core chain kernels as they will sit in shared memory: tf32 (nearest, ties away),
    // K-major rows of 32 values, 16-byte chunks XOR-swizzled with the row index modulo 8.
    if (c->chain_tc) {
        const bool lit = c->literal;
        const float* wz = host.data() + off[8];                  // first layers, [H][D]: Wz; W1 or Wg1; W3 or Wh1; Wi1
        const float* wa = host.data() + off[15];
        const float* wb = host.data() + off[19];
        const float* wi1 = lit ? host.data() + off[27] : nullptr;
        const float* wmu = host.data() + off[10];                // second layers, [D][H] ([2D][H] for W2): Wmu; W2 or Wg2; Wh2
        const float* wc = host.data() + off[17];
        const float* wh2 = lit ? host.data() + off[21] : nullptr;
        const float* ws = lit ? host.data() + off[25] : nullptr; // [D][D]
        const size_t tile = H * 32, bytes = tc::chain_tc_image_bytes(c->D, c->H, lit);
        std::vector<uint8_t> img(bytes + tc::chain_tc_tail_floats(c->D, c->H) * sizeof(float), 0);
        float* const first = reinterpret_cast<float*>(img.data());
        if (D == 16) {                                           // two matrices share a tile (columns 0..15 and 16..31)
            put_first_layer(first, wz, H, D, 0);
            put_first_layer(first, wa, H, D, 16);
            put_first_layer(first + tile, wb, H, D, 0);
            if (lit) put_first_layer(first + tile, wi1, H, D, 16);
        } else {
            put_first_layer(first, wz, H, D, 0);
            put_first_layer(first + tile, wa, H, D, 0);
            put_first_layer(first + 2 * tile, wb, H, D, 0);
            if (lit) put_first_layer(first + 3 * tile, wi1, H, D, 0);
        }
        const size_t rows = tc::chain_tc_row_bytes(c->D, c->H);
        uint8_t* const guide = img.data() + tc::chain_tc_first_bytes(c->D, c->H, lit);
        uint8_t* const out = guide + 3 * rows;
        float* const inv = reinterpret_cast<float*>(img.data() + bytes);
        put_second_layer_half(guide, inv, wmu, D, H, 3 * D);
        {
            // Wsig Wmu as the sum of two halves; with Wsig bmu + bsig also in fp32
            const float *wsig = host.data() + off[12], *bmu = host.data() + off[11], *bsig = host.data() + off[13];
            std::vector<double> map(D * H, 0.0), rest(D * H);
            for (size_t d = 0; d < D; ++d)
                for (size_t e = 0; e < D; ++e)
                    for (size_t k = 0; k < H; ++k) map[d * H + k] += static_cast<double>(wsig[d * D + e]) * wmu[e * H + k];
            put_second_layer_half(guide, inv, map.data(), D, H, D, 3 * D, rest.data());
            put_second_layer_half(guide, inv, rest.data(), D, H, 2 * D, 3 * D);
            float* const plain = inv + 5 * D;
            for (size_t d = 0; d < D; ++d) {
                double b = bsig[d];
                for (size_t e = 0; e < D; ++e) b += static_cast<double>(wsig[d * D + e]) * bmu[e];
                plain[d] = static_cast<float>(b);
                for (size_t k = 0; k < H; ++k) plain[D + d * H + k] = static_cast<float>(map[d * H + k]);
            }
        }
        if (lit) {
            put_second_layer_half(out, inv + 3 * D, wc, D, H, D);
            put_second_layer_half(out + rows, inv + 4 * D, wh2, D, H, D);
            put_first_layer(reinterpret_cast<float*>(out + 2 * rows), ws, D, D, 0);
        } else {
            put_second_layer_half(out, inv + 3 * D, wc, 2 * D, H, 2 * D);
        }
        CU_CHECK(c, upload(c, c->d_chain_image, img.data(), img.size()));
    }

    ModelDev& m = c->m;
    m.N = c->N; m.D = c->D; m.H = c->H; m.W = c->W;
    const float* b = c->d_blob;
    m.Wxf = b + off[0]; m.Whf = b + off[1]; m.bf = b + off[2]; m.a0 = b + off[3];
    m.Wxb = b + off[4]; m.Whb = b + off[5]; m.bb = b + off[6]; m.b0 = b + off[7];
    m.WzT = c->d_WT; m.bz = b + off[9]; m.Wmu = b + off[10]; m.bmu = b + off[11];
    m.Wsig = b + off[12]; m.bsig = b + off[13]; m.z0 = b + off[14];
    if (c->literal) {
        if (c->use_tc) {
            // I = Wi2 u + bi2 is affine in u, so Wj1 I + bj1 = M u + b' with M = Wj1 Wi2 [H][H] and b' = Wj1 bi2 + bj1:
            // formed here once, in double, from the weights as the tensor cores see them; M is rounded to tf32.
            const size_t N = c->N;
            const float* wj1 = host.data() + off[31];    // [H][N]
            const float* wi2 = host.data() + off[29];    // [N][H]
            const float* bi2 = host.data() + off[30];
            const float* bj1 = host.data() + off[32];
            std::vector<float> big_m(H * H), mb(H);
            std::vector<double> acc(H);
            for (size_t i = 0; i < H; ++i) {
                std::fill(acc.begin(), acc.end(), 0.0);
                double bacc = bj1[i];
                for (size_t k = 0; k < N; ++k) {
                    const double w = wj1[i * N + k];
                    const float* row = wi2 + k * H;
                    for (size_t j = 0; j < H; ++j) acc[j] += w * row[j];
                    bacc += w * bi2[k];
                }
                for (size_t j = 0; j < H; ++j) big_m[i * H + j] = host_tf32(static_cast<float>(acc[j]));
                mb[i] = static_cast<float>(bacc);
            }
            float bound[2];
            layer_bound(big_m.data(), mb.data(), H, H, true, bound);
            CU_CHECK(c, upload(c, c->d_bound + 2, bound, sizeof(bound)));
            CU_CHECK(c, upload(c, c->d_Mb, mb.data(), mb.size() * sizeof(float)));
            CU_CHECK(c, upload(c, c->d_M, big_m.data(), big_m.size() * sizeof(float)));
            half_rows(c, c->d_M, c->H, 2 * c->N);
            CU_CHECK(c, cudaGetLastError());
        } else {
            // Wj1 [H][N] with rows padded with zeros to ldx floats (rows then start on 32 bytes for any N)
            std::vector<float> wj1p(H * static_cast<size_t>(c->ldx), 0.0f);
            for (size_t i = 0; i < H; ++i)
                std::memcpy(wj1p.data() + i * c->ldx, host.data() + off[31] + i * c->N, sizeof(float) * c->N);
            CU_CHECK(c, upload(c, c->d_Wj1p, wj1p.data(), wj1p.size() * sizeof(float)));
        }
        LiteralDev& l = c->lit;
        l.Wg1T = c->d_WT + H * D; l.bg1 = b + off[16]; l.Wg2 = b + off[17]; l.bg2 = b + off[18];
        l.Wh1T = c->d_WT + 2 * H * D; l.bh1 = b + off[20]; l.Wh2 = b + off[21]; l.bh2 = b + off[22];
        l.Wl = b + off[23]; l.bl = b + off[24]; l.Ws = b + off[25]; l.bs = b + off[26];
        l.Wi1T = c->d_WT + 3 * H * D; l.bi1 = b + off[28];
        l.Wi2 = b + off[29]; l.bi2 = b + off[30];
        l.Wj1 = c->d_Wj1p; l.bj1 = b + off[32]; l.ldn = c->ldx;
        l.Wj2 = b + off[33]; l.bj2 = b + off[34];
        m.W1T = m.b1 = m.W2 = m.b2 = m.W3T = m.b3 = m.W4 = m.b4 = nullptr;
        c->weights_loaded = true;
        c->proj_stale = true;
        return CUTOFF_OK;
    }
    m.W1T = c->d_WT + H * D; m.b1 = b + off[16]; m.W2 = b + off[17]; m.b2 = b + off[18];
    m.W3T = c->d_WT + 2 * H * D; m.b3 = b + off[20]; m.W4 = b + off[21]; m.b4 = b + off[22];
    c->weights_loaded = true;
    c->proj_stale = true;
    return CUTOFF_OK;
}

// With `report` the device state as the push leaves it goes to h_state, for a call that waits for the push.  The others leave h_state to
// the decisions: one that is in flight reports its own state to cutoff_fetch, not what a push behind it found.
static void launch_push(cutoff_ctx* c, const float* src, bool report) {
    launch_dependent(k_push, dim3(1), dim3(kPushThreads), 0, c->stream, src, c->d_ring, c->d_state, c->N, c->W, report ? c->h_state : nullptr);
    c->launches += 1;
}

static int push_common(cutoff_ctx* c, const float* src, bool report) {
    launch_push(c, src, report);
    if (c->weights_loaded && !c->proj_stale) launch_projection(c, true);     // else every slot is redone before the next decision
    CU_CHECK(c, cudaGetLastError());
    c->pushes += 1;
    return CUTOFF_OK;
}

int cutoff_push_async(cutoff_ctx* c, const float* runtimes_sec_device) {
    if (!c || !runtimes_sec_device) return CUTOFF_ERR_BAD_ARG;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    return push_common(c, runtimes_sec_device, false);
}

// Push with a censoring mask: land run-times and mask on the device, replace the censored entries by
// draws from the truncated predictive distribution of the last decision, then push as usual.
static int push_censored(cutoff_ctx* c, const float* runtimes_sec, int on_device, const uint8_t* censored) {
    if (!c->draws_valid) return CUTOFF_ERR_STATE;          // no decision yet whose draws could be used
    if (c->cfg.sample_offset != 0 || (c->cfg.total_samples > 0 && c->cfg.total_samples != c->S))
        return CUTOFF_ERR_UNSUPPORTED;                      // a context that holds only part of the draws
    const float* src = runtimes_sec;
    const uint8_t* mask = censored;
    if (!on_device) {
        int finished = 0;
        for (int j = 0; j < c->N; ++j) {
            if (censored[j]) continue;
            if (!(runtimes_sec[j] > 0.0f) || !std::isfinite(runtimes_sec[j])) return CUTOFF_ERR_BAD_VALUE;
            ++finished;
        }
        if (finished == 0) return CUTOFF_ERR_BAD_ARG;
        CU_CHECK(c, cudaStreamSynchronize(c->stream));     // the landing buffers may still be in use
        for (int j = 0; j < c->N; ++j) c->h_stage[j] = censored[j] ? 1.0f : runtimes_sec[j];
        std::memcpy(c->h_mask, censored, c->N);
        src = c->h_stage;
        mask = c->h_mask;
    }
    const NoiseKey key{static_cast<uint32_t>(c->cfg.seed), static_cast<uint32_t>(c->cfg.seed >> 32)};
    k_impute<<<c->N < kImputeCtas ? c->N : kImputeCtas, kImputeThreads, 0, c->stream>>>(src, mask, c->d_stage, c->d_x, c->ldx, c->S, c->N, c->d_state, key);
    c->launches += 1;
    c->draws_valid = false;                                 // one step's draws serve one push
    int rc = push_common(c, c->d_stage, true);
    if (rc) return rc;
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    if (c->h_state->error_flags & (kErrBadValue | kErrNoFinisher)) {
        c->pushes = c->h_state->push_count;
        CU_CHECK(c, cudaMemsetAsync(&c->d_state->error_flags, 0, sizeof(int32_t), c->stream));
        return CUTOFF_ERR_BAD_VALUE;
    }
    return CUTOFF_OK;
}

int cutoff_push(cutoff_ctx* c, const float* runtimes_sec, int on_device, const uint8_t* censored) {
    if (!c || !runtimes_sec) return CUTOFF_ERR_BAD_ARG;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    if (censored) return push_censored(c, runtimes_sec, on_device, censored);
    if (!on_device) {
        for (int j = 0; j < c->N; ++j)
            if (!(runtimes_sec[j] > 0.0f) || !std::isfinite(runtimes_sec[j])) return CUTOFF_ERR_BAD_VALUE;
        CU_CHECK(c, cudaStreamSynchronize(c->stream));       // the landing buffer may still be in use
        std::memcpy(c->h_stage, runtimes_sec, sizeof(float) * c->N);
        const int rc = push_common(c, c->h_stage, false);
        c->stage_in_use = true;
        return rc;
    }
    const int rc = push_common(c, runtimes_sec, true);
    if (rc) return rc;
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    if (c->h_state->error_flags & kErrBadValue) {
        // the kernel left the window untouched; clear the flag and undo the host-side count
        c->pushes = c->h_state->push_count;
        CU_CHECK(c, cudaMemsetAsync(&c->d_state->error_flags, 0, sizeof(int32_t), c->stream));
        return CUTOFF_ERR_BAD_VALUE;
    }
    return CUTOFF_OK;
}

int cutoff_predict_async(cutoff_ctx* c) {
    if (!c) return CUTOFF_ERR_BAD_ARG;
    if (!c->weights_loaded) return CUTOFF_ERR_STATE;
    if (c->pending || c->partial_pending) return CUTOFF_ERR_STATE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    c->pending = true;
    c->pending_warmup = c->pushes < static_cast<uint32_t>(c->W);
    if (c->pending_warmup) {
        // nothing to compute; still read the state so that a bad device push is reported
        CU_CHECK(c, cudaMemcpyAsync(c->h_state, c->d_state, sizeof(DevState), cudaMemcpyDeviceToHost, c->stream));
        return CUTOFF_OK;
    }
    const int rc = enqueue_decision(c);
    if (rc) c->pending = false;
    return rc;
}

int cutoff_fetch(cutoff_ctx* c, int32_t* c_out) {
    if (!c || !c_out) return CUTOFF_ERR_BAD_ARG;
    if (!c->pending) return CUTOFF_ERR_STATE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    c->pending = false;
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    if (c->h_state->error_flags & kErrBadValue) {
        c->pushes = c->h_state->push_count;
        CU_CHECK(c, cudaMemsetAsync(&c->d_state->error_flags, 0, sizeof(int32_t), c->stream));
        return CUTOFF_ERR_BAD_VALUE;
    }
    if (c->h_state->error_flags & kErrTimeout) return CUTOFF_ERR_TIMEOUT;
    if (c->pending_warmup) {
        *c_out = c->N;
        return CUTOFF_WARMUP;
    }
    const int rc = collect_timing(c);
    if (rc) return rc;
    c->have_result = true;
    c->decided_once = true;
    c->draws_valid = c->n_chunks == 1;
    *c_out = c->h_state->c_star;
    return c->h_state->code == 2 ? CUTOFF_DEGENERATE : CUTOFF_OK;
}

int cutoff_predict(cutoff_ctx* c, int32_t* c_out) {
    if (!c || !c_out) return CUTOFF_ERR_BAD_ARG;
    const int rc = cutoff_predict_async(c);
    if (rc < 0) return rc;
    return cutoff_fetch(c, c_out);
}

// Capture "push, decide" once, the run-times read from the pinned landing buffer or from the one on the device; replays need no
// changing argument because the window position, the normaliser and the decision counter live
// in device memory.
static int build_graph(cutoff_ctx* c, bool from_host) {
    refresh_projections(c);                        // not part of the graph: replays only project the vector they push
    const int64_t launches_before = c->launches;
    CU_CHECK(c, cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
    launch_push(c, from_host ? c->h_stage : c->d_stage, false);
    launch_projection(c, true);
    const bool timing = c->timing;
    c->timing = false;
    const int rc = enqueue_decision(c);
    c->timing = timing;
    cudaGraph_t g = nullptr;
    const cudaError_t end = cudaStreamEndCapture(c->stream, &g);
    c->graph_kernels = static_cast<int>(c->launches - launches_before);
    c->launches = launches_before;                 // nothing ran yet
    if (rc != CUTOFF_OK || end != cudaSuccess || !g) {
        if (g) cudaGraphDestroy(g);
        c->last_error = std::string("graph capture failed: ") + cudaGetErrorString(end);
        cudaGetLastError();
        return CUTOFF_ERR_CUDA;
    }
    if (from_host) {
        c->graph = g;
        CU_CHECK(c, cudaGraphInstantiate(&c->graph_exec, c->graph, 0));
    } else {
        c->graph_dev = g;
        CU_CHECK(c, cudaGraphInstantiate(&c->graph_dev_exec, c->graph_dev, 0));
    }
    return CUTOFF_OK;
}

int cutoff_step(cutoff_ctx* c, const float* runtimes_sec, int32_t* c_out) {
    if (!c || !runtimes_sec || !c_out) return CUTOFF_ERR_BAD_ARG;
    if (!c->weights_loaded || c->pending) return CUTOFF_ERR_STATE;
    const bool replay = (c->cfg.flags & CUTOFF_FLAG_GRAPH) && c->decided_once &&
                        c->pushes + 1 >= static_cast<uint32_t>(c->W);
    if (!replay) {
        const int rc = cutoff_push(c, runtimes_sec, 0, nullptr);
        if (rc < 0) return rc;
        return cutoff_predict(c, c_out);
    }
    for (int j = 0; j < c->N; ++j)
        if (!(runtimes_sec[j] > 0.0f) || !std::isfinite(runtimes_sec[j])) return CUTOFF_ERR_BAD_VALUE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    if (!c->graph_exec) {
        CU_CHECK(c, cudaStreamSynchronize(c->stream));
        const int rc = build_graph(c, true);
        if (rc) return rc;
    }
    if (c->stage_in_use) CU_CHECK(c, cudaStreamSynchronize(c->stream));   // cutoff_push returns while its kernel has yet to read the buffer
    c->stage_in_use = false;
    std::memcpy(c->h_stage, runtimes_sec, sizeof(float) * c->N);
    refresh_projections(c);                        // after a restore or new weights; the replay then adds the new vector
    CU_CHECK(c, cudaGraphLaunch(c->graph_exec, c->stream));
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    c->launches += c->graph_kernels;
    c->pushes += 1;
    c->draws_valid = c->n_chunks == 1;
    if (c->h_state->error_flags & kErrTimeout) return CUTOFF_ERR_TIMEOUT;
    c->have_result = true;
    *c_out = c->h_state->c_star;
    return c->h_state->code == 2 ? CUTOFF_DEGENERATE : CUTOFF_OK;
}

int cutoff_step_device(cutoff_ctx* c, const float* runtimes_sec_device, int32_t* c_out) {
    if (!c || !runtimes_sec_device || !c_out) return CUTOFF_ERR_BAD_ARG;
    if (!c->weights_loaded || c->pending) return CUTOFF_ERR_STATE;
    const bool replay = (c->cfg.flags & CUTOFF_FLAG_GRAPH) && c->decided_once &&
                        c->pushes + 1 >= static_cast<uint32_t>(c->W);
    if (!replay) {
        const int rc = cutoff_push(c, runtimes_sec_device, 1, nullptr);
        if (rc < 0) return rc;
        return cutoff_predict(c, c_out);
    }
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    if (!c->graph_dev_exec) {
        CU_CHECK(c, cudaStreamSynchronize(c->stream));
        const int rc = build_graph(c, false);
        if (rc) return rc;
    }
    refresh_projections(c);
    CU_CHECK(c, cudaMemcpyAsync(c->d_stage, runtimes_sec_device, sizeof(float) * c->N, cudaMemcpyDeviceToDevice, c->stream));
    CU_CHECK(c, cudaGraphLaunch(c->graph_dev_exec, c->stream));
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    c->launches += c->graph_kernels;
    if (c->h_state->error_flags & kErrBadValue) {
        // the push kernel left the window untouched, but the decision that followed it ran on the old window and
        // advanced the decision counter: put the counter back, clear the flag, report the bad value
        const uint32_t step_before = c->h_state->step - 1u;
        CU_CHECK(c, cudaMemcpyAsync(&c->d_state->step, &step_before, sizeof(uint32_t), cudaMemcpyHostToDevice, c->stream));
        CU_CHECK(c, cudaMemsetAsync(&c->d_state->error_flags, 0, sizeof(int32_t), c->stream));
        CU_CHECK(c, cudaStreamSynchronize(c->stream));
        c->draws_valid = false;
        return CUTOFF_ERR_BAD_VALUE;
    }
    c->pushes += 1;
    c->draws_valid = c->n_chunks == 1;
    if (c->h_state->error_flags & kErrTimeout) return CUTOFF_ERR_TIMEOUT;
    c->have_result = true;
    *c_out = c->h_state->c_star;
    return c->h_state->code == 2 ? CUTOFF_DEGENERATE : CUTOFF_OK;
}

int cutoff_get_stats(cutoff_ctx* c, float* e_out, float* omega_out) {
    if (!c) return CUTOFF_ERR_BAD_ARG;
    if (!c->have_result) return CUTOFF_ERR_STATE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    if (c->pending || c->partial_pending) CU_CHECK(c, cudaStreamSynchronize(c->stream));   // a later decision is writing them
    if (e_out) std::memcpy(e_out, c->h_E, sizeof(float) * c->N);
    if (omega_out) std::memcpy(omega_out, c->h_omega, sizeof(float) * c->N);
    return CUTOFF_OK;
}

int cutoff_get_order_stat_std(cutoff_ctx* c, float* std_sec) {
    if (!c || !std_sec) return CUTOFF_ERR_BAD_ARG;
    if (!c->have_result || !c->have_std) return CUTOFF_ERR_STATE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    CU_CHECK(c, cudaMemcpyAsync(std_sec, c->d_std, sizeof(float) * c->N, cudaMemcpyDeviceToHost, c->stream));
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    return CUTOFF_OK;
}

int cutoff_get_partial_sums(cutoff_ctx* c, double* sums) {
    if (!c || !sums) return CUTOFF_ERR_BAD_ARG;
    if (!c->have_result) return CUTOFF_ERR_STATE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    CU_CHECK(c, cudaMemcpyAsync(sums, c->d_sums, sizeof(double) * c->N, cudaMemcpyDeviceToHost, c->stream));
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    return CUTOFF_OK;
}

int cutoff_decide_from_sums(cutoff_ctx* c, const double* sums, int32_t* c_out) {
    if (!c || !sums || !c_out) return CUTOFF_ERR_BAD_ARG;
    if (c->pending) return CUTOFF_ERR_STATE;
    if (c->pushes < static_cast<uint32_t>(c->W)) return CUTOFF_ERR_STATE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    CU_CHECK(c, cudaMemcpyAsync(c->d_sums, sums, sizeof(double) * c->N, cudaMemcpyHostToDevice, c->stream));
    const int64_t total = c->cfg.total_samples > 0 ? c->cfg.total_samples : c->S;
    k_decide<<<1, kDecideThreads, 0, c->stream>>>(c->d_sums, c->N, 1.0 / static_cast<double>(total), c->d_state, 0,
                                                  c->h_E, c->h_omega, c->h_state);
    c->launches += 1;
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    c->have_result = true;
    *c_out = c->h_state->c_star;
    return c->h_state->code == 2 ? CUTOFF_DEGENERATE : CUTOFF_OK;
}

int cutoff_predict_partial_async(cutoff_ctx* c) {
    if (!c) return CUTOFF_ERR_BAD_ARG;
    if (!c->weights_loaded) return CUTOFF_ERR_STATE;
    if (c->pending || c->partial_pending) return CUTOFF_ERR_STATE;
    if (c->pushes < static_cast<uint32_t>(c->W)) return CUTOFF_WARMUP;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    const int rc = enqueue_decision(c, false);
    if (rc == CUTOFF_OK) c->partial_pending = true;
    return rc;
}

int cutoff_partial_sums_device(cutoff_ctx* c, double** sums_device) {
    if (!c || !sums_device) return CUTOFF_ERR_BAD_ARG;
    *sums_device = c->d_sums;
    return CUTOFF_OK;
}

int cutoff_decide_from_device_sums(cutoff_ctx* c, const double* sums_device, int32_t* c_out) {
    if (!c || !sums_device || !c_out) return CUTOFF_ERR_BAD_ARG;
    if (c->pending) return CUTOFF_ERR_STATE;
    if (c->pushes < static_cast<uint32_t>(c->W)) return CUTOFF_ERR_STATE;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    if (sums_device != c->d_sums)
        CU_CHECK(c, cudaMemcpyAsync(c->d_sums, sums_device, sizeof(double) * c->N, cudaMemcpyDeviceToDevice, c->stream));
    const int64_t total = c->cfg.total_samples > 0 ? c->cfg.total_samples : c->S;
    // the decision counter moves on here if the sums came from cutoff_predict_partial_async (which left it alone)
    k_decide<<<1, kDecideThreads, 0, c->stream>>>(c->d_sums, c->N, 1.0 / static_cast<double>(total), c->d_state,
                                                  c->partial_pending ? 1 : 0, c->h_E, c->h_omega, c->h_state);
    c->launches += 1;
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    if (c->h_state->error_flags & kErrBadValue) {
        // a bad asynchronous push came before this decision: as cutoff_fetch reports it
        c->pushes = c->h_state->push_count;
        CU_CHECK(c, cudaMemsetAsync(&c->d_state->error_flags, 0, sizeof(int32_t), c->stream));
        c->partial_pending = false;
        return CUTOFF_ERR_BAD_VALUE;
    }
    if (c->h_state->error_flags & kErrTimeout) return CUTOFF_ERR_TIMEOUT;
    if (c->partial_pending) {
        const int rc = collect_timing(c);
        if (rc) return rc;
        c->partial_pending = false;
        c->decided_once = true;
    }
    c->have_result = true;
    *c_out = c->h_state->c_star;
    return c->h_state->code == 2 ? CUTOFF_DEGENERATE : CUTOFF_OK;
}

int cutoff_measure_pipe_rates(int device, float* rates_out) {
    if (device < 0 || !rates_out) return CUTOFF_ERR_BAD_ARG;
    cutoff_ctx* none = nullptr;
    DeviceGuard guard(device);
    CU_CHECK(none, guard.err);
    cudaDeviceProp prop;
    CU_CHECK(none, cudaGetDeviceProperties(&prop, device));
    const int sms = prop.multiProcessorCount;
    long long* d_cycles = nullptr;
    float* d_sink = nullptr;
    if (cudaMalloc(&d_cycles, sizeof(long long) * sms) != cudaSuccess || cudaMalloc(&d_sink, sizeof(float)) != cudaSuccess) {
        cudaFree(d_cycles);
        return CUTOFF_ERR_NOMEM;
    }
    std::vector<long long> h(sms);
    int rc = CUTOFF_OK;
    for (int kind = 0; kind < 3 && rc == CUTOFF_OK; ++kind) {
        double best = 0.0;
        for (int rep = 0; rep < 4 && rc == CUTOFF_OK; ++rep) {         // the first repetition warms the clocks up
            if (kind == 0) k_pipe_rate<0><<<sms, kRateThreads>>>(1.25f, d_cycles, d_sink);
            if (kind == 1) k_pipe_rate<1><<<sms, kRateThreads>>>(1.25f, d_cycles, d_sink);
            if (kind == 2) k_pipe_rate<2><<<sms, kRateThreads>>>(1.25f, d_cycles, d_sink);
            if (cudaMemcpy(h.data(), d_cycles, sizeof(long long) * sms, cudaMemcpyDeviceToHost) != cudaSuccess) {
                rc = CUTOFF_ERR_CUDA;
                break;
            }
            long long worst = 1;
            for (long long v : h) worst = v > worst ? v : worst;
            const double warp_instr = static_cast<double>(kRateThreads / 32) * kRateChains * kRateIters;
            const double rate = warp_instr / static_cast<double>(worst);
            if (rep > 0 && rate > best) best = rate;
        }
        rates_out[kind] = static_cast<float>(best);
    }
    cudaFree(d_cycles);
    cudaFree(d_sink);
    return rc;
}

int cutoff_measure_operand_stream(int device, float* gbs_out) {
    if (device < 0 || !gbs_out) return CUTOFF_ERR_BAD_ARG;
    cutoff_ctx* none = nullptr;
    DeviceGuard guard(device);
    CU_CHECK(none, guard.err);
    cudaDeviceProp prop;
    CU_CHECK(none, cudaGetDeviceProperties(&prop, device));
    const int sms = prop.multiProcessorCount;
    CU_CHECK(none, cudaFuncSetAttribute(k_operand_stream, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        static_cast<int>(kStreamSmemBytes)));
    constexpr int kCols = 256;
    const int rows_of[2] = {2048, 65536};                // 2 MB that every SM re-reads; 64 MB
    float* d_src = nullptr;
    int* d_err = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaMalloc(&d_src, sizeof(float) * rows_of[1] * kCols) != cudaSuccess) return CUTOFF_ERR_NOMEM;
    int rc = CUTOFF_OK;
    if (cudaMalloc(&d_err, sizeof(int)) != cudaSuccess) rc = CUTOFF_ERR_NOMEM;
    if (rc == CUTOFF_OK && (cudaMemset(d_src, 0, sizeof(float) * rows_of[1] * kCols) != cudaSuccess ||
                            cudaMemset(d_err, 0, sizeof(int)) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
                            cudaEventCreate(&e1) != cudaSuccess))
        rc = CUTOFF_ERR_CUDA;
    for (int which = 0; which < 2 && rc == CUTOFF_OK; ++which) {
        CUtensorMap map;
        rc = make_tile_map(nullptr, &map, d_src, rows_of[which], kCols);
        if (rc != CUTOFF_OK) break;
        const int iters = static_cast<int>((4096ll << 20) / sms / kStreamStageBytes);    // 4 GB per launch in all
        float best = 0.0f;
        for (int rep = 0; rep < 3; ++rep) {              // the first repetition fills the L2 and warms the clocks up
            cudaEventRecord(e0);
            k_operand_stream<<<sms, 32, kStreamSmemBytes>>>(map, rows_of[which], kCols / 32, iters, d_err);
            cudaEventRecord(e1);
            float ms = 0.0f;
            if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess || ms <= 0.0f) {
                rc = CUTOFF_ERR_CUDA;
                break;
            }
            const float gbs = static_cast<float>(static_cast<double>(iters) * kStreamStageBytes * sms / (ms * 1e6));
            if (rep > 0 && gbs > best) best = gbs;
        }
        gbs_out[which] = best;
    }
    int h_err = 0;
    if (rc == CUTOFF_OK && cudaMemcpy(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) rc = CUTOFF_ERR_CUDA;
    if (rc == CUTOFF_OK && h_err) rc = CUTOFF_ERR_TIMEOUT;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(d_src);
    cudaFree(d_err);
    return rc;
}

int cutoff_reset(cutoff_ctx* c) {
    if (!c) return CUTOFF_ERR_BAD_ARG;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    CU_CHECK(c, cudaMemsetAsync(c->d_state, 0, sizeof(DevState), c->stream));
    CU_CHECK(c, cudaMemsetAsync(c->d_ring, 0, sizeof(float) * c->W * c->N, c->stream));
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    c->pushes = 0;
    c->pending = false;
    c->partial_pending = false;
    c->have_result = false;
    c->draws_valid = false;
    c->proj_stale = true;
    return CUTOFF_OK;
}

int cutoff_save_state(cutoff_ctx* c, void* buf, size_t* nbytes) {
    if (!c || !nbytes) return CUTOFF_ERR_BAD_ARG;
    const size_t need = 4 * sizeof(uint32_t) + sizeof(DevState) + sizeof(float) * c->W * c->N;
    if (!buf) { *nbytes = need; return CUTOFF_OK; }
    if (*nbytes < need) return CUTOFF_ERR_BAD_ARG;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    char* p = static_cast<char*>(buf);
    const uint32_t hdr[4] = {0x53465443u /* "CTFS" */, 1u, static_cast<uint32_t>(c->N), static_cast<uint32_t>(c->W)};
    std::memcpy(p, hdr, sizeof(hdr));
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    CU_CHECK(c, cudaMemcpy(p + sizeof(hdr), c->d_state, sizeof(DevState), cudaMemcpyDeviceToHost));
    CU_CHECK(c, cudaMemcpy(p + sizeof(hdr) + sizeof(DevState), c->d_ring, sizeof(float) * c->W * c->N,
                           cudaMemcpyDeviceToHost));
    *nbytes = need;
    return CUTOFF_OK;
}

int cutoff_restore_state(cutoff_ctx* c, const void* buf, size_t nbytes) {
    if (!c || !buf) return CUTOFF_ERR_BAD_ARG;
    const size_t need = 4 * sizeof(uint32_t) + sizeof(DevState) + sizeof(float) * c->W * c->N;
    if (nbytes != need) return CUTOFF_ERR_BAD_ARG;
    const char* p = static_cast<const char*>(buf);
    uint32_t hdr[4];
    std::memcpy(hdr, p, sizeof(hdr));
    if (hdr[0] != 0x53465443u || hdr[1] != 1u || hdr[2] != static_cast<uint32_t>(c->N) ||
        hdr[3] != static_cast<uint32_t>(c->W))
        return CUTOFF_ERR_BAD_ARG;
    DevState s;
    std::memcpy(&s, p + sizeof(hdr), sizeof(s));
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    CU_CHECK(c, upload(c, c->d_state, &s, sizeof(DevState)));
    CU_CHECK(c, upload(c, c->d_ring, p + sizeof(hdr) + sizeof(DevState), sizeof(float) * c->W * c->N));
    c->pushes = s.push_count;
    c->pending = false;
    c->partial_pending = false;
    c->have_result = false;
    c->draws_valid = false;            // the retained draws belong to a decision on the state that was replaced
    c->proj_stale = true;
    return CUTOFF_OK;
}

int cutoff_set_timing(cutoff_ctx* c, int on) {
    if (!c) return CUTOFF_ERR_BAD_ARG;
    if (on && (c->cfg.flags & CUTOFF_FLAG_GRAPH)) return CUTOFF_ERR_UNSUPPORTED;
    c->timing = on != 0;
    return CUTOFF_OK;
}

int cutoff_get_timing(cutoff_ctx* c, float* ms, int cap) {
    if (!c || !ms || cap < 0) return CUTOFF_ERR_BAD_ARG;
    for (int i = 0; i < kNumStages && i < cap; ++i) ms[i] = c->stage_ms[i];
    return kNumStages;
}

int64_t cutoff_launch_count(cutoff_ctx* c) { return c ? c->launches : 0; }

int cutoff_set_option(cutoff_ctx* c, const char* name, int64_t value) {
    if (!c || !name) return CUTOFF_ERR_BAD_ARG;
    if (c->pending) return CUTOFF_ERR_STATE;
    if (std::strcmp(name, "order_stat_std") == 0) {
        if (value != 0 && value != 1) return CUTOFF_ERR_BAD_ARG;
        if (value && c->cfg.total_samples > 0 && c->cfg.total_samples != c->S) return CUTOFF_ERR_UNSUPPORTED;
        if (c->graph_exec || c->graph_dev_exec) return CUTOFF_ERR_STATE;   // the captured graph has the other sort kernel in it
        if (value && c->N > 1024 && !c->d_sq_totals) {
            DeviceGuard guard(c->cfg.device);
            CU_CHECK(c, guard.err);
            const size_t ctas = static_cast<size_t>(c->sm_count) * bucket_wide_ctas(c->N);
            if (cudaMalloc(&c->d_sq_totals, sizeof(float) * ctas * 128 * keys_per_thread(c->N, 128)) != cudaSuccess) {
                cudaGetLastError();
                return CUTOFF_ERR_NOMEM;
            }
        }
        c->want_std = value != 0;
        return CUTOFF_OK;
    }
    if (std::strcmp(name, "pair_emission") == 0) {
        if (value != 0 && value != 1) return CUTOFF_ERR_BAD_ARG;
        if (value && (c->literal || !c->use_tc || c->pair_clusters == 0)) return CUTOFF_ERR_UNSUPPORTED;
        if (c->graph_exec || c->graph_dev_exec) return CUTOFF_ERR_STATE;   // the captured graph has the other kernel in it
        c->pair_emission = value != 0;
        return CUTOFF_OK;
    }
    if (std::strcmp(name, "pass_rows") == 0) {
        if (value < 1024 || value > 0x7fffffffll) return CUTOFF_ERR_BAD_ARG;
        if (c->graph_exec || c->graph_dev_exec) return CUTOFF_ERR_STATE;   // the captured graph replays the old split
        DeviceGuard guard(c->cfg.device);
        CU_CHECK(c, guard.err);
        plan_chunks(c, static_cast<int>(value));
        c->draws_valid = false;
        CU_CHECK(c, set_pass_attributes(c));
        return CUTOFF_OK;
    }
    return CUTOFF_ERR_BAD_ARG;
}

// ---- test hooks --------------------------------------------------------------------------------

namespace {
__global__ void k_debug_normals(uint32_t seed_lo, uint32_t seed_hi, uint32_t step, uint32_t stream, uint32_t k0,
                                int64_t count, int nq, int n_elems, float* __restrict__ normals,
                                uint32_t* __restrict__ words) {
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= count * nq) return;
    const int64_t k = idx / nq;
    const int q = static_cast<int>(idx % nq);
    const Philox4 r = philox4x32_10(q, k0 + static_cast<uint32_t>(k), stream, step, seed_lo, seed_hi);
    if (words) {
        uint32_t* w = words + idx * 4;
        w[0] = r.x; w[1] = r.y; w[2] = r.z; w[3] = r.w;
    }
    if (normals) {
        float e[4];
        box_muller(r.x, r.y, e[0], e[1]);
        box_muller(r.z, r.w, e[2], e[3]);
        for (int c = 0; c < 4; ++c)
            if (4 * q + c < n_elems) normals[k * n_elems + 4 * q + c] = e[c];
    }
}
}  // namespace

int cutoff_debug_normals(int device, uint64_t seed, uint32_t step, uint32_t stream, int64_t k0, int64_t count,
                         int32_t n_elems, float* normals_out, uint32_t* words_out) {
    if (device < 0 || k0 < 0 || count < 1 || n_elems < 1 || k0 + count > (1ll << 32)) return CUTOFF_ERR_BAD_ARG;
    if (!normals_out && !words_out) return CUTOFF_ERR_BAD_ARG;
    cutoff_ctx* none = nullptr;
    DeviceGuard guard(device);
    CU_CHECK(none, guard.err);
    const int nq = (n_elems + 3) / 4;
    float* d_n = nullptr;
    uint32_t* d_w = nullptr;
    int rc = CUTOFF_OK;
    if (normals_out && cudaMalloc(&d_n, sizeof(float) * count * n_elems) != cudaSuccess) rc = CUTOFF_ERR_NOMEM;
    if (!rc && words_out && cudaMalloc(&d_w, sizeof(uint32_t) * count * nq * 4) != cudaSuccess) rc = CUTOFF_ERR_NOMEM;
    if (!rc) {
        const int64_t threads = count * nq;
        k_debug_normals<<<static_cast<unsigned>(ceil_div64(threads, 256)), 256>>>(
            static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32), step, stream, static_cast<uint32_t>(k0),
            count, nq, n_elems, d_n, d_w);
        if (cudaDeviceSynchronize() != cudaSuccess) rc = CUTOFF_ERR_CUDA;
    }
    if (!rc && normals_out &&
        cudaMemcpy(normals_out, d_n, sizeof(float) * count * n_elems, cudaMemcpyDeviceToHost) != cudaSuccess)
        rc = CUTOFF_ERR_CUDA;
    if (!rc && words_out &&
        cudaMemcpy(words_out, d_w, sizeof(uint32_t) * count * nq * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
        rc = CUTOFF_ERR_CUDA;
    cudaFree(d_n);
    cudaFree(d_w);
    return rc;
}

int cutoff_debug_samples(cutoff_ctx* c, int64_t k0, int64_t count, float* x_out) {
    if (!c || !x_out || k0 < 0 || count < 1 || k0 + count > c->S) return CUTOFF_ERR_BAD_ARG;
    if (!c->weights_loaded || c->pending) return CUTOFF_ERR_STATE;
    if (c->pushes < static_cast<uint32_t>(c->W)) return CUTOFF_WARMUP;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    c->draws_valid = false;                                 // the sample matrix is about to be overwritten
    launch_encoder(c);
    for (int64_t done = 0; done < count; done += c->chunk_rows) {
        const int n = static_cast<int>(count - done < c->chunk_rows ? count - done : c->chunk_rows);
        const uint32_t base = static_cast<uint32_t>(c->cfg.sample_offset + k0 + done);
        CU_CHECK(c, set_call_attributes(c, n));
        launch_chain(c, base, n);
        launch_emission(c, base, n);
        CU_CHECK(c, cudaMemcpy2DAsync(x_out + done * c->N, sizeof(float) * c->N, c->d_x, sizeof(float) * c->ldx,
                                      sizeof(float) * c->N, n, cudaMemcpyDeviceToHost, c->stream));
        CU_CHECK(c, cudaStreamSynchronize(c->stream));
    }
    CU_CHECK(c, cudaGetLastError());
    return CUTOFF_OK;
}

int cutoff_debug_window(cutoff_ctx* c, float* window_out) {
    if (!c || !window_out) return CUTOFF_ERR_BAD_ARG;
    if (c->pending) return CUTOFF_ERR_STATE;
    if (c->pushes < static_cast<uint32_t>(c->W)) return CUTOFF_WARMUP;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    CU_CHECK(c, cudaStreamSynchronize(c->stream));
    for (int t = 0; t < c->W; ++t) {                       // position t (0 = oldest) sits in slot (pushes + t) mod W
        const size_t slot = (static_cast<size_t>(c->pushes) + t) % c->W;
        CU_CHECK(c, cudaMemcpy(window_out + static_cast<size_t>(t) * c->N, c->d_ring + slot * c->N, sizeof(float) * c->N,
                               cudaMemcpyDeviceToHost));
    }
    return CUTOFF_OK;
}

int cutoff_debug_sort(cutoff_ctx* c, const float* rows, int64_t n_rows, int32_t n, float* keys_out, int32_t* perm_out) {
    if (!c || !rows || !keys_out || !perm_out || n_rows < 1 || n < 1 || n > 4096 || n_rows > (1 << 24))
        return CUTOFF_ERR_BAD_ARG;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    const size_t elems = static_cast<size_t>(n_rows) * n;
    float *d_rows = nullptr, *d_keys = nullptr;
    int* d_perm = nullptr;
    int rc = CUTOFF_OK;
    if (cudaMalloc(&d_rows, elems * 4) != cudaSuccess || cudaMalloc(&d_keys, elems * 4) != cudaSuccess ||
        cudaMalloc(&d_perm, elems * 4) != cudaSuccess)
        rc = CUTOFF_ERR_NOMEM;
    if (!rc && cudaMemcpyAsync(d_rows, rows, elems * 4, cudaMemcpyHostToDevice, c->stream) != cudaSuccess)
        rc = CUTOFF_ERR_CUDA;
    if (!rc) {
        const int P = next_pow2(n) < 32 ? 32 : next_pow2(n);
        const int rows_i = static_cast<int>(n_rows);
        const int grid_w = ceil_div(rows_i, kSortWarps) < 4 * c->sm_count ? ceil_div(rows_i, kSortWarps) : 4 * c->sm_count;
        const int grid_c = rows_i < 4 * c->sm_count ? rows_i : 4 * c->sm_count;
        switch (P) {
            case 32: k_debug_sort_warp<1><<<grid_w, kSortWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm); break;
            case 64: k_debug_sort_warp<2><<<grid_w, kSortWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm); break;
            case 128: k_debug_sort_warp<4><<<grid_w, kSortWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm); break;
            case 256: k_debug_sort_warp<8><<<grid_w, kSortWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm); break;
            case 512: k_debug_sort_warp<16><<<grid_w, kSortWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm); break;
            case 1024: k_debug_sort_warp<32><<<grid_w, kSortWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm); break;
            case 2048: k_debug_sort_cta<2><<<grid_c, 64, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm); break;
            default: k_debug_sort_cta<4><<<grid_c, 128, 0, c->stream>>>(d_rows, n, rows_i, d_keys, d_perm);
        }
        c->launches += 1;
        if (cudaMemcpyAsync(keys_out, d_keys, elems * 4, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
            cudaMemcpyAsync(perm_out, d_perm, elems * 4, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
            cudaStreamSynchronize(c->stream) != cudaSuccess)
            rc = CUTOFF_ERR_CUDA;
    }
    if (rc == CUTOFF_ERR_CUDA) c->last_error = cudaGetErrorString(cudaGetLastError());
    cudaFree(d_rows); cudaFree(d_keys); cudaFree(d_perm);
    return rc;
}

int cutoff_debug_sort_values(cutoff_ctx* c, const float* rows, int64_t n_rows, int32_t n, float* keys_out) {
    if (!c || !rows || !keys_out || n_rows < 1 || n < 1 || n > 4096 || n_rows > (1 << 24)) return CUTOFF_ERR_BAD_ARG;
    DeviceGuard guard(c->cfg.device);
    CU_CHECK(c, guard.err);
    const size_t elems = static_cast<size_t>(n_rows) * n;
    float *d_rows = nullptr, *d_keys = nullptr;
    int rc = CUTOFF_OK;
    if (cudaMalloc(&d_rows, elems * 4) != cudaSuccess || cudaMalloc(&d_keys, elems * 4) != cudaSuccess) rc = CUTOFF_ERR_NOMEM;
    if (!rc && cudaMemcpyAsync(d_rows, rows, elems * 4, cudaMemcpyHostToDevice, c->stream) != cudaSuccess) rc = CUTOFF_ERR_CUDA;
    if (!rc) {
        const int rows_i = static_cast<int>(n_rows);
        const auto grid = [&](int rows_per_cta) { return std::min(ceil_div(rows_i, rows_per_cta), 4 * c->sm_count); };
        const auto network = [&](auto* kernel) { kernel<<<grid(kSortWarps), kSortWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys); };
        const auto warps = [&](auto* kernel) { kernel<<<grid(8 * kDebugBucketWarps), kDebugBucketWarps * 32, 0, c->stream>>>(d_rows, n, rows_i, d_keys); };
        const auto ctas = [&](auto* kernel) { kernel<<<grid(8), 128, 0, c->stream>>>(d_rows, n, rows_i, d_keys); };
        if (n > 1024) {
            switch (keys_per_thread(n, 128)) {
                case 12: ctas(k_debug_bucket_cta<12>); break;
                case 16: ctas(k_debug_bucket_cta<16>); break;
                case 20: ctas(k_debug_bucket_cta<20>); break;
                case 24: ctas(k_debug_bucket_cta<24>); break;
                case 28: ctas(k_debug_bucket_cta<28>); break;
                default: ctas(k_debug_bucket_cta<32>); break;
            }
        } else if (by_buckets(n, n_rows)) {
            switch (keys_per_thread(n, 32)) {
                case 8: warps(k_debug_bucket_warp<8>); break;
                case 12: warps(k_debug_bucket_warp<12>); break;
                case 16: warps(k_debug_bucket_warp<16>); break;
                case 20: warps(k_debug_bucket_warp<20>); break;
                case 24: warps(k_debug_bucket_warp<24>); break;
                case 28: warps(k_debug_bucket_warp<28>); break;
                default: warps(k_debug_bucket_warp<32>); break;
            }
        } else {
            switch (n <= 32 ? 32 : next_pow2(n)) {
                case 32: network(k_debug_sort_values_warp<1>); break;
                case 64: network(k_debug_sort_values_warp<2>); break;
                case 128: network(k_debug_sort_values_warp<4>); break;
                default: network(k_debug_sort_values_warp<8>); break;
            }
        }
        c->launches += 1;
        if (cudaMemcpyAsync(keys_out, d_keys, elems * 4, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
            cudaStreamSynchronize(c->stream) != cudaSuccess)
            rc = CUTOFF_ERR_CUDA;
    }
    if (rc == CUTOFF_ERR_CUDA) c->last_error = cudaGetErrorString(cudaGetLastError());
    cudaFree(d_rows); cudaFree(d_keys);
    return rc;
}

// Device memory for the duration of one call that has no context: taken from and returned to a memory pool of the
// library's own, in the order of the call's stream, so calls on other threads and streams do not meet in it.  The pool keeps at
// most kPoolKeeps bytes between calls, until the process ends (what exceeds that goes back to the driver at the next
// synchronisation): cudaMalloc and cudaFree took 1 to 10 ms per call, the kernels 60 us.
namespace {
constexpr uint64_t kPoolKeeps = 64ull << 20;
constexpr int kPoolDevices = 64;

cudaMemPool_t scratch_pool(int device) {
    static std::mutex lock;
    static cudaMemPool_t pools[kPoolDevices] = {};
    if (device < 0 || device >= kPoolDevices) return nullptr;
    std::lock_guard<std::mutex> hold(lock);
    if (!pools[device]) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        uint64_t keep = kPoolKeeps;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        pools[device] = pool;
    }
    return pools[device];
}

struct Scratch {
    void* p = nullptr;
    cudaStream_t stream;
    Scratch(int device, cudaStream_t s, size_t bytes) : stream(s) {
        cudaMemPool_t pool = bytes ? scratch_pool(device) : nullptr;
        if (pool && cudaMallocFromPoolAsync(&p, bytes, pool, s) != cudaSuccess) { cudaGetLastError(); p = nullptr; }
    }
    ~Scratch() { if (p) cudaFreeAsync(p, stream); }
    Scratch(const Scratch&) = delete;
    Scratch& operator=(const Scratch&) = delete;
};
}  // namespace

// ---- evaluation of cutoff rules on recorded run-times ------------------------------------------------------

int cutoff_eval_trace(int device, const float* trace, int64_t n_steps, int32_t n, int32_t ld, const int32_t* cutoffs,
                      int32_t n_rules, int32_t* best_c, float* best, float* all, float* achieved, float* step_time,
                      int32_t* static_c, void* stream) {
    if (device < 0 || !trace || n_steps < 1 || n_steps > (1ll << 31) - 1 || n < 1 || n > 4096 || ld < n || n_rules < 0 ||
        !best_c || !best || !all || (n_rules > 0 && (!cutoffs || !achieved || !step_time)))
        return CUTOFF_ERR_BAD_ARG;
    cutoff_ctx* none = nullptr;
    DeviceGuard guard(device);
    CU_CHECK(none, guard.err);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int sms = 0;
    CU_CHECK(none, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    // scratch only for the static cutoff: the sorted rows and the columns' totals
    Scratch scratch(device, s, static_c ? sizeof(double) * n + sizeof(float) * static_cast<size_t>(n_steps) * n : 0);
    if (static_c && !scratch.p) return CUTOFF_ERR_NOMEM;
    double* d_totals = static_cast<double*>(scratch.p);
    float* d_sorted = static_c ? reinterpret_cast<float*>(d_totals + n) : nullptr;
    const int P = next_pow2(n) < 32 ? 32 : next_pow2(n);
    const int cap = 8 * sms;
    const int64_t want_w = ceil_div64(n_steps, kEvalWarps);
    const int grid_w = static_cast<int>(want_w < 2 * cap ? want_w : 2 * cap);
    const int grid_c = static_cast<int>(n_steps < cap ? n_steps : cap);
#define EVAL_ARGS trace, n_steps, n, ld, cutoffs, n_rules, best_c, best, all, achieved, step_time, d_sorted
    switch (P) {
        case 32: k_eval_trace_warp<1><<<grid_w, kEvalWarps * 32, 0, s>>>(EVAL_ARGS); break;
        case 64: k_eval_trace_warp<2><<<grid_w, kEvalWarps * 32, 0, s>>>(EVAL_ARGS); break;
        case 128: k_eval_trace_warp<4><<<grid_w, kEvalWarps * 32, 0, s>>>(EVAL_ARGS); break;
        case 256: k_eval_trace_warp<8><<<grid_w, kEvalWarps * 32, 0, s>>>(EVAL_ARGS); break;
        case 512: k_eval_trace_warp<16><<<grid_w, kEvalWarps * 32, 0, s>>>(EVAL_ARGS); break;
        case 1024: k_eval_trace_warp<32><<<grid_w, kEvalWarps * 32, 0, s>>>(EVAL_ARGS); break;
        case 2048: k_eval_trace_cta<2><<<grid_c, 64, 0, s>>>(EVAL_ARGS); break;
        default: k_eval_trace_cta<4><<<grid_c, 128, 0, s>>>(EVAL_ARGS); break;
    }
#undef EVAL_ARGS
    if (static_c) {
        launch_dependent(k_static_totals, dim3(ceil_div(n, 32)), dim3(32 * kStaticSlices), 0, s, d_sorted, n_steps, n, d_totals);
        launch_dependent(k_best_static, dim3(1), dim3(1024), 0, s, d_totals, n, static_c);
    }
    const cudaError_t launched = cudaGetLastError();
    const cudaError_t err = cudaStreamSynchronize(s);
    return err == cudaSuccess && launched == cudaSuccess ? CUTOFF_OK : CUTOFF_ERR_CUDA;
}

int cutoff_order_baseline(int device, const float* trace, int64_t n_steps, int32_t n, int32_t ld, int32_t* cutoffs_out,
                          void* stream) {
    if (device < 0 || !trace || n_steps < 1 || n_steps > (1ll << 31) - 1 || n < 1 || ld < n || !cutoffs_out)
        return CUTOFF_ERR_BAD_ARG;
    cutoff_ctx* none = nullptr;
    DeviceGuard guard(device);
    CU_CHECK(none, guard.err);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // [T] sums / means, [T] sums of squares / deviations, [n] normal quantiles
    Scratch scratch(device, s, sizeof(double) * (2 * static_cast<size_t>(n_steps) + n));
    if (!scratch.p) return CUTOFF_ERR_NOMEM;
    double* d1 = static_cast<double*>(scratch.p);
    double* d2 = d1 + n_steps;
    double* dq = d1 + 2 * n_steps;
    const unsigned step_ctas = static_cast<unsigned>(ceil_div64(n_steps, kMomentWarps));
    k_step_moments<<<step_ctas + ceil_div(n, kMomentWarps * 32), kMomentWarps * 32, 0, s>>>(trace, n_steps, n, ld, d1, d2, dq, step_ctas);
    launch_dependent(k_running_moments, dim3(1), dim3(1024), 0, s, n_steps, n, d1, d2);
    launch_dependent(k_order_cutoffs, dim3(static_cast<unsigned>(ceil_div64(n_steps, 8))), dim3(256), 0, s, n_steps, n, d1, d2, dq, cutoffs_out);
    const cudaError_t launched = cudaGetLastError();
    const cudaError_t err = cudaStreamSynchronize(s);
    return err == cudaSuccess && launched == cudaSuccess ? CUTOFF_OK : CUTOFF_ERR_CUDA;
}

// ---- learning the model: ELBO, gradient, Adam -------------------------------------------------------------------

int64_t cutoff_fit_param_count(int32_t n_workers, int32_t latent_dim, int32_t hidden) {
    if (n_workers < 1 || latent_dim < 1 || hidden < 1) return 0;
    return fit::layout(n_workers, latent_dim, hidden).off[fit::kTensors];
}

int64_t cutoff_fit_workspace_bytes(int32_t n_workers, int32_t latent_dim, int32_t hidden, int32_t lag, int32_t batch) {
    if (n_workers < 1 || latent_dim < 1 || hidden < 1 || lag < 0 || batch < 1) return 0;
    return static_cast<int64_t>(sizeof(float)) * fit::workspace_floats(n_workers, latent_dim, hidden, lag + 1, batch);
}

int cutoff_elbo_grad(int device, int32_t n_workers, int32_t latent_dim, int32_t hidden, int32_t lag, int32_t batch,
                     const float* params, const float* xhat, const float* eps, float* elbo, float* grads, void* workspace,
                     size_t workspace_bytes, void* stream) {
    if (device < 0 || n_workers < 1 || n_workers > 4096 || latent_dim < 1 || latent_dim > 64 || hidden < 1 || hidden > 1024 ||
        lag < 0 || lag > 255 || batch < 1 || batch > 65535 || !params || !xhat || !eps || !elbo || !workspace)
        return CUTOFF_ERR_BAD_ARG;
    if (workspace_bytes < static_cast<size_t>(cutoff_fit_workspace_bytes(n_workers, latent_dim, hidden, lag, batch)))
        return CUTOFF_ERR_BAD_ARG;
    cutoff_ctx* none = nullptr;
    DeviceGuard guard(device);
    CU_CHECK(none, guard.err);
    fit::elbo_grad(n_workers, latent_dim, hidden, lag + 1, batch, params, xhat, eps, elbo, grads,
                   static_cast<float*>(workspace), static_cast<cudaStream_t>(stream));
    return cudaGetLastError() == cudaSuccess ? CUTOFF_OK : CUTOFF_ERR_CUDA;
}

int cutoff_adam_step(int device, int64_t n, float* params, const float* grads, float* m, float* v, int32_t t, float lr,
                     float beta1, float beta2, float eps, float clip_norm, float grad_scale, float* norm_out, void* workspace,
                     size_t workspace_bytes, void* stream) {
    if (device < 0 || n < 1 || !params || !grads || !m || !v || t < 1 || !(lr > 0.f) || !(beta1 >= 0.f && beta1 < 1.f) ||
        !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f) || !(clip_norm > 0.f) || !norm_out || !workspace ||
        workspace_bytes < fit::kNormParts * sizeof(double))
        return CUTOFF_ERR_BAD_ARG;
    cutoff_ctx* none = nullptr;
    DeviceGuard guard(device);
    CU_CHECK(none, guard.err);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    double* partial = static_cast<double*>(workspace);
    const int64_t want = (n + fit::kNormThreads - 1) / fit::kNormThreads;
    const int parts = static_cast<int>(want < fit::kNormParts ? want : fit::kNormParts);
    fit::k_sumsq_partial<<<parts, fit::kNormThreads, 0, s>>>(grads, n, grad_scale, partial);
    const float corr1 = 1.f - std::pow(beta1, static_cast<float>(t)), corr2 = 1.f - std::pow(beta2, static_cast<float>(t));
    const int64_t most = 8 * 148;                     // a few CTAs per SM: each adds the partial sums up first
    fit::k_adam<<<static_cast<unsigned>(want < most ? want : most), fit::kNormThreads, 0, s>>>(
        params, grads, m, v, n, grad_scale, partial, parts, norm_out, clip_norm, lr, beta1, beta2, eps, corr1, corr2);
    return cudaGetLastError() == cudaSuccess ? CUTOFF_OK : CUTOFF_ERR_CUDA;
}

}  // extern "C"

// ---- allocation-free entry point -------------------------------------------------------------

namespace {
constexpr int kStaticParts = 256;     // partial rows (= most CTAs the sort kernel may use here)
constexpr int kStaticRowsPerWarp = 64;                                                  // rows a warp adds in fp32
constexpr int64_t kStaticBlockRows = static_cast<int64_t>(kStaticParts) * kSortWarps * kStaticRowsPerWarp;   // 131072
static_assert(kStaticParts * CUTOFF_STATIC_MAX_N * sizeof(float) == CUTOFF_STATIC_SCRATCH_BYTES, "scratch size");

// Scratch of cutoff_sorted_row_sums_static: one partial sum row per CTA.  Lives in the library
// image, one copy per GPU.  In host code this name is only a handle for cudaGetSymbolAddress;
// the kernels get the device address found at set-up.
static __device__ __align__(256) float g_static_partial[kStaticParts * CUTOFF_STATIC_MAX_N];

constexpr int kMaxDevices = 64;
float* g_static_partial_addr[kMaxDevices] = {};   // device address per GPU, filled on first use
int g_static_sms[kMaxDevices] = {};               // its SMs

// Returns the number of partial rows (CTAs).
template <int E>
int launch_static_network(const float* x, int ldx, int n, int n_rows, float* partial, cudaStream_t stream) {
    const int want = ceil_div(n_rows, kSortWarps), grid = want < kStaticParts ? want : kStaticParts;
    k_sort_sum_warp<E><<<grid, kSortWarps * 32, 0, stream>>>(x, ldx, n, n_rows, partial);
    return grid;
}

// Rows that all start on 16 bytes come in as 16-byte chunks, others word by word (700 keys x 32768 rows: 63 against 65 us).
template <int E>
int launch_static_bucket(const float* x, int ldx, int n, int n_rows, float* partial, cudaStream_t stream, int sms) {
    const int most = sms < kStaticParts ? sms : kStaticParts, grid = n_rows < most ? n_rows : most;
    const size_t smem = bucket_smem_bytes<E>();
    DevState* const none = nullptr;
    const bool chunks = (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && ldx % 4 == 0;
    if (chunks) k_bucket_sum_warp<E, false, 16><<<grid, kBucketWarps<E> * 32, smem, stream>>>(x, ldx, n, n_rows, partial, nullptr, none);
    else k_bucket_sum_warp<E, false, 4><<<grid, kBucketWarps<E> * 32, smem, stream>>>(x, ldx, n, n_rows, partial, nullptr, none);
    return grid;
}

template <int E>
cudaError_t allow_smem_static() {
    cudaError_t e = allow_smem(k_bucket_sum_warp<E, false, 16>, bucket_smem_bytes<E>());
    if (e == cudaSuccess) e = allow_smem(k_bucket_sum_warp<E, false, 4>, bucket_smem_bytes<E>());
    return e;
}
cudaError_t allow_smem_static_all() {
    cudaError_t e = allow_smem_static<8>();
    if (e == cudaSuccess) e = allow_smem_static<12>();
    if (e == cudaSuccess) e = allow_smem_static<16>();
    if (e == cudaSuccess) e = allow_smem_static<20>();
    if (e == cudaSuccess) e = allow_smem_static<24>();
    if (e == cudaSuccess) e = allow_smem_static<28>();
    if (e == cudaSuccess) e = allow_smem_static<32>();
    return e;
}
}  // namespace

extern "C" int cutoff_sorted_row_sums_static(int device, const float* x, int64_t n_rows, int32_t n, int32_t ldx,
                                             double* sums, void* stream) {
    if (device < 0 || device >= kMaxDevices || !x || !sums || n_rows < 1 || n_rows > CUTOFF_STATIC_MAX_ROWS || n < 1 ||
        ldx < n)
        return CUTOFF_ERR_BAD_ARG;
    if (n > CUTOFF_STATIC_MAX_N) return CUTOFF_ERR_TOO_LARGE;
    DeviceGuard guard(device);
    if (guard.err != cudaSuccess) return CUTOFF_ERR_CUDA;
    if (!g_static_partial_addr[device]) {
        // once per device, with that device current: translate the symbol into a device address, let the kernels
        // have the shared memory they need
        float* addr = nullptr;
        if (cudaGetSymbolAddress(reinterpret_cast<void**>(&addr), g_static_partial) != cudaSuccess || !addr)
            return CUTOFF_ERR_CUDA;
        if (allow_smem_static_all() != cudaSuccess ||
            cudaDeviceGetAttribute(&g_static_sms[device], cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
            return CUTOFF_ERR_CUDA;
        g_static_partial_addr[device] = addr;
    }
    float* partial = g_static_partial_addr[device];
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int P = next_pow2(n) < 32 ? 32 : next_pow2(n);
    // The rows go through in blocks: within a block a warp adds at most kStaticRowsPerWarp sorted rows in fp32 (the bucket sort has a
    // CTA per SM, so its blocks are shorter on a GPU of less than 128 SMs), then the block's partial rows are added to `sums`
    // in double.  The blocks run one after the other on the stream, so they can share the scratch array.
    const int sms = g_static_sms[device];
    const int64_t bucket_rows = static_cast<int64_t>(kStaticRowsPerWarp) * kBucketFewestWarps * (sms < kStaticParts ? sms : kStaticParts);
    const int64_t block_rows = n > 128 && bucket_rows < kStaticBlockRows ? bucket_rows : kStaticBlockRows;
    for (int64_t r0 = 0; r0 < n_rows; r0 += block_rows) {
        const int rows = static_cast<int>(n_rows - r0 < block_rows ? n_rows - r0 : block_rows);
        const float* xb = x + static_cast<size_t>(r0) * ldx;
        // every CTA of the grid writes its whole partial row (zeros if it had no sample), and the
        // column sum reads exactly `grid` rows: stale contents of the shared array are never read
        int grid = 0;
        if (by_buckets(n, rows)) {
            switch (keys_per_thread(n, 32)) {
                case 8: grid = launch_static_bucket<8>(xb, ldx, n, rows, partial, s, sms); break;
                case 12: grid = launch_static_bucket<12>(xb, ldx, n, rows, partial, s, sms); break;
                case 16: grid = launch_static_bucket<16>(xb, ldx, n, rows, partial, s, sms); break;
                case 20: grid = launch_static_bucket<20>(xb, ldx, n, rows, partial, s, sms); break;
                case 24: grid = launch_static_bucket<24>(xb, ldx, n, rows, partial, s, sms); break;
                case 28: grid = launch_static_bucket<28>(xb, ldx, n, rows, partial, s, sms); break;
                default: grid = launch_static_bucket<32>(xb, ldx, n, rows, partial, s, sms); break;
            }
        } else {
            switch (P) {
                case 32: grid = launch_static_network<1>(xb, ldx, n, rows, partial, s); break;
                case 64: grid = launch_static_network<2>(xb, ldx, n, rows, partial, s); break;
                case 128: grid = launch_static_network<4>(xb, ldx, n, rows, partial, s); break;
                default: grid = launch_static_network<8>(xb, ldx, n, rows, partial, s); break;
            }
        }
        launch_dependent(k_colsum, dim3(ceil_div(n, 32)), dim3(32 * kPlainSlices), 0, s, partial, grid, n, sums, r0 > 0 ? 1 : 0);
    }
    return cudaGetLastError() == cudaSuccess ? CUTOFF_OK : CUTOFF_ERR_CUDA;
}
