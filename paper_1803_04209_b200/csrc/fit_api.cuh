// Host side of the learning entry points (see include/cutoff.h): lays the forward and backward pass of fit.cuh out
// as launches on one stream.  The parameter vector is the weight blob's tensors, in its order, without the header.
#pragma once
#include "fit.cuh"

namespace cutoff {
namespace fit {

enum { iWxf, iWhf, ibf, ia0, iWxb, iWhb, ibb, ib0, iWz, ibz, iWmu, ibmu, iWsig, ibsig, iz0, iW1, ib1, iW2, ib2, iW3, ib3, iW4, ib4, kTensors };

struct Layout {
    long long off[kTensors + 1];
};

inline Layout layout(long long N, long long D, long long H) {
    const long long size[kTensors] = {H * N, H * H, H, H, H * N, H * H, H, H, H * D, H, D * H, D, D * D, D, D,
                                      H * D, H, 2 * D * H, 2 * D, H * D, H, 2 * N * H, 2 * N};
    Layout l;
    l.off[0] = 0;
    for (int i = 0; i < kTensors; ++i) l.off[i + 1] = l.off[i] + size[i];
    return l;
}

inline long long tiles_of(long long n, int tile) { return (n + tile - 1) / tile; }

// Everything the passes keep, as offsets (floats, multiples of 4) into the workspace.
struct Workspace {
    long long proj, a, b, comb, hout, mu, presig, z, u, v, dhz, dzt, path, dhx, part, dv_raw, dv, du, dpc, dh, dmu, dps, gz0,
        dpf, dpb, ca, cb, total;
};

inline Workspace workspace(long long N, long long D, long long H, long long W, long long B) {
    const long long R = B * W, rh = R * H, rd = R * D, sh = B * (W + 1) * H, sd = B * (W + 1) * D;
    Workspace w;
    long long o = 0;
    const auto take = [&](long long n) { const long long r = o; o += (n + 3) / 4 * 4; return r; };
    w.proj = take(2 * rh);
    w.a = take(sh); w.b = take(sh);
    w.comb = take(rh); w.hout = take(rh); w.mu = take(rd); w.presig = take(rd); w.z = take(sd); w.u = take(rh); w.v = take(rh);
    w.dhz = take(2 * rd); w.dzt = take(rd); w.path = take(B);
    w.dhx = take(R * 2 * N);
    w.part = take(tiles_of(N, kHeadWorkers) * R);
    w.dv_raw = take(rh);
    w.dv = take(rh); w.du = take(rh); w.dpc = take(rh); w.dh = take(rh); w.dmu = take(rd); w.dps = take(rd); w.gz0 = take(B * D);
    w.dpf = take(rh); w.dpb = take(rh); w.ca = take(B * H); w.cb = take(B * H);
    w.total = o;
    return w;
}

inline long long workspace_floats(long long N, long long D, long long H, long long W, long long B) { return workspace(N, D, H, W, B).total; }

// A kernel that may begin while the one before it is still running (it waits by itself before it touches its results).
template <typename... KArgs, typename... Args>
inline void launch(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t s, bool dependent, int cluster, Args... args) {
    if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (dependent) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename T>
struct ProductBuilder {
    ProductList list{};
    int tiles = 0;
    ProductBuilder() { list.n = 0; }
    void add(const Operand& a, const Operand& b, float* c, long long ldc, float* a_sums, int K, int n_seg = 1) {
        Product& p = list.p[list.n++];
        p.a = a; p.b = b; p.c = c; p.ldc = ldc; p.a_sums = a_sums; p.K = K; p.n_seg = n_seg;
        p.tile0 = tiles;
        p.tiles_n = b.rows > 0 ? static_cast<int>(tiles_of(b.rows, T::TN)) : 1;
        tiles += static_cast<int>(tiles_of(a.rows, T::TM)) * p.tiles_n;
    }
    template <bool AK, bool BK, bool SEG>
    void run(bool vec, cudaStream_t s, bool dependent) {
        if (vec) launch(k_products<T, AK, BK, true, SEG>, dim3(tiles), T::kThreads, 0, s, dependent, 1, list);
        else launch(k_products<T, AK, BK, false, SEG>, dim3(tiles), T::kThreads, 0, s, dependent, 1, list);
    }
};

// 64 x 64 tiles only where they fill the GPU: below that the small ones finish earlier.
constexpr int kFillTiles = 148, kManyTiles = 4 * kFillTiles;

// One product per direction of a dense layer over all rows: C[a.rows][b.rows] = A B with B k-major (X W^T) or m-major (dY W).
template <typename T, bool BK>
inline void run_rows_product(const Operand& a, const Operand* b, float* const* c, long long ldc, int n, int K, bool vec, cudaStream_t s, bool dependent) {
    ProductBuilder<T> q;
    for (int i = 0; i < n; ++i) q.add(a, b[i], c[i], ldc, nullptr, K);
    q.template run<true, BK, false>(vec, s, dependent);
}
template <bool BK>
inline void rows_product(const Operand& a, const Operand* b, float* const* c, long long ldc, int n, int K, bool vec, cudaStream_t s, bool dependent) {
    if (n * tiles_of(a.rows, LargeTile::TM) * tiles_of(b[0].rows, LargeTile::TN) >= kFillTiles)
        run_rows_product<LargeTile, BK>(a, b, c, ldc, n, K, vec, s, dependent);
    else
        run_rows_product<SmallTile, BK>(a, b, c, ldc, n, K, vec, s, dependent);
}

// How a recurrence is laid out: the fewest CTAs per cluster whose shares of the matrix fit, or eight and the matrix in chunks;
// two windows per cluster if the clusters then still fit the GPU at once, else four.
struct RnnPlan {
    int rw, cluster, units, chunk, threads;
    size_t smem;
    dim3 grid;
};
inline RnnPlan rnn_plan(int B, int H) {
    constexpr size_t kMost = 200 * 1024;
    RnnPlan p;
    p.cluster = 1;
    while (p.cluster < 8 && rnn_smem_bytes(H, (H + p.cluster - 1) / p.cluster, H, 4) > kMost) p.cluster *= 2;
    p.units = (H + p.cluster - 1) / p.cluster;
    p.chunk = rnn_smem_bytes(H, p.units, H, 4) <= kMost ? H : 128;
    p.rw = (B + 1) / 2 * 2 * p.cluster <= 148 ? 2 : 4;
    p.threads = (p.units + 31) / 32 * 32;                    // at most 224: a matrix of more units does not fit one CTA
    p.smem = rnn_smem_bytes(H, p.units, p.chunk, p.rw);
    p.grid = dim3((B + p.rw - 1) / p.rw * p.cluster, 2);
    return p;
}

// Whether the forward recurrence runs as products over all windows, a launch per step (k_rnn_step), instead: where the clusters
// would take several turns on the GPU.  Forward passes of five steps, N=64, D=4, clusters and products: H=192 1024 windows 226 and
// 225 us, 4096 744 and 537; H=256 256 windows 176 and 204, 512 250 and 225; H=512 64 windows 302 and 306, 256 698 and 328; H=1024 16
// windows 483 and 493, 64 776 and 532, 1024 6038 and 2387; H=128 4096 windows 369 and 382.
inline bool rnn_by_steps(int B, int H) { return H >= 192 && static_cast<long long>(B) * H * H > 40 << 20; }

// Enqueue forward (+ backward if grads) on `stream`.  All pointers are device pointers.
inline void elbo_grad(int N, int D, int H, int W, int B, const float* p, const float* xhat, const float* eps, float* elbo,
                      float* grads, float* ws, cudaStream_t stream) {
    const Layout L = layout(N, D, H);
    const Workspace o = workspace(N, D, H, W, B);
    const auto w = [&](int i) { return p + L.off[i]; };
    const auto g = [&](int i) { return grads + L.off[i]; };
    const int R = B * W;
    const bool back = grads != nullptr;
    const auto aligned = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    // 16-byte loads: every tensor and every row then starts on 16 bytes
    const bool vec = N % 4 == 0 && D % 4 == 0 && H % 4 == 0 && aligned(p) && aligned(xhat) && aligned(ws);

    // ---- forward -------------------------------------------------------------------------------------------------
    {
        const Operand b[2] = {Operand{w(iWxf), N, 0, H}, Operand{w(iWxb), N, 0, H}};     // input projections of both RNNs
        float* const c[2] = {ws + o.proj, ws + o.proj + H};
        rows_product<true>(Operand{xhat, N, 0, R}, b, c, 2 * H, 2, N, vec, stream, false);
    }
    RnnArgs r{};
    r.proj = ws + o.proj;
    r.Wh[0] = w(iWhf); r.Wh[1] = w(iWhb); r.bias[0] = w(ibf); r.bias[1] = w(ibb); r.init[0] = w(ia0); r.init[1] = w(ib0);
    r.state[0] = ws + o.a; r.state[1] = ws + o.b; r.g = ws + o.dh;
    r.d_pre[0] = ws + o.dpf; r.d_pre[1] = ws + o.dpb; r.carry_out[0] = ws + o.ca; r.carry_out[1] = ws + o.cb;
    const RnnPlan rp = rnn_plan(B, H);
    r.B = B; r.W = W; r.H = H; r.cluster = rp.cluster; r.units = rp.units; r.chunk = rp.chunk;
    if (rnn_by_steps(B, H)) {
        const dim3 grid(static_cast<unsigned>(tiles_of(B, LargeTile::TM) * tiles_of(H, LargeTile::TN)), 2);
        for (int s = 0; s < W; ++s)
            launch(vec ? k_rnn_step<LargeTile, true> : k_rnn_step<LargeTile, false>, grid, LargeTile::kThreads, 0, stream, true, 1, r, s);
    } else {
        launch(rp.rw == 2 ? k_rnn_forward<2> : k_rnn_forward<4>, rp.grid, rp.threads, rp.smem, stream, true, rp.cluster, r);
    }
    PathArgs a{};
    a.Wz = w(iWz); a.bz = w(ibz); a.Wmu = w(iWmu); a.bmu = w(ibmu); a.Wsig = w(iWsig); a.bsig = w(ibsig); a.z0 = w(iz0);
    a.W1 = w(iW1); a.b1 = w(ib1); a.W2 = w(iW2); a.b2 = w(ib2); a.W3 = w(iW3); a.b3 = w(ib3);
    a.a = ws + o.a; a.b = ws + o.b; a.eps = eps;
    a.comb = ws + o.comb; a.hout = ws + o.hout; a.mu = ws + o.mu; a.presig = ws + o.presig; a.z = ws + o.z; a.u = ws + o.u;
    a.v = ws + o.v; a.dhz = ws + o.dhz; a.dzt = ws + o.dzt; a.path = ws + o.path;
    const int head_tiles = static_cast<int>(tiles_of(N, kHeadWorkers));
    a.part = ws + o.part; a.n_part = head_tiles; a.elbo = elbo; a.dv_raw = ws + o.dv_raw;
    a.dv = ws + o.dv; a.du = ws + o.du; a.dpc = ws + o.dpc; a.dh = ws + o.dh; a.dmu = ws + o.dmu; a.dps = ws + o.dps;
    a.gz0 = ws + o.gz0; a.B = B; a.W = W; a.D = D; a.H = H;
    const size_t path_scratch = path_scratch_floats(D, H) * sizeof(float);
    const size_t path_full = path_scratch + path_weight_floats(D, H) * sizeof(float);
    const bool staged = path_full <= 200 * 1024;
    const size_t path_smem = staged ? path_full : path_scratch;
    if (staged) launch(k_path_forward<true>, dim3(B), kPathThreads, path_full, stream, true, 1, a);
    else launch(k_path_forward<false>, dim3(B), kPathThreads, path_scratch + kPathBuffer * sizeof(float), stream, true, 1, a);
    {
        float* dhx = back ? ws + o.dhx : nullptr;
        const auto run = [&](auto tile) {
            using T = decltype(tile);
            launch(vec ? k_emission_density<T, true> : k_emission_density<T, false>, dim3(static_cast<unsigned>(head_tiles * tiles_of(R, T::TM))),
                   T::kThreads, 0, stream, true, 1, ws + o.v, w(iW4), w(ib4), xhat, R, N, H, dhx, ws + o.part);
        };
        if (head_tiles * tiles_of(R, LargeTile::TM) >= kManyTiles) run(LargeTile{});
        else run(MediumTile{});
    }
    if (!back) {
        launch(k_elbo_finish, dim3((B + 3) / 4), 128, 0, stream, true, 1, ws + o.part, head_tiles, R, W, B, ws + o.path, elbo);
        return;
    }
    // ---- backward ------------------------------------------------------------------------------------------------
    {
        const Operand b{w(iW4), H, 0, H};                     // d v = d_head W4
        float* const c = ws + o.dv_raw;
        rows_product<false>(Operand{ws + o.dhx, 2ll * N, 0, R}, &b, &c, H, 1, 2 * N, vec, stream, true);
    }
    launch(k_path_backward, dim3(B), kPathThreads, path_smem, stream, true, 1, a, staged);
    launch(rp.rw == 2 ? k_rnn_backward<2> : k_rnn_backward<4>, rp.grid, rp.threads, rp.smem, stream, true, rp.cluster, r);
    {
        // every weight gradient d W = d_out^T in, one segment of B rows per step, and the biases as sums of d_out; the
        // largest first.  Descending steps, as the reverse pass reaches them; the backward RNN is reversed in ascending ones.
        const auto run = [&](auto tile) {
            ProductBuilder<decltype(tile)> q;
            const auto rows = [&](const float* base, int ld, bool ascending, int slots, int first) {      // of [B][slots][ld]
                return Operand{base + static_cast<long long>(first + (ascending ? 0 : W - 1)) * ld, static_cast<long long>(slots) * ld, ascending ? ld : -ld, ld};
            };
            const auto down = [&](long long off, int ld) { return rows(ws + off, ld, false, W, 0); };
            const Operand none{nullptr, 0, 0, 0};
            q.add(down(o.dhx, 2 * N), down(o.v, H), g(iW4), H, g(ib4), B, W);
            q.add(down(o.dpf, H), rows(xhat, N, false, W, 0), g(iWxf), N, g(ibf), B, W);
            q.add(rows(ws + o.dpb, H, true, W, 0), rows(xhat, N, true, W, 0), g(iWxb), N, g(ibb), B, W);
            q.add(down(o.dpf, H), rows(ws + o.a, H, false, W + 1, 0), g(iWhf), H, nullptr, B, W);
            q.add(rows(ws + o.dpb, H, true, W, 0), rows(ws + o.b, H, true, W + 1, 1), g(iWhb), H, nullptr, B, W);
            q.add(down(o.dv, H), rows(ws + o.z, D, false, W + 1, 1), g(iW3), D, g(ib3), B, W);
            q.add(down(o.du, H), rows(ws + o.z, D, false, W + 1, 0), g(iW1), D, g(ib1), B, W);
            q.add(down(o.dpc, H), rows(ws + o.z, D, false, W + 1, 0), g(iWz), D, g(ibz), B, W);
            q.add(down(o.dhz, 2 * D), down(o.u, H), g(iW2), H, g(ib2), B, W);
            q.add(down(o.dmu, D), down(o.hout, H), g(iWmu), H, g(ibmu), B, W);
            q.add(down(o.dps, D), down(o.mu, D), g(iWsig), D, g(ibsig), B, W);
            q.add(Operand{ws + o.ca, H, 0, H}, none, nullptr, 0, g(ia0), B);
            q.add(Operand{ws + o.cb, H, 0, H}, none, nullptr, 0, g(ib0), B);
            q.add(Operand{ws + o.gz0, D, 0, D}, none, nullptr, 0, g(iz0), B);
            q.template run<false, false, true>(vec, stream, true);
        };
        // the head's gradient has the most tiles
        if (tiles_of(2 * N, LargeTile::TM) * tiles_of(H, LargeTile::TN) >= kFillTiles) run(LargeTile{});
        else run(MediumTile{});
    }
}

}  // namespace fit
}  // namespace cutoff
