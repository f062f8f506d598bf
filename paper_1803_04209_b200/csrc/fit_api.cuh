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

inline long long tiles_of(long long n) { return (n + kTile - 1) / kTile; }

// Parts a product's K is split into so that its tiles fill the GPU about twice (a tile of 64 x 64 alone takes
// K * 32 clocks of an SM), at least 128 long each.
inline int k_part_of(long long tiles, long long K) {
    long long parts = (2 * 148 + tiles - 1) / tiles;
    if (parts > 16) parts = 16;
    long long len = (K + parts - 1) / parts;
    if (len < 128) len = 128;
    return static_cast<int>((len + kTileK - 1) / kTileK * kTileK);
}
inline int parts_of(long long K, int k_part) { return static_cast<int>((K + k_part - 1) / k_part); }

// Everything the passes keep, as offsets (floats, multiples of 4) into the workspace.
struct Workspace {
    long long proj, a, b, comb, hout, mu, presig, z, u, v, dhz, dzt, path, dhx, part, dv_parts, dv, du, dpc, dh, dmu, dps, gz0,
        dpf, dpb, ca, cb, total;
    int proj_k, proj_parts, dv_k, dv_parts_n;
};

inline Workspace workspace(long long N, long long D, long long H, long long W, long long B) {
    const long long R = B * W, rh = R * H, rd = R * D, sh = B * (W + 1) * H, sd = B * (W + 1) * D;
    Workspace w;
    w.proj_k = k_part_of(tiles_of(R) * 2 * tiles_of(H), N);
    w.proj_parts = parts_of(N, w.proj_k);
    w.dv_k = k_part_of(tiles_of(R) * tiles_of(H), 2 * N);
    w.dv_parts_n = parts_of(2 * N, w.dv_k);
    long long o = 0;
    const auto take = [&](long long n) { const long long r = o; o += (n + 3) / 4 * 4; return r; };
    w.proj = take(w.proj_parts * 2 * rh);
    w.a = take(sh); w.b = take(sh);
    w.comb = take(rh); w.hout = take(rh); w.mu = take(rd); w.presig = take(rd); w.z = take(sd); w.u = take(rh); w.v = take(rh);
    w.dhz = take(2 * rd); w.dzt = take(rd); w.path = take(B);
    w.dhx = take(R * 2 * N);
    w.part = take((N + kHeadWorkers - 1) / kHeadWorkers * R);
    w.dv_parts = take(w.dv_parts_n * rh);
    w.dv = take(rh); w.du = take(rh); w.dpc = take(rh); w.dh = take(rh); w.dmu = take(rd); w.dps = take(rd); w.gz0 = take(B * D);
    w.dpf = take(rh); w.dpb = take(rh); w.ca = take(B * H); w.cb = take(B * H);
    w.total = o;
    return w;
}

inline long long workspace_floats(long long N, long long D, long long H, long long W, long long B) { return workspace(N, D, H, W, B).total; }

// A kernel that may begin while the one before it is still running (it waits by itself before it touches its results).
template <typename... KArgs, typename... Args>
inline void launch(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t s, bool dependent, Args... args) {
    if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

struct ProductBuilder {
    ProductList list{};
    int tiles = 0;
    ProductBuilder() { list.n = 0; }
    void add(const Operand& a, const Operand& b, float* c, long long ldc, float* a_sums, int K) {
        Product& p = list.p[list.n++];
        p.a = a; p.b = b; p.c = c; p.ldc = ldc; p.a_sums = a_sums; p.K = K;
        p.tile0 = tiles;
        p.tiles_n = b.rows > 0 ? static_cast<int>(tiles_of(b.rows)) : 1;
        tiles += static_cast<int>(tiles_of(a.rows)) * p.tiles_n;
    }
    template <bool AK, bool BK>
    void run(bool vec, int k_part, int parts, long long part_stride, cudaStream_t s, bool dependent) {
        list.k_part = k_part;
        list.part_stride = part_stride;
        if (vec) launch(k_products<AK, BK, true>, dim3(tiles, parts), kGemmThreads, 0, s, dependent, list);
        else launch(k_products<AK, BK, false>, dim3(tiles, parts), kGemmThreads, 0, s, dependent, list);
    }
};

// Enqueue forward (+ backward if grads) on `stream`.  All pointers are device pointers.
inline void elbo_grad(int N, int D, int H, int W, int B, const float* p, const float* xhat, const float* eps, float* elbo,
                      float* grads, float* ws, cudaStream_t stream) {
    const Layout L = layout(N, D, H);
    const Workspace o = workspace(N, D, H, W, B);
    const auto w = [&](int i) { return p + L.off[i]; };
    const auto g = [&](int i) { return grads + L.off[i]; };
    const int R = B * W;
    const long long rh = static_cast<long long>(R) * H;
    const bool back = grads != nullptr;
    const auto aligned = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    // 16-byte loads: every tensor and every row then starts on 16 bytes
    const bool vec = N % 4 == 0 && D % 4 == 0 && H % 4 == 0 && aligned(p) && aligned(xhat) && aligned(ws);
    const bool vec_h = H % 4 == 0 && vec;

    // ---- forward -------------------------------------------------------------------------------------------------
    {
        ProductBuilder q;                                     // input projections of both RNNs, K = N in parts
        const Operand x{xhat, N, R, 0, 0};
        q.add(x, Operand{w(iWxf), N, H, 0, 0}, ws + o.proj, 2 * H, nullptr, N);
        q.add(x, Operand{w(iWxb), N, H, 0, 0}, ws + o.proj + H, 2 * H, nullptr, N);
        q.run<true, true>(vec, o.proj_k, o.proj_parts, 2 * rh, stream, false);
    }
    const bool wh_staged = H <= kRnnSmemH;
    {
        RnnArgs a{};
        a.proj = ws + o.proj; a.n_parts = o.proj_parts; a.part_stride = 2 * rh;
        a.Wh[0] = w(iWhf); a.Wh[1] = w(iWhb); a.bias[0] = w(ibf); a.bias[1] = w(ibb); a.init[0] = w(ia0); a.init[1] = w(ib0);
        a.state[0] = ws + o.a; a.state[1] = ws + o.b; a.B = B; a.W = W; a.H = H;
        const dim3 grid((B + kRnnRows - 1) / kRnnRows, 2);
        const size_t smem = rnn_smem_bytes(H, wh_staged);
        if (vec_h) launch(k_rnn_forward<true>, grid, kRnnThreads, smem, stream, true, a, wh_staged ? 1 : 0);
        else launch(k_rnn_forward<false>, grid, kRnnThreads, smem, stream, true, a, wh_staged ? 1 : 0);
    }
    PathArgs a{};
    a.Wz = w(iWz); a.bz = w(ibz); a.Wmu = w(iWmu); a.bmu = w(ibmu); a.Wsig = w(iWsig); a.bsig = w(ibsig); a.z0 = w(iz0);
    a.W1 = w(iW1); a.b1 = w(ib1); a.W2 = w(iW2); a.b2 = w(ib2); a.W3 = w(iW3); a.b3 = w(ib3);
    a.a = ws + o.a; a.b = ws + o.b; a.eps = eps;
    a.comb = ws + o.comb; a.hout = ws + o.hout; a.mu = ws + o.mu; a.presig = ws + o.presig; a.z = ws + o.z; a.u = ws + o.u;
    a.v = ws + o.v; a.dhz = ws + o.dhz; a.dzt = ws + o.dzt; a.path = ws + o.path;
    a.dv_parts = ws + o.dv_parts; a.n_parts = o.dv_parts_n; a.part_stride = rh;
    a.dv = ws + o.dv; a.du = ws + o.du; a.dpc = ws + o.dpc; a.dh = ws + o.dh; a.dmu = ws + o.dmu; a.dps = ws + o.dps;
    a.gz0 = ws + o.gz0; a.B = B; a.W = W; a.D = D; a.H = H;
    const size_t path_scratch = path_scratch_floats(D, H) * sizeof(float);
    const size_t path_full = path_scratch + path_weight_floats(D, H) * sizeof(float);
    const int staged = path_full <= 200 * 1024 ? 1 : 0;
    const size_t path_smem = staged ? path_full : path_scratch;
    launch(k_path_forward, dim3(B), kPathThreads, path_smem, stream, true, a, staged);
    const int head_tiles = (N + kHeadWorkers - 1) / kHeadWorkers;
    {
        const dim3 grid(static_cast<unsigned>(head_tiles * tiles_of(R)));
        float* dhx = back ? ws + o.dhx : nullptr;
        if (vec) launch(k_emission_density<true>, grid, kGemmThreads, 0, stream, true, ws + o.v, w(iW4), w(ib4), xhat, R, N, H, dhx, ws + o.part);
        else launch(k_emission_density<false>, grid, kGemmThreads, 0, stream, true, ws + o.v, w(iW4), w(ib4), xhat, R, N, H, dhx, ws + o.part);
    }
    launch(k_elbo_finish, dim3((B + 3) / 4), 128, 0, stream, true, ws + o.part, head_tiles, R, W, B, ws + o.path, elbo);
    if (!back) return;
    // ---- backward ------------------------------------------------------------------------------------------------
    {
        ProductBuilder q;                                     // d v = d_head W4, K = 2N in parts
        q.add(Operand{ws + o.dhx, 2ll * N, R, 0, 0}, Operand{w(iW4), H, H, 0, 0}, ws + o.dv_parts, H, nullptr, 2 * N);
        q.run<true, false>(vec, o.dv_k, o.dv_parts_n, rh, stream, true);
    }
    launch(k_path_backward, dim3(B), kPathThreads, path_smem, stream, true, a, staged);
    {
        RnnBackArgs r{};
        r.g = ws + o.dh; r.state[0] = ws + o.a; r.state[1] = ws + o.b; r.Wh[0] = w(iWhf); r.Wh[1] = w(iWhb);
        r.d_pre[0] = ws + o.dpf; r.d_pre[1] = ws + o.dpb; r.carry_out[0] = ws + o.ca; r.carry_out[1] = ws + o.cb;
        r.B = B; r.W = W; r.H = H;
        const dim3 grid((B + kRnnRows - 1) / kRnnRows, 2);
        const size_t smem = rnn_back_smem_bytes(H, wh_staged);
        if (vec_h) launch(k_rnn_backward<true>, grid, kRnnThreads, smem, stream, true, r, wh_staged ? 1 : 0);
        else launch(k_rnn_backward<false>, grid, kRnnThreads, smem, stream, true, r, wh_staged ? 1 : 0);
    }
    {
        // every weight gradient d W = d_out^T in over the R rows, and the biases as column sums of d_out; the largest first
        ProductBuilder q;
        const auto rows = [&](long long off, int ld) { return Operand{ws + off, ld, ld, 0, 0}; };
        const auto before = [&](long long off, int ld, int first) { return Operand{ws + off, ld, ld, W, first}; };   // of [B][W + 1]
        const Operand none{nullptr, 0, 0, 0, 0};
        q.add(rows(o.dhx, 2 * N), rows(o.v, H), g(iW4), H, g(ib4), R);
        q.add(rows(o.dpf, H), Operand{xhat, N, N, 0, 0}, g(iWxf), N, g(ibf), R);
        q.add(rows(o.dpb, H), Operand{xhat, N, N, 0, 0}, g(iWxb), N, g(ibb), R);
        q.add(rows(o.dpf, H), before(o.a, H, 0), g(iWhf), H, nullptr, R);
        q.add(rows(o.dpb, H), before(o.b, H, 1), g(iWhb), H, nullptr, R);
        q.add(rows(o.dv, H), before(o.z, D, 1), g(iW3), D, g(ib3), R);
        q.add(rows(o.du, H), before(o.z, D, 0), g(iW1), D, g(ib1), R);
        q.add(rows(o.dpc, H), before(o.z, D, 0), g(iWz), D, g(ibz), R);
        q.add(rows(o.dhz, 2 * D), rows(o.u, H), g(iW2), H, g(ib2), R);
        q.add(rows(o.dmu, D), rows(o.hout, H), g(iWmu), H, g(ibmu), R);
        q.add(rows(o.dps, D), rows(o.mu, D), g(iWsig), D, g(ibsig), R);
        q.add(rows(o.ca, H), none, nullptr, 0, g(ia0), B);
        q.add(rows(o.cb, H), none, nullptr, 0, g(ib0), B);
        q.add(rows(o.gz0, D), none, nullptr, 0, g(iz0), B);
        q.run<false, false>(vec, (R + kTileK - 1) / kTileK * kTileK, 1, 0, stream, true);
    }
}

}  // namespace fit
}  // namespace cutoff
