// Per-sample chain (guide steps, transition, first emission layer) on the tcgen05 tensor cores,
// for latent size 16 and hidden width 64..256, or latent size 32 and hidden width up to 512.  One kernel template serves both model
// variants: the compact one (transition = one hidden layer with a [mean | logvar] head, then the emission's
// hidden layer v) and the networks as Section 3.1.3 prints them (LITERAL: gated transition
//      g = sigmoid(Wg2 relu(Wg1 z + bg1) + bg2)        h = Wh2 relu(Wh1 z + bh1) + bh2
//      G = (1 - g) * (Wl z + bl) + g * h               H = softplus(Ws relu(G) + bs)        z' = G + H * eps
// then the affine first layer of the emission mean, u = Wi1 z' + bi1).
//
// A CTA walks over tiles of samples; a sample is a TMEM lane.  Every layer pair
//      hidden = act(A z + a)          (M=128, N=H, K=D, tf32)
//      out    = B hidden (+ b)        (M=128, N=D to 3D, K=H, halves)
// is two UMMA groups.  The first writes the hidden pre-activations to TMEM columns [0, H) of the tile's slot.  Each
// epilogue warp reads its lanes' quarter of the columns, applies bias and activation and writes the result as packed
// halves over the columns that it has just read: the hidden layer is the A operand of the second product straight from tensor
// memory and never passes through shared memory.  The second result (mu; mean | logvar; gate; proposal) is read back by all
// epilogue warps, which draw the noise, form the next latent and store it as the next A operand of a first layer (shared
// memory, tf32).  In the literal variant the proposal's result is combined with the gate and the linear map (computed by the
// epilogue threads from the latent tile) into G, relu(G) then takes the place of the latent tile and one more small product
// with Ws gives the scale.
//
// The halves carry the 11 bits of a tf32 value (half_operand.cuh): hidden values of the guide lie in [-1, 1] and are scaled by
// 2^14, those of the other layers by a power of two from the sample's largest |latent|, rows of weights by one each.  Of the
// guide's h_out = (tanh + h_left + h_right) / 3 only the tanh differs between samples, so only it is an operand:
//      mu = (Wmu tanh) / 3 + [Wmu (h_left + h_right) / 3 + bmu],
// the bracket, one vector of 16 per step, is formed in fp32 from the unrounded weights when the kernel starts.  The scale's linear
// map Wsig mu + bsig comes out of the same product: its rows are those of Wsig Wmu, formed in double and split into two halves
// each (together 22 bits), and a bracket of its own.  The first step starts from one latent for all samples, so its tanh is one vector
// too and joins the bracket: that step is only noise.
//
// What bounds it: each step's round trip, two products and the noise in between, which a second tile covers in part; no unit is busy.  Of
// them the special-function pipe is the first (256 tanh per sample and step and about 60 logarithms, sines and the like for its
// noise): S=65536, D=16, H=256, lag 4 66 us, special-function pipe 37 % busy, issue slots 44 %, shared-memory wavefronts 29 %, tensor pipe
// 11 %.  With the hidden layer through shared memory as tf32, 64 units at a time, four steps of handshakes each, it took 108.  With
// one tile per SM, S=8192 41 -> 27 us (35 with tiles of 128).  D=32, with one tile per SM: S=32768, H=512, lag 4 162 -> 92 us,
// S=8192, H=256 60 -> 35 us; its weights were copied by the epilogue's threads before.
//
// The host prepares a swizzled image of the weight operands once.  Latent rows are 128 bytes wide (32 tf32).  D = 16: all operands live in
// shared memory for the whole kernel, and two first-layer matrices share one tile (columns 0..15 and 16..31: [Wz | W1], or
// [Wz | Wg1] and [Wh1 | Wi1]), so the MMA for the second of them simply starts 64 bytes into the rows.  D = 32: they are too large
// (352 KB at H = 512), so one first-layer and one second-layer matrix are there at a time and the issuing warp has each replaced by
// the next phase's as soon as its last product is done, while the epilogue is still at work on the result.
// The last layer's hidden vector (v, or u) goes to global memory as halves for the emission output GEMMs.
//
// A tile is the work of one warp that issues its MMAs and of 8 or 16 epilogue warps: warp w serves TMEM lanes 32*(w%4).. and one of
// two or four column groups, that is its share of the hidden units and 8 or 4 of the latent dimensions (whole Philox calls).  Two tiles
// of 8 warps each run side by side without knowing of each other, so that one's tanh meets the other's noise, products and waits;
// a CTA with only one tile gives it all 16 warps.
// Every mbarrier wait is bounded (see async.cuh).
#pragma once
#include "emit_tc.cuh"

namespace cutoff {
namespace tc {

constexpr int kChainEpiWarps = 16;
constexpr int kChainTcThreads = (2 + kChainEpiWarps) * 32;
constexpr int kChainD = 16, kChain32D = 32;
constexpr float kTanhScale = 16384.0f;       // a tanh as an operand: normal halves down to 2^-28

struct ChainTcArgs {
    // swizzled operand tiles: first-layer matrices in floats (D = 16: [Wz|W1], [W3] or [Wz|Wg1], [Wh1|Wi1]; D = 32: Wz, W1, W3 or Wz, Wg1,
    // Wh1, Wi1; H x 32 each), then second-layer ones in halves, K blocks of 64: Wmu and the two parts of Wsig Wmu (3D rows), W2 (2D rows) or
    // Wg2 and Wh2 (D rows each); literal: Ws (D x 32 floats).  Behind them, floats: the inverse scales of the rows of halves, in that order
    // (5D), then Wsig bmu + bsig (D) and Wsig Wmu (D x H).
    const uint8_t* image;
    // compact: b1, b3 = biases of the transition's and the emission's hidden layer, b2 = [mean | logvar] bias (2D);
    // literal: b1 = bg1, b3 = bh1, b2 unused
    const float *bz, *b1, *b3, *bmu, *b2, *z0;
    const float *bi1, *bg2, *bh2, *Wl, *bl, *bs;       // literal variant only
    const float *WzT, *Wmu;     // [D][H] each, fp32
    const float* hlr;           // [2][W][H] h_left, h_right
    const float* bounds;        // [2][2] of the transition's hidden layer (literal: of the gate's and the proposal's), as HalfRows::bound
    DevState* st;
    NoiseKey key;
    uint32_t sample_base;
    int count, H, W;
    HalfRows v_out;             // v (literal: u), scaled
};

// Bytes of D rows of halves (whole K blocks), of the first-layer tiles, of all operand tiles, and floats behind them.
__host__ __device__ constexpr uint32_t chain_tc_row_bytes(int D, int H) { return static_cast<uint32_t>((H + 63) / 64) * 128u * static_cast<uint32_t>(D); }
__host__ __device__ constexpr uint32_t chain_tc_first_bytes(int D, int H, bool literal) { return static_cast<uint32_t>(H) * 128u * (D == 16 ? 2u : (literal ? 4u : 3u)); }
__host__ __device__ constexpr uint32_t chain_tc_image_bytes(int D, int H, bool literal) {
    return chain_tc_first_bytes(D, H, literal) + 5u * chain_tc_row_bytes(D, H) + (literal ? static_cast<uint32_t>(D) * 128u : 0u);
}
inline size_t chain_tc_tail_floats(int D, int H) { return 6 * static_cast<size_t>(D) + static_cast<size_t>(D) * H; }
// What of them is in shared memory at a time: D = 16 all, D = 32 one first-layer tile, the guide's second layer or a smaller one, and Ws.
__host__ __device__ constexpr uint32_t chain_tc_operand_bytes(int D, int H, bool literal) {
    return D == 16 ? chain_tc_image_bytes(D, H, literal) : static_cast<uint32_t>(H) * 128u + 3u * chain_tc_row_bytes(D, H) + (literal ? 4096u : 0u);
}
constexpr int kChainLatentBytes = 2 * 16384;      // latent tiles of two slots

inline size_t chain_tc_smem_bytes(int D, int H, int W, bool literal) {
    const size_t floats = (literal ? 4 : 3) * static_cast<size_t>(H) + 2 * 4 * 128 + 2 * static_cast<size_t>(W) * D + (literal ? D * D : 0) + 5 * D +
                          (literal ? 4 : 2) * D + 32;
    return 1024 + chain_tc_operand_bytes(D, H, literal) + kChainLatentBytes + floats * 4;
}

// The longest window, in steps: D = 16 13 at H = 256 (literal 9), 56 (51) at 192, 141 (134) at 128; D = 32 96 at H = 256, 14 at 512.  The line is
// one of precision, not of room: longer windows have always been computed by the fp32 kernels (the RNN states of these, W H floats, used
// to stand beside the operands), and what is computed in fp32 stays so.  This kernel itself would take longer ones (D = 16, H = 256, 13 steps:
// 150 of 227 KB).
inline int chain_tc_longest_window(int D, int H, bool literal) {
    return D == 32 ? 42144 / H - 68 : literal ? 32080 / H - 116 : 32880 / H - 115;
}
inline bool chain_tc_window(int D, int H, int W, bool literal) {
    return W <= chain_tc_longest_window(D, H, literal) && chain_tc_smem_bytes(D, H, W, literal) <= 227 * 1024;
}

// byte offset of the 16-byte chunk `chunk` of row `row` in a K-major tile with 128-byte swizzled rows
__device__ __forceinline__ uint32_t sw128(int row, int chunk) {
    return static_cast<uint32_t>((row >> 3) * 1024 + (row & 7) * 128 + ((chunk ^ (row & 7)) << 4));
}

__device__ __forceinline__ uint32_t instr_desc_tf32(int n) {      // D = f32, A = B = tf32, K-major, M = 128
    return (1u << 4) | (2u << 7) | (2u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | ((128u >> 4) << 24);
}

// Round to tf32 (nearest, ties away from zero) with two integer instructions instead of the conversion instruction,
// which shares the slow special-function pipe with tanh: add half a unit of the 13 dropped bits to the magnitude,
// clear them.  The same bits as cvt.rna.tf32.f32 for every finite value (an overflow of the mantissa carries into
// the exponent, as it should).
__device__ __forceinline__ float tf32_rna(float x) {
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

__device__ __forceinline__ float softplus_fast(float x) {          // ln(1 + e^x)
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * 1.4426950408889634f));
    return x > 15.0f ? x : 0.6931471805599453f * log2_fast(1.0f + e);
}

__device__ __forceinline__ float sigmoid_fast(float x) {
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * -1.4426950408889634f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(e + 1.0f));
    return r;
}

__device__ __forceinline__ float4 ld_shared_v4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

// The largest |latent| of a thread's dimensions.
template <int N>
__device__ __forceinline__ void put_largest(uint32_t addr, const float (&z)[N]) {
    float m = 0.0f;
#pragma unroll
    for (int c = 0; c < N; ++c) m = fmaxf(m, fabsf(z[c]));
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(m) : "memory");
}

// 16 consecutive halves: one sector.
__device__ __forceinline__ void store8(__half* p, const uint32_t (&w)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
}

// Sixteen consecutive accumulator columns of a warp's 32 lanes as they are spread by .32x32b (a lane's 16 columns in its thread), or
// of its first 16 lanes by .16x256b: the thread's rows are lane / 4 and lane / 4 + 8, its columns 2 (lane % 4) and the one behind it, of each 8.
// What is written back as packed halves takes the .32x32b and .16x128b spreads, under which a thread owns the pairs that it has read.
__device__ __forceinline__ void tmem_ld16_half(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_st8_half(uint32_t taddr, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.16x128b.x2.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_dims(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_dims(uint32_t taddr, uint32_t (&r)[8]) { tmem_ld8(taddr, r); }

// D += A B with A in tensor memory (lanes = rows, two halves per column).
__device__ __forceinline__ void umma_f16_tmem(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

__device__ __forceinline__ float tanh_hw(float x) {
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(x));
    return t;
}
// tanh of two biased accumulators as a word of two scaled halves.
__device__ __forceinline__ uint32_t tanh_pair(uint32_t acc0, uint32_t acc1, unsigned long long bias) {
    float x0, x1;
    unpack2(add2(pack2(__uint_as_float(acc0), __uint_as_float(acc1)), bias), x0, x1);
    unpack2(mul2(pack2(tanh_hw(x0), tanh_hw(x1)), pack2(kTanhScale, kTanhScale)), x0, x1);
    return pack_half2(x0, x1);
}
// The same of a ReLU layer (or an affine one), scaled by the sample's power of two.
template <bool RELU>
__device__ __forceinline__ uint32_t scaled_pair(uint32_t acc0, uint32_t acc1, unsigned long long bias, unsigned long long scale) {
    float x0, x1;
    unpack2(mul2(add2(pack2(__uint_as_float(acc0), __uint_as_float(acc1)), bias), scale), x0, x1);
    return RELU ? pack_half2(fmaxf(x0, 0.0f), fmaxf(x1, 0.0f)) : pack_half2(x0, x1);
}
// Biases of 16 columns, from shared memory.
__device__ __forceinline__ void load_bias(const float* bias, ulonglong2 (&b)[4]) {
#pragma unroll
    for (int g = 0; g < 4; ++g) b[g] = *reinterpret_cast<const ulonglong2*>(bias + 4 * g);
}
// Eight words from 16 columns of one lane.  act(acc0, acc1, bias pair).
template <typename Act>
__device__ __forceinline__ void pack_columns(const uint32_t (&acc)[16], const ulonglong2 (&b)[4], uint32_t (&w)[8], Act act) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        w[2 * g] = act(acc[4 * g], acc[4 * g + 1], b[g].x);
        w[2 * g + 1] = act(acc[4 * g + 2], acc[4 * g + 3], b[g].y);
    }
}

// WARPS: epilogue warps of a tile.  HALF: tiles of 64 samples, 16 lanes of each quarter of the tensor memory, for decisions that leave SMs
// without a tile of 128.  A warp then spreads the 16 lanes' guide columns over its 32 threads; all else runs as in a full tile, the
// other lanes on values that nobody reads.  The results of a sample are the same to the last bit in every shape.
template <int D, bool LITERAL, int WARPS, bool HALF>
__global__ void __launch_bounds__(kChainTcThreads, 1) k_chain_tc(ChainTcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    constexpr int kRows = HALF ? 64 : 128;                        // samples per tile
    constexpr int kSlots = kChainEpiWarps / WARPS, kGroups = WARPS / 4, kDims = D / kGroups;
    constexpr bool kStaged = D == 32;
    static_assert(!kStaged || kSlots == 1, "operands that come and go serve one tile");
    const int H = a.H, W = a.W;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gen = smem_raw + (base - raw);
    // weight operand tiles
    const uint32_t first_bytes = chain_tc_first_bytes(D, H, LITERAL);
    const uint32_t image_bytes = chain_tc_image_bytes(D, H, LITERAL), operand_bytes = chain_tc_operand_bytes(D, H, LITERAL);
    const uint32_t t_first = base;
    const uint32_t t_guide = t_first + (kStaged ? H * 128u : first_bytes);    // Wmu and the parts of Wsig Wmu; staged: any second layer
    const uint32_t row_bytes = chain_tc_row_bytes(D, H);
    const uint32_t t_out1 = t_guide + 3 * row_bytes;              // W2 (2D rows per K block) or Wg2 (D rows)
    const uint32_t t_out2 = t_out1 + row_bytes;                   // literal: Wh2
    const uint32_t t_ws = base + operand_bytes - D * 128u;        // literal: Ws, D rows x 128 bytes
    const uint32_t t_act = base + operand_bytes;                  // latent tiles, one per slot
    // fp32 side tables
    float* sbzs = reinterpret_cast<float*>(gen + operand_bytes + kChainLatentBytes);     // bz
    float* sb1 = sbzs + H;
    float* sb3 = sb1 + H;
    float* sbi1 = sb3 + H;                   // literal only
    // [guide, transition][slot][column group][row] largest |latent| of a thread's dimensions.  Two arrays, because nobody waits between the
    // last layer's reads of the transition's and, in a window of one step, the next tile's writes of the guide's: a warp that is ahead would
    // change what another has yet to read.  So both arrays' writes are a barrier that all warps arrive at away from their readers: the guide's are
    // read before the arrivals on bar_z that the last layer's product waits for, the transition's before those on bar_h of the next tile.
    float* szmax = sb3 + (LITERAL ? 2 : 1) * H;
    float* sct = szmax + 2 * 4 * 128;        // [W][D]  Wmu (h_left + h_right) / 3 + bmu
    float* spt = sct + W * D;                // [W][D]  the same of the scale: Wsig times that, + bsig
    float* sWl = spt + W * D;                // [D][D], literal only
    // what the products of halves are multiplied with: mu D, the two parts of the scale's map D each, then W2 2D or Wg2, Wh2 D each
    float* sscale = sWl + (LITERAL ? D * D : 0);
    float* sb2 = sscale + 5 * D;             // compact: [2D]
    float* sbg2 = sb2;                       // literal: bg2, bh2, bl, bs, D each
    float* sbh2 = sbg2 + D;
    float* sbl = sbh2 + D;
    float* sbs = sbl + D;
    float* sbar = sb2 + (LITERAL ? 4 : 2) * D;
    const uint32_t bars = smem_u32(sbar);                         // 2 slots x 5 barriers
    const uint32_t bar_img = bars + 2 * 40, bar_second = bar_img + 8;      // the operand image has landed; staged: a first layer, a second layer
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sbar + 24);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sbar + 25);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // Staged operands.  First layers in the order of the image, one per kind of phase: guide, transition (gate), last layer (proposal), - (last
    // layer).  Second layers: guide, W2 (Wg2), - (Wh2).
    const auto phase_kind = [&](int ph) { return ph < W ? 0 : ph - W + 1; };
    const auto load_operand = [&](uint32_t dst, uint32_t offset, uint32_t bytes, uint32_t bar) {
        mbar_arrive_expect_tx(bar, bytes);
        for (uint32_t off = 0; off < bytes; off += 32768u) bulk_load_1d(dst + off, a.image + offset + off, min(bytes - off, 32768u), bar);
    };
    const auto load_first = [&](int kind) { load_operand(t_first, static_cast<uint32_t>(kind) * H * 128u, H * 128u, bar_img); };
    const auto load_second = [&](int kind) {
        load_operand(t_guide, first_bytes + (kind == 0 ? 0u : kind == 1 ? 3u : 4u) * row_bytes, (kind == 0 ? 3u : (LITERAL ? 1u : 2u)) * row_bytes, bar_second);
    };

    // ---- one-time set-up: barriers, operand image (bulk copies, while the side tables are filled), TMEM ----------
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < 2; ++s) {
            const uint32_t b0 = bars + 40 * s;
            mbar_init(b0, WARPS);                    // latent tile (or relu(G)) ready
            mbar_init(b0 + 8, 1);                    // hidden pre-activations ready
            mbar_init(b0 + 16, WARPS);               // hidden layer written
            mbar_init(b0 + 24, 1);                   // second result ready
            mbar_init(b0 + 32, 1);                   // drained
        }
        mbar_init(bar_img, 1);
        mbar_init(bar_second, 1);
        *abort_flag = 0;
        fence_barrier_init();
        if (kStaged) {
            load_first(phase_kind(1));
            load_second(phase_kind(1));
        } else {
            load_operand(base, 0u, image_bytes, bar_img);
        }
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(const_cast<uint32_t*>(tmem_slot))), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const float* const tail = reinterpret_cast<const float*>(a.image + image_bytes);
    for (int i = threadIdx.x; i < H; i += kChainTcThreads) {
        sbzs[i] = a.bz[i];
        sb1[i] = a.b1[i];
        sb3[i] = a.b3[i];
        if (LITERAL) sbi1[i] = a.bi1[i];
    }
    if (LITERAL) {
        for (int i = threadIdx.x; i < D * D; i += kChainTcThreads) sWl[i] = a.Wl[i];
        if (kStaged)                                              // Ws stays
            for (int i = threadIdx.x; i < D * 32; i += kChainTcThreads)
                reinterpret_cast<float*>(gen + operand_bytes - D * 128)[i] = reinterpret_cast<const float*>(a.image + image_bytes - D * 128)[i];
        if (threadIdx.x < D) {
            sbg2[threadIdx.x] = a.bg2[threadIdx.x];
            sbh2[threadIdx.x] = a.bh2[threadIdx.x];
            sbl[threadIdx.x] = a.bl[threadIdx.x];
            sbs[threadIdx.x] = a.bs[threadIdx.x];
        }
    } else if (threadIdx.x < 2 * D) {
        sb2[threadIdx.x] = a.b2[threadIdx.x];
    }
    if (threadIdx.x < 5 * D) {
        const float inv = tail[threadIdx.x];
        sscale[threadIdx.x] = threadIdx.x < 3 * D ? inv * (1.0f / (3.0f * kTanhScale)) : inv;
    }
    // hidden unit i of the first step, the same for every sample
    float first_tanh = 0.0f;
    if (threadIdx.x < H) {
        float s = a.bz[threadIdx.x];
#pragma unroll 16
        for (int d = 0; d < D; ++d) s = fmaf(a.WzT[d * H + threadIdx.x], a.z0[d], s);
        first_tanh = tanhf(s);
    }
    // epilogue warp 2 + w: rows w, w + 16 of Wmu and of Wsig Wmu, for the parts of mu and of the scale that no sample changes
    constexpr int kPer = D == 16 ? 8 : 16;                        // hidden units per lane at most
    float wmu[kPer], wsm[kPer];
    const auto load_row = [&](int d) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int at = d * H + 32 * i + lane;
            wmu[i] = 32 * i < H ? a.Wmu[at] : 0.0f;
            wsm[i] = 32 * i < H ? tail[6 * D + at] : 0.0f;
        }
    };
    if (warp > 1) load_row(warp - 2);
    // up to here nothing an earlier kernel of the stream writes has been touched (the image and the biases are
    // weights): the encoder's states and the device state come after this point
    dependency_wait();
    launch_dependents();
    // h_left + h_right (first step: + tanh) of as many steps as the place of the latent tiles holds, then the steps' vectors from them.
    // Nothing is unrolled over steps or rows: a launch finds the instruction caches cold, and this code runs once.
    float* const slr = reinterpret_cast<float*>(gen + operand_bytes);
    const int per_round = kChainLatentBytes / 4 / H;
#pragma unroll 1
    for (int t0 = 0; t0 < W; t0 += per_round) {
        const int steps = min(per_round, W - t0);
        if (t0 > 0) __syncthreads();
        for (int i = threadIdx.x; i < steps * H; i += kChainTcThreads)
            slr[i] = a.hlr[t0 * H + i] + a.hlr[(W + t0) * H + i] + (t0 == 0 && i < H ? first_tanh : 0.0f);
        __syncthreads();
        if (warp > 1) {
#pragma unroll 1
            for (int d = warp - 2; d < D; d += 16) {
                if (d != warp - 2 || (D == 32 && t0 > 0)) load_row(d);
                const float bmu = a.bmu[d], bsm = tail[5 * D + d];
#pragma unroll 1
                for (int t = 0; t < steps; ++t) {
                    float s = 0.0f, p = 0.0f;
#pragma unroll
                    for (int i = 0; i < kPer; ++i)
                        if (32 * i < H) {
                            const float v = slr[t * H + 32 * i + lane];
                            s = fmaf(wmu[i], v, s);
                            p = fmaf(wsm[i], v, p);
                        }
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) {
                        s += __shfl_xor_sync(0xffffffffu, s, off);
                        p += __shfl_xor_sync(0xffffffffu, p, off);
                    }
                    if (lane == 0) {
                        sct[(t0 + t) * D + d] = fmaf(s, 1.0f / 3.0f, bmu);
                        spt[(t0 + t) * D + d] = fmaf(p, 1.0f / 3.0f, bsm);
                    }
                }
            }
        }
    }
    if (LITERAL && kStaged) fence_proxy_async();                  // Ws was written with ordinary stores
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // nothing starts before the weights are in place; if they never arrive every role skips its loop (staged: the issuing warp waits for each)
    const bool image_ok = kStaged || mbar_wait(bar_img, 0u, abort_flag, a.st);
    const int n_tiles = image_ok ? ceil_div(a.count, kRows) : 0;
    // phases: W guide steps, then transition and emission hidden layer -- or gate, proposal (+ scale), first emission layer
    const int n_phases = LITERAL ? W + 3 : W + 2;
    const int ph_last = n_phases - 1;                             // its hidden layer goes to global memory, no second GEMM
    // The hidden units go to the column groups in blocks of 16.  A group's stand, packed, in the first half of the columns of its
    // pre-activations, group 1's in the second half.  The second result (at most 3D columns) takes columns that hold neither: those behind the
    // hidden layer, or the other halves of groups 0 and 1.
    const int blocks = H / 16;
    const auto group_block = [&](int g) { return g * blocks / kGroups; };
    const auto packed_col = [&](int g) { return 16 * group_block(g) + (g == 1 ? 8 * (group_block(2) - group_block(1)) : 0); };
    const uint32_t acc2_col = H + 3 * D <= 512 / kSlots ? H : 8 * group_block(1);

    const int slot = warp < 2 ? warp : (warp - 2) / WARPS;
    const uint32_t t_z = t_act + slot * 16384u;                   // latent A operand [128 x 128 B]
    const uint32_t tmem = tmem_base + slot * 256u;                // first of the slot's 256 TMEM columns
    const uint32_t bar_z = bars + 40 * slot, bar_p = bar_z + 8, bar_h = bar_z + 16, bar_acc2 = bar_z + 24, bar_drain = bar_z + 32;
    const int tile0 = static_cast<int>(blockIdx.x) + slot * static_cast<int>(gridDim.x), tile_step = kSlots * static_cast<int>(gridDim.x);
    bool ok = true;
    if (warp < kSlots) {
        // ---------------- MMA issuer of the slot ---------------------------------------------------------
        const int n_lo = H < 256 ? H : 256, n_hi = H - n_lo;
        const uint32_t idesc_lo = instr_desc_tf32(n_lo), idesc_hi = instr_desc_tf32(n_hi);
        uint32_t nz = 0, nh = 0, np = 0, na = 0, n_first = 0, n_second = 0;
        int first_kind = -1, second_kind = -1;                     // staged: the operands that have been waited for
        for (int tile = tile0; ok && tile < n_tiles; tile += tile_step) {
            const bool last_tile = tile + tile_step >= n_tiles;
            for (int ph = 1; ph < n_phases; ++ph) {
                const int kind = phase_kind(ph);
                ok = mbar_wait(bar_z, nz & 1u, abort_flag, a.st);
                if (!ok) break;
                ++nz;
                if (kStaged && first_kind != kind) {
                    ok = mbar_wait(bar_img, n_first & 1u, abort_flag, a.st);
                    if (!ok) break;
                    ++n_first;
                    first_kind = kind;
                }
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t b_tile = kStaged || kind == 0 ? t_first : t_first + (kind >> 1) * H * 128u + (kind & 1) * 64u;
                    const uint64_t a_desc = make_smem_desc(t_z), b_lo = make_smem_desc(b_tile);
#pragma unroll
                    for (int k = 0; k < D / 8; ++k) umma_tf32(tmem, a_desc + 2 * k, b_lo + 2 * k, idesc_lo, k != 0 ? 1u : 0u);
                    if (D == 32 && n_hi > 0) {
                        const uint64_t b_hi = make_smem_desc(b_tile + 256u * 128u);
#pragma unroll
                        for (int k = 0; k < D / 8; ++k) umma_tf32(tmem + 256u, a_desc + 2 * k, b_hi + 2 * k, idesc_hi, k != 0 ? 1u : 0u);
                    }
                    umma_commit(bar_p);
                }
                __syncwarp();
                if (kStaged) {
                    const int next = ph < ph_last ? phase_kind(ph + 1) : (last_tile ? kind : phase_kind(1));
                    if (next != kind) {
                        ok = mbar_wait(bar_p, np & 1u, abort_flag, a.st);
                        if (!ok) break;
                        if (elect_one()) load_first(next);
                        __syncwarp();
                    }
                    ++np;
                }
                if (ph == ph_last) continue;                       // the last hidden layer has no second GEMM here
                ok = mbar_wait(bar_h, nh & 1u, abort_flag, a.st);
                if (!ok) break;
                ++nh;
                if (kStaged && second_kind != kind) {
                    ok = mbar_wait(bar_second, n_second & 1u, abort_flag, a.st);
                    if (!ok) break;
                    ++n_second;
                    second_kind = kind;
                }
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t b_base = kStaged || kind == 0 ? t_guide : (kind == 1 ? t_out1 : t_out2);
                    const uint32_t out_rows = kind == 0 ? 3u * D : (LITERAL ? D : 2u * D), idesc2 = instr_desc_f16(out_rows, 128);
                    uint64_t b_desc = make_smem_desc(b_base);
                    uint32_t more = 0, k = 0;
                    for (int g = 0; g < kGroups; ++g) {
                        uint32_t packed = tmem + packed_col(g);
                        for (int c = group_block(g); c < group_block(g + 1); ++c) {       // 16 hidden units: 8 columns, 32 bytes of a row of B
                            umma_f16_tmem(tmem + acc2_col, packed, b_desc, idesc2, more);
                            more = 1;
                            packed += 8;
                            k += 16;
                            b_desc += k & 63 ? 2 : out_rows * 8 - 6;         // the next 32 bytes, or the next K block
                        }
                    }
                    umma_commit(bar_acc2);
                }
                __syncwarp();
                if (kStaged) {
                    const int next = ph + 1 < ph_last ? phase_kind(ph + 1) : (last_tile ? kind : phase_kind(1));
                    if (next != kind) {
                        ok = mbar_wait(bar_acc2, na & 1u, abort_flag, a.st);
                        if (!ok) break;
                        if (elect_one()) load_second(next);
                        __syncwarp();
                    }
                    ++na;
                }
                if (!LITERAL || ph != W + 1) continue;
                // scale: Ws relu(G), relu(G) sits in the latent tile
                ok = mbar_wait(bar_z, nz & 1u, abort_flag, a.st);
                if (!ok) break;
                ++nz;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t a_desc = make_smem_desc(t_z), b_desc = make_smem_desc(t_ws);
#pragma unroll
                    for (int k = 0; k < D / 8; ++k) umma_tf32(tmem + acc2_col, a_desc + 2 * k, b_desc + 2 * k, instr_desc_tf32(D), k != 0 ? 1u : 0u);
                    umma_commit(bar_acc2);
                }
                __syncwarp();
                ++na;
            }
        }
        if (kStaged && !ok) {
            // wind down: let a copy that was asked for land before the CTA leaves (bounded)
            mbar_wait_quiet(bar_img, n_first & 1u);
            mbar_wait_quiet(bar_second, n_second & 1u);
        }
        __syncwarp();
    } else if (warp >= 2) {
        // ---------------- epilogue ---------------------------------------------------------------------
        const int q = warp & 3, cg = ((warp - 2) % WARPS) >> 2;
        const int row = q * 32 + lane;                                            // TMEM lane, row of the latent tile
        const int sample_row = HALF ? q * 16 + lane : row;                        // sample of the tile (HALF: lanes 0 .. 15)
        const bool mine = !HALF || lane < 16;
        const uint32_t lane_off = static_cast<uint32_t>(q * 32) << 16;
        const uint32_t step = a.st->step;
        // 16 columns at a time, packed over columns that have been read: group 1 from its last ones on, towards the end of its columns
        const int hidden0 = 16 * group_block(cg), batches = group_block(cg + 1) - group_block(cg), first = cg == 1 ? batches - 1 : 0, dir = cg == 1 ? -1 : 1;
        const uint32_t cols = tmem + lane_off + hidden0, packed = tmem + lane_off + packed_col(cg);
        const uint32_t res = tmem + lane_off + acc2_col + kDims * cg;             // this thread's columns of a second result
        const int d0 = kDims * cg;                                                // its latent dimensions
        float* const z_largest = szmax + slot * kGroups * 128 + row;              // [column group][128]: the guide's latent
        float* const t_largest = z_largest + 4 * 128;                             // the transition's
        float gate_own[kDims], lin_own[kDims], G_own[kDims];                      // literal
        uint32_t np = 0, na = 0;
        // A wait that gave up changes nothing here: all lanes and warps take the same way through the work that is left, without purpose and,
        // the abort flag being up, without waiting for long, so that none is missing where the others need it.  (A vote on every
        // result: S=65536 67.9 us instead of 66.3; one per tile: S=8192 28.4 us instead of 27.3.)
        const auto wait = [&](uint32_t bar, uint32_t& n) { mbar_wait_lane(bar, n++ & 1u, abort_flag, a.st); };
        const auto arrive = [&](uint32_t bar) {                     // our reads and writes precede the MMAs that this unblocks
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        const auto store_latent = [&](const float (&z)[kDims]) {
#pragma unroll
            for (int c = 0; c < kDims; c += 4)
                st_shared_v4(t_z + sw128(row, (d0 + c) / 4), tf32_rna(z[c]), tf32_rna(z[c + 1]), tf32_rna(z[c + 2]), tf32_rna(z[c + 3]));
            fence_proxy_async();
            arrive(bar_z);
        };
        for (int tile = tile0; tile < n_tiles; tile += tile_step) {
            const int k = tile * kRows + sample_row;
            const uint32_t sample = a.sample_base + static_cast<uint32_t>(k);
            float z_own[kDims], eps[kDims];
            Philox4 words[kDims / 4];
            const auto draw_words = [&](uint32_t stream) {
#pragma unroll
                for (int c = 0; c < kDims / 4; ++c) words[c] = philox4x32_10(static_cast<uint32_t>(d0 / 4 + c), sample, stream, step, a.key.seed_lo, a.key.seed_hi);
            };
            const auto draw_normals = [&] {
#pragma unroll
                for (int c = 0; c < kDims; c += 4) {
                    float four[4];
                    box_muller_fast(words[c / 4], four);
#pragma unroll
                    for (int i = 0; i < 4; ++i) eps[c + i] = four[i];
                }
            };
            draw_words(0u);                                                       // the first guide step
            draw_normals();
#pragma unroll
            for (int c = 0; c < kDims; ++c) z_own[c] = fmaf(softplus_fast(spt[d0 + c]), eps[c], sct[d0 + c]);
            if (W == 1) put_largest(smem_u32(z_largest + cg * 128), z_own);
            store_latent(z_own);
            float h_inv = 1.0f;                                                   // inverse scale of the hidden layer
            for (int ph = 1; ph < n_phases; ++ph) {
                const float* bias = (ph < W ? sbzs : (ph == W ? sb1 : (ph == W + 1 ? sb3 : sbi1))) + hidden0;
                // the generator's words while the pre-activations are formed: they depend on nothing (literal: the gate draws nothing)
                if (ph != ph_last && (!LITERAL || ph != W)) draw_words(ph < W ? static_cast<uint32_t>(ph) : kStreamTransition);
                // ---- hidden layer: bias, activation, next A operand (or v) -----------------
                wait(bar_p, np);
                tc_fence_after();
                if (HALF && ph < W) {
                    const float* thread_bias = bias + 2 * (lane & 3);
                    uint32_t acc[2][8];
                    if (batches > 0) tmem_ld16_half(cols + 16 * first, acc[0]);
#pragma unroll 1
                    for (int b = 0; b < batches; b += 2) {
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            if (b + u >= batches) break;
                            const int at = first + dir * (b + u);
                            tmem_ld_wait();
                            if (b + u + 1 < batches) tmem_ld16_half(cols + 16 * (at + dir), acc[u ^ 1]);
                            uint32_t w[4];
#pragma unroll
                            for (int g = 0; g < 2; ++g) {
                                const unsigned long long bv = *reinterpret_cast<const unsigned long long*>(thread_bias + 16 * at + 8 * g);
                                w[2 * g] = tanh_pair(acc[u][4 * g], acc[u][4 * g + 1], bv);
                                w[2 * g + 1] = tanh_pair(acc[u][4 * g + 2], acc[u][4 * g + 3], bv);
                            }
                            tmem_st8_half(packed + 8 * at, w);
                        }
                    }
                } else {
                    unsigned long long scale2 = 0;
                    if (ph >= W) {                                  // the column groups' largest |latent| of this sample
                        const float* const largest = ph == ph_last ? t_largest : z_largest;
                        float zm = 0.0f, scale;
#pragma unroll
                        for (int gg = 0; gg < kGroups; ++gg) zm = fmaxf(zm, largest[gg * 128]);
                        const float* bound = ph == ph_last ? a.v_out.bound : a.bounds + 2 * (ph - W);
                        half_scale(1.01f * fmaf(__ldg(bound), zm, __ldg(bound + 1)), scale, h_inv);
                        scale2 = pack2(scale, scale);
                        if (ph == ph_last && cg == 0 && mine && k < a.count) a.v_out.inv_scale[k] = h_inv;
                    }
                    const auto act16 = [&](const uint32_t (&acc)[16], const ulonglong2 (&bv)[4], int at) {
                        uint32_t w[8];
                        if (ph < W) {
                            pack_columns(acc, bv, w, [](uint32_t x0, uint32_t x1, unsigned long long b) { return tanh_pair(x0, x1, b); });
                        } else if (LITERAL && ph == ph_last) {  // u = Wi1 z' + bi1: no activation
                            pack_columns(acc, bv, w, [&](uint32_t x0, uint32_t x1, unsigned long long b) { return scaled_pair<false>(x0, x1, b, scale2); });
                        } else {
                            pack_columns(acc, bv, w, [&](uint32_t x0, uint32_t x1, unsigned long long b) { return scaled_pair<true>(x0, x1, b, scale2); });
                        }
                        if (ph != ph_last) tmem_st8(packed + 8 * at, w);
                        else if (mine && k < a.count) store8(a.v_out.p + static_cast<size_t>(k) * a.v_out.ld + hidden0 + 16 * at, w);   // one sector
                    };
                    uint32_t acc[2][16];
                    ulonglong2 bv[2][4];
                    if constexpr (WARPS == 8) {
                        // 32 columns at a time (D = 16: a group has a multiple of 32): two warps per scheduler keep the special-function pipe busy only with that
                        // many independent values each
#pragma unroll 1
                        for (int b = 0; b < batches; b += 2) {
                            const int at = first + dir * b;
                            tmem_ld16(cols + 16 * at, acc[0]);
                            tmem_ld16(cols + 16 * (at + dir), acc[1]);
                            load_bias(bias + 16 * at, bv[0]);
                            load_bias(bias + 16 * (at + dir), bv[1]);
                            tmem_ld_wait();
                            act16(acc[0], bv[0], at);
                            act16(acc[1], bv[1], at + dir);
                        }
                    } else {
                        if (batches > 0) tmem_ld16(cols + 16 * first, acc[0]);
                        load_bias(bias + 16 * first, bv[0]);
#pragma unroll 1
                        for (int b = 0; b < batches; b += 2) {
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                if (b + u >= batches) break;
                                const int at = first + dir * (b + u);
                                tmem_ld_wait();
                                if (b + u + 1 < batches) {
                                    tmem_ld16(cols + 16 * (at + dir), acc[u ^ 1]);
                                    load_bias(bias + 16 * (at + dir), bv[u ^ 1]);
                                }
                                act16(acc[u], bv[u], at);
                            }
                        }
                    }
                }
                if (ph == ph_last) continue;
                tmem_st_wait();
                arrive(bar_h);
                // ---- second result: the next latent (literal: gate, then G and relu(G), then the scale) ------------
                if (!LITERAL || ph != W) draw_normals();
                wait(bar_acc2, na);
                tc_fence_after();
                uint32_t r0[kDims];
                tmem_ld_dims(res, r0);
                if (ph < W) {
                    // guide: z = mu + softplus(Wsig mu + bsig) * eps
                    uint32_t hi[kDims], lo[kDims];
                    tmem_ld_dims(res + D, hi);
                    tmem_ld_dims(res + 2 * D, lo);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < kDims; ++c) {
                        const int d = d0 + c;
                        const float pre = fmaf(__uint_as_float(hi[c]), sscale[D + d], fmaf(__uint_as_float(lo[c]), sscale[2 * D + d], spt[ph * D + d]));
                        z_own[c] = fmaf(softplus_fast(pre), eps[c], fmaf(__uint_as_float(r0[c]), sscale[d], sct[ph * D + d]));
                    }
                    if (ph == W - 1) put_largest(smem_u32(z_largest + cg * 128), z_own);      // the next layer scales its halves by it
                } else if constexpr (!LITERAL) {
                    uint32_t lv[kDims];
                    tmem_ld_dims(res + D, lv);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < kDims; ++c) {
                        const int d = d0 + c;
                        z_own[c] = fmaf(exp_half_fast(fmaf(__uint_as_float(lv[c]) * h_inv, sscale[4 * D + d], sb2[D + d])), eps[c],
                                        fmaf(__uint_as_float(r0[c]) * h_inv, sscale[3 * D + d], sb2[d]));
                    }
                    put_largest(smem_u32(t_largest + cg * 128), z_own);
                } else {
                    tmem_ld_wait();
                    if (ph == W) {
                        // gate g, and the linear map Wl z + bl from the latent tile (it stays as it is for the proposal)
                        float lin[kDims];
#pragma unroll
                        for (int c = 0; c < kDims; ++c) lin[c] = sbl[d0 + c];
#pragma unroll
                        for (int e4 = 0; e4 < D / 4; ++e4) {
                            const float4 z = ld_shared_v4(t_z + sw128(row, e4));
#pragma unroll
                            for (int c = 0; c < kDims; ++c) {
                                const float4 w = *reinterpret_cast<const float4*>(sWl + (d0 + c) * D + 4 * e4);
                                lin[c] = fmaf(w.w, z.w, fmaf(w.z, z.z, fmaf(w.y, z.y, fmaf(w.x, z.x, lin[c]))));
                            }
                        }
#pragma unroll
                        for (int c = 0; c < kDims; ++c) {
                            gate_own[c] = sigmoid_fast(fmaf(__uint_as_float(r0[c]) * h_inv, sscale[3 * D + d0 + c], sbg2[d0 + c]));
                            lin_own[c] = lin[c];
                        }
                        arrive(bar_z);
                        continue;
                    }
                    // proposal h -> G = (1 - g) * lin + g * h; relu(G) replaces the latent tile for the scale product
#pragma unroll
                    for (int c = 0; c < kDims; ++c) {
                        const float prop = fmaf(__uint_as_float(r0[c]) * h_inv, sscale[4 * D + d0 + c], sbh2[d0 + c]);
                        G_own[c] = fmaf(gate_own[c], prop - lin_own[c], lin_own[c]);
                        z_own[c] = fmaxf(G_own[c], 0.0f);
                    }
                    store_latent(z_own);
                    // z' = G + softplus(Ws relu(G) + bs) * eps
                    wait(bar_acc2, na);
                    tc_fence_after();
                    tmem_ld_dims(res, r0);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < kDims; ++c) z_own[c] = fmaf(softplus_fast(__uint_as_float(r0[c]) + sbs[d0 + c]), eps[c], G_own[c]);
                    put_largest(smem_u32(t_largest + cg * 128), z_own);
                }
                store_latent(z_own);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {                                            // nobody has waited for the last products: let them end (bounded)
        if (warp < kSlots) {
            if (elect_one()) umma_commit(bar_drain);
            __syncwarp();
            mbar_wait_quiet(bar_drain, 0u);
        }
        __syncthreads();
    }
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

}  // namespace tc
}  // namespace cutoff
