// Emission output layer on the 5th-generation tensor cores (tcgen05), with the noise drawn in
// the epilogue:   [mean | logvar] = W4 v + b4,   x_j = mean_j + exp(logvar_j / 2) * eps_j.
//
// One persistent CTA per SM walks over output tiles of 128 samples x 128 workers.  A tile is one
// accumulator of 128 TMEM lanes (samples) x 256 fp32 columns (128 means, then 128 log-variances),
// filled by UMMA instructions of shape M=128, N=256, K=16 in kind::f16: the operands are tf32 (or bf16) values stored as
// halves with a power of two per row taken out (half_operand.cuh), which the epilogue multiplies back.  The accumulator
// is double-buffered (2 x 256 of the 512 TMEM columns) so that the epilogue of one tile runs while the next tile is multiplied.
//
// Operands arrive by TMA (plain, per-CTA loads) as 128-byte-swizzled K-major tiles of 64 halves.  A CTA's tiles are
// consecutive, samples first, so that it works on the same 128 workers for most of its time.  For H <= 256 their weights
// (32 KB per K block) are loaded once per change of workers and stay in shared memory beside a ring of sample tiles;
// beyond that they would leave no room for the ring, and both operands go through it.
//
// Warp roles: warp 0 issues TMA loads, warp 1 owns TMEM and issues the MMAs, warps 2..17 are the
// epilogue (warp w reads TMEM lanes 32*(w%4).., the 32 workers of column group (w-2)/4).
//
// What bounds it, at N = 1024, S = 65536, H = 256 and at N = 4096, S = 32768, H = 512: as four-byte operands, the stream from
// L2 to shared memory (0.148 and 0.432 ms); as halves, with the weights resident (H = 256) and the
// MMAs issued at their rate, it takes 0.118 and 0.282 ms.  Now no
// single resource: shared-memory and store wavefronts 67 %, issue slots 47 %, special-function pipe 45 %, tensor pipe 29 % (N = 1024).  Shares,
// of an earlier version that took 0.113 and 0.290: streamed weights 0.122 and 0.297, the drawing alone, without operands and
// products, 0.104 and 0.200, without the stores 0.111 and 0.295, without the products 0.112 and 0.241.
// 28 epilogue warps of 64 registers, with the generator's words in tables of the whole CTA, were slower (0.142 and 0.330 ms):
// more instructions for the indexing than the occupancy gives.
//
// Every wait on an mbarrier is bounded: after about two seconds it records kErrTimeout in the
// device state, raises a CTA-wide abort flag and the kernel winds down (outstanding copies are
// waited for, again bounded, and TMEM is released).
#pragma once
#include <cuda.h>

#include "async.cuh"
#include "common.cuh"
#include "half_operand.cuh"
#include "rng.cuh"

namespace cutoff {
namespace tc {

using namespace cutoff::async;

constexpr int kBM = 128;                 // samples per tile (TMEM lanes)
constexpr int kBW = 128;                 // workers per tile
constexpr int kBK = 64;                  // halves per 128-byte swizzle row
constexpr int kABytes = kBM * kBK * 2;           // 16 KB
constexpr int kBBytes = 2 * kBW * kBK * 2;       // 32 KB: two blocks of 128 rows (mean rows, then log-variance rows)
constexpr int kMaxStages = 8;
constexpr int kMaxResident = 4;                  // K blocks of weights that can stay in shared memory (H <= 256)
constexpr int kOperandBytes = 13 * kABytes;      // 208 KB of shared memory for operands
constexpr int kEpiWarps = 16;
constexpr int kThreads = (2 + kEpiWarps) * 32;
constexpr int kTmemCols = 512;
constexpr int kAccCols = 2 * kBW;                // 256 columns per accumulator
constexpr int kTableFloats = 128 + 32;           // per epilogue warp: biases of its 32 + 32 columns, their inverse scales, and the
constexpr int kBiasBytes = kEpiWarps * kTableFloats * 4;   // generator's part of its 8 groups of four workers
constexpr size_t kSmemBytes = kOperandBytes + 1024 /*alignment slack*/ + 256 /*barriers*/ + kBiasBytes;

// instruction descriptor: D = f32, A = B = f16, both K-major, N columns, M rows
__host__ __device__ constexpr uint32_t instr_desc_f16(uint32_t n, uint32_t m) { return (1u << 4) | ((n >> 3) << 17) | ((m >> 4) << 24); }

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}

// K-major operand tile, 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);      // start address
    d |= static_cast<uint64_t>(1) << 16;                           // leading byte offset (unused here)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;                   // stride byte offset
    d |= static_cast<uint64_t>(1) << 46;                           // descriptor version
    d |= static_cast<uint64_t>(2) << 61;                           // SWIZZLE_128B
    return d;
}

// True in one lane of the warp, always the same; takes all 32 lanes.  MMAs are issued from a branch on it: their operands are uniform
// registers, and only of such a branch does the compiler know that one thread runs it; from a branch on a lane number every MMA takes longer to
// issue (emission at N = 4096, S = 32768, H = 512: 301 us so, 282 with the election; of the literal networks at N = 1024, S = 65536: 165 and
// 152; N = 1024, H = 256: 121 and 119; the chain of D = 32, H = 512, S = 32768: 174 and 162).
__device__ __forceinline__ bool elect_one() {
    uint32_t yes;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(yes));
    return yes != 0;
}
__device__ __forceinline__ void umma_tf32(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// One 256-bit store: eight consecutive floats at a 32-byte aligned address.
__device__ __forceinline__ void store8(float* p, const float* v) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}

// Tiles of CTA b of the grid: first_tile(b) .. first_tile(b + 1) - 1, as equal as they can be.
__device__ __forceinline__ int first_tile(unsigned b, int total) { return static_cast<int>(static_cast<unsigned long long>(total) * b / gridDim.x); }

struct EmitArgs {
    const float* b4;        // [2N]
    const float* v_inv;     // [count] inverse scales of the samples' hidden vectors
    const float* w_inv;     // [2N] inverse scales of the rows of W4
    float* x;               // [count][ldx]
    DevState* st;
    NoiseKey key;
    uint32_t sample_base;
    int count, N, H, ldx;
};

// Epilogue of one 128 x 128 output tile for one warp: 32 samples (its TMEM lanes) x 32 workers, eight workers at a time.
// The noise of the eight is drawn while their accumulators are on their way from tensor memory, without a branch between
// the two generator calls: the generator is a chain of ten dependent rounds, and one call after the other, behind the loads,
// left the issue slots 54 % empty (N = 1024, S = 65536: 0.165 ms with half-precision operands).
// finish(first 8 columns' words, second 8 columns' words, 8 normals, column of the warp, 8 results): the variant's own arithmetic.
template <typename Finish>
__device__ __forceinline__ void noise_epilogue_tile(float* __restrict__ x, int ldx, int N, bool row_ok, int row, uint32_t sample, NoiseKey key,
                                                    const float* table, uint32_t taddr, int jw0, int lane, uint32_t bar_acc_empty, Finish finish) {
    const PhiloxRow noise = philox_row(sample, kStreamEmission, key.seed_lo);
    const uint4* columns = reinterpret_cast<const uint4*>(table + 128);
#pragma unroll
    for (int c8 = 0; c8 < 32; c8 += 8) {
        uint32_t lo[8], hi[8];
        tmem_ld8(taddr + c8, lo);
        tmem_ld8(taddr + kBW + c8, hi);
        const int jw = jw0 + c8;
        float eps[2][4], out[8];
        normal4_row_column_fast(noise, columns[c8 / 4], key.seed_lo, key.seed_hi, eps[0]);
        normal4_row_column_fast(noise, columns[c8 / 4 + 1], key.seed_lo, key.seed_hi, eps[1]);
        tmem_ld_wait();
        if (c8 == 24) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty);              // accumulator is free again
        }
        finish(lo, hi, eps, c8, out);
        if (!row_ok || jw >= N) continue;
        // whole sectors (the row pitch is a multiple of 8 floats), 16-byte or scalar stores on the ragged edge
        float* dst = x + static_cast<size_t>(row) * ldx + jw;
        if (jw + 7 < N) {
            store8(dst, out);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (jw + i < N) dst[i] = out[i];
        }
    }
}

// The generator's column words of a warp's 32 workers from j0 on (j0 a multiple of 32): lanes 0 .. 7.
__device__ __forceinline__ void put_noise_columns(float* table, int j0, int lane, uint32_t step, NoiseKey key) {
    if (lane < 8)
        reinterpret_cast<uint4*>(table + 128)[lane] = philox_column(static_cast<uint32_t>((j0 >> 2) + lane), kStreamEmission, step, key.seed_lo, key.seed_hi);
}

// Eight floats of a table as pairs.
__device__ __forceinline__ void load8(unsigned long long (&r)[4], const float* p) {
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p), b = *reinterpret_cast<const ulonglong2*>(p + 4);
    r[0] = a.x; r[1] = a.y; r[2] = b.x; r[3] = b.y;
}
// acc * row * column + bias of two accumulators, in this order.
__device__ __forceinline__ unsigned long long unscale2(uint32_t acc0, uint32_t acc1, unsigned long long row, unsigned long long column, unsigned long long bias) {
    fma2(bias, mul2(pack2(__uint_as_float(acc0), __uint_as_float(acc1)), row), column);
    return bias;
}

// A warp's table for the 32 workers from j0 on: mean and log-variance biases, then the inverse scales of the same rows of W4
// (zero beyond worker N), then the generator's column words.
__device__ __forceinline__ void stage_emission_tables(const EmitArgs& a, float* table, int j0, int lane, uint32_t step) {
    const int j = j0 + lane;
    table[lane] = j < a.N ? __ldg(a.b4 + j) : 0.f;
    table[32 + lane] = j < a.N ? __ldg(a.b4 + a.N + j) : 0.f;
    table[64 + lane] = j < a.N ? __ldg(a.w_inv + j) : 0.f;
    table[96 + lane] = j < a.N ? __ldg(a.w_inv + a.N + j) : 0.f;
    put_noise_columns(table, j0, lane, step, a.key);
}

// x = mean + exp(logvar / 2) * eps for one warp's 32 samples x 32 workers from j0 on.  v_inv: inverse scale of this thread's sample.
__device__ __forceinline__ void emit_epilogue_tile(const EmitArgs& a, uint32_t taddr, int row, int j0, int lane, uint32_t bar_acc_empty,
                                                   const float* table, float v_inv) {
    noise_epilogue_tile(a.x, a.ldx, a.N, row < a.count, row, a.sample_base + static_cast<uint32_t>(row), a.key, table, taddr, j0, lane, bar_acc_empty,
                        [&](const uint32_t (&mean)[8], const uint32_t (&logvar)[8], const float (&eps)[2][4], int c8, float (&out)[8]) {
        unsigned long long bm[4], bl[4], sm[4], sl[4];
        load8(bm, table + c8);
        load8(bl, table + 32 + c8);
        load8(sm, table + 64 + c8);
        load8(sl, table + 96 + c8);
        const unsigned long long row_inv = pack2(v_inv, v_inv);
#pragma unroll
        for (int c = 0; c < 8; c += 2)
            unpack2(scale_noise2(unscale2(logvar[c], logvar[c + 1], row_inv, sl[c / 2], bl[c / 2]), eps[c / 4][c % 4], eps[c / 4][c % 4 + 1],
                                 unscale2(mean[c], mean[c + 1], row_inv, sm[c / 2], bm[c / 2])), out[c], out[c + 1]);
    });
}

// The pipeline that the kernels of this file and of gemm_tc.cuh share: operands -> MMA -> double-buffered accumulators.
// A tile is 128 rows of the A operand(s) by two blocks of 128 rows of B.  With one A operand both blocks are one MMA of
// N = 256; with two, the first meets the first block and the second the second, each an MMA of N = 128.
template <int A>
struct Operands {
    const CUtensorMap* a[A];
    const CUtensorMap* b[2];
    int b_row[2];                        // first row of each block of B, for worker tile 0
    int b_step;                          // rows from one worker tile to the next
};

struct Pipeline {
    uint32_t tiles, bars, tmem_base;
    volatile int* abort_flag;
    DevState* st;
    int k_blocks, stages, stage_bytes, tile_begin, tile_end, n_tiles_m;
    bool resident;                       // the weights stay in shared memory, at the front of the operand area
    float* tables;                       // [kEpiWarps][kTableFloats]

    __device__ __forceinline__ uint32_t full(uint32_t s) const { return bars + 8 * s; }
    __device__ __forceinline__ uint32_t empty(uint32_t s) const { return bars + 8 * (kMaxStages + s); }
    __device__ __forceinline__ uint32_t acc_full(uint32_t b) const { return bars + 8 * (2 * kMaxStages + b); }
    __device__ __forceinline__ uint32_t acc_empty(uint32_t b) const { return bars + 8 * (2 * kMaxStages + 2 + b); }
    __device__ __forceinline__ uint32_t w_full(uint32_t kb) const { return bars + 8 * (2 * kMaxStages + 4 + kb); }
    __device__ __forceinline__ uint32_t w_empty() const { return bars + 8 * (2 * kMaxStages + 4 + kMaxResident); }
    __device__ __forceinline__ uint32_t drain() const { return bars + 8 * (2 * kMaxStages + 5 + kMaxResident); }
    __device__ __forceinline__ uint32_t ring(uint32_t s) const { return tiles + (resident ? k_blocks * kBBytes : 0) + s * stage_bytes; }
};
constexpr int kBarriers = 2 * kMaxStages + 6 + kMaxResident;
static_assert(8 * kBarriers + 16 <= 256, "barriers, tensor-memory address and abort flag");

// One K block of weights: the two blocks of 128 rows of worker tile wt.
template <int A>
__device__ __forceinline__ void load_weight_block(const Operands<A>& o, uint32_t dst, int kb, int wt, uint32_t bar) {
    tma_load_2d(dst, o.b[0], kb * kBK, o.b_row[0] + wt * o.b_step, bar);
    tma_load_2d(dst + kBBytes / 2, o.b[1], kb * kBK, o.b_row[1] + wt * o.b_step, bar);
}
// All K blocks of worker tile wt into their place at the front of the operand area (one thread).
template <int A>
__device__ __forceinline__ void load_weights(const Pipeline& p, const Operands<A>& o, int wt) {
    for (int kb = 0; kb < p.k_blocks; ++kb) {
        mbar_arrive_expect_tx(p.w_full(kb), kBBytes);
        load_weight_block(o, p.tiles + kb * kBBytes, kb, wt, p.w_full(kb));
    }
}

// Everything before the first wait: barriers, tensor memory, and the weights of the first tile (they are nobody's output).
template <int A>
__device__ __forceinline__ Pipeline open_pipeline(uint8_t* smem_raw, const Operands<A>& o, DevState* st, int rows, int n_tiles_w, int K) {
    Pipeline p;
    const uint32_t raw = smem_u32(smem_raw);
    p.tiles = (raw + 1023u) & ~1023u;                                  // 1024-byte aligned
    p.bars = p.tiles + kOperandBytes;
    uint8_t* gen = smem_raw + (p.tiles - raw) + kOperandBytes;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen + 8 * kBarriers);
    p.abort_flag = reinterpret_cast<volatile int*>(gen + 8 * kBarriers + 8);
    p.tables = reinterpret_cast<float*>(gen + 256);
    p.st = st;
    p.n_tiles_m = ceil_div(rows, kBM);
    p.tile_begin = first_tile(blockIdx.x, n_tiles_w * p.n_tiles_m);
    p.tile_end = first_tile(blockIdx.x + 1, n_tiles_w * p.n_tiles_m);
    p.k_blocks = ceil_div(K, kBK);
    p.resident = p.k_blocks <= kMaxResident;
    p.stage_bytes = A * kABytes + (p.resident ? 0 : kBBytes);
    p.stages = min(kMaxStages, (kOperandBytes - (p.resident ? p.k_blocks * kBBytes : 0)) / p.stage_bytes);

    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(p.full(s), 1);
            mbar_init(p.empty(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(p.acc_full(b), 1);
            mbar_init(p.acc_empty(b), kEpiWarps);
        }
        for (int kb = 0; kb < kMaxResident; ++kb) mbar_init(p.w_full(kb), 1);
        mbar_init(p.w_empty(), 1);
        mbar_init(p.drain(), 1);
        *p.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (p.resident && p.tile_begin < p.tile_end) load_weights(p, o, p.tile_begin / p.n_tiles_m);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(const_cast<uint32_t*>(tmem_slot))), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    p.tmem_base = *tmem_slot;
    return p;
}

__device__ __forceinline__ void close_pipeline(const Pipeline& p) {
    tc_fence_before();
    __syncthreads();
    if ((threadIdx.x >> 5) == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(p.tmem_base), "r"(kTmemCols) : "memory");
    }
}

// Warp 0: the TMA loads.
template <int A>
__device__ __forceinline__ void load_operands(const Pipeline& p, const Operands<A>& o, int lane) {
    uint32_t stage = 0, phase = 0;
    uint32_t armed_mask = 0, parity_mask = 0;      // per stage: armed at least once / parity of its last phase
    int w_tile = p.tile_begin / p.n_tiles_m;       // the worker tile whose weights are resident
    uint32_t w_loads = 1;
    bool ok = true;
    for (int t = p.tile_begin; ok && t < p.tile_end; ++t) {
        const int m0 = (t % p.n_tiles_m) * kBM, wt = t / p.n_tiles_m;
        if (p.resident && wt != w_tile) {
            ok = mbar_wait(p.w_empty(), (w_loads + 1) & 1u, p.abort_flag, p.st);     // the previous worker tile's products are done
            if (!ok) break;
            if (lane == 0) load_weights(p, o, wt);
            __syncwarp();
            w_tile = wt;
            ++w_loads;
        }
        for (int kb = 0; kb < p.k_blocks; ++kb) {
            ok = mbar_wait(p.empty(stage), phase ^ 1u, p.abort_flag, p.st);
            if (!ok) break;
            if (lane == 0) {
                const uint32_t dst = p.ring(stage);
                mbar_arrive_expect_tx(p.full(stage), p.stage_bytes);
#pragma unroll
                for (int i = 0; i < A; ++i) tma_load_2d(dst + i * kABytes, o.a[i], kb * kBK, m0, p.full(stage));
                if (!p.resident) load_weight_block(o, dst + A * kABytes, kb, wt, p.full(stage));
            }
            __syncwarp();
            armed_mask |= 1u << stage;
            parity_mask = (parity_mask & ~(1u << stage)) | (phase << stage);
            if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
        }
    }
    if (!ok) {
        // wind down: let every copy that was issued land before the CTA leaves (bounded)
        for (int s = 0; s < p.stages; ++s)
            if ((armed_mask >> s) & 1u) mbar_wait_quiet(p.full(s), (parity_mask >> s) & 1u);
        if (p.resident)
            for (int kb = 0; kb < p.k_blocks; ++kb) mbar_wait_quiet(p.w_full(kb), (w_loads + 1) & 1u);
    }
}

// Warp 1: the MMAs.
template <int A>
__device__ __forceinline__ void multiply_operands(const Pipeline& p, int lane) {
    uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0, w_phase = 0;
    bool ok = true;
    for (int t = p.tile_begin; ok && t < p.tile_end; ++t) {
        ok = mbar_wait(p.acc_empty(acc), acc_phase ^ 1u, p.abort_flag, p.st);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = p.tmem_base + acc * kAccCols;
        const bool first_use = t == p.tile_begin || t % p.n_tiles_m == 0;                     // of this worker tile's weights
        const bool last_use = t + 1 < p.tile_end && (t + 1) % p.n_tiles_m == 0;
        for (int kb = 0; kb < p.k_blocks; ++kb) {
            ok = (!p.resident || !first_use || mbar_wait(p.w_full(kb), w_phase, p.abort_flag, p.st)) &&
                 mbar_wait(p.full(stage), phase, p.abort_flag, p.st);
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t a_addr = p.ring(stage), b_addr = p.resident ? p.tiles + kb * kBBytes : a_addr + A * kABytes;
                const uint64_t a_desc = make_smem_desc(a_addr), b_desc = make_smem_desc(b_addr);
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k) {           // 16 halves = 32 bytes per instruction
                    if constexpr (A == 1) {
                        umma_f16(d_tmem, a_desc + 2 * k, b_desc + 2 * k, instr_desc_f16(256, 128), (kb | k) != 0);
                    } else {
                        umma_f16(d_tmem, a_desc + 2 * k, b_desc + 2 * k, instr_desc_f16(128, 128), (kb | k) != 0);
                        umma_f16(d_tmem + kBW, a_desc + (kABytes >> 4) + 2 * k, b_desc + (kBBytes >> 5) + 2 * k, instr_desc_f16(128, 128),
                                 (kb | k) != 0);
                    }
                }
                umma_commit(p.empty(stage));                   // frees the stage when these MMAs are done
                if (kb == p.k_blocks - 1) {
                    umma_commit(p.acc_full(acc));
                    if (p.resident && last_use) umma_commit(p.w_empty());
                }
            }
            __syncwarp();
            if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
        }
        if (first_use) w_phase ^= 1u;
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (!ok) {
        // make sure no MMA is still running before TMEM is released (bounded)
        if (elect_one()) umma_commit(p.drain());
        __syncwarp();
        mbar_wait_quiet(p.drain(), 0u);
    }
    __syncwarp();
}

// Warps 2..17.  stage_tables(table, worker tile): this warp's tables, once per worker tile.
// row_values(first row): what belongs to this thread's row, on its way while the accumulator is waited for.
// tile(row values, accumulator's tensor-memory address of this warp's lanes, first row, worker tile, "accumulator free" barrier, table).
template <typename StageTables, typename RowValues, typename Tile>
__device__ __forceinline__ void read_accumulators(const Pipeline& p, int warp, StageTables stage_tables, RowValues row_values, Tile tile) {
    float* table = p.tables + (warp - 2) * kTableFloats;
    const uint32_t lanes = p.tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    int staged = -1;
    uint32_t acc = 0, acc_phase = 0;
    for (int t = p.tile_begin; t < p.tile_end; ++t) {
        const int m0 = (t % p.n_tiles_m) * kBM, wt = t / p.n_tiles_m;
        if (wt != staged) {
            __syncwarp();                                      // the previous tile's readers are done
            stage_tables(table, wt);
            __syncwarp();
            staged = wt;
        }
        const auto values = row_values(m0);
        if (!mbar_wait(p.acc_full(acc), acc_phase, p.abort_flag, p.st)) break;
        tc_fence_after();
        tile(values, lanes + acc * kAccCols, m0, wt, p.acc_empty(acc), table);
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
}

__global__ void __launch_bounds__(kThreads, 1) k_emit_tc(const __grid_constant__ CUtensorMap map_v,
                                                          const __grid_constant__ CUtensorMap map_w4, EmitArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const Operands<1> o{{&map_v}, {&map_w4, &map_w4}, {0, a.N}, kBW};
    const Pipeline p = open_pipeline(smem_raw, o, a.st, a.count, ceil_div(a.N, kBW), a.H);
    // no launch_dependents: a row sort with several CTAs per SM would place them as the SMs come free, unevenly (N=4096, S=32768:
    // 858 us per decision with it, 851 without; N=2175: 139.2 and 137.8; with one CTA per SM no difference)
    dependency_wait();            // the hidden vectors and the device state are an earlier kernel's
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        load_operands(p, o, lane);
    } else if (warp == 1) {
        multiply_operands<1>(p, lane);
    } else {
        const int q = warp & 3, cg = (warp - 2) >> 2;
        const uint32_t step = a.st->step;
        read_accumulators(
            p, warp, [&](float* table, int wt) { stage_emission_tables(a, table, wt * kBW + cg * 32, lane, step); },
            [&](int m0) { return m0 + q * 32 + lane < a.count ? a.v_inv[m0 + q * 32 + lane] : 0.f; },
            [&](float v_inv, uint32_t taddr, int m0, int wt, uint32_t bar_free, const float* table) {
                emit_epilogue_tile(a, taddr + cg * 32, m0 + q * 32 + lane, wt * kBW + cg * 32, lane, bar_free, table, v_inv);
            });
    }
    close_pipeline(p);
}

}  // namespace tc
}  // namespace cutoff
