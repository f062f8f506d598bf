// Emission output layer on the 5th-generation tensor cores (tcgen05), with the noise drawn in
// the epilogue:   [mean | logvar] = W4 v + b4,   x_j = mean_j + exp(logvar_j / 2) * eps_j.
//
// One persistent CTA per SM walks over output tiles of 128 samples x 128 workers.  A tile is one
// accumulator of 128 TMEM lanes (samples) x 256 fp32 columns (128 means, then 128 log-variances),
// filled by UMMA instructions of shape M=128, N=256, K=16 in kind::f16: the operands are tf32 (or bf16) values stored as
// halves with a power of two per row taken out (half_operand.cuh), which the epilogue multiplies back.  Operands arrive by TMA
// (plain, per-CTA loads) into a 4-stage ring of 128-byte-swizzled K-major tiles; the accumulator
// is double-buffered (2 x 256 of the 512 TMEM columns) so that the epilogue of one tile runs
// while the next tile is multiplied.
//
// Warp roles: warp 0 issues TMA loads, warp 1 owns TMEM and issues the MMAs, warps 2..17 are the
// epilogue (warp w reads TMEM lanes 32*(w%4).., the 32 workers of column group (w-2)/4).
//
// What bounds it: as four-byte operands it was the stream L2 -> shared memory, 384 KB per tile (N = 1024, S = 65536: 0.148 ms); as
// halves the stream and the tensor time halve and the epilogue sets the pace, about 150 instructions per four draws.
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
constexpr int kStages = 4;
constexpr int kABytes = kBM * kBK * 2;           // 16 KB
constexpr int kBBytes = 2 * kBW * kBK * 2;       // 32 KB: mean rows, then log-variance rows
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kEpiWarps = 16;
constexpr int kThreads = (2 + kEpiWarps) * 32;
constexpr int kTmemCols = 512;
constexpr int kAccCols = 2 * kBW;                // 256 columns per accumulator
constexpr int kTableFloats = 128 + 32;           // per epilogue warp: biases of its 32 + 32 columns, their inverse scales, and the
constexpr int kBiasBytes = kEpiWarps * kTableFloats * 4;   // generator's part of its 8 groups of four workers
constexpr size_t kSmemBytes = kStages * kStageBytes + 1024 /*alignment slack*/ + 256 /*barriers*/ + kBiasBytes;

// instruction descriptor: D = f32, A = B = f16, both K-major, N columns, M rows
constexpr uint32_t instr_desc_f16(uint32_t n, uint32_t m) { return (1u << 4) | ((n >> 3) << 17) | ((m >> 4) << 24); }
constexpr uint32_t kInstrDesc = instr_desc_f16(256, 128);

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

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
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
        float eps[8], out[8];
        normal4_row_column_fast(noise, columns[c8 / 4], key.seed_lo, key.seed_hi, eps);
        normal4_row_column_fast(noise, columns[c8 / 4 + 1], key.seed_lo, key.seed_hi, eps + 4);
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

__device__ __forceinline__ void load8(float (&r)[8], const float* p) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    r[0] = a.x; r[1] = a.y; r[2] = a.z; r[3] = a.w; r[4] = b.x; r[5] = b.y; r[6] = b.z; r[7] = b.w;
}

// x = mean + exp(logvar / 2) * eps.  bias_s: this warp's 32 mean biases, then its 32 log-variance biases, then the inverse scales
// of the same columns, in shared memory (zero beyond worker N).  v_inv: inverse scale of this thread's sample.
__device__ __forceinline__ void emit_epilogue_tile(const EmitArgs& a, uint32_t tmem_base, uint32_t acc, int q, int cg,
                                                   int lane, int m0, int w0, uint32_t bar_acc_empty,
                                                   const float* bias_s, float v_inv) {
    const int row = m0 + q * 32 + lane;
    noise_epilogue_tile(a.x, a.ldx, a.N, row < a.count, row, a.sample_base + static_cast<uint32_t>(row), a.key, bias_s,
                        tmem_base + (static_cast<uint32_t>(q * 32) << 16) + acc * kAccCols + cg * 32, w0 + cg * 32, lane, bar_acc_empty + 8 * acc,
                        [&](const uint32_t (&mean)[8], const uint32_t (&logvar)[8], const float (&eps)[8], int c8, float (&out)[8]) {
        float bm[8], bl[8], sm[8], sl[8];
        load8(bm, bias_s + c8);
        load8(bl, bias_s + 32 + c8);
        load8(sm, bias_s + 64 + c8);
        load8(sl, bias_s + 96 + c8);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            out[c] = fmaf(exp_half_fast(fmaf(__uint_as_float(logvar[c]) * v_inv, sl[c], bl[c])), eps[c],
                          fmaf(__uint_as_float(mean[c]) * v_inv, sm[c], bm[c]));
    });
}

__global__ void __launch_bounds__(kThreads, 1) k_emit_tc(const __grid_constant__ CUtensorMap map_v,
                                                          const __grid_constant__ CUtensorMap map_w4, EmitArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;                     // operand ring, 1024-byte aligned
    const uint32_t bars = tiles + kStages * kStageBytes;
    // barrier layout (8 bytes each): full[4], empty[4], acc_full[2], acc_empty[2], drain; then tmem base, abort flag
    const uint32_t bar_full = bars, bar_empty = bars + 8 * kStages;
    const uint32_t bar_acc_full = bar_empty + 8 * kStages, bar_acc_empty = bar_acc_full + 16;
    const uint32_t bar_drain = bar_acc_empty + 16;
    uint8_t* gen = smem_raw + (tiles - raw) + kStages * kStageBytes;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen + 8 * (2 * kStages + 5));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gen + 8 * (2 * kStages + 5) + 8);
    float* bias_all = reinterpret_cast<float*>(gen + 256);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_tiles_w = ceil_div(a.N, kBW);
    const int n_tiles_m = ceil_div(a.count, kBM);
    // consecutive tiles, samples first: a CTA stays with its workers, whose biases and generator words are staged once or twice
    const int tile_begin = first_tile(blockIdx.x, n_tiles_w * n_tiles_m), tile_end = first_tile(blockIdx.x + 1, n_tiles_w * n_tiles_m);
    const int k_blocks = ceil_div(a.H, kBK);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_acc_full + 8 * b, 1);
            mbar_init(bar_acc_empty + 8 * b, kEpiWarps);
        }
        mbar_init(bar_drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(const_cast<uint32_t*>(tmem_slot))), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    dependency_wait();            // the hidden vectors and the device state are an earlier kernel's
    launch_dependents();

    if (warp == 0) {
        // ---------------- TMA producer ----------------------------------------------------------
        uint32_t stage = 0, phase = 0;
        uint32_t armed_mask = 0, parity_mask = 0;      // per stage: armed at least once / parity of its last phase
        bool ok = true;
        for (int t = tile_begin; ok && t < tile_end; ++t) {
            const int m0 = (t % n_tiles_m) * kBM, w0 = (t / n_tiles_m) * kBW;
            for (int kb = 0; kb < k_blocks; ++kb) {
                ok = mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, a.st);
                if (!ok) break;
                if (lane == 0) {
                    const uint32_t full = bar_full + 8 * stage;
                    const uint32_t dst = tiles + stage * kStageBytes;
                    mbar_arrive_expect_tx(full, kStageBytes);
                    tma_load_2d(dst, &map_v, kb * kBK, m0, full);
                    tma_load_2d(dst + kABytes, &map_w4, kb * kBK, w0, full);
                    tma_load_2d(dst + kABytes + kBBytes / 2, &map_w4, kb * kBK, a.N + w0, full);
                }
                __syncwarp();
                armed_mask |= 1u << stage;
                parity_mask = (parity_mask & ~(1u << stage)) | (phase << stage);
                if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok) {
            // wind down: let every copy that was issued land before the CTA leaves (bounded)
            for (uint32_t s = 0; s < static_cast<uint32_t>(kStages); ++s) {
                if (!((armed_mask >> s) & 1u)) continue;
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(bar_full + 8 * s, (parity_mask >> s) & 1u) && global_ns() - t0 < kWaitLimitNs) {}
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer -------------------------------------------------------------
        uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
        bool ok = true;
        for (int t = tile_begin; ok && t < tile_end; ++t) {
            ok = mbar_wait(bar_acc_empty + 8 * acc, acc_phase ^ 1u, abort_flag, a.st);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * kAccCols;
            for (int kb = 0; kb < k_blocks; ++kb) {
                ok = mbar_wait(bar_full + 8 * stage, phase, abort_flag, a.st);
                if (!ok) break;
                tc_fence_after();
                if (lane == 0) {
                    const uint32_t a_addr = tiles + stage * kStageBytes;
                    const uint64_t a_desc = make_smem_desc(a_addr);
                    const uint64_t b_desc = make_smem_desc(a_addr + kABytes);
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k)         // 16 halves = 32 bytes per instruction
                        umma_f16(d_tmem, a_desc + 2 * k, b_desc + 2 * k, kInstrDesc, (kb | k) != 0);
                    umma_commit(bar_empty + 8 * stage);         // frees the stage when these MMAs are done
                    if (kb == k_blocks - 1) umma_commit(bar_acc_full + 8 * acc);
                }
                __syncwarp();
                if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (!ok) {
            // make sure no MMA is still running before TMEM is released (bounded)
            if (lane == 0) umma_commit(bar_drain);
            __syncwarp();
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(bar_drain, 0u) && global_ns() - t0 < kWaitLimitNs) {}
        }
        __syncwarp();
    } else {
        // ---------------- epilogue ---------------------------------------------------------------
        const int q = warp & 3, cg = (warp - 2) >> 2;
        const uint32_t step = a.st->step;
        float* bias_s = bias_all + (warp - 2) * kTableFloats;
        int w_staged = -1;
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        for (int t = tile_begin; ok && t < tile_end; ++t) {
            const int m0 = (t % n_tiles_m) * kBM, w0 = (t / n_tiles_m) * kBW;
            if (w0 != w_staged) {                       // biases of this warp's 32 workers, read once per worker tile
                const int j = w0 + cg * 32 + lane;
                const float bm = j < a.N ? __ldg(a.b4 + j) : 0.f;
                const float bl = j < a.N ? __ldg(a.b4 + a.N + j) : 0.f;
                const float sm = j < a.N ? __ldg(a.w_inv + j) : 0.f;
                const float sl = j < a.N ? __ldg(a.w_inv + a.N + j) : 0.f;
                __syncwarp();                           // the previous tile's readers are done
                bias_s[lane] = bm;
                bias_s[32 + lane] = bl;
                bias_s[64 + lane] = sm;
                bias_s[96 + lane] = sl;
                put_noise_columns(bias_s, w0 + cg * 32, lane, step, a.key);
                __syncwarp();
                w_staged = w0;
            }
            const int row = m0 + q * 32 + lane;
            const float v_inv = row < a.count ? a.v_inv[row] : 0.f;      // on its way while the accumulator is waited for
            ok = mbar_wait(bar_acc_full + 8 * acc, acc_phase, abort_flag, a.st);
            if (!ok) break;
            tc_fence_after();
            emit_epilogue_tile(a, tmem_base, acc, q, cg, lane, m0, w0, bar_acc_empty, bias_s, v_inv);
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

}  // namespace tc
}  // namespace cutoff
