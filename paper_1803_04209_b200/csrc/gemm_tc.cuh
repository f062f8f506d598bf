// The emission of the literal model variant (Section 3.1.3) on the 5th-generation tensor cores (tcgen05), operands as in
// half_operand.cuh:
//   I = Wi2 u + bi2        r = relu(Wj1 I + bj1)        x = I + softplus(Wj2 r + bj2) * eps,      u = Wi1 z' + bi1.
// I = MLP_2(z, Identity, Identity) is affine in u, so the hidden layer of the scale does not need I:
//   Wj1 I + bj1 = (Wj1 Wi2) u + (Wj1 bi2 + bj1) = M u + b',
// with the H x H matrix M and the vector b' formed once when the weights are loaded.  Two kernels remain:
//   k_gemm_relu_tc   r = relu(u M^T + b')                       (K = H instead of K = N)
//   k_emit_dual_tc   x = (u Wi2^T + bi2) + softplus(r Wj2^T + bj2) * eps,  both products in one accumulator.
//
// Both run on the pipeline of emit_tc.cuh: its warp roles, its operands (rows or columns outside the matrices read as zero),
// its accumulators and its bounded waits.  Epilogue warp w reads TMEM lanes 32*(w%4).. and the columns
// 32*cg .. 32*cg+31 and 128+32*cg .. 128+32*cg+31 of the tile, cg = (w-2)/4.
#pragma once
#include "chain_tc.cuh"      // softplus_fast
#include "emit_tc.cuh"
#include "kernels_literal.cuh"

namespace cutoff {
namespace tc {

constexpr int kGemmBN = 256;              // output columns per tile

struct GemmTcArgs {
    const float* bias;      // [Nout]
    const float* a_inv;     // [M] inverse scales of the rows of A
    const float* b_inv;     // [Nout] inverse scales of the rows of B
    HalfRows out;           // relu(A B^T + bias), rounded to tf32 and scaled: the next product's operand.  Its bound per row
                            // follows from A's, whose entries are below 2^15 times their inverse scale
    DevState* st;
    int M, Nout, K;
};

__device__ __forceinline__ void gemm_epilogue_tile(const GemmTcArgs& a, uint32_t taddr, int cg, int row, int lane, int w0,
                                                   uint32_t bar_acc_empty, const float* bias_s, float a_inv) {
    const bool row_ok = row < a.M;
    float scale, inv;
    half_scale(a.out, 32768.0f * a_inv, scale, inv);
    if (row_ok && w0 == 0 && cg == 0) a.out.inv_scale[row] = inv;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        uint32_t bits[2][16];
        tmem_ld16(taddr + 16 * half, bits[0]);
        tmem_ld16(taddr + 128 + 16 * half, bits[1]);
        tmem_ld_wait();
        if (half == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty);    // accumulator is free again
        }
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            const int jw = w0 + 128 * part + cg * 32 + 16 * half;
            if (!row_ok || jw >= a.Nout) continue;
            uint32_t out[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 bv = *reinterpret_cast<const float4*>(bias_s + 32 * part + 16 * half + 4 * i);
                const float4 sv = *reinterpret_cast<const float4*>(bias_s + 64 + 32 * part + 16 * half + 4 * i);
                const float b[4] = {bv.x, bv.y, bv.z, bv.w}, sc[4] = {sv.x, sv.y, sv.z, sv.w};
                float v[4];
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    v[c] = scale * round_tf32(fmaxf(fmaf(__uint_as_float(bits[part][4 * i + c]) * a_inv, sc[c], b[c]), 0.0f));
                out[2 * i] = pack_half2(v[0], v[1]);
                out[2 * i + 1] = pack_half2(v[2], v[3]);
            }
            // rows are a multiple of 8 halves long, the pitch too: whole 16-byte chunks, the last of them short on the ragged edge
            __half* dst = a.out.p + static_cast<size_t>(row) * a.out.ld + jw;
#pragma unroll
            for (int p = 0; p < 2; ++p)
                if (jw + 8 * p < a.out.ld)
                    *reinterpret_cast<uint4*>(dst + 8 * p) = make_uint4(out[4 * p], out[4 * p + 1], out[4 * p + 2], out[4 * p + 3]);
        }
    }
}

__global__ void __launch_bounds__(kThreads, 1) k_gemm_relu_tc(const __grid_constant__ CUtensorMap map_a,
                                                          const __grid_constant__ CUtensorMap map_b, GemmTcArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const Operands<1> o{{&map_a}, {&map_b, &map_b}, {0, kGemmBN / 2}, kGemmBN};
    const Pipeline p = open_pipeline(smem_raw, o, a.st, a.M, ceil_div(a.Nout, kGemmBN), a.K);
    dependency_wait();            // the A operand and the device state are an earlier kernel's
    launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        load_operands(p, o, lane);
    } else if (warp == 1) {
        multiply_operands<1>(p, lane);
    } else {
        const int q = warp & 3, cg = (warp - 2) >> 2;
        read_accumulators(
            p, warp,
            [&](float* table, int wt) {                        // biases and inverse scales of this warp's 2 x 32 columns
                const int j = wt * kGemmBN + cg * 32 + lane;
                table[lane] = j < a.Nout ? __ldg(a.bias + j) : 0.f;
                table[32 + lane] = j + 128 < a.Nout ? __ldg(a.bias + j + 128) : 0.f;
                table[64 + lane] = j < a.Nout ? __ldg(a.b_inv + j) : 0.f;
                table[96 + lane] = j + 128 < a.Nout ? __ldg(a.b_inv + j + 128) : 0.f;
            },
            [&](int m0) { return m0 + q * 32 + lane < a.M ? a.a_inv[m0 + q * 32 + lane] : 1.f; },
            [&](float a_inv, uint32_t taddr, int m0, int wt, uint32_t bar_free, const float* table) {
                gemm_epilogue_tile(a, taddr + cg * 32, cg, m0 + q * 32 + lane, lane, wt * kGemmBN, bar_free, table, a_inv);
            });
    }
    close_pipeline(p);
}

// ---------------------------------------------------------------------------------------------
// x = I + softplus(r Wj2^T + bj2) * eps  with  I = u Wi2^T + bi2, both products in one accumulator, so that I
// never goes through memory (an earlier version wrote I out and read it back element by element in the epilogue of
// the scale product: that alone cost 0.14 ms at N=1024, S=65536).  Tiles of 128 samples x 128 workers; the
// accumulator holds I in columns 0..127 and the scale pre-activation in columns 128..255, from two MMAs per
// K step with different operands: (u, Wi2 rows) and (r, Wj2 rows).  The epilogue is k_emit_tc's with softplus in place of
// exp(logvar / 2).
// ---------------------------------------------------------------------------------------------
struct EmitDualArgs {
    const float* bias_mean;     // bi2 [N]
    const float* bias_scale;    // bj2 [N]
    const float *u_inv, *r_inv; // [count] inverse scales of the samples' rows of u and r
    const float *wi_inv, *wj_inv;   // [N] inverse scales of the rows of Wi2 and Wj2
    float* x;                   // [count][ldx]
    DevState* st;
    NoiseKey key;
    uint32_t sample_base;
    int count, N, H, ldx;
};

// x = I + softplus(scale) * eps
__device__ __forceinline__ void dual_epilogue_tile(const EmitDualArgs& a, uint32_t taddr, int row, int j0, int lane, uint32_t bar_acc_empty,
                                                   const float* table, float u_inv, float r_inv) {
    noise_epilogue_tile(a.x, a.ldx, a.N, row < a.count, row, a.sample_base + static_cast<uint32_t>(row), a.key, table, taddr, j0, lane, bar_acc_empty,
                        [&](const uint32_t (&mean)[8], const uint32_t (&scale)[8], const float (&eps)[2][4], int c8, float (&out)[8]) {
        unsigned long long bm[4], bs[4], im[4], is[4];
        load8(bm, table + c8);
        load8(bs, table + 32 + c8);
        load8(im, table + 64 + c8);
        load8(is, table + 96 + c8);
        const unsigned long long u2 = pack2(u_inv, u_inv), r2 = pack2(r_inv, r_inv);
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
            float s0, s1;
            unpack2(unscale2(scale[c], scale[c + 1], r2, is[c / 2], bs[c / 2]), s0, s1);
            unsigned long long x = unscale2(mean[c], mean[c + 1], u2, im[c / 2], bm[c / 2]);
            fma2(x, pack2(softplus_fast(s0), softplus_fast(s1)), pack2(eps[c / 4][c % 4], eps[c / 4][c % 4 + 1]));
            unpack2(x, out[c], out[c + 1]);
        }
    });
}

__global__ void __launch_bounds__(kThreads, 1) k_emit_dual_tc(const __grid_constant__ CUtensorMap map_u,
                                                               const __grid_constant__ CUtensorMap map_r,
                                                               const __grid_constant__ CUtensorMap map_wi2,
                                                               const __grid_constant__ CUtensorMap map_wj2, EmitDualArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const Operands<2> o{{&map_u, &map_r}, {&map_wi2, &map_wj2}, {0, 0}, kBW};
    const Pipeline p = open_pipeline(smem_raw, o, a.st, a.count, ceil_div(a.N, kBW), a.H);
    dependency_wait();            // the rows of u and r and the device state are an earlier kernel's (no launch_dependents: as in k_emit_tc)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        load_operands(p, o, lane);
    } else if (warp == 1) {
        multiply_operands<2>(p, lane);
    } else {
        const int q = warp & 3, cg = (warp - 2) >> 2;
        const uint32_t step = a.st->step;
        read_accumulators(
            p, warp,
            [&](float* table, int wt) {                        // biases and inverse scales of this warp's 32 workers, the generator's words
                const int j0 = wt * kBW + cg * 32, j = j0 + lane;
                table[lane] = j < a.N ? __ldg(a.bias_mean + j) : 0.f;
                table[32 + lane] = j < a.N ? __ldg(a.bias_scale + j) : 0.f;
                table[64 + lane] = j < a.N ? __ldg(a.wi_inv + j) : 0.f;
                table[96 + lane] = j < a.N ? __ldg(a.wj_inv + j) : 0.f;
                put_noise_columns(table, j0, lane, step, a.key);
            },
            [&](int m0) {
                const int row = m0 + q * 32 + lane;
                return row < a.count ? make_float2(a.u_inv[row], a.r_inv[row]) : make_float2(0.f, 0.f);
            },
            [&](float2 inv, uint32_t taddr, int m0, int wt, uint32_t bar_free, const float* table) {
                dual_epilogue_tile(a, taddr + cg * 32, m0 + q * 32 + lane, wt * kBW + cg * 32, lane, bar_free, table, inv.x, inv.y);
            });
    }
    close_pipeline(p);
}

}  // namespace tc
}  // namespace cutoff
