// Tiled products C[m][n] = sum_k A(m, k) B(n, k) in fp32, one chain of fused multiply-adds over ascending k per result whatever the
// tile.  An operand is either "k-major" (element (m, k) at m*ld + k) or "m-major" (at k*ld + m), so the three orientations a
// dense layer needs are X W^T, dY W and dY^T X.  With n_seg > 1 the product is a sum of n_seg products over K, segment s at
// p + s * seg; the segments' sums are added in order.
// Slabs of TK k arrive by asynchronous copies, kSlabs in flight (a slab is multiplied in a fraction of the time its copies
// take), and keep the operand's own orientation: k-major rows are read four k at a time, m-major ones several m at a time,
// pitches chosen so that neither conflicts.
#pragma once
#include "common.cuh"

namespace cutoff {
namespace fma32 {

template <int TM_, int TN_, int RM_, int RN_, int TK_> struct Tile {
    static constexpr int TM = TM_, TN = TN_, RM = RM_, RN = RN_, TK = TK_;
    static constexpr int TX = TN / RN, TY = TM / RM, kThreads = TX * TY;
    __host__ __device__ static constexpr int pitch(int t, bool k_major) { return (k_major ? TK : t) + 4; }
    __host__ __device__ static constexpr int floats(int t, bool k_major) { return (k_major ? t : TK) * pitch(t, k_major); }
};
constexpr int kSlabs = 4;

struct Operand {
    const float* p;
    long long ld, seg;
    int rows;            // valid m (the other dimension of the product is bounded by its K)
};
// Four consecutive values of an operand into shared memory, zero where they do not exist.
template <bool VEC>
__device__ __forceinline__ void copy4(uint32_t dst, const float* src, int valid) {
    if (VEC) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid > 0 ? 16 : 0) : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * i), "l"(i < valid ? src + i : src), "r"(i < valid ? 4 : 0) : "memory");
    }
}
__device__ __forceinline__ void copy1(uint32_t dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const float* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void copies_landed() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// n consecutive floats, by all threads of the CTA
__device__ __forceinline__ void copy_vector(float* dst, const float* src, int n) {
    const uint32_t d = smem_addr(dst);
    for (int i = threadIdx.x; i < n; i += blockDim.x) copy1(d + 4 * i, src + i);
}
// rows x cols of a row-major matrix (pitch ld) to shared memory with another pitch, or transposed; a warp per row.  All
// copies are in flight at once: loaded through registers the matrices took longer to arrive than the steps that use them.
__device__ __forceinline__ void copy_matrix(float* dst, int pitch, const float* src, long long ld, int rows, int cols) {
    for (int r = threadIdx.x >> 5; r < rows; r += blockDim.x >> 5) {
        const uint32_t d = smem_addr(dst + r * pitch);
        for (int c = threadIdx.x & 31; c < cols; c += 32) copy1(d + 4 * c, src + r * ld + c);
    }
}
__device__ __forceinline__ void copy_matrix_transposed(float* dst, int pitch, const float* src, long long ld, int rows, int cols) {
    for (int r = threadIdx.x >> 5; r < rows; r += blockDim.x >> 5) {
        const uint32_t d = smem_addr(dst + r);
        for (int c = threadIdx.x & 31; c < cols; c += 32) copy1(d + 4 * c * pitch, src + r * ld + c);
    }
}
// One slab of an operand, T rows (m) x TK k.
template <typename T, int ROWS, bool K_MAJOR, bool VEC>
__device__ __forceinline__ void copy_slab(uint32_t dst, const float* base, long long ld, int rows, int m0, int k0, int K) {
    constexpr int kVecs = ROWS * T::TK / 4, P = T::pitch(ROWS, K_MAJOR);
#pragma unroll
    for (int v = threadIdx.x; v < kVecs; v += T::kThreads) {
        const int r = K_MAJOR ? v / (T::TK / 4) : v / (ROWS / 4), c = K_MAJOR ? v % (T::TK / 4) * 4 : v % (ROWS / 4) * 4;
        const int m = m0 + (K_MAJOR ? r : c), k = k0 + (K_MAJOR ? c : r);
        const int valid = K_MAJOR ? (m < rows ? K - k : 0) : (k < K ? rows - m : 0);
        copy4<VEC>(dst + 4 * (r * P + c), valid > 0 ? base + (K_MAJOR ? m * ld + k : k * ld + m) : base, valid);
    }
}
// r[i][q]: the thread's R values of four consecutive k.  k-major: rows at, at + STEP, ..; m-major: R consecutive from at * R.
template <int R, int STEP, int PITCH, bool K_MAJOR>
__device__ __forceinline__ void load_four_k(float (&r)[R][4], const float* slab, int at, int k) {
    if (K_MAJOR) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const float4 q = *reinterpret_cast<const float4*>(slab + (at + i * STEP) * PITCH + k);
            r[i][0] = q.x; r[i][1] = q.y; r[i][2] = q.z; r[i][3] = q.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float* p = slab + (k + q) * PITCH + at * R;
            if constexpr (R % 4 == 0) {
#pragma unroll
                for (int i = 0; i < R; i += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(p + i);
                    r[i][q] = v.x; r[i + 1][q] = v.y; r[i + 2][q] = v.z; r[i + 3][q] = v.w;
                }
            } else {
                const float2 v = *reinterpret_cast<const float2*>(p);
                r[0][q] = v.x; r[1][q] = v.y;
            }
        }
    }
}
// Tile row (column) of a thread's i-th result.
template <int R, int STEP, bool K_MAJOR>
__device__ __forceinline__ int result_at(int at, int i) { return K_MAJOR ? at + i * STEP : at * R + i; }

template <typename T, bool A_KMAJOR, bool B_KMAJOR> struct Slabs {
    static constexpr int kA = T::floats(T::TM, A_KMAJOR), kB = T::floats(T::TN, B_KMAJOR);
    float f[kSlabs * (kA + kB)];
};

// acc[i][j] = sum over segments and k of A(m0 + .., k) B(n0 + .., k).  copy_b(dst, k0, s) requests B's slab.
template <typename T, bool A_KMAJOR, bool B_KMAJOR, bool VEC, bool SUMS, bool SEGMENTS, typename CopyB>
__device__ __forceinline__ void tile_product(Slabs<T, A_KMAJOR, B_KMAJOR>& sm, const Operand& a, int m0, int K, int n_seg, CopyB copy_b,
                                             float (&acc)[T::RM][T::RN], float& a_sum) {
    using S = Slabs<T, A_KMAJOR, B_KMAJOR>;
    const int tid = threadIdx.x, tx = tid % T::TX, ty = tid / T::TX;
    const uint32_t smem = static_cast<uint32_t>(__cvta_generic_to_shared(sm.f));
    const int per_seg = (K + T::TK - 1) / T::TK, slabs = per_seg * (SEGMENTS ? n_seg : 1);
    int k_req = 0, s_req = 0, buf_req = 0;
    const auto request = [&] {
        if (s_req < (SEGMENTS ? n_seg : 1)) {
            const uint32_t dst = smem + 4 * buf_req * (S::kA + S::kB);
            copy_slab<T, T::TM, A_KMAJOR, VEC>(dst, a.p + (SEGMENTS ? s_req * a.seg : 0), a.ld, a.rows, m0, k_req, K);
            copy_b(dst + 4 * S::kA, k_req, s_req);
            k_req += T::TK;
            if (k_req >= K) { k_req = 0; ++s_req; }
            if (++buf_req == kSlabs) buf_req = 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < kSlabs - 1; ++i) request();
    float total[T::RM][T::RN] = {};
    int buf = 0, left = per_seg;
    for (int it = 0; it < slabs; ++it) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kSlabs - 2) : "memory");
        __syncthreads();                 // the slab is there for everyone, and everyone has finished with the one before it
        request();
        const float* sa = sm.f + buf * (S::kA + S::kB);
        const float* sb = sa + S::kA;
#pragma unroll
        for (int k = 0; k < T::TK; k += 4) {
            float x[T::RM][4], y[T::RN][4];
            load_four_k<T::RM, T::TY, T::pitch(T::TM, A_KMAJOR), A_KMAJOR>(x, sa, ty, k);
            load_four_k<T::RN, T::TX, T::pitch(T::TN, B_KMAJOR), B_KMAJOR>(y, sb, tx, k);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < T::RM; ++i)
#pragma unroll
                    for (int j = 0; j < T::RN; ++j) acc[i][j] = fmaf(x[i][q], y[j][q], acc[i][j]);
        }
        if (SUMS && tid < T::TM) {
#pragma unroll
            for (int k = 0; k < T::TK; ++k) a_sum += sa[k * T::pitch(T::TM, false) + tid];
        }
        if (SEGMENTS && --left == 0) {
            left = per_seg;
#pragma unroll
            for (int i = 0; i < T::RM; ++i)
#pragma unroll
                for (int j = 0; j < T::RN; ++j) { total[i][j] += acc[i][j]; acc[i][j] = 0.f; }
        }
        if (++buf == kSlabs) buf = 0;
    }
    if (SEGMENTS) {
#pragma unroll
        for (int i = 0; i < T::RM; ++i)
#pragma unroll
            for (int j = 0; j < T::RN; ++j) acc[i][j] = total[i][j];
    }
}

}  // namespace fma32
}  // namespace cutoff
