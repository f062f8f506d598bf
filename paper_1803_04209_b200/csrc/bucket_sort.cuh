// Sorting one row by distribution: count the keys per bucket in shared memory, turn the counts into positions, scatter
// the keys there, and finish with as many odd-even transposition passes as the fullest bucket has keys.
#pragma once
#include <cmath>

#include "async.cuh"
#include "common.cuh"

namespace cutoff {

// Where a key goes: a monotone map onto [0, 1] made of two saturated straight lines, one over the whole range of the
// row and one over its middle (without its outermost 1/32 on either side), so that neither a far outlier nor the dense
// middle of a bell-shaped row crowds a few buckets.  Each step (fused multiply-add, saturation, sum of
// non-decreasing terms) is monotone in the key, rounding included, so a smaller key never gets a later bucket; the map
// only decides how many keys share one.  It is taken from the row the same warp sorted before (its own extremes for
// the first one): the sorted values do not depend on it.
struct BucketMap {
    float s_all, o_all, s_mid, o_mid;
};
constexpr float kMidShare = 0.75f;       // of the buckets; with it a normal row fills its fullest spots evenly

__device__ __forceinline__ void bucket_line(float lo, float hi, float& s, float& o) {
    const float width = hi - lo;
    s = width > 0.0f && width < INFINITY ? __frcp_rn(width) : 0.0f;
    s = s < INFINITY ? s : 0.0f;                     // a width so small that its reciprocal overflows
    o = -lo * s;
    o = fabsf(o) < INFINITY ? o : 0.0f;
}

// Words of the counters: two 16-bit counters each.  A lane owns kBucketWords consecutive words in the prefix sum; an odd
// multiple of 4 makes the lanes' 16-byte accesses fall into different banks.
template <int E> struct BucketShape {
    static constexpr int kLaneWords = E <= 4 ? 4 : (E <= 16 ? 12 : 20);
    static constexpr int kWords = 32 * kLaneWords;
    static constexpr int kSwizzle = E == 32 ? 0x70 : (E == 16 ? 0x30 : (E == 8 ? 0x10 : 0));
};

// Byte address (relative) of sorted position p: lane L later reads positions L*E .. L*E + E - 1 as 16-byte chunks,
// which are XOR-swizzled so that the lanes of a quarter warp read different banks.
template <int E>
__device__ __forceinline__ uint32_t bucket_pos_bytes(uint32_t p) {
    const uint32_t b = p * 4u;
    return BucketShape<E>::kSwizzle ? b ^ ((b >> 3) & BucketShape<E>::kSwizzle) : b;
}
template <int E>
__device__ __forceinline__ int bucket_chunk(int lane, int i) {
    if (E == 32) return i ^ (lane & 7);
    if (E == 16) return i ^ ((lane >> 1) & 3);
    if (E == 8) return i ^ ((lane >> 2) & 1);
    return i;
}

// m: position of the key's counter in quarters of a word: bits 2.. = word, bit 1 = which half.
template <int WORDS>
__device__ __forceinline__ uint32_t bucket_of(float x, const BucketMap& map) {
    const float all = __saturatef(fmaf(x, map.s_all, map.o_all)), mid = __saturatef(fmaf(x, map.s_mid, map.o_mid));
    const float u = fmaf(mid, kMidShare * (WORDS - 0.25f), fmaf(all, (1.0f - kMidShare) * (WORDS - 0.25f), 2097152.0f));
    return __float_as_uint(u) & (4u * 2048u - 1u);
}

__device__ __forceinline__ uint32_t atom_add_shared(uint32_t addr, uint32_t v) {
    uint32_t old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void red_add_shared(uint32_t addr, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// One odd-even transposition step pair over the warp's 32 E keys (lane L holds positions L*E ..).
template <int E>
__device__ __forceinline__ void transpose_pair(float (&v)[E], int lane) {
#pragma unroll
    for (int r = 0; r < E; r += 2) {
        const float a = v[r], c = v[r + 1];
        v[r] = fminf(a, c);
        v[r + 1] = fmaxf(a, c);
    }
    float up = __shfl_down_sync(0xffffffffu, v[0], 1), dn = __shfl_up_sync(0xffffffffu, v[E - 1], 1);
    up = lane == 31 ? INFINITY : up;
    dn = lane == 0 ? -INFINITY : dn;
#pragma unroll
    for (int r = 1; r + 1 < E; r += 2) {
        const float a = v[r], c = v[r + 1];
        v[r] = fminf(a, c);
        v[r + 1] = fmaxf(a, c);
    }
    v[E - 1] = fminf(v[E - 1], up);
    v[0] = fmaxf(v[0], dn);
}

// v: the row's keys, key e = r*32 + lane valid if e < n.  row: 32 E floats of shared memory (may be where the keys came
// from), hist: kWords zeroed words (zero again on exit).  On exit v is sorted, position lane*E + r (beyond n: +infinity).
template <int E, bool FULL>
__device__ __forceinline__ uint32_t warp_bucket_sort(float (&v)[E], uint32_t row, uint32_t hist, int n, int lane, BucketMap map) {
    using S = BucketShape<E>;
    constexpr int LW = S::kLaneWords;
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const uint32_t m = bucket_of<S::kWords>(v[r], map);
        if ((FULL ? 0 : r * 32) + lane < n) red_add_shared(hist + (m & 0x1ffcu), (m & 2u) ? 0x10000u : 1u);
    }
    __syncwarp();
    uint32_t fullest;
    {
        uint32_t c[LW], total = 0, mx = 0;
        const uint32_t mine = hist + lane * LW * 4;
#pragma unroll
        for (int i = 0; i < LW; i += 4)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(c[i]), "=r"(c[i + 1]), "=r"(c[i + 2]), "=r"(c[i + 3]) : "r"(mine + 4 * i) : "memory");
#pragma unroll
        for (int i = 0; i < LW; ++i) {
            const uint32_t w = c[i];
            mx = __vmaxu2(mx, w);
            c[i] = total * 0x10001u + (w << 16);          // exclusive positions of the two buckets, without the lanes before
            total += (w & 0xffffu) + (w >> 16);
        }
        uint32_t inc = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        const uint32_t before = (inc - total) * 0x10001u;
#pragma unroll
        for (int i = 0; i < LW; i += 4)
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(mine + 4 * i), "r"(c[i] + before), "r"(c[i + 1] + before), "r"(c[i + 2] + before), "r"(c[i + 3] + before) : "memory");
        fullest = __reduce_max_sync(0xffffffffu, max(mx & 0xffffu, mx >> 16));
    }
    __syncwarp();
    // the buckets are computed a second time: kept from the first pass they would take E registers more
    asm volatile("" : "+f"(map.s_all), "+f"(map.o_all), "+f"(map.s_mid), "+f"(map.o_mid));
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const uint32_t m = bucket_of<S::kWords>(v[r], map);
        if ((FULL ? 0 : r * 32) + lane < n) {
            const uint32_t old = atom_add_shared(hist + (m & 0x1ffcu), (m & 2u) ? 0x10000u : 1u);
            const uint32_t p = (m & 2u) ? old >> 16 : old & 0xffffu;
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + bucket_pos_bytes<E>(p)), "f"(v[r]) : "memory");
        }
    }
    if (!FULL)
        for (int p = n + lane; p < 32 * E; p += 32) asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + bucket_pos_bytes<E>(p)), "f"(INFINITY) : "memory");
    __syncwarp();
#pragma unroll
    for (int i = 0; i < LW; i += 4)
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(hist + lane * LW * 4 + 4 * i), "r"(0u) : "memory");
#pragma unroll
    for (int i = 0; i < E / 4; ++i)
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[4 * i]), "=f"(v[4 * i + 1]), "=f"(v[4 * i + 2]), "=f"(v[4 * i + 3])
                     : "r"(row + (lane * E + 4 * bucket_chunk<E>(lane, i)) * 4) : "memory");
#pragma unroll 1
    for (uint32_t p = 0; p < fullest; p += 2) transpose_pair<E>(v, lane);
    return fullest;
}

// The map of the next row from a sorted one of n keys.
template <int E, bool FULL>
__device__ __forceinline__ void bucket_map_from_sorted(const float (&v)[E], int n, BucketMap& map) {
    const int last = FULL ? 31 : (n - 1) / E;        // lane of the largest key
    float top = v[E - 1];
    if (!FULL) {
        top = v[0];
#pragma unroll
        for (int r = 1; r < E; ++r) top = v[r] < INFINITY ? v[r] : top;
    }
    bucket_line(__shfl_sync(0xffffffffu, v[0], 0), __shfl_sync(0xffffffffu, top, last), map.s_all, map.o_all);
    bucket_line(__shfl_sync(0xffffffffu, v[0], last > 1 ? 1 : 0), __shfl_sync(0xffffffffu, v[0], last), map.s_mid, map.o_mid);
}

// The first map of a warp: the extremes of the row's own keys.
template <int E, bool FULL>
__device__ __forceinline__ void bucket_map_from_keys(const float (&v)[E], int n, int lane, BucketMap& map) {
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int r = 0; r < E; ++r)
        if (FULL || r * 32 + lane < n) { lo = fminf(lo, v[r]); hi = fmaxf(hi, v[r]); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    bucket_line(lo, hi, map.s_all, map.o_all);
    bucket_line(lo, hi, map.s_mid, map.o_mid);
}

}  // namespace cutoff
