// Sorting rows by distribution, in shared memory: count the keys per bucket, turn the counts into positions, scatter
// the keys there, read them back as consecutive positions per lane and finish with as many odd-even transposition steps
// as the fullest bucket has keys (keys of different buckets are in order, so no key is further from its place than that).
//
// What bounds it: the shared-memory pipe.  The counting and the scattering touch shared memory three times per key at
// random banks (3.7 wavefronts per warp instruction, measured, atomics and stores alike), about 500 wavefronts per row
// of 1024 keys with the scan and the read-back; the instructions (about 1700 per row against 2930 of the network, of
// which 2 in 3 were min/max) come second.  65536 rows of 1024 keys of the benchmark: 0.253 ms by the register network,
// 0.152 ms this way.
#pragma once
#include <cmath>

#include "async.cuh"
#include "common.cuh"
#include "kernels_sort.cuh"

namespace cutoff {

// Where a key goes: a monotone map onto the counters made of two saturated straight lines, one over the whole range of
// the row and one over its middle (without its outermost 1/32 on either side), so that neither a far outlier nor the
// dense middle of a bell-shaped row crowds a few buckets.  Each operation (fused multiply-add, saturation, sum of
// non-decreasing terms) is monotone in the key, rounding included, so a smaller key never gets a later bucket; the map
// only decides how many keys share one.  It is taken from the row the same warps sorted before (from the extremes of
// its own keys for the first one): the sorted values do not depend on it.
struct BucketMap {
    float s_all, o_all, s_mid, o_mid;
};
constexpr float kMidShare = 0.75f;       // of the buckets

__device__ __forceinline__ void bucket_line(float lo, float hi, float& s, float& o) {
    const float width = hi - lo;
    s = width > 0.0f && width < INFINITY ? __frcp_rn(width) : 0.0f;
    s = s < INFINITY ? s : 0.0f;                     // a width so small that its reciprocal overflows
    o = -lo * s;
    o = fabsf(o) < INFINITY ? o : 0.0f;
}

// Shared-memory byte address of the key's counter.  The sum is formed around 2^21, where a float's last bit is worth a
// quarter: the mantissa then holds 4 x (first counter's word address + word) plus a fraction that is masked off.
// base = 2^21 + (byte address of the counters) / 4; an address below 256 KB keeps the sum inside the binade.
template <int WORDS>
__device__ __forceinline__ uint32_t bucket_of(float x, const BucketMap& map, float base) {
    constexpr float kTop = WORDS - 0.75f;
    const float all = __saturatef(fmaf(x, map.s_all, map.o_all)), mid = __saturatef(fmaf(x, map.s_mid, map.o_mid));
    return __float_as_uint(fmaf(mid, kMidShare * kTop, fmaf(all, (1.0f - kMidShare) * kTop, base))) & 0x3fffcu;
}

// E keys per lane.  A lane owns kLaneWords consecutive counters in the prefix sum; four times an odd number makes the
// lanes' 16-byte accesses fall into different banks, and about 0.9 counters per key is where fewer passes and a longer scan
// balance (1024 keys, 65536 rows: 20 words 0.156 ms with half-word counters, 28 words 0.152, 36 words 0.157).
template <int E> struct BucketShape {
    static constexpr int kLaneWords = E <= 4 ? 4 : (E <= 16 ? 12 : (E <= 24 ? 20 : 28));
    // read-back chunks are XOR-swizzled where 4E bytes per lane would put the lanes of a quarter warp into the same banks
    static constexpr uint32_t kSwizzle = E == 32 ? 0x70u : (E == 16 ? 0x30u : (E == 8 ? 0x10u : 0u));
};

// Address of sorted position p in a row that starts at a multiple of 128 bytes.
template <int E>
__device__ __forceinline__ uint32_t bucket_slot(uint32_t row, uint32_t p) {
    const uint32_t b = row + 4u * p;
    return BucketShape<E>::kSwizzle ? b ^ ((p >> 1) & BucketShape<E>::kSwizzle) : b;
}
// The 16-byte chunk of the lane's own E positions that holds its positions 4i .. 4i + 3.
template <int E>
__device__ __forceinline__ int bucket_chunk(int lane, int i) {
    if (E == 32) return i ^ (lane & 7);
    if (E == 16) return i ^ ((lane >> 1) & 3);
    if (E == 8) return i ^ ((lane >> 2) & 1);
    return i;
}

__device__ __forceinline__ uint32_t atom_add_shared(uint32_t addr, uint32_t v) {
    uint32_t old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void red_add_shared(uint32_t addr, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_f32(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }
__device__ __forceinline__ float lds_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

// Which of a thread's E keys exist: element r * THREADS + thread of a row of n.  E is N / THREADS rounded up to a multiple
// of 4, so only the last four can be missing.
template <int E>
__device__ __forceinline__ bool key_exists(int r, int threads, int thread, int n) {
    return r < E - 4 || r * threads + thread < n;
}

// The lane's counters: read, prefix-summed within the lane, total and fullest returned.
template <int LW>
__device__ __forceinline__ void lane_scan(uint32_t mine, uint32_t (&c)[LW], uint32_t& total, uint32_t& fullest) {
#pragma unroll
    for (int i = 0; i < LW; i += 4)
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(c[i]), "=r"(c[i + 1]), "=r"(c[i + 2]), "=r"(c[i + 3]) : "r"(mine + 4 * i) : "memory");
    total = 0;
    fullest = 0;
#pragma unroll
    for (int i = 0; i < LW; ++i) {
        const uint32_t w = c[i];
        fullest = max(fullest, w);
        c[i] = total;
        total += w;
    }
}
template <int LW>
__device__ __forceinline__ void lane_store_positions(uint32_t mine, const uint32_t (&c)[LW], uint32_t before) {
#pragma unroll
    for (int i = 0; i < LW; i += 4)
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(mine + 4 * i), "r"(c[i] + before), "r"(c[i + 1] + before), "r"(c[i + 2] + before), "r"(c[i + 3] + before) : "memory");
}
__device__ __forceinline__ uint32_t warp_inclusive_sum(uint32_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Two odd-even transposition steps over the warp's 32 E keys (lane L holds positions L*E ..).
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

// Count the thread's keys.  `lane < n` always holds: the predicate keeps the compiler from computing every key's counter
// before it issues the first addition, which would take E registers more (1024 keys: 0.202 ms with the spills, 0.162 without).
template <int E, int WORDS>
__device__ __forceinline__ void bucket_count(const float (&v)[E], const BucketMap& map, float base, int threads, int thread, int n) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const uint32_t a = bucket_of<WORDS>(v[r], map, base);
        if (r < E - 4 ? (thread & 31) < n : r * threads + thread < n) red_add_shared(a, 1u);
    }
}
// Take a position for each key and put it there.  The counters' addresses are formed a second time (see above).
template <int E, int WORDS>
__device__ __forceinline__ void bucket_scatter(const float (&v)[E], BucketMap map, float base, uint32_t row, int threads, int thread, int n) {
    asm volatile("" : "+f"(map.s_all), "+f"(map.o_all), "+f"(map.s_mid), "+f"(map.o_mid));
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const uint32_t a = bucket_of<WORDS>(v[r], map, base);
        if (r < E - 4 ? (thread & 31) < n : r * threads + thread < n) sts_f32(bucket_slot<E>(row, atom_add_shared(a, 1u)), v[r]);
    }
}
// Read the thread's consecutive positions back and clear its counters.
template <int E, int LW>
__device__ __forceinline__ void bucket_read_back(float (&v)[E], uint32_t row, uint32_t mine, int thread) {
#pragma unroll
    for (int i = 0; i < LW; i += 4)
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(mine + 4 * i), "r"(0u) : "memory");
#pragma unroll
    for (int i = 0; i < E / 4; ++i)
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[4 * i]), "=f"(v[4 * i + 1]), "=f"(v[4 * i + 2]), "=f"(v[4 * i + 3])
                     : "r"(row + (thread * E + 4 * bucket_chunk<E>(thread & 31, i)) * 4) : "memory");
}
// The next row's map from a row whose keys stand in the order of their buckets.
template <int E>
__device__ __forceinline__ void bucket_map_from_row(uint32_t row, int n, BucketMap& map) {
    const uint32_t last = n - 1, trim = n >> 5;
    bucket_line(lds_f32(bucket_slot<E>(row, 0)), lds_f32(bucket_slot<E>(row, last)), map.s_all, map.o_all);
    bucket_line(lds_f32(bucket_slot<E>(row, trim)), lds_f32(bucket_slot<E>(row, last - trim)), map.s_mid, map.o_mid);
}
// Extremes of a thread's keys.
template <int E>
__device__ __forceinline__ void key_extremes(const float (&v)[E], int threads, int thread, int n, float& lo, float& hi) {
    lo = INFINITY;
    hi = -INFINITY;
#pragma unroll
    for (int r = 0; r < E; ++r)
        if (key_exists<E>(r, threads, thread, n)) { lo = fminf(lo, v[r]); hi = fmaxf(hi, v[r]); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
}

// Rows the map does not spread (ties, clusters far apart): the register network, on the keys as they stand in the row
// buffer, put back in order.  A call of its own: the keys of the caller need not be kept in registers for it.
// Such a row costs the counting, the scan and one more pass through shared memory than a kernel that only has the network.  32768
// rows, all of them like that, against that kernel: 160 keys 59 and 56 us, 300 keys 107 and 90, 700 keys 185 and 170, 1024 keys 181 and
// 173; of rows the map spreads 40 and 55, 46 and 92, 74 and 170, 92 and 173.  (Not counting the 15 rows after one that was not
// spread took 57, 104, 181 and 176 us, but 1 to 3 % more where all are spread, and half as much again where a few are not.)
template <int E>
__device__ __noinline__ void warp_network_row(uint32_t row, int n, int lane) {
    constexpr int EP = E <= 8 ? 8 : (E <= 16 ? 16 : 32);
    float v[EP];
#pragma unroll
    for (int r = 0; r < EP; ++r) v[r] = r * 32 + lane < n ? lds_f32(row + (r * 32 + lane) * 4) : INFINITY;
    __syncwarp();
    warp_bitonic_sort<float, EP, true>(v, lane);
#pragma unroll
    for (int r = 0; r < EP; ++r)
        if (lane * EP + r < 32 * E) sts_f32(bucket_slot<E>(row, lane * EP + r), v[r]);
    __syncwarp();
}
template <int E>
__device__ __noinline__ void cta_network_row(uint32_t row, float* row_p, int n) {
    const int t = threadIdx.x;
    float v[32];
#pragma unroll
    for (int r = 0; r < 32; ++r) v[r] = r * 128 + t < n ? lds_f32(row + (r * 128 + t) * 4) : INFINITY;
    __syncthreads();
    cta_bitonic_sort<float, 4>(v, row_p);                    // the row buffer holds 4096 keys: it is the exchange buffer
#pragma unroll
    for (int r = 0; r < 32; ++r)
        if (t * 32 + r < 128 * E) sts_f32(bucket_slot<E>(row, t * 32 + r), v[r]);
    __syncthreads();
}

// Up to how many keys in the fullest bucket the transposition steps beat the network (35 against 3000 instructions); for
// rows shared by four warps a bucket must also fit one warp (see below).
constexpr uint32_t kWarpMostPasses = 64, kCtaMostPasses = 32;

// One warp's row of n <= 32 E keys, in shared memory at `row` (128-byte aligned, 32 E floats), counters at `hist`
// (32 * kLaneWords words, zero on entry and on exit).  On exit v holds the sorted positions lane*E + r (+infinity beyond n)
// and nothing in the row buffer is needed any more once `released` has been called.
template <int E, typename Released>
__device__ __forceinline__ void warp_bucket_sort(float (&v)[E], uint32_t row, uint32_t hist, int n, int lane, bool first,
                                                 BucketMap& map, Released released) {
    constexpr int LW = BucketShape<E>::kLaneWords, WORDS = 32 * LW;
    const float base = 2097152.0f + static_cast<float>(hist >> 2);
    const uint32_t mine = hist + lane * LW * 4;
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = key_exists<E>(r, 32, lane, n) ? lds_f32(row + (r * 32 + lane) * 4) : 0.0f;
    if (first) {
        float lo, hi;
        key_extremes<E>(v, 32, lane, n, lo, hi);
        bucket_line(lo, hi, map.s_all, map.o_all);
        map.s_mid = map.s_all;
        map.o_mid = map.o_all;
    }
    bucket_count<E, WORDS>(v, map, base, 32, lane, n);
    __syncwarp();
    uint32_t fullest;
    {
        uint32_t c[LW], total;
        lane_scan<LW>(mine, c, total, fullest);
        lane_store_positions<LW>(mine, c, warp_inclusive_sum(total, lane) - total);
        fullest = __reduce_max_sync(0xffffffffu, fullest);
    }
    __syncwarp();
    if (fullest <= kWarpMostPasses) {
        bucket_scatter<E, WORDS>(v, map, base, row, 32, lane, n);
        for (int p = n + lane; p < 32 * E; p += 32) sts_f32(bucket_slot<E>(row, p), INFINITY);
        __syncwarp();
    } else {
        warp_network_row<E>(row, n, lane);
        fullest = 0;
    }
    bucket_read_back<E, LW>(v, row, mine, lane);
    bucket_map_from_row<E>(row, n, map);
    released();
#pragma unroll 1
    for (uint32_t p = 0; p < fullest; p += 2) transpose_pair<E>(v, lane);
}

// The same for a row shared by the four warps of a CTA: n <= 128 E keys, row buffer of 4096 floats, counters at `hist`
// (128 * kLaneWords words).  `red`: 16 words of shared memory.  A bucket that lies across the border between two warps'
// positions is put in order by one warp beforehand (it has at most 32 keys), so that the transposition steps never have
// to cross a border.  Returns false if any thread says its keys did not arrive.
template <int E, typename Released>
__device__ __forceinline__ bool cta_bucket_sort(float (&v)[E], uint32_t row, float* row_p, uint32_t hist, uint32_t* red, int n,
                                                bool arrived, bool first, BucketMap& map, Released released) {
    constexpr int LW = BucketShape<E>::kLaneWords, WORDS = 128 * LW;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const float base = 2097152.0f + static_cast<float>(hist >> 2);
    const uint32_t mine = hist + t * LW * 4;
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = key_exists<E>(r, 128, t, n) ? lds_f32(row + (r * 128 + t) * 4) : 0.0f;
    if (first) {
        float lo, hi;
        key_extremes<E>(v, 128, t, n, lo, hi);
        if (lane == 0) { red[warp] = __float_as_uint(lo); red[4 + warp] = __float_as_uint(hi); }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 4; ++w) { lo = fminf(lo, __uint_as_float(red[w])); hi = fmaxf(hi, __uint_as_float(red[4 + w])); }
        bucket_line(lo, hi, map.s_all, map.o_all);
        map.s_mid = map.s_all;
        map.o_mid = map.o_all;
    }
    bucket_count<E, WORDS>(v, map, base, 128, t, n);
    if (__syncthreads_or(!arrived)) return false;
    uint32_t c[LW], total, fullest;
    lane_scan<LW>(mine, c, total, fullest);
    const uint32_t inc = warp_inclusive_sum(total, lane);
    fullest = __reduce_max_sync(0xffffffffu, fullest);
    if (lane == 31) { red[8 + warp] = inc; red[12 + warp] = fullest; }
    __syncthreads();
    uint32_t before = inc - total;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        if (w < warp) before += red[8 + w];
        fullest = max(fullest, red[12 + w]);
    }
    lane_store_positions<LW>(mine, c, before);
    __syncthreads();
    if (fullest <= kCtaMostPasses) {
        bucket_scatter<E, WORDS>(v, map, base, row, 128, t, n);
        for (int p = n + t; p < 128 * E; p += 128) sts_f32(bucket_slot<E>(row, p), INFINITY);
        __syncthreads();
        const int border = 32 * E * warp;
        if (warp > 0 && border < n) {
            // every counter now holds the end of its bucket
            const uint32_t a = bucket_of<WORDS>(lds_f32(bucket_slot<E>(row, border)), map, base);
            const uint32_t end = lds_u32(a), begin = a == hist ? 0u : lds_u32(a - 4);
            if (begin < static_cast<uint32_t>(border)) {
                const uint32_t slot = bucket_slot<E>(row, begin + lane);
                const bool has = begin + lane < end;
                float k = has ? lds_f32(slot) : INFINITY;
                float one[1] = {k};
                warp_bitonic_sort<float, 1>(one, lane);
                if (has) sts_f32(slot, one[0]);
            }
        }
        __syncthreads();
    } else {
        cta_network_row<E>(row, row_p, n);
        fullest = 0;
    }
    bucket_read_back<E, LW>(v, row, mine, t);
    bucket_map_from_row<E>(row, n, map);
    released();                                              // holds the barrier behind which the row buffer may be refilled
#pragma unroll 1
    for (uint32_t p = 0; p < fullest; p += 2) transpose_pair<E>(v, lane);
    return true;
}

// ---------------------------------------------------------------------------------------------
// Sort + accumulate, one warp per row, 32 (E - 4) < n <= 32 E.  The next row is requested as soon as the current one has
// left its buffer and lands under the transposition steps.  Running sums in registers; a CTA (one per SM) adds its
// warps in a fixed order and writes one partial row.
// COPY says how rows come in: kBulk by the bulk-copy engine (ldx and the matrix base multiples of 16 bytes), 16 or 4 by
// asynchronous copies of that many bytes per lane (no mbarrier, so no device state to report a timeout to).
// ---------------------------------------------------------------------------------------------
constexpr int kBulk = 0;
// Warps per SM the registers allow: two arrays of E (keys and sums) and about 60 more.  The variant that also sums squares
// (SQ) keeps the same split of the rows, so that the means do not depend on it; its third array is spilled in part.
constexpr int kBucketFewestWarps = 16;
template <int E> constexpr int kBucketWarps = E >= 24 ? kBucketFewestWarps : 24;

template <int E> __host__ __device__ constexpr size_t bucket_warp_floats() { return 32 * (E + BucketShape<E>::kLaneWords); }
template <int E> constexpr size_t bucket_smem_bytes() { return 128 + kBucketWarps<E> * (bucket_warp_floats<E>() * 4 + 8) + 16; }

// Add the CTA's warps position by position: stage[warp][32 E] -> one row of n.
template <int E, int WARPS>
__device__ __forceinline__ void store_partial_row(const float (&acc)[E], float* stage, int n, float* __restrict__ out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();                                   // every buffer is dead: reuse them as the stage
#pragma unroll
    for (int r = 0; r < E; ++r) stage[warp * 32 * E + lane * E + r] = acc[r];
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += WARPS * 32) out[j] = add_warps<WARPS>(stage, 32 * E, j);
}

template <int E, bool SQ, int COPY>
__global__ void __launch_bounds__(kBucketWarps<E> * 32, 1)
k_bucket_sum_warp(const float* __restrict__ x, int ldx, int n, int count, float* __restrict__ partial,
                  float* __restrict__ partial_sq, DevState* st) {
    using namespace cutoff::async;
    extern __shared__ __align__(16) uint8_t sm_bucket[];
    constexpr size_t kWarpFloats = bucket_warp_floats<E>();
    constexpr int kWarps = kBucketWarps<E>;
    float* data = reinterpret_cast<float*>(sm_bucket + (128u - (smem_u32(sm_bucket) & 127u)) % 128u);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t row_s = smem_u32(data + warp * kWarpFloats), hist = row_s + 32 * E * 4;
    uint64_t* bars = reinterpret_cast<uint64_t*>(data + kWarps * kWarpFloats);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + kWarps);
    const uint32_t bar = smem_u32(bars + warp);
    if (COPY == kBulk) {
        if (threadIdx.x == 0) *abort_flag = 0;
        if (lane == 0) {
            mbar_init(bar, 1);
            fence_barrier_init();
            fence_proxy_async();
        }
    }
    for (int i = lane; i < 32 * BucketShape<E>::kLaneWords; i += 32) data[warp * kWarpFloats + 32 * E + i] = 0.0f;
    __syncthreads();
    dependency_wait();            // the sample matrix is an earlier kernel's
    launch_dependents();

    float acc[E], acc_sq[SQ ? E : 1];
#pragma unroll
    for (int r = 0; r < E; ++r) acc[r] = 0.0f;
#pragma unroll
    for (int r = 0; r < (SQ ? E : 1); ++r) acc_sq[r] = 0.0f;
    const int stride = gridDim.x * kWarps, row0 = blockIdx.x + gridDim.x * warp;   // a few rows spread over all SMs
    const auto request = [&](int row) {
        const float* src = x + static_cast<size_t>(row) * ldx;
        if (COPY == kBulk) {
            if (lane == 0) {
                mbar_arrive_expect_tx(bar, static_cast<uint32_t>(ldx) * 4u);
                bulk_load_1d(row_s, src, static_cast<uint32_t>(ldx) * 4u, bar);
            }
        } else if (COPY == 16) {
            for (int e = 4 * lane; e < n; e += 128)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(row_s + 4 * e), "l"(src + e) : "memory");
        } else {
            for (int e = lane; e < n; e += 32)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(row_s + 4 * e), "l"(src + e) : "memory");
        }
    };
    if (row0 < count) request(row0);
    BucketMap map{};
    uint32_t parity = 0;
    for (int row = row0; row < count; row += stride, parity ^= 1u) {
        if (COPY == kBulk) {
            if (!mbar_wait(bar, parity, abort_flag, st)) {
                mbar_wait_quiet(bar, parity);          // wind down: give the copy in flight time to land (bounded)
                break;
            }
        } else {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
        }
        float v[E];
        warp_bucket_sort<E>(v, row_s, hist, n, lane, row == row0, map, [&] {
            if (row + stride < count) {
                if (COPY == kBulk) fence_proxy_async();   // our reads of the buffer before the engine's write
                __syncwarp();
                request(row + stride);
            }
        });
#pragma unroll
        for (int r = 0; r < E; ++r) acc[r] += v[r];
        if (SQ) {
#pragma unroll
            for (int r = 0; r < E; ++r) acc_sq[SQ ? r : 0] = fmaf(v[r], v[r], acc_sq[SQ ? r : 0]);
        }
    }
    store_partial_row<E, kWarps>(acc, data, n, partial + static_cast<size_t>(blockIdx.x) * n);
    if constexpr (SQ) store_partial_row<E, kWarps>(acc_sq, data, n, partial_sq + static_cast<size_t>(blockIdx.x) * n);
}

// ---------------------------------------------------------------------------------------------
// Sort + accumulate, four warps per row, 128 (E - 4) < N <= 128 E; otherwise as above, one partial row per CTA.
// A thread's running sums go through at most kWideRun rows in registers, then into the thread's own totals: of the sums in shared
// memory, of the squares (SQ: there is no room for both) at sq_totals [CTA][128 E].  One chain through all of a CTA's rows, twice
// as long as with the eight CTAs per SM of a register sort, has twice its error (rms relative to the sum of magnitudes, N=4096:
// S=32768 4.4e-9 against 2.2e-9, S=8192 2.3e-9 against 1.3e-9); runs of 8 rows 1.2e-9 and 1.7e-9, of 4 rows 1.1e-9 and 1.3e-9.  The
// decision of N=4096, S=32768 takes 0.4 % longer for it (864 and 868 us); more CTAs instead would cost 10 us in the column sums.
// ---------------------------------------------------------------------------------------------
template <int E> constexpr int kBucketWideCtas = E >= 24 ? 4 : (E >= 16 ? 5 : 6);
constexpr int kWideRun = 4;

template <int E> constexpr size_t bucket_wide_smem_bytes() {
    return 128 + (4096 + 128 * BucketShape<E>::kLaneWords + 128 * E) * 4 + 16 * 4 + 8 + 8;
}

// The thread's entries of a CTA's totals: entry r at total[r * 128] (coalesced, free of conflicts).  What the addition rounds away
// stays in the running sum (Dekker 1971), so that the totals add no error of their own.
template <int E>
__device__ __forceinline__ void add_to_totals(float* total, float (&acc)[E], bool first) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const float old = first ? 0.0f : total[r * 128], sum = old + acc[r];
        total[r * 128] = sum;
        acc[r] = fabsf(sum) < INFINITY ? acc[r] - (sum - old) : 0.0f;
    }
}

template <int E, bool SQ>
__global__ void __launch_bounds__(128, kBucketWideCtas<E>)
k_bucket_sum_cta(const float* __restrict__ x, int ldx, int n, int count, float* __restrict__ partial,
                 float* __restrict__ partial_sq, float* __restrict__ sq_totals, DevState* st) {
    using namespace cutoff::async;
    extern __shared__ __align__(16) uint8_t sm_bucket[];
    constexpr int kCounters = 128 * BucketShape<E>::kLaneWords;
    float* data = reinterpret_cast<float*>(sm_bucket + (128u - (smem_u32(sm_bucket) & 127u)) % 128u);
    const int t = threadIdx.x;
    const uint32_t row_s = smem_u32(data), hist = row_s + 4096 * 4;
    float* total = data + 4096 + kCounters + t;
    uint32_t* red = reinterpret_cast<uint32_t*>(data + 4096 + kCounters + 128 * E);
    float* total_sq = SQ ? sq_totals + static_cast<size_t>(blockIdx.x) * 128 * E + t : nullptr;
    const uint32_t bar = smem_u32(red + 16);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(red + 18);
    const uint32_t row_bytes = static_cast<uint32_t>(ldx) * 4u;
    if (t == 0) {
        *abort_flag = 0;
        mbar_init(bar, 1);
        fence_barrier_init();
        fence_proxy_async();
    }
    for (int i = t; i < kCounters; i += 128) data[4096 + i] = 0.0f;
    __syncthreads();
    dependency_wait();
    launch_dependents();

    float acc[E], acc_sq[SQ ? E : 1];
#pragma unroll
    for (int r = 0; r < E; ++r) acc[r] = 0.0f;
#pragma unroll
    for (int r = 0; r < (SQ ? E : 1); ++r) acc_sq[r] = 0.0f;
    const auto request = [&](int row) {
        if (t == 0) {
            mbar_arrive_expect_tx(bar, row_bytes);
            bulk_load_1d(row_s, x + static_cast<size_t>(row) * ldx, row_bytes, bar);
        }
    };
    const int row0 = blockIdx.x;
    if (row0 < count) request(row0);
    BucketMap map{};
    uint32_t done = 0;                                       // rows; the barrier's parity is that of their number
    for (int row = row0; row < count; row += gridDim.x) {
        const bool arrived = mbar_wait(bar, done & 1u, abort_flag, st);
        float v[E];
        if (!cta_bucket_sort<E>(v, row_s, data, hist, red, n, arrived, row == row0, map, [&] {
                const int next = row + static_cast<int>(gridDim.x);
                fence_proxy_async();
                __syncthreads();
                if (next < count) request(next);
            })) {
            mbar_wait_quiet(bar, done & 1u);
            break;
        }
#pragma unroll
        for (int r = 0; r < E; ++r) acc[r] += v[r];
        if constexpr (SQ) {
#pragma unroll
            for (int r = 0; r < E; ++r) acc_sq[r] = fmaf(v[r], v[r], acc_sq[r]);
        }
        ++done;
        if (done % kWideRun == 0) {
            add_to_totals<E>(total, acc, done == kWideRun);
            if constexpr (SQ) add_to_totals<E>(total_sq, acc_sq, done == kWideRun);
        }
    }
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int j = t * E + r;
        if (j < n) {
            partial[static_cast<size_t>(blockIdx.x) * n + j] = done < kWideRun ? acc[r] : total[r * 128] + acc[r];
            if constexpr (SQ) partial_sq[static_cast<size_t>(blockIdx.x) * n + j] = done < kWideRun ? acc_sq[r] : total_sq[r * 128] + acc_sq[r];
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Test hook: the sorts above, the sorted rows written out instead of summed.  Rows come in by plain copies; a warp (a CTA) sorts
// several rows one after the other, so that a row meets the map of the one before it.
// ---------------------------------------------------------------------------------------------
constexpr int kDebugBucketWarps = 4;

template <int E>
__global__ void __launch_bounds__(kDebugBucketWarps * 32) k_debug_bucket_warp(const float* __restrict__ rows, int n, int n_rows,
                                                                              float* __restrict__ keys) {
    constexpr size_t kWarpFloats = bucket_warp_floats<E>();
    __shared__ __align__(128) float data[kDebugBucketWarps * kWarpFloats];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* const mine = data + warp * kWarpFloats;
    const uint32_t row_s = async::smem_u32(mine), hist = row_s + 32 * E * 4;
    for (int i = lane; i < 32 * BucketShape<E>::kLaneWords; i += 32) mine[32 * E + i] = 0.0f;
    BucketMap map{};
    const int row0 = blockIdx.x * kDebugBucketWarps + warp;
    for (int row = row0; row < n_rows; row += gridDim.x * kDebugBucketWarps) {
        for (int e = lane; e < n; e += 32) mine[e] = rows[static_cast<size_t>(row) * n + e];
        __syncwarp();
        float v[E];
        warp_bucket_sort<E>(v, row_s, hist, n, lane, row == row0, map, [] { __syncwarp(); });
#pragma unroll
        for (int r = 0; r < E; ++r)
            if (lane * E + r < n) keys[static_cast<size_t>(row) * n + lane * E + r] = v[r];
    }
}

template <int E>
__global__ void __launch_bounds__(128) k_debug_bucket_cta(const float* __restrict__ rows, int n, int n_rows, float* __restrict__ keys) {
    constexpr int kCounters = 128 * BucketShape<E>::kLaneWords;
    __shared__ __align__(128) float data[4096 + kCounters];
    __shared__ uint32_t red[16];
    const int t = threadIdx.x;
    for (int i = t; i < kCounters; i += 128) data[4096 + i] = 0.0f;
    BucketMap map{};
    for (int row = blockIdx.x; row < n_rows; row += gridDim.x) {
        for (int e = t; e < n; e += 128) data[e] = rows[static_cast<size_t>(row) * n + e];
        __syncthreads();
        float v[E];
        cta_bucket_sort<E>(v, async::smem_u32(data), data, async::smem_u32(data + 4096), red, n, true, row == static_cast<int>(blockIdx.x), map,
                           [] { __syncthreads(); });
#pragma unroll
        for (int r = 0; r < E; ++r)
            if (t * E + r < n) keys[static_cast<size_t>(row) * n + t * E + r] = v[r];
    }
}

}  // namespace cutoff
