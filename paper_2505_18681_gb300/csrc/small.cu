// Small-array path of the dispatcher (Algorithm 5, AdaptivePartitionSort):
// the paper hands arrays below its threshold T_np to a library sort instead
// of running its parallel sorts on them.  On the GPU the device-wide radix
// sort of a few thousand keys is all fixed cost, so arrays of at most
// small_cap keys are sorted by ONE CTA in shared memory in a single launch
// that needs no scratch memory: the keys are loaded into registers, mapped to
// the order-preserving key space, sorted by bins over their own range
// (bin_sort.cuh), mapped back and stored.  Key/value sorts order the keys with
// their input positions, so equal keys keep their input order and each value
// is fetched once at the end (the stable argsort); where the range does not
// separate the keys they take stable radix passes over the range in shared
// memory, or the merge sort of Algorithm 3 (insertion-sorted base runs, then
// pairwise merges with merge-path splits), whichever has fewer rounds.
//
// What bounds it is latency: some ten barriers and the accesses between them.
// The merge sort had six to nine rounds, each a binary search and a serial
// merge per thread; the bins have one scan.  Device time of one sort, from a
// replayed graph: see kSmallRun below for the merge sort's.
#include <cfloat>
#include <type_traits>

#include "evosort.h"
#include "api_internal.h"
#include "bin_sort.cuh"
#include "common.cuh"
#include "smem_sort.cuh"

namespace evosort {
namespace {

constexpr int kSmallThreads = 512;
static_assert(kSmallMax <= 16 * kSmallThreads, "largest compiled shape");
__host__ __device__ constexpr size_t small_up(size_t x) { return (x + 15) / 16 * 16; }
constexpr int kSmallRun = 16;   // longest insertion-sorted base run

// Position of a float key by its value: (value - smallest) * scale.  Floats of
// an even spread crowd into the few bit patterns of the largest exponents, so
// equal stretches of the mapped keys would leave most bins empty; equal
// stretches of the values do not.  Rounding keeps the order: subtraction,
// multiplication and the narrowing of doubles never turn two values around.
// NaNs, which have no value, go to their end of the order, infinities clamp.
template <typename U>
__device__ __forceinline__ float key_value(U k, const KeyMap& map);
template <>
__device__ __forceinline__ float key_value<uint32_t>(uint32_t k, const KeyMap& map) {
    return __uint_as_float(map_inv(k, map));
}
template <>
__device__ __forceinline__ float key_value<uint64_t>(uint64_t k, const KeyMap& map) {
    return __double2float_rn(__longlong_as_double((long long)map_inv(k, map)));
}
template <typename U>
struct ValuePosition {
    static constexpr bool linear = false;
    KeyMap map;
    float low, scale;   // of half the value, so that the widest range stays finite
    bool descending;
    __device__ __forceinline__ uint32_t operator()(U k) const {
        const float f = key_value<U>(k, map);
        if (f != f) return descending ? 0u : 0xFFFFFFFFu;
        const float h = 0.5f * f;
        const float x = (descending ? low - h : h - low) * scale;
        return x <= 0.f ? 0u : (x >= 4294967040.f ? 0xFFFFFFFFu : (uint32_t)x);
    }
};

// KPT keys per thread at most, WPT words of four bins per thread.
template <typename U, bool PAIRS, bool FLT, int KPT, int WPT>
__global__ void __launch_bounds__(kSmallThreads) small_sort_kernel(const U* in, U* out, const uint32_t* vin,
                                                                    uint32_t* vout, int n, KeyMap map, int tins) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NT = kSmallThreads;
    __shared__ BinShared<U, NT> sh;
    // keys, the bins' words or the merge sort's second array, values and
    // input positions or the merge sort's second values
    U* k0 = (U*)smem;
    U* k1 = (U*)(smem + small_up(n * sizeof(U)));
    uint32_t* v0 = (uint32_t*)((char*)k1 + small_up(bin_scratch_bytes(n, (int)sizeof(U), WPT * NT)));
    uint32_t* v1 = v0 + (PAIRS ? n : 0);
    uint16_t* x0 = (uint16_t*)v1;
    uint16_t* counts = (uint16_t*)(v1 + (PAIRS ? n : 0));   // of the radix passes
    const int tid = threadIdx.x;
    U key[KPT];
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        if (i * NT + tid < n) {
            key[i] = in[i * NT + tid];
            if (PAIRS) v0[i * NT + tid] = vin[i * NT + tid];
        }
    }
    bin_zero<NT, WPT>(k1);
#pragma unroll
    for (int i = 0; i < KPT; ++i)
        if (i * NT + tid < n) key[i] = map_fwd(key[i], map);
    U lo, hi;
    block_extent<U, NT, KPT>(key, n, sh, &lo, &hi);   // (its barrier also ends the clearing)
    const unsigned long long width = (unsigned long long)(U)(hi - lo);
    const U* ks;
    if (width == 0) {   // equal keys: in order as they are
        for (int i = tid; i < n; i += NT) {
            out[i] = map_inv(lo, map);
            if (PAIRS) vout[i] = v0[i];   // (written before block_extent's barrier)
        }
        return;
    }
    if (FLT) {
        // smallest and largest finite value, then the same bins by value
        __shared__ float s_f[2][NT / 32];
        float a = INFINITY, b = -INFINITY;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            if (i * NT + tid < n) {
                const float f = key_value<U>(key[i], map);
                if (fabsf(f) < INFINITY) {
                    a = fminf(a, f);
                    b = fmaxf(b, f);
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a = fminf(a, __shfl_xor_sync(0xffffffffu, a, o));
            b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
        }
        if ((tid & 31) == 0) {
            s_f[0][tid >> 5] = a;
            s_f[1][tid >> 5] = b;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) {
            a = fminf(a, s_f[0][w]);
            b = fmaxf(b, s_f[1][w]);
        }
        const bool desc = map.x != 0;
        const float range = 0.5f * b - 0.5f * a;   // negative or NaN if no value is finite: one bin
        const float scale = range > 0.f ? fminf(4294967040.f / range, FLT_MAX) : 0.f;
        const ValuePosition<U> pos{map, 0.5f * (desc ? b : a), scale, desc};
        ks = block_bin_sort<U, NT, KPT, WPT, PAIRS, true>(key, n, lo, width, pos, (uint32_t)(4 * WPT * NT), k0, k1, sh,
                                                          []() {}, x0);
    } else {
        int lz;
        uint32_t mult;
        cut_range_near(width, (uint32_t)(4 * WPT * NT), &lz, &mult);
        ks = block_bin_sort<U, NT, KPT, WPT, PAIRS, true>(key, n, lo, width, KeyPosition<U>{lo, lz}, mult, k0, k1,
                                                          sh, []() {}, x0);
    }
    const uint32_t* vs = v0;
    bool by_position = true;
    if (ks == nullptr) {
        // frequent values, or keys crowded into a small part of their range:
        // radix passes over the range, or the merge rounds where they are fewer
        // (a pass takes about as long as a round: 1.2 us at 1,000 keys)
        __syncthreads();
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (i * NT + tid < n) k0[i * NT + tid] = key[i];
        __syncthreads();
        const int passes = (64 - __clzll((long long)width) + 7) / 8;
        int rounds = 1;
        while ((kSmallRun << rounds) < n) ++rounds;
        const int which = passes <= rounds
                              ? smem_radix_sort<U, PAIRS, NT, KPT>(k0, k1, v0, v1, n, lo, passes, counts, sh.wsum)
                              : smem_merge_sort<U, PAIRS, kSmallRun>(k0, k1, v0, v1, n, tins);
        ks = which ? k1 : k0;
        vs = which ? v1 : v0;
        by_position = false;
    }
    // in place (in == out) is safe: every input was read before the sort
    for (int i = tid; i < n; i += NT) {
        out[i] = map_inv(ks[i], map);
        if (PAIRS) vout[i] = vs[by_position ? (int)x0[i] : i];
    }
}

// Most keys of each compiled shape (keys per thread, words per thread).
#define EVOSORT_SMALL_SHAPES(X) X(2, 4) X(8, 12) X(16, 12)

template <typename U, bool PAIRS, bool FLT, int KPT, int WPT>
cudaError_t launch_small_shape(const void* in, void* out, const uint32_t* vin, uint32_t* vout, int n, KeyMap map,
                               int tins, cudaStream_t s) {
    auto kern = small_sort_kernel<U, PAIRS, FLT, KPT, WPT>;
    auto bytes = [](int m) {
        return small_up(m * sizeof(U)) + small_up(bin_scratch_bytes(m, (int)sizeof(U), WPT * kSmallThreads)) +
               (PAIRS ? (size_t)m * 8 : 0) + (size_t)kSmallThreads / 32 * 512;
    };
    static bool configured = false;
    if (!configured) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)bytes(KPT * kSmallThreads));
        if (e != cudaSuccess) return e;
        configured = true;
    }
    kern<<<1, kSmallThreads, bytes(n), s>>>((const U*)in, (U*)out, vin, vout, n, map, tins);
    return cudaGetLastError();
}

template <typename U, bool PAIRS, bool FLT>
cudaError_t launch_small(const void* in, void* out, const uint32_t* vin, uint32_t* vout, int n, KeyMap map,
                         int tins, cudaStream_t s) {
#define EVOSORT_CASE(K, W) \
    if (n <= K * kSmallThreads) return launch_small_shape<U, PAIRS, FLT, K, W>(in, out, vin, vout, n, map, tins, s);
    EVOSORT_SMALL_SHAPES(EVOSORT_CASE)
#undef EVOSORT_CASE
    return cudaErrorInvalidValue;
}

}  // namespace

int small_sort(const void* in, void* out, const uint32_t* vin, uint32_t* vout, size_t n, int dt, const Plan& pl,
               cudaStream_t s, std::string* err) {
    const int w = dtype_bytes(dt);
    const bool pairs = vout != nullptr;
    if (n > (size_t)kSmallMax) {
        *err = "small-array path: more keys than it holds";
        return EVOSORT_ERR_INVALID;
    }
    const KeyMap map = key_map_for(dt, pl.descending);
    // base runs: the insertion threshold, capped at kSmallRun (runs are
    // insertion-sorted in registers, then merged by every thread): a replayed
    // graph of int32 sorts takes 8.1 us per 1000 keys and 18.2 us per 4096
    // keys with 16-key runs, against 9.0 / 20.8 us with 4-key runs
    const int tins = pl.insertion_threshold > kSmallRun ? kSmallRun : pl.insertion_threshold;
    const int call = prof_call_begin(nullptr, 0, s);
    cudaError_t e;
    {
        ProfScope ps(call, EVOSORT_K_SMALL, -1, 2.0 * (double)n * (w + (pairs ? 4 : 0)), n, s);
        auto go = [&](auto u, auto flt) {
            using U = decltype(u);
            return pairs ? launch_small<U, true, flt.value>(in, out, vin, vout, (int)n, map, tins, s)
                         : launch_small<U, false, flt.value>(in, out, vin, vout, (int)n, map, tins, s);
        };
        switch (dt) {
            case EVOSORT_F32: e = go(uint32_t(), std::true_type()); break;
            case EVOSORT_F64: e = go(uint64_t(), std::true_type()); break;
            default: e = w == 4 ? go(uint32_t(), std::false_type()) : go(uint64_t(), std::false_type());
        }
    }
    prof_call_end(call, s, nullptr);
    count_launches(1);
    if (e != cudaSuccess) {
        *err = std::string("small-array sort launch: ") + cudaGetErrorString(e);
        return EVOSORT_ERR_CUDA;
    }
    return EVOSORT_OK;
}

}  // namespace evosort
