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
// replayed graph, merge sort -> bins: 1,000 uniform int32 keys 8.2 -> 3.1 us,
// 4,096 18.8 -> 5.5, int64 11.1 -> 3.5 and 29.5 -> 7.0, 4,096 int32 pairs 29.9
// -> 6.9; where the bins do not separate the keys (Zipf) 4,096 int32 keys 18.9
// -> 15.3.
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
// A second size of CTA for 32-bit keys alone (64-bit keys and values leave no
// room in 64 registers, or in shared memory).
constexpr int kSmallWideThreads = 1024;
constexpr int kSmallWideKpt = 15;   // (a place in the bins has 14 bits)
__host__ __device__ constexpr size_t small_up(size_t x) { return (x + 15) / 16 * 16; }
constexpr int kSmallRun = 16;   // longest insertion-sorted base run

// KPT keys per thread at most, WPT words of four bins per thread.
template <typename U, bool PAIRS, bool FLT, int NT, int KPT, int WPT>
__global__ void __launch_bounds__(NT) small_sort_kernel(const U* in, U* out, const uint32_t* vin,
                                                                    uint32_t* vout, int n, KeyMap map, int tins) {
    extern __shared__ __align__(16) unsigned char smem[];
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
        // the same bins by value
        __shared__ float s_f[2][NT / 32];
        const auto pos = block_value_position<U, NT, KPT>(key, n, GeneralOut<U>(map), map.x != 0, s_f);
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
        // radix passes over the range, or where they are many, for pairs the
        // merge rounds if they are fewer (a pass takes about as long as a round:
        // 1.2 us at 1,000 keys), for keys alone bitonic runs and their merge rounds
        __syncthreads();
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (i * NT + tid < n) k0[i * NT + tid] = key[i];
        __syncthreads();
        const int bits = 64 - __clzll((long long)width), passes = (bits + 7) / 8;
        // Over a wide range two passes over the leading 16 bits may do: a few
        // frequent values rarely share these.  Tried if the first keys of each
        // warp share them only with equal keys; one look at the neighbours
        // shows whether the keys are in order (16 values, 3,000 int64 keys:
        // 27 us by eight passes, 11 so).
        bool lead = false, sorted = false;
        const bool runs = !PAIRS && NT == kSmallThreads && (n <= 512 || passes > 4 || (passes > 3 && n <= 4096));
        if (passes > 3 && !(runs && n <= 512)) {
            bool other = false;
            const uint32_t m = __ballot_sync(0xffffffffu, tid < n);
            if (tid < n) {
                const uint32_t peers = __match_any_sync(m, digit_of((U)(key[0] - lo), bits - 16, 0xFFFFu));
                other = k0[tid / 32 * 32 + __ffs((int)peers) - 1] != key[0];
            }
            lead = !__syncthreads_or(other);
        }
        int which = 0;
        if (lead) {
            smem_radix_sort<U, PAIRS, NT, KPT>(k0, k1, v0, v1, n, lo, bits - 16, 2, counts, sh.wsum);   // back in k0
            // the few keys that share them and differ: exchanges of neighbours,
            // which keep equal keys in order (90% zeros among 10,000 int32 keys)
            bool quiet = false;
            for (int r = 0; r < 12 && !sorted; ++r) {
                bool moved = false;
                for (int i = 2 * tid + (r & 1); i + 1 < n; i += 2 * NT) {
                    const U a = k0[i], b = k0[i + 1];
                    if (b < a) {
                        k0[i] = b;
                        k0[i + 1] = a;
                        if (PAIRS) {
                            const uint32_t va = v0[i];
                            v0[i] = v0[i + 1];
                            v0[i + 1] = va;
                        }
                        moved = true;
                    }
                }
                const bool still = !__syncthreads_or(moved);
                sorted = still && quiet;   // neither the even nor the odd pairs moved
                quiet = still;
            }
        }
        ks = nullptr;
        if constexpr (!PAIRS && NT == kSmallThreads)
            if (runs && !sorted) ks = smem_sort_any(k0, k1, n);
        if (!sorted && ks == nullptr) {   // (equal keys are still in input order)
            int rounds = 1;
            while ((kSmallRun << rounds) < n) ++rounds;
            which = passes <= rounds
                        ? smem_radix_sort<U, PAIRS, NT, KPT>(k0, k1, v0, v1, n, lo, 0, passes, counts, sh.wsum)
                        : smem_merge_sort<U, PAIRS, kSmallRun>(k0, k1, v0, v1, n, tins);
        }
        if (ks == nullptr) ks = which ? k1 : k0;
        vs = which ? v1 : v0;
        by_position = false;
    }
    // in place (in == out) is safe: every input was read before the sort
    for (int i = tid; i < n; i += NT) {
        out[i] = map_inv(ks[i], map);
        if (PAIRS) vout[i] = vs[by_position ? (int)x0[i] : i];
    }
}

// Most keys of each compiled shape (keys per thread, words per thread); 32-bit
// keys alone have one more, of 1,024 threads.
#define EVOSORT_SMALL_SHAPES(X) X(2, 4) X(8, 12) X(16, 12)

template <typename U, bool PAIRS, bool FLT, int NT, int KPT, int WPT>
cudaError_t launch_small_shape(const void* in, void* out, const uint32_t* vin, uint32_t* vout, int n, KeyMap map,
                               int tins, cudaStream_t s) {
    auto kern = small_sort_kernel<U, PAIRS, FLT, NT, KPT, WPT>;
    auto bytes = [](int m) {
        return small_up(m * sizeof(U)) + small_up(bin_scratch_bytes(m, (int)sizeof(U), WPT * NT)) +
               (PAIRS ? (size_t)m * 8 : 0) + (size_t)NT / 32 * 512;
    };
    static bool configured = false;
    if (!configured) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)bytes(KPT * NT));
        if (e != cudaSuccess) return e;
        configured = true;
    }
    kern<<<1, NT, bytes(n), s>>>((const U*)in, (U*)out, vin, vout, n, map, tins);
    return cudaGetLastError();
}

template <typename U, bool PAIRS, bool FLT>
cudaError_t launch_small(const void* in, void* out, const uint32_t* vin, uint32_t* vout, int n, KeyMap map,
                         int tins, cudaStream_t s) {
#define EVOSORT_CASE(K, W) \
    if (n <= K * kSmallThreads) return launch_small_shape<U, PAIRS, FLT, kSmallThreads, K, W>(in, out, vin, vout, n, map, tins, s);
    EVOSORT_SMALL_SHAPES(EVOSORT_CASE)
#undef EVOSORT_CASE
    if constexpr (sizeof(U) == 4 && !PAIRS)
        if (n <= kSmallWideKpt * kSmallWideThreads)
            return launch_small_shape<U, PAIRS, FLT, kSmallWideThreads, kSmallWideKpt, 12>(in, out, vin, vout, n, map,
                                                                                           tins, s);
    return cudaErrorInvalidValue;
}

}  // namespace

// Against the one-launch radix sort, whose barriers over the grid take it 37 us
// for 32-bit and 57 to 64 us for 64-bit keys at these sizes: 10,000 uniform
// int32 keys 9.5 us, 15,360 12.0, 8,192 uniform int64 keys 11.4, with values
// 15.5.  Keys that the bins do not separate lose to it from some 8,000 on, whatever
// repeats or crowds together in them (int32, one CTA and one launch, us): 8,192 keys
// Zipf 29 and 27, exponential 46 and 33; 12,000 of a thousand small values 27 and 15;
// 15,360 Zipf 46 and 31, half of them equal 54 and 38, magnitudes of every order 56
// and 37.  (The chain of launches that such sorts took before: 75 to 90.)
size_t small_auto_keys(int w, bool pairs) {
    return w == 4 && !pairs ? (size_t)kSmallWideKpt * kSmallWideThreads : (size_t)kSmallMax;
}

int small_sort(const void* in, void* out, const uint32_t* vin, uint32_t* vout, size_t n, int dt, const Plan& pl,
               cudaStream_t s, std::string* err) {
    const int w = dtype_bytes(dt);
    const bool pairs = vout != nullptr;
    if (n > small_auto_keys(w, pairs)) {
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
