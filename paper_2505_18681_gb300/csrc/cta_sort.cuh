// Sort of one long run of keys by one CTA (keys only): segments of a batch
// that shared memory does not hold, and buckets of the partition sort that
// came out too large for it.
//
//   cta_vote         says by a sample which of the two below the run gets;
//   cta_split_sort   cuts the run's sampled key range into equal parts, moves
//                    the keys to their parts through the other buffer (one
//                    read to count, one read and one write to move, unstable:
//                    one shared atomic per key), then sorts runs of whole
//                    parts in shared memory (bin_sort.cuh).  A part that is
//                    still too large is cut once more, over its own range;
//   cta_radix_sort   the LSD radix passes of Algorithms 4a/4b by one CTA, for
//                    what two cuts do not separate (many equal keys among
//                    others) and for runs longer than 32-bit counters hold.
//                    The CTA walks the tiles in order, so running digit
//                    offsets replace a look-back.
#pragma once

#include <type_traits>

#include "bin_sort.cuh"
#include "common.cuh"
#include "seg_tiers.h"

namespace evosort {

constexpr int kCtaThreads = 512;
constexpr int kCtaWarps = kCtaThreads / 32;
constexpr int kCtaParts = 1024;      // most parts of one cut
constexpr int kCtaWords = 12;        // words of four bins per thread of a local sort
constexpr int kCtaFewWords = 4;      // the same for short runs
constexpr int kCtaFewKeys = 1536;    // longest run they are used for

// keys per thread of a local sort, and of a tile on its way to the parts
template <typename U>
__host__ __device__ constexpr int cta_kpt() { return sizeof(U) == 4 ? 16 : 12; }
template <typename U>
__host__ __device__ constexpr int cta_cap() { return kCtaThreads * cta_kpt<U>(); }
// keys per part aimed at: several parts per local sort
template <typename U>
__host__ __device__ constexpr int cta_target() { return sizeof(U) == 4 ? 1536 : 1024; }
// Dynamic shared memory: two buffers of a local sort (the radix passes use
// them too), then the ends of the parts of both cuts.
template <typename U>
__host__ __device__ constexpr size_t cta_buf_bytes() {
    return (size_t)cta_cap<U>() * sizeof(U) + bin_scratch_bytes(cta_cap<U>(), (int)sizeof(U), kCtaWords * kCtaThreads);
}
template <typename U>
__host__ __device__ constexpr size_t cta_smem_bytes() { return cta_buf_bytes<U>() + (size_t)kCtaParts * 8; }

template <typename U>
struct CtaShared {
    BinShared<U, kCtaThreads> bin;
    uint32_t scan[kCtaWarps + 1];
    uint32_t next, end, below, above, longest;
    float value[2][kCtaWarps];
};

struct AsIs {
    template <typename U>
    __device__ __forceinline__ U operator()(U k) const { return k; }
};
// Whether keys that are left where they are, in their own array, need out().
template <typename MI>
constexpr bool kMapsBack = !std::is_same<MI, AsIs>::value;

// Local sort of n <= cta_cap() keys held in registers (mapped); out maps back,
// store(position, key) receives the sorted keys, still mapped.  Bins by the
// keys' range, or by their values' for floats.
template <typename U, typename MO, typename S>
__device__ __forceinline__ void cta_local_sort(const U (&key)[cta_kpt<U>()], int n, const MO& out, unsigned char* smem,
                                               CtaShared<U>& sh, const S& store) {
    constexpr int KPT = cta_kpt<U>();
    U* k0 = (U*)smem;
    U* k1 = k0 + cta_cap<U>();
    if (n <= kCtaFewKeys)
        bin_zero<kCtaThreads, kCtaFewWords>(k1);
    else
        bin_zero<kCtaThreads, kCtaWords>(k1);
    U lo, hi;
    block_extent<U, kCtaThreads, KPT>(key, n, sh.bin, &lo, &hi);   // (its barrier also ends the clearing)
    const unsigned long long width = (unsigned long long)(U)(hi - lo);
    const U* r;
    auto none = []() {};
    if constexpr (MO::is_float) {
        const auto pos = block_value_position<U, kCtaThreads, KPT>(key, n, out, out.descending(), sh.value);
        r = n <= kCtaFewKeys
                ? block_bin_sort<U, kCtaThreads, KPT, kCtaFewWords>(key, n, lo, width, pos,
                                                                    4u * kCtaFewWords * kCtaThreads, k0, k1, sh.bin, none)
                : block_bin_sort<U, kCtaThreads, KPT, kCtaWords>(key, n, lo, width, pos, 4u * kCtaWords * kCtaThreads, k0,
                                                                 k1, sh.bin, none);
    } else {
        int lz;
        uint32_t mult;
        cut_range_near(width, (uint32_t)(4 * (n <= kCtaFewKeys ? kCtaFewWords : kCtaWords) * kCtaThreads), &lz, &mult);
        const KeyPosition<U> pos{lo, lz};
        r = n <= kCtaFewKeys
                ? block_bin_sort<U, kCtaThreads, KPT, kCtaFewWords>(key, n, lo, width, pos, mult, k0, k1, sh.bin, none)
                : block_bin_sort<U, kCtaThreads, KPT, kCtaWords>(key, n, lo, width, pos, mult, k0, k1, sh.bin, none);
    }
    for (int i = threadIdx.x; i < n; i += kCtaThreads) store(i, r[i]);
    __syncthreads();
}

// LSD radix sort of the len keys in a (other buffer b): out() maps a key on its
// last store, and out.forward() on its first load unless it is mapped already
// (MAPPED); the sorted keys end in fin (a or b).
// 8-bit digits; digits that are equal in all keys are skipped.  I counts keys:
// 32 bits for runs of at most kSegCutKeys, 64 bits for any.
template <typename I, bool MAPPED, typename U, typename M>
__device__ __noinline__ void cta_radix_sort(U* a, U* b, U* fin, I len, M out) {
    auto in = [&](U k) { return MAPPED ? k : out.forward(k); };
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_scan[kCtaWarps + 1];
    __shared__ int s_active[sizeof(U)];
    constexpr int NP = sizeof(U);
    constexpr int BINS = 256;
    constexpr int KPT = 8;
    constexpr uint32_t TILE = kCtaThreads * KPT;
    static_assert(sizeof(I) == 8 || kSegCutKeys + 4u * kCtaThreads <= 0xFFFFFFFFull, "an unrolled step past the end");
    static_assert(sizeof(I) == 8 || kSegCutKeys + TILE <= 0xFFFFFFFFull, "a tile past the end");
    static_assert((NP + 1) * BINS * sizeof(I) + BINS * 8 + kCtaWarps * BINS * 6 + TILE * sizeof(U) <= cta_buf_bytes<U>(),
                  "shared memory");
    static_assert(NP <= kCtaWarps, "the long runs' counts in the match masks' room");
    I* s_hist = (I*)smem;                               // NP * BINS
    I* s_run = s_hist + NP * BINS;                      // BINS running offsets
    uint32_t* s_excl = (uint32_t*)(s_run + BINS);       // BINS tile offsets
    uint32_t* s_tcnt = s_excl + BINS;                   // BINS tile counts
    uint32_t* s_match = s_tcnt + BINS;                  // warps * BINS match masks
    uint16_t* s_whist = (uint16_t*)(s_match + kCtaWarps * BINS);   // warps * BINS
    U* s_r = (U*)(s_whist + kCtaWarps * BINS);          // TILE keys
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < NP * BINS; i += kCtaThreads) s_hist[i] = 0;
    if (tid < NP) s_active[tid] = 0;
    __syncthreads();
    auto count = [&](const U* keys, uint32_t m, uint32_t* hist) {
#pragma unroll 4
        for (uint32_t i = tid; i < m; i += kCtaThreads) {
            const U k = in(keys[i]);
#pragma unroll
            for (int p = 0; p < NP; ++p) atomicAdd(&hist[p * BINS + digit_of(k, 8 * p, 0xFFu)], 1u);
        }
        __syncthreads();
    };
    if constexpr (sizeof(I) == 4) {
        count(a, len, s_hist);
    } else {
        // 32-bit counts of a stretch at a time, in the room of the match masks
        // (64-bit shared atomics queue up on a digit that is equal in all
        // keys: 2^31 keys of 600 values took 84 s)
        for (int i = tid; i < NP * BINS; i += kCtaThreads) s_match[i] = 0u;
        __syncthreads();
        for (I at = 0; at < len; at += kSegCutKeys) {
            count(a + at, (uint32_t)(len - at < kSegCutKeys ? len - at : kSegCutKeys), s_match);
            for (int i = tid; i < NP * BINS; i += kCtaThreads) {
                s_hist[i] += s_match[i];
                s_match[i] = 0u;
            }
            __syncthreads();
        }
    }
    for (int i = tid; i < NP * BINS; i += kCtaThreads)
        if (s_hist[i] != 0 && s_hist[i] != len) s_active[i / BINS] = 1;
    __syncthreads();
    int nact = 0;
    for (int p = 0; p < NP; ++p) nact += s_active[p];
    if (nact == 0) {   // equal keys
        if (fin != a || MAPPED)
            for (I i = tid; i < len; i += kCtaThreads) fin[i] = out(in(a[i]));
        __syncthreads();
        return;
    }
    int done = 0;
    U* src = a;
    U* dst = b;
    const uint32_t lt = lanemask_lt();
    for (int p = 0; p < NP; ++p) {
        if (!s_active[p]) continue;
        const int shift = 8 * p;
        const bool first = done == 0, last = ++done == nact;
        {
            const I c = tid < BINS ? s_hist[p * BINS + tid] : (I)0;
            I tot;
            I* scan;
            if constexpr (sizeof(I) == 4)
                scan = s_scan;
            else
                scan = (I*)s_match;   // (cleared again by the first tile)
            const I ex = block_exclusive_scan<kCtaThreads, I>(c, scan, &tot);
            if (tid < BINS) s_run[tid] = ex;
        }
        __syncthreads();
        for (I t0 = 0; t0 < len; t0 += TILE) {
            const int valid = len - t0 < TILE ? (int)(len - t0) : (int)TILE;
            uint16_t* wh = s_whist + warp * BINS;
            uint32_t* wm = s_match + warp * BINS;
            for (int i = lane; i < BINS; i += 32) {
                wm[i] = 0u;
                if ((i & 1) == 0) ((uint32_t*)wh)[i >> 1] = 0u;
            }
            __syncwarp();
            U key[KPT];
            uint32_t rk[KPT / 2];   // rank in the warp, two 16-bit fields per register
            const int wofs = warp * 32 * KPT + lane;
            if (tid == 0 && t0 + TILE < len)   // the next tile, while this one is ranked
                prefetch_l2_inner(src + t0 + TILE, (size_t)(len - t0 - TILE < TILE ? len - t0 - TILE : (I)TILE) * sizeof(U));
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const int s = wofs + 32 * i;
                key[i] = s < valid ? src[t0 + s] : ~(U)0;
            }
            if (first) {
#pragma unroll
                for (int i = 0; i < KPT; ++i) key[i] = wofs + 32 * i < valid ? in(key[i]) : ~(U)0;
            }
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const uint32_t dig = digit_of(key[i], shift, 0xFFu);
                atomicOr(&wm[dig], 1u << lane);
                __syncwarp();
                const uint32_t peers = wm[dig];
                __syncwarp();
                const int leader = 31 - __clz(peers);
                uint32_t old = 0;
                if (lane == leader) {
                    old = wh[dig];
                    wh[dig] = (uint16_t)(old + __popc(peers));
                    wm[dig] = 0u;
                }
                old = __shfl_sync(0xffffffffu, old, leader) + __popc(peers & lt);
                rk[i / 2] = i & 1 ? __byte_perm(rk[i / 2], old, 0x5410) : old;
                __syncwarp();
            }
            __syncthreads();
            uint32_t tc = 0;
            if (tid < BINS) {
                for (int w = 0; w < kCtaWarps; ++w) {
                    const uint32_t c = s_whist[w * BINS + tid];
                    s_whist[w * BINS + tid] = (uint16_t)tc;
                    tc += c;
                }
                s_tcnt[tid] = tc;
            }
            {
                uint32_t tot;
                const uint32_t ex = block_exclusive_scan<kCtaThreads>(tc, s_scan, &tot);
                if (tid < BINS) s_excl[tid] = ex;
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                if (wofs + 32 * i < valid) {
                    const uint32_t dig = digit_of(key[i], shift, 0xFFu);
                    s_r[s_excl[dig] + wh[dig] + (i & 1 ? rk[i / 2] >> 16 : rk[i / 2] & 0xFFFFu)] = key[i];
                }
            }
            __syncthreads();
            for (int s = tid; s < valid; s += kCtaThreads) {
                const U k = s_r[s];
                const uint32_t dig = digit_of(k, shift, 0xFFu);
                dst[s_run[dig] + (s - s_excl[dig])] = last ? out(k) : k;
            }
            __syncthreads();
            if (tid < BINS) s_run[tid] += s_tcnt[tid];
            __syncthreads();
        }
        U* t = src;
        src = dst;
        dst = t;
    }
    if (src != fin)
        for (I i = tid; i < len; i += kCtaThreads) fin[i] = src[i];
    __syncthreads();
}

// Whether a run of len keys is better sorted by radix passes than cut.  A cut
// moves a key once and sorts it on chip, which costs about as much as two
// (32-bit keys) or three passes.  It costs more where the keys crowd together
// (uneven parts are cut again), where one value holds much of them (its counters
// queue up) and, while the keys of a value fit a local sort, where values repeat
// (the bins fill up); it costs less where a part holds one value.  Read off the
// CTA's sample: x is one of this thread's sampled keys, vary the bits in which
// they differ from the smallest, width their range.  kCtaVoters warps compare
// their keys (all of them took 6 % of segments of 7,000 keys).
// 300 segments of up to 40,000 keys, cut in any case -> so: float64 keys of 1,000
// values 2,378 -> 376 us, int64 keys of 7 values 271 -> 152 us, float32 keys of 100
// values 327 -> 185 us; passes in any case: uniform int64 keys 555 us, 216 so.
constexpr int kCtaVoters = 4;   // warps
template <typename U, typename P>
__device__ __noinline__ bool cta_vote(U x, bool have, U vary, uint32_t len, unsigned long long width, P position,
                                      CtaShared<U>& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t vl = __reduce_or_sync(0xffffffffu, (uint32_t)vary);
    const uint32_t vh = __reduce_or_sync(0xffffffffu, (uint32_t)((unsigned long long)vary >> 32));
    uint32_t said = 0;   // which digits vary (8 bits), then counts of up to 32
#pragma unroll
    for (int b = 0; b < 4; ++b)
        said |= (((vl >> (8 * b)) & 0xFFu) != 0u ? 1u << b : 0u) | (((vh >> (8 * b)) & 0xFFu) != 0u ? 16u << b : 0u);
    if (warp < kCtaVoters) {
        const KeyVotes v = key_votes(x, have, position);
        said |= (uint32_t)__popc(__ballot_sync(0xffffffffu, v.crowded)) << 8 |
                (uint32_t)__popc(__ballot_sync(0xffffffffu, v.repeated)) << 16 |
                (uint32_t)__popc(__ballot_sync(0xffffffffu, v.frequent)) << 24;
    }
    if (lane == 0) sh.scan[warp] = said;
    __syncthreads();
    uint32_t crowded = 0, repeated = 0, frequent = 0;
#pragma unroll
    for (int w = 0; w < kCtaVoters; ++w) {
        crowded += (sh.scan[w] >> 8) & 0xFFu;
        repeated += (sh.scan[w] >> 16) & 0xFFu;
        frequent += sh.scan[w] >> 24;
    }
    const int digits = __popc(__reduce_or_sync(0xffffffffu, lane < kCtaWarps ? sh.scan[lane] : 0u) & 0xFFu);
    __syncthreads();   // (scan is used again)
    constexpr uint32_t voters = kCtaVoters * 32;
    if (crowded > voters / 3 || frequent > voters / 4 || digits == 1) return true;
    // values with more keys each than a local sort holds: from the distinct keys
    // among a warp's 32, v distinct values are at most kinds / (1 - kinds / 32)
    const float kinds = (float)(voters - repeated) / (float)kCtaVoters;
    if ((float)len * (32.f - kinds) > 32.f * kinds * (float)cta_cap<U>()) return false;
    if (repeated >= 2u && digits <= (sizeof(U) == 8 ? 3 : 2)) return true;
    return P::linear && sizeof(U) == 8 && digits <= 2 && width < (unsigned long long)len;
}
template <typename U, typename P>
__device__ __forceinline__ bool cta_wants_passes(const U (&k)[8], int m, uint32_t len, U lo, unsigned long long width,
                                                 const P& position, CtaShared<U>& sh) {
    const int tid = threadIdx.x, row = (tid & 31) % ((m + kCtaThreads - 1) / kCtaThreads);
    U x = k[0], vary = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (row == i) x = k[i];
        if (i * kCtaThreads + tid < m) vary |= k[i] ^ lo;
    }
    return cta_vote<U, P>(x, row * kCtaThreads + tid < m, vary, len, width, position, sh);
}

// Sort of the len keys of src: in() maps a key on its load, out() on its last
// store.  The parts are laid out in part (as long as src); the sorted keys end
// in fin, which is src or part.  LEVEL 0 cuts too large parts again.  len is at
// most kSegCutKeys: the counters are of 32 bits.  False, and src as it was, where
// the run is better left to radix passes.
template <typename U, int LEVEL, typename MI, typename MO>
__device__ __forceinline__ bool cta_split_impl(U* src, U* part, U* fin, uint32_t len, MI in, MO out,
                                               unsigned char* smem, CtaShared<U>& sh);
template <typename U, typename MO>
__device__ __noinline__ void cta_split_again(U* src, U* part, U* fin, uint32_t len, MO out, unsigned char* smem,
                                             CtaShared<U>& sh) {
    if (!cta_split_impl<U, 1>(src, part, fin, len, AsIs(), out, smem, sh))
        cta_radix_sort<uint32_t, true>(src, part, fin, len, out);
}
template <typename U, typename MI, typename MO>
__device__ __forceinline__ void cta_split_sort(U* src, U* part, U* fin, uint32_t len, MI in, MO out,
                                               unsigned char* smem, CtaShared<U>& sh) {
    if (!cta_split_impl<U, 0>(src, part, fin, len, in, out, smem, sh))
        cta_radix_sort<uint32_t, false>(src, part, fin, len, out);
}

template <typename U, int LEVEL, typename MI, typename MO>
__device__ __forceinline__ bool cta_split_impl(U* src, U* part, U* fin, uint32_t len, MI in, MO out,
                                               unsigned char* smem, CtaShared<U>& sh) {
    constexpr int KPT = cta_kpt<U>();
    constexpr int CAP = cta_cap<U>();
    constexpr uint32_t TILE = CAP;
    static_assert(kSegCutKeys + TILE <= 0xFFFFFFFFull && kSegCutKeys + 16u * kCtaThreads <= 0xFFFFFFFFull,
                  "a step past the end");
    U* s_key = (U*)smem;                                                  // tile buffer, or a local sort's first
    uint32_t* s_cnt = (uint32_t*)(smem + (size_t)CAP * sizeof(U));        // tile counts (the second buffer)
    uint32_t* s_at = s_cnt + kCtaParts;
    uint32_t* s_to = s_at + kCtaParts;
    // next free place of a part, at last its end
    uint32_t* s_cur = (uint32_t*)(smem + cta_buf_bytes<U>()) + LEVEL * kCtaParts;
    const int tid = threadIdx.x, lane = tid & 31;

    // ---- range of the keys, from a sample, and whether to cut them at all
    U lo, hi;
    float low = 0.f, scale = 0.f;   // floats: the cut of the sampled values
    bool passes = false;   // (asked of whole runs only)
    {
        U k[8];
        const uint32_t stride = len / (8 * kCtaThreads);
        const int m = stride ? 8 * kCtaThreads : (int)len;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            k[i] = in(i * kCtaThreads + tid < m ? src[(uint32_t)(i * kCtaThreads + tid) * (stride ? stride : 1u)] : (U)0);
        block_extent<U, kCtaThreads, 8>(k, m, sh.bin, &lo, &hi);
        const int wlz = __clzll((long long)((unsigned long long)(U)(hi - lo) | 1ull));
        if constexpr (MO::is_float) {
            const auto pos = block_value_position<U, kCtaThreads, 8>(k, m, out, out.descending(), sh.value);
            low = pos.low;
            scale = pos.scale;
            if (LEVEL == 0) passes = cta_wants_passes<U>(k, m, len, lo, 0ull, pos, sh);
        } else {
            if (LEVEL == 0)
                passes = cta_wants_passes<U>(k, m, len, lo, (unsigned long long)(U)(hi - lo), KeyPosition<U>{lo, wlz}, sh);
        }
    }
    const unsigned long long width = (unsigned long long)(U)(hi - lo);
    if (width == 0) {   // one value, as far as the sample shows
        bool other = false;
        uint32_t i = tid;
        for (; i + 7u * kCtaThreads < len; i += 8u * kCtaThreads) {
            U k[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) k[u] = src[i + (uint32_t)(u * kCtaThreads)];
#pragma unroll
            for (int u = 0; u < 8; ++u) other |= in(k[u]) != lo;
        }
        for (; i < len; i += kCtaThreads) other |= in(src[i]) != lo;
        if (!__syncthreads_or(other)) {
            if (fin != src || !kMapsBack<MI>) {
                const U k = out(lo);
                for (i = tid; i < len; i += kCtaThreads) fin[i] = k;
                __syncthreads();
            }
            return true;
        }
    } else if (passes) {
        return false;
    }
    uint32_t want = (len + (uint32_t)cta_target<U>() - 1u) / (uint32_t)cta_target<U>();
    if (want > (uint32_t)kCtaParts) want = (uint32_t)kCtaParts;
    int lz;
    uint32_t mult;
    uint32_t np = cut_range(width, want, &lz, &mult);
    bool one_value = width < (unsigned long long)np;
    if (MO::is_float) {
        np = want;
        one_value = false;
    }
    // keys outside the sampled range go to the first and the last part
    auto part_of = [&](U k) {
        if constexpr (MO::is_float) {
            ValuePosition<U, MO> pos(out, 0.f, 0.f, out.descending());
            pos.low = low;
            pos.scale = scale;
            return __umulhi(pos(k), np);
        } else {
            const U d = (k > lo ? k : lo) - lo;
            return __umulhi(norm32(d < (U)width ? d : (U)width, lz), mult);
        }
    };

    // ---- count
    for (int i = tid; i < kCtaParts; i += kCtaThreads) s_cnt[i] = 0u;
    if (tid == 0) sh.below = sh.above = sh.longest = 0u;
    __syncthreads();
    {
        bool below = false, above = false;
        auto one = [&](U raw) {
            const U k = in(raw);
            below |= k < lo;
            above |= k > hi;
            atomicAdd(&s_cnt[part_of(k)], 1u);
        };
        uint32_t i = tid;
        for (; i + 7u * kCtaThreads < len; i += 8u * kCtaThreads) {
            U k[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) k[u] = src[i + (uint32_t)(u * kCtaThreads)];
#pragma unroll
            for (int u = 0; u < 8; ++u) one(k[u]);
        }
        for (; i < len; i += kCtaThreads) one(src[i]);
        if (below) sh.below = 1u;
        if (above) sh.above = 1u;
    }
    __syncthreads();
    {
        uint32_t c[2], sum = 0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            c[j] = s_cnt[tid * 2 + j];
            s_cnt[tid * 2 + j] = 0u;
            sum += c[j];
        }
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<kCtaThreads>(sum, sh.scan, &tot);
        s_cur[tid * 2] = ex;
        s_cur[tid * 2 + 1] = ex + c[0];
        atomicMax(&sh.longest, max(c[0], c[1]));
    }
    __syncthreads();
    const bool low_end = sh.below != 0u, high_end = sh.above != 0u;
    // most keys in one part: not separated by its range
    if (!one_value && sh.longest > (uint32_t)CAP && sh.longest > len / 2u) return false;

    // ---- move the keys to their parts, a tile at a time
    {
        U key[KPT];
        auto load = [&](uint32_t t0) {
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const uint32_t j = t0 + (uint32_t)(i * kCtaThreads + tid);
                key[i] = j < len ? src[j] : (U)0;
            }
        };
        load(0);
        for (uint32_t t0 = 0; t0 < len; t0 += TILE) {
            const uint32_t valid = min(len - t0, TILE);
            uint32_t rk[(KPT + 1) / 2];
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                if ((uint32_t)(i * kCtaThreads + tid) < valid) {
                    key[i] = in(key[i]);
                    const uint32_t r = atomicAdd(&s_cnt[part_of(key[i])], 1u);
                    rk[i / 2] = i & 1 ? __byte_perm(rk[i / 2], r, 0x5410) : r;
                }
            }
            __syncthreads();
            const uint32_t c0 = s_cnt[tid * 2], c1 = s_cnt[tid * 2 + 1];
            s_cnt[tid * 2] = 0u;
            s_cnt[tid * 2 + 1] = 0u;
            uint32_t tot;
            const uint32_t ex = block_exclusive_scan<kCtaThreads>(c0 + c1, sh.scan, &tot);
            const uint32_t g0 = s_cur[tid * 2], g1 = s_cur[tid * 2 + 1];
            s_at[tid * 2] = ex;
            s_at[tid * 2 + 1] = ex + c0;
            s_to[tid * 2] = g0 - ex;
            s_to[tid * 2 + 1] = g1 - (ex + c0);
            s_cur[tid * 2] = g0 + c0;
            s_cur[tid * 2 + 1] = g1 + c1;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < KPT; ++i)
                if ((uint32_t)(i * kCtaThreads + tid) < valid)
                    s_key[s_at[part_of(key[i])] + (i & 1 ? rk[i / 2] >> 16 : rk[i / 2] & 0xFFFFu)] = key[i];
            if (t0 + TILE < len) load(t0 + TILE);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const uint32_t s = (uint32_t)(i * kCtaThreads + tid);
                if (s < valid) {
                    const U k = s_key[s];
                    part[s_to[part_of(k)] + s] = k;
                }
            }
            // (the next tile writes s_key, s_at and s_to only after two barriers)
        }
        __syncthreads();
    }

    // ---- runs of whole parts that fit, sorted in shared memory
    uint32_t f = 0, s = 0;
    while (f < np) {
        if (tid < 32) {
            uint32_t g = f, e = s;
            for (;;) {
                const uint32_t i = g + (uint32_t)lane;
                const uint32_t x = i < np ? s_cur[i] : 0u;
                const uint32_t m = __ballot_sync(0xffffffffu, i < np && x - s <= (uint32_t)CAP);
                const int k = m == 0xffffffffu ? 32 : __ffs((int)~m) - 1;
                if (k > 0) e = __shfl_sync(0xffffffffu, x, k - 1);
                g += (uint32_t)k;
                if (k < 32) break;
            }
            if (g == f) {   // one part too large
                e = s_cur[f];
                g = f + 1u;
            }
            if (lane == 0) {
                sh.next = g;
                sh.end = e;
                if (e < len) prefetch_l2_inner(part + e, (size_t)min(len - e, (uint32_t)CAP) * sizeof(U));
            }
        }
        __syncthreads();
        const uint32_t g = sh.next, e = sh.end, n = e - s;
        if (n > (uint32_t)CAP) {
            U* const other = (fin == part ? src : fin) + s;
            if (one_value && !(f == 0u && low_end) && !(f + 1u == np && high_end)) {
                for (uint32_t i = s + tid; i < e; i += kCtaThreads) fin[i] = out(part[i]);
                __syncthreads();
            } else if (LEVEL == 0) {
                __syncthreads();   // (sh is used again)
                cta_split_again<U>(part + s, other, fin + s, n, out, smem, sh);
            } else {
                __syncthreads();
                cta_radix_sort<uint32_t, true>(part + s, other, fin + s, n, out);
            }
        } else if (n > 0) {
            U key[KPT];
#pragma unroll
            for (int i = 0; i < KPT; ++i)
                key[i] = (uint32_t)(i * kCtaThreads + tid) < n ? part[s + (uint32_t)(i * kCtaThreads + tid)] : (U)0;
            cta_local_sort<U>(key, (int)n, out, smem, sh, [&](int i, U k) { fin[s + (uint32_t)i] = out(k); });
        } else {
            __syncthreads();
        }
        f = g;
        s = e;
    }
    return true;
}

}  // namespace evosort
