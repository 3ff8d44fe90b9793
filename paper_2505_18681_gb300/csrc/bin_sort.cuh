// Bin sort of a few thousand keys by one CTA in shared memory (keys only).
//
// The keys are spread over equal stretches of their range, several times more
// of them than there are keys, so most bins hold no key or one.  One shared
// atomic per key counts its bin and gives the key a place in it, a scan of the
// bins gives each bin its start, every key is written once to its place, and
// the few bins with two or more keys are sorted by the thread that owns them.
// Equal keys are identical bit patterns, so the places inside a bin may be
// given in any order: no match masks, no per-warp counters and no second pass
// are needed, which the stable radix passes spend most of their shared-memory
// wavefronts on.
//
// Four bins share a 32-bit word: 8-bit counts while the keys are counted,
// then the first place of the word's first bin (14 bits) and the offsets of
// the other three (6 bits each), so that a key's place is one read away.  A
// quarter of the words of 32-bit counters are zeroed, scanned and rewritten,
// or, seen the other way, four times as many bins cost the same and leave
// fewer keys to sort inside bins.  1e9 int32 / int64 keys, all groups: 5.3 /
// 7.3 ms with 10,240 32-bit counters.
//
// Where the stretches do not separate the keys (a bin of 16 keys or more),
// the caller's own way (OWN) or block_bin_sort_fine or _wide takes over: counters
// of 16 or 32 bits, bins of equal keys left as they are, others of up to 32 *
// kBinWarpKeys keys sorted by one warp each (bitonic), and if some bin is longer
// still, or the keys crowd together from the start, bitonic runs and the merge
// rounds of Algorithm 3, so any input is sorted in bounded time.
#pragma once

#include <cfloat>

#include "common.cuh"
#include "smem_sort.cuh"

namespace evosort {

constexpr int kBinMax = 1 << 16;     // most bins
constexpr int kBinThreadKeys = 31;   // longest bin one thread sorts (2^k - 1)
constexpr int kBinWarpKeys = 16;     // keys per lane of the warp sort
constexpr int kBinOdd = 32;          // keys beside the frequent one of a longer bin

// Bytes of the second buffer of n keys: the words of the bins, or the merge
// sort's other array.
__host__ __device__ constexpr size_t bin_scratch_bytes(int n, int w, int words) {
    return (size_t)n * w > (size_t)words * 4 ? (size_t)n * w : (size_t)words * 4;
}

// Position of d = key - low in [0, 2^32): d shifted so that the widest one
// (lz leading zeros, of 64 bits) starts at bit 31.
__device__ __forceinline__ uint32_t norm32(uint32_t d, int lz) { return d << (lz - 32); }
__device__ __forceinline__ uint32_t norm32(uint64_t d, int lz) {
    const uint32_t lo = (uint32_t)d, hi = (uint32_t)(d >> 32);
    return lz < 32 ? __funnelshift_l(lo, hi, lz) : lo << (lz - 32);
}
// Smallest d whose position is at least x.
__device__ __forceinline__ unsigned long long denorm32(uint32_t x, int lz) {
    if (lz < 32) return (unsigned long long)x << (32 - lz);
    const int s = lz - 32;
    return ((unsigned long long)x + ((1ull << s) - 1ull)) >> s;
}
// Cuts [0, width] into at most parts equal stretches: part = umulhi(position,
// mult), below the returned count.  With width < parts every part is one
// value (part = d).
__device__ __forceinline__ uint32_t cut_range(unsigned long long width, uint32_t parts, int* lz, uint32_t* mult) {
    if (width == 0 || parts <= 1u) {
        *lz = 63;
        *mult = 0u;
        return 1u;
    }
    const int z = __clzll((long long)width);
    *lz = z;
    if (width < (unsigned long long)parts) {   // (parts <= kBinMax, so z >= 48)
        *mult = 1u << (64 - z);
        return (uint32_t)width + 1u;
    }
    const uint32_t x = norm32((uint64_t)width, z);   // in [2^31, 2^32)
    *mult = (uint32_t)(((unsigned long long)parts << 32) / ((unsigned long long)x + 1ull));
    return parts;
}
// The same for many cuts of one value each in turn, where a few parts fewer do
// not matter: one float division instead of a 64-bit one.
__device__ __forceinline__ void cut_range_near(unsigned long long width, uint32_t parts, int* lz, uint32_t* mult) {
    if (width == 0) {
        *lz = 63;
        *mult = 0u;
        return;
    }
    const int z = __clzll((long long)width);
    *lz = z;
    if (width < (unsigned long long)parts) {
        *mult = 1u << (64 - z);
        return;
    }
    // below the exact quotient by more than the float roundings add up to
    const float x = (float)norm32((uint64_t)width, z);
    *mult = (uint32_t)(__fdividef((float)parts * 65536.0f, x) * 65535.9f * 0.999999f);
}
// Smallest position of part j >= 1.
__device__ __forceinline__ uint32_t part_start(uint32_t j, uint32_t mult) {
    return (uint32_t)((((unsigned long long)j << 32) + mult - 1ull) / mult);
}

// Position of a key in [lo, lo + width].
template <typename U>
struct KeyPosition {
    static constexpr bool linear = true;   // few enough values: one per bin
    U lo;
    int lz;
    __device__ __forceinline__ uint32_t operator()(U k) const { return norm32((U)(k - lo), lz); }
};

// Key maps of a first load and a last store, as function objects: integers are
// mapped by one xor (which is its own inverse), floats by the general map.
template <typename U>
struct XorMap {
    static constexpr bool is_float = false;
    U c;
    __device__ __forceinline__ explicit XorMap(const KeyMap& m) : c((U)(m.s ^ m.x)) {}
    __device__ __forceinline__ U operator()(U k) const { return k ^ c; }
    __device__ __forceinline__ U forward(U k) const { return k ^ c; }   // the map of the load
};
template <typename U>
struct FloatIn {
    KeyMap m;
    __device__ __forceinline__ explicit FloatIn(const KeyMap& k) : m(k) {}
    __device__ __forceinline__ U operator()(U k) const { return map_fwd(k, m); }
};
template <typename U>
struct GeneralOut {   // any key type
    static constexpr bool is_float = false;
    KeyMap m;
    __device__ __forceinline__ explicit GeneralOut(const KeyMap& k) : m(k) {}
    __device__ __forceinline__ U operator()(U k) const { return map_inv(k, m); }
    __device__ __forceinline__ U forward(U k) const { return map_fwd(k, m); }
};
template <typename U>
struct FloatOut : GeneralOut<U> {
    static constexpr bool is_float = true;
    __device__ __forceinline__ explicit FloatOut(const KeyMap& k) : GeneralOut<U>(k) {}
    __device__ __forceinline__ bool descending() const { return this->m.x != 0; }
};

// Position of a float key by its value: (value - smallest) * scale.  Floats of
// an even spread crowd into the few bit patterns of the largest exponents, so
// equal stretches of the mapped keys would leave most bins empty; equal
// stretches of the values do not.  Rounding keeps the order: subtraction,
// multiplication and the narrowing of doubles never turn two values around.
// NaNs, which have no value, go to their end of the order, infinities and
// values outside the range clamp.  (34.9e6 doubles in 3,000 segments: 2.41 ms
// by equal stretches of the mapped keys, 0.79 ms by value.)
__device__ __forceinline__ float float_of(uint32_t bits) { return __uint_as_float(bits); }
__device__ __forceinline__ float float_of(uint64_t bits) {
    return __double2float_rn(__longlong_as_double((long long)bits));
}
template <typename U, typename MO>
struct ValuePosition {
    static constexpr bool linear = false;
    MO out;
    float low, scale;   // of half the value, so that the widest range stays finite
    bool descending;
    // a, b: smallest and largest value of the range (a > b if there is none)
    __device__ __forceinline__ ValuePosition(const MO& o, float a, float b, bool desc)
        : out(o), low(0.5f * (desc ? b : a)), scale(0.f), descending(desc) {
        const float range = 0.5f * b - 0.5f * a;
        if (range > 0.f) scale = fminf(4294967040.f / range, FLT_MAX);
    }
    __device__ __forceinline__ uint32_t operator()(U k) const {
        const float f = float_of(out(k));
        if (f != f) return descending ? 0u : 0xFFFFFFFFu;
        const float h = 0.5f * f;
        const float x = (descending ? low - h : h - low) * scale;
        return x <= 0.f ? 0u : (x >= 4294967040.f ? 0xFFFFFFFFu : (uint32_t)x);
    }
};
// The position over the finite values of the CTA's keys (element i * NT +
// thread < n, mapped; out maps back).
template <typename U, int NT, int KPT, typename MO>
__device__ __forceinline__ ValuePosition<U, MO> block_value_position(const U (&key)[KPT], int n, const MO& out, bool desc,
                                                                     float (&s_f)[2][NT / 32]) {
    const int tid = threadIdx.x;
    float a = INFINITY, b = -INFINITY;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        if (i * NT + tid < n) {
            const float f = float_of(out(key[i]));
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
    return ValuePosition<U, MO>(out, a, b, desc);
}

template <typename U, int NT>
struct BinShared {
    U mn[NT / 32], mx[NT / 32];   // extents; later the keys of a long bin that are not its frequent one
    uint32_t wsum[NT / 32 + 1];
    uint32_t nlist, nodd;
    uint32_t list[512];   // bins left to the warps: first position | length << 16
};

// Smallest and largest of the CTA's keys (element i * NT + thread < n).
template <typename U, int NT, int KPT>
__device__ __forceinline__ void block_extent(const U (&key)[KPT], int n, BinShared<U, NT>& sh, U* lo, U* hi) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    U mn = ~(U)0, mx = 0;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        if (i * NT + tid < n) {
            mn = key[i] < mn ? key[i] : mn;
            mx = key[i] > mx ? key[i] : mx;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const U a = __shfl_xor_sync(0xffffffffu, mn, o), b = __shfl_xor_sync(0xffffffffu, mx, o);
        mn = a < mn ? a : mn;
        mx = b > mx ? b : mx;
    }
    if (lane == 0) {
        sh.mn[warp] = mn;
        sh.mx[warp] = mx;
    }
    __syncthreads();
    mn = lane < NW ? sh.mn[lane] : ~(U)0;
    mx = lane < NW ? sh.mx[lane] : (U)0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const U a = __shfl_xor_sync(0xffffffffu, mn, o), b = __shfl_xor_sync(0xffffffffu, mx, o);
        mn = a < mn ? a : mn;
        mx = b > mx ? b : mx;
    }
    *lo = mn;
    *hi = mx;
}

// Insertion sort of k[0..c) in shared memory by one thread.
template <typename U>
__device__ __forceinline__ void bin_insertion(U* k, int c) {
    const U a = k[0], b = k[1];
    if (b < a) {
        k[0] = b;
        k[1] = a;
    }
    for (int i = 2; i < c; ++i) {
        const U x = k[i];
        int j = i;
        while (j > 0) {
            const U y = k[j - 1];
            if (!(y > x)) break;
            k[j] = y;
            --j;
        }
        if (j < i) k[j] = x;
    }
}

// The same for keys with their input positions (x), in the order (key,
// position): equal keys keep their input order.
template <typename U>
__device__ __forceinline__ void bin_insertion_indexed(U* k, uint16_t* x, int c) {
    for (int i = 1; i < c; ++i) {
        const U a = k[i];
        const uint16_t xa = x[i];
        int j = i;
        while (j > 0) {
            const U y = k[j - 1];
            const uint16_t xy = x[j - 1];
            if (!(y > a || (y == a && xy > xa))) break;
            k[j] = y;
            x[j] = xy;
            --j;
        }
        if (j < i) {
            k[j] = a;
            x[j] = xa;
        }
    }
}

// Sort of k[0..c), c <= 32 * kBinWarpKeys, by one warp.
template <typename U>
__device__ __noinline__ void bin_warp_sort(U* k, int c) {
    const int lane = threadIdx.x & 31;
    U x[kBinWarpKeys];
#pragma unroll
    for (int r = 0; r < kBinWarpKeys; ++r) x[r] = r * 32 + lane < c ? k[r * 32 + lane] : ~(U)0;
    warp_bitonic_sort<U, kBinWarpKeys>(x);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kBinWarpKeys; ++r) {
        const int i = lane * kBinWarpKeys + r;
        if (i < c) k[i] = x[r];
    }
}

// Sort of k[0..m) by the CTA if all but kBinOdd of the keys are one value: the
// others go around it.  False, and nothing moved, if they are not.
template <typename U, int NT>
__device__ __forceinline__ bool bin_one_value(U* k, int m, BinShared<U, NT>& sh) {
    static_assert(kBinOdd <= 2 * (NT / 32), "room of the extents");
    const int tid = threadIdx.x;
    U* const odds = sh.mn;   // (mx lies behind it)
    const U a = k[0], b = k[m / 2], c = k[m - 1];
    const U most = a == b || a == c ? a : b;
    if (tid == 0) sh.nodd = 0u;
    __syncthreads();
    for (int i = tid; i < m; i += NT) {
        const U x = k[i];
        if (x != most) {
            const uint32_t at = atomicAdd(&sh.nodd, 1u);
            if (at < (uint32_t)kBinOdd) odds[at] = x;
        }
    }
    __syncthreads();
    const int odd = (int)sh.nodd;
    if (odd > kBinOdd) return false;
    if (odd > 0) {
        int less = 0;
        for (int i = 0; i < odd; ++i) less += odds[i] < most;
        for (int i = tid; i < m - odd; i += NT) k[less + i] = most;
        if (tid < odd) {
            const U x = odds[tid];
            int rank = 0;
            for (int i = 0; i < odd; ++i) rank += odds[i] < x || (odds[i] == x && i < tid);
            k[x < most ? rank : m - odd + rank] = x;
        }
    }
    __syncthreads();
    return true;
}

// The keys of k0 stand in their bins (starts in k1, of type C, ends of a thread's
// last bin in run, multi: its bins of two or more keys): sorts the bins.  A thread
// sorts its short ones, up to kBinThreadWork steps or so in all: where keys crowd
// together the bins of one thread may hold hundreds.  The others are sorted by a
// warp each, or everything if some bin is very long and holds several frequent
// values.
constexpr int kBinThreadWork = 256;
template <typename U, int NT, int BPT, typename C>
__device__ __forceinline__ const U* bin_finish(U* k0, U* k1, int n, uint32_t multi, uint32_t run, BinShared<U, NT>& sh) {
    constexpr int ROOM = sizeof(sh.list) / sizeof(sh.list[0]);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const C* const own = (const C*)k1 + tid * BPT;
    if (tid == 0) sh.nlist = sh.nodd = 0u;
    __syncthreads();
    int work = 0;
    while (multi) {
        const int q = __ffs((int)multi) - 1;
        multi &= multi - 1u;
        const uint32_t at = own[q], next = q + 1 < BPT ? own[q + 1] : run;
        const int m = (int)(next - at);
        work += m * m / 4;
        // (bins of more than kBinThreadKeys: n / (kBinThreadKeys + 1) at most, which is half the room)
        bool mine = m <= kBinThreadKeys && (work <= kBinThreadWork || m <= 4);
        if (!mine) {
            const uint32_t e = atomicAdd(m <= kBinThreadKeys ? &sh.nodd : &sh.nlist, 1u);
            if (m > kBinThreadKeys)
                sh.list[e] = at | (uint32_t)m << 16;
            else if (e < ROOM / 2)
                sh.list[ROOM - 1 - e] = at | (uint32_t)m << 16;
            else
                mine = true;
        }
        if (mine) bin_insertion(k0 + at, m);
    }
    __syncthreads();
    const int listed = (int)sh.nlist, shorter = min((int)sh.nodd, ROOM / 2);
    __syncthreads();   // (nodd is used again)
    for (int e = 0; e < listed; ++e) {
        const int m = (int)(sh.list[e] >> 16);
        if (m > 32 * kBinWarpKeys && !bin_one_value<U, NT>(k0 + (sh.list[e] & 0xFFFFu), m, sh))
            return smem_sort_any(k0, k1, n);   // (k1's starts are not needed any more)
    }
    for (int e = warp; e < listed + shorter; e += NT / 32) {
        const uint32_t x = e < listed ? sh.list[e] : sh.list[ROOM - 1 - (e - listed)];
        U* const k = k0 + (x & 0xFFFFu);
        const int m = (int)(x >> 16);
        if (m > 32 * kBinWarpKeys) continue;
        if (m <= 32) {
            U one[1] = {lane < m ? k[lane] : ~(U)0};
            __syncwarp();
            warp_bitonic_sort<U, 1>(one);
            if (lane < m) k[lane] = one[0];
            continue;
        }
        const U first = k[0];
        bool other = false;
        for (int i = lane; i < m; i += 32) other |= k[i] != first;
        if (__any_sync(0xffffffffu, other)) bin_warp_sort(k, m);
    }
    if (listed + shorter) __syncthreads();
    return k0;
}

// What the keys of a warp say of all: x is a sampled key of each lane that
// have()s one, from all over the array.  near: lanes whose key shares a 1024th of
// the range; a lane's key is compared with the first of them.
struct KeyVotes {
    bool crowded, repeated, frequent;   // another key there; the same key; and a third of the warp with it
};
template <typename U, typename P>
__device__ __forceinline__ KeyVotes key_votes(U x, bool have, const P& position) {
    const uint32_t some = __ballot_sync(0xffffffffu, have);
    KeyVotes v = {false, false, false};
    if (have) {
        const uint32_t near = __match_any_sync(some, position(x) >> 22);
        const int first = __ffs((int)near) - 1;
        const bool same = __shfl_sync(near, x, first) == x;
        v.crowded = !same;
        v.repeated = same && first != (int)(threadIdx.x & 31);
        v.frequent = same && __popc(near) >= 10;
    }
    return v;
}

template <int NT, int BPT, typename U>
__device__ __forceinline__ void bin_zero(U* k1) {
    uint4* const mine = (uint4*)k1 + threadIdx.x * (BPT / 4);
#pragma unroll
    for (int j = 0; j < BPT / 4; ++j) mine[j] = make_uint4(0u, 0u, 0u, 0u);
}

// The position as block_bin_sort_wide is given it: one of the keys' range is
// made from the range (as an argument its registers cost 1.5 % of 10,000 segments
// of int32 keys, which never need it).
template <typename P>
struct WidePosition {
    P p;
    __device__ __forceinline__ explicit WidePosition(const P& position) : p(position) {}
    template <typename U>
    __device__ __forceinline__ P get(U, unsigned long long) const { return p; }
};
template <typename U>
struct WidePosition<KeyPosition<U>> {
    __device__ __forceinline__ WidePosition() {}
    __device__ __forceinline__ explicit WidePosition(const KeyPosition<U>&) {}
    __device__ __forceinline__ KeyPosition<U> get(U lo, unsigned long long width) const {
        return {lo, __clzll((long long)(width | 1ull))};
    }
};

// The same sort with 32-bit counters and any distribution of the keys, which
// lie in k0 (element i * NT + thread of a thread, n in all).  BPT bins per
// thread: the words of block_bin_sort, so that k1 is as large as there.  Unless a
// bin is one value, one key of each thread tells first whether bins can separate
// them at all (a quarter of these keys share a 1024th of the range with a different
// one: they cannot), and whether some value is so frequent that a warp's equal bins
// are better added up before the counters see them (it costs more where they
// differ: 2,000 segments of 4,000 int32 keys of 7 values 95 -> 109 us).  Floats whose
// values crowd together are tried once more by their bit patterns, which spread
// magnitudes evenly.  Bins of one value are left as they are: 1e8 int64 keys with
// some 40 keys of each value, partition sort, 23.2 -> 3.6 ms (every bin by a warp
// before, or everything merged).
template <typename U, int NT, int KPT, int BPT, typename P>
__device__ __noinline__ const U* block_bin_sort_wide(int n, U lo, unsigned long long width, WidePosition<P> given,
                                                     U* k0, U* k1, BinShared<U, NT>& sh) {
    const P position = given.get(lo, width);
    static_assert(BPT % 8 == 4 && BPT * NT <= kBinMax, "bins per thread");
    static_assert(KPT * NT <= 256 * (kBinThreadKeys + 1), "half of the list");
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool one_value = P::linear && width < (unsigned long long)(BPT * NT);   // per bin: nothing left to sort
    bool add_up = false;
    if (!one_value) {
        const int at = lane % ((n + NT - 1) / NT) * NT + tid;
        const KeyVotes v = key_votes(at < n ? k0[at] : (U)0, at < n, position);
        const int most = min(n, NT);
        if (4 * __syncthreads_count(v.crowded) > most) {
            if constexpr (P::linear)
                return smem_sort_any(k0, k1, n);
            else
                return block_bin_sort_wide<U, NT, KPT, BPT, KeyPosition<U>>(
                    n, lo, width, WidePosition<KeyPosition<U>>(), k0, k1, sh);
        }
        add_up = 4 * __syncthreads_count(v.frequent) > most;
    }
    uint32_t* const bins = (uint32_t*)k1;
    // A thread's BPT bins are consecutive and read four at a time; with BPT / 4
    // odd, a quarter-warp's 16-byte reads fall in different banks.
    uint4* const mine = (uint4*)bins + tid * (BPT / 4);
    bin_zero<NT, BPT>(k1);
    U key[KPT];
#pragma unroll
    for (int i = 0; i < KPT; ++i) key[i] = i * NT + tid < n ? k0[i * NT + tid] : (U)0;
    int lz;
    uint32_t mult = (uint32_t)(BPT * NT);
    if (P::linear) cut_range(width, (uint32_t)(BPT * NT), &lz, &mult);
    const uint32_t lt = lanemask_lt();
    __syncthreads();
    // ---- count; the old count is the key's place in its bin
    uint32_t br[KPT];   // bin | place << 16
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const bool have = i * NT + tid < n;
        const uint32_t some = __ballot_sync(0xffffffffu, have);
        if (have) {
            // (in range for every key of [lo, lo + width]; never out of the array for any other)
            const uint32_t b = min(__umulhi(position(key[i]), mult), (uint32_t)(BPT * NT - 1));
            uint32_t place;
            if (add_up) {
                const uint32_t peers = __match_any_sync(some, b);
                const int leader = __ffs((int)peers) - 1;
                place = 0u;
                if (lane == leader) place = atomicAdd(&bins[b], (uint32_t)__popc(peers));
                place = __shfl_sync(peers, place, leader) + (uint32_t)__popc(peers & lt);
            } else {
                place = atomicAdd(&bins[b], 1u);
            }
            br[i] = b | place << 16;
        }
    }
    __syncthreads();

    // ---- exclusive scan of the bins
    uint32_t sum = 0, multi = 0;   // multi: bins of two or more keys
#pragma unroll
    for (int j = 0; j < BPT / 4; ++j) {
        const uint4 q = mine[j];
        sum += q.x + q.y + q.z + q.w;
        if (q.x > 1u) multi |= 1u << (4 * j);
        if (q.y > 1u) multi |= 2u << (4 * j);
        if (q.z > 1u) multi |= 4u << (4 * j);
        if (q.w > 1u) multi |= 8u << (4 * j);
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sh.wsum[warp] = inc;
    __syncthreads();
    uint32_t run = inc - sum;
    {
        uint32_t v = lane < NW ? sh.wsum[lane] : 0u;
        v = lane < warp ? v : 0u;
        run += __reduce_add_sync(0xffffffffu, v);
    }
#pragma unroll
    for (int j = 0; j < BPT / 4; ++j) {
        uint4 q = mine[j];   // read again: registers hold the keys
        const uint32_t a = run + q.x, b = a + q.y, c = b + q.z, d = c + q.w;
        q = make_uint4(run, a, b, c);
        mine[j] = q;
        run = d;
    }
    __syncthreads();

    // ---- every key to its place
#pragma unroll
    for (int i = 0; i < KPT; ++i)
        if (i * NT + tid < n) k0[bins[br[i] & 0xFFFFu] + (br[i] >> 16)] = key[i];
    __syncthreads();
    if (one_value) return k0;
    return bin_finish<U, NT, BPT, uint32_t>(k0, k1, n, multi, run, sh);
}

// The same for keys of which no bin of block_bin_sort held 32: two 16-bit counters
// to a word, so that fewer values share a bin.  (Not for frequent keys: the shared
// atomic that adds one constant counts equal ones of a warp at once, this one
// does not.)  1e8 keys with some ten copies of each value: int32 2.21 -> 2.07 ms,
// int64 3.06 -> 2.87 ms.
template <typename U, int NT, int KPT, int WPT, typename P>
__device__ __noinline__ const U* block_bin_sort_fine(int n, U lo, unsigned long long width, WidePosition<P> given,
                                                     U* k0, U* k1, BinShared<U, NT>& sh) {
    const P position = given.get(lo, width);
    static_assert(WPT % 8 == 4 && 2 * WPT <= 32 && 2 * WPT * NT <= kBinMax, "words per thread");
    static_assert(KPT * NT <= 256 * (kBinThreadKeys + 1), "half of the list");
    constexpr uint32_t BINS = 2 * WPT * NT;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* const words = (uint32_t*)k1;
    // A thread's WPT words are consecutive and read four at a time; with WPT / 4
    // odd, a quarter-warp's 16-byte reads fall in different banks.
    uint4* const mine = (uint4*)words + tid * (WPT / 4);
    bin_zero<NT, WPT>(k1);
    U key[KPT];
#pragma unroll
    for (int i = 0; i < KPT; ++i) key[i] = i * NT + tid < n ? k0[i * NT + tid] : (U)0;
    int lz;
    uint32_t mult = BINS;
    if (P::linear) cut_range(width, BINS, &lz, &mult);
    __syncthreads();
    // ---- count; the old count is the key's place in its bin
    uint32_t br[KPT];   // bin | place << 16
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        if (i * NT + tid < n) {
            // (in range for every key of [lo, lo + width]; never out of the array for any other)
            const uint32_t b = min(__umulhi(position(key[i]), mult), BINS - 1u), half = 16u * (b & 1u);
            br[i] = b | (atomicAdd(&words[b >> 1], 1u << half) >> half & 0xFFFFu) << 16;
        }
    }
    __syncthreads();

    // ---- exclusive scan of the bins
    uint32_t sum = 0, multi = 0;   // multi: bins of two or more keys
#pragma unroll
    for (int j = 0; j < WPT / 4; ++j) {
        const uint4 q = mine[j];
        auto word = [&](uint32_t x, int at) {
            sum += (x & 0xFFFFu) + (x >> 16);
            if (x & 0xFFFEu) multi |= 1u << at;
            if (x >> 17) multi |= 2u << at;
        };
        word(q.x, 8 * j);
        word(q.y, 8 * j + 2);
        word(q.z, 8 * j + 4);
        word(q.w, 8 * j + 6);
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sh.wsum[warp] = inc;
    __syncthreads();
    uint32_t run = inc - sum;
    {
        uint32_t v = lane < NW ? sh.wsum[lane] : 0u;
        v = lane < warp ? v : 0u;
        run += __reduce_add_sync(0xffffffffu, v);
    }
#pragma unroll
    for (int j = 0; j < WPT / 4; ++j) {
        uint4 q = mine[j];   // read again: registers hold the keys
        auto word = [&](uint32_t x) {   // counts -> first places (n < 2^14)
            const uint32_t v = run | (run + (x & 0xFFFFu)) << 16;
            run += (x & 0xFFFFu) + (x >> 16);
            return v;
        };
        q.x = word(q.x);
        q.y = word(q.y);
        q.z = word(q.z);
        q.w = word(q.w);
        mine[j] = q;
    }
    const bool one_value = P::linear && width < (unsigned long long)BINS;   // per bin: nothing left to sort
    __syncthreads();

    // ---- every key to its place
#pragma unroll
    for (int i = 0; i < KPT; ++i)
        if (i * NT + tid < n) k0[((const uint16_t*)k1)[br[i] & 0xFFFFu] + (br[i] >> 16)] = key[i];
    __syncthreads();
    if (one_value) return k0;
    return bin_finish<U, NT, 2 * WPT, uint16_t>(k0, k1, n, multi, run, sh);
}

// Sorts the n keys that the CTA's NT threads hold in registers (key i of a
// thread is element i * NT + thread; elements from n on are ignored), all in
// [lo, lo + width].  The words in k1 are zero (bin_zero) and every thread
// knows it.  WPT words of four bins per thread: bin = umulhi(position(key),
// mult), where position is a KeyPosition (mult and lz from cut_range(width, 4 *
// WPT * NT)) or any other function that never falls as the keys rise.  k0 holds n keys, k1 bin_scratch_bytes(n, w,
// WPT * NT) bytes, both 16-byte aligned; n < 2^14.  placed() runs once the
// registers' keys are in shared memory (the caller may reload them, all of
// them).  Returns the sorted array (k0 or k1), complete for every thread.
// With IDX, x0 receives the input position of each sorted key, equal keys in
// input order.  With OWN it returns null, and has sorted nothing, where the
// stretches do not separate the keys: the caller has its own way then.
template <typename U, int NT, int KPT, int WPT, bool IDX = false, bool OWN = IDX, typename P, typename F>
__device__ __forceinline__ const U* block_bin_sort(const U (&key)[KPT], int n, U lo, unsigned long long width,
                                                   const P& position, uint32_t mult, U* k0, U* k1,
                                                   BinShared<U, NT>& sh, const F& placed, uint16_t* x0 = nullptr) {
    static_assert(WPT % 8 == 4 && 4 * WPT * NT <= kBinMax && KPT * NT < (1 << 14), "words per thread");
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* const words = (uint32_t*)k1;
    // A thread's WPT words are consecutive and read four at a time; with WPT /
    // 4 odd, a quarter-warp's 16-byte reads fall in different banks.
    uint4* const mine = (uint4*)words + tid * (WPT / 4);

    // ---- count; the old count is the key's place in its bin
    uint32_t br[KPT];   // place | bin << 8
#pragma unroll
    for (int c = 0; c < KPT; c += 4) {
        if (c * NT < n) {   // (four columns at a time, so that a short run skips the others)
#pragma unroll
            for (int i = c; i < c + 4 && i < KPT; ++i) {
                if (i * NT + tid < n) {
                    // (in range for every key of [lo, lo + width]; never out of the array for any other)
                    const uint32_t b = min(__umulhi(position(key[i]), mult), (uint32_t)(4 * WPT * NT - 1));
                    const uint32_t old = atomicAdd(&words[b >> 2], __funnelshift_l(0u, 1u, 8u * b));   // by 8 (b mod 4)
                    br[i] = b << 8 | (__funnelshift_r(old, 0u, 8u * b) & 0xFFu);
                }
            }
        }
    }
    __syncthreads();

    // ---- exclusive scan of the bins.  A count that ran over its 8 bits shows
    // in the total: it takes 256 from its own and gives at most one away.
    uint32_t sum = 0, any = 0, widest = 0, multi = 0;   // multi: words with a bin of two or more keys
#pragma unroll
    for (int j = 0; j < WPT / 4; ++j) {
        const uint4 q = mine[j];
        if constexpr (OWN) {
            const uint32_t x = __dp4a(q.x, 0x01010101u, 0u), y = __dp4a(q.y, 0x01010101u, 0u);
            const uint32_t z = __dp4a(q.z, 0x01010101u, 0u), t = __dp4a(q.w, 0x01010101u, 0u);
            sum += (x + y) + (z + t);
            widest = max(max(widest, max(x, y)), max(z, t));
        } else {
            sum = __dp4a(q.x, 0x01010101u, sum);
            sum = __dp4a(q.y, 0x01010101u, sum);
            sum = __dp4a(q.z, 0x01010101u, sum);
            sum = __dp4a(q.w, 0x01010101u, sum);
        }
        any |= q.x | q.y | q.z | q.w;
        if (q.x & 0xFEFEFEFEu) multi |= 1u << (4 * j);
        if (q.y & 0xFEFEFEFEu) multi |= 2u << (4 * j);
        if (q.z & 0xFEFEFEFEu) multi |= 4u << (4 * j);
        if (q.w & 0xFEFEFEFEu) multi |= 8u << (4 * j);
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sh.wsum[warp] = inc;
    // a word's counts must stay below 64 in all: bins below 16, or, where the
    // other way is the slower one, every word counted
    // With positions equal keys have to be put in order too, and a narrow range
    // takes the caller two radix passes at most: bins below 8 there (4,000
    // floats with 8 to 15 equal ones among them: 14.3 us by insertion, 22.5 by passes).
    // Positions arrive in no order, which insertion pays for with the square of
    // the bin: bins below 16 where the other way is short too (16 values among
    // 300 pairs: 5.0 us by passes, 16.7 by insertion; 8,192 pairs of floats with
    // 20 equal ones at most: 36 and 16.5).
    const bool few = IDX && width < 65536ull, strict = !OWN || few || (IDX && n <= 4096);
    // Up to 1,024 keys a thread that sorts a word of many is what the others wait
    // for, and the other way is short: words of up to 24 there, of up to 12 in up to
    // 128 keys, unless a bin is one value and nothing is left to sort (50 floats of
    // every magnitude: 27.8 us with up to 63, 5.9 so).
    const bool one_value = !IDX && P::linear && width < (unsigned long long)(4 * WPT * NT);
    const uint32_t most = !OWN || NT > 512 || n > 1024 || one_value ? 63u : (n > 128 ? 24u : 12u);
    const bool heavy = __syncthreads_or(strict ? (any & (few ? 0xF8F8F8F8u : 0xF0F0F0F0u)) != 0u : widest > most);
    uint32_t run = inc - sum;
    {
        const uint32_t v = lane < NW ? sh.wsum[lane] : 0u;
        run += __reduce_add_sync(0xffffffffu, lane < warp ? v : 0u);
        if (heavy || __reduce_add_sync(0xffffffffu, v) != (uint32_t)n) {   // the same for every thread
            if constexpr (OWN) {
                return nullptr;
            } else {
#pragma unroll
                for (int i = 0; i < KPT; ++i)
                    if (i * NT + tid < n) k0[i * NT + tid] = key[i];
                // (bins of fewer than 32 keys; one value each needs no sort at all)
                const bool single = P::linear && width < (unsigned long long)(WPT * NT);
                const bool mild = !single && !__syncthreads_or((any & 0xE0E0E0E0u) != 0u) &&
                                  __reduce_add_sync(0xffffffffu, v) == (uint32_t)n;
                const WidePosition<P> given(position);
                const U* r = mild ? block_bin_sort_fine<U, NT, KPT, WPT, P>(n, lo, width, given, k0, k1, sh)
                                  : block_bin_sort_wide<U, NT, KPT, WPT, P>(n, lo, width, given, k0, k1, sh);
                placed();
                return r;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < WPT / 4; ++j) {
        uint4 q = mine[j];   // read again: registers hold the keys
        auto word = [&](uint32_t w) {   // counts -> first place and offsets
            const uint32_t p = w * 0x01010101u;   // prefix sums of the four counts
            const uint32_t v = run << 18 | (p & 0x3Fu) | ((p >> 2) & 0xFC0u) | ((p >> 4) & 0x3F000u);
            run += p >> 24;
            return v;
        };
        q.x = word(q.x);
        q.y = word(q.y);
        q.z = word(q.z);
        q.w = word(q.w);
        mine[j] = q;
    }
    __syncthreads();

    // ---- every key to its place
#pragma unroll
    for (int c = 0; c < KPT; c += 4) {
        if (c * NT < n) {
#pragma unroll
            for (int i = c; i < c + 4 && i < KPT; ++i) {
                if (i * NT + tid < n) {
                    const uint32_t b = br[i] >> 8, w = words[b >> 2];
                    const uint32_t before = ((w << 6) >> (6u * (b & 3u))) & 0x3Fu;   // keys of the word's earlier bins
                    const uint32_t at = (w >> 18) + before + (br[i] & 0xFFu);
                    k0[at] = key[i];
                    if (IDX) x0[at] = (uint16_t)(i * NT + tid);
                }
            }
        }
    }
    placed();
    __syncthreads();
    if (one_value) return k0;

    // ---- words with several keys in a bin: first the pairs, which are most of
    // them, so that a warp's lanes stay together; then the longer ones
    const uint32_t* const own = words + tid * WPT;
    uint32_t more = 0;
    while (multi) {
        const int q = __ffs((int)multi) - 1;
        multi &= multi - 1u;
        const uint32_t at = own[q] >> 18, next = q + 1 < WPT ? own[q + 1] >> 18 : run;
        if (next - at == 2u) {
            const U a = k0[at], b = k0[at + 1];
            if (IDX) {
                const uint16_t xa = x0[at], xb = x0[at + 1];
                if (b < a || (b == a && xb < xa)) {
                    k0[at] = b;
                    k0[at + 1] = a;
                    x0[at] = xb;
                    x0[at + 1] = xa;
                }
            } else if (b < a) {
                k0[at] = b;
                k0[at + 1] = a;
            }
        } else {
            more |= 1u << q;
        }
    }
    while (more) {
        const int q = __ffs((int)more) - 1;
        more &= more - 1u;
        const uint32_t at = own[q] >> 18, next = q + 1 < WPT ? own[q + 1] >> 18 : run;
        if (IDX)
            bin_insertion_indexed(k0 + at, x0 + at, (int)(next - at));
        else
            bin_insertion(k0 + at, (int)(next - at));
    }
    __syncthreads();
    return k0;
}

}  // namespace evosort
