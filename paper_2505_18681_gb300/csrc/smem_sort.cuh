// Sorting building blocks that work on data already on chip: a warp bitonic
// sort of keys held in registers and a CTA merge sort of a tile held in
// shared memory (insertion-sorted base runs, then pairwise merges with
// merge-path splits per thread, as in Algorithm 3).
#pragma once

#include <type_traits>

#include "common.cuh"

namespace evosort {

// Merge-path split: number of keys of run A among the first k outputs of the
// stable merge of A (length la) and B (length lb).
template <typename U, typename I = size_t, typename AccA, typename AccB>
__device__ __forceinline__ I merge_path(AccA A, std::common_type_t<I> la, AccB B, std::common_type_t<I> lb,
                                        std::common_type_t<I> k) {
    I lo = k > lb ? k - lb : 0;
    I hi = k < la ? k : la;
    while (lo < hi) {
        const I mid = (lo + hi) >> 1;
        if ((U)B(k - 1 - mid) < (U)A(mid))
            hi = mid;
        else
            lo = mid + 1;
    }
    return lo;
}

// Longest base run sorted in registers: 32 keys of 4 bytes, 16 of 8 bytes
// (with their values); longer runs are insertion-sorted in shared memory.
template <typename U>
__host__ __device__ constexpr int reg_run_max() { return sizeof(U) == 4 ? 32 : 16; }

// Insertion sort of the first len <= R keys (and values) of a register array:
// key i moves left past every strictly greater key, one neighbour exchange at
// a time, so equal keys keep their order (stable).  The loops are unrolled
// over R, so the arrays stay in registers; positions len..R-1 are not touched.
template <typename U, bool PAIRS, int R>
__device__ __forceinline__ void reg_insertion_sort(U (&k)[R], uint32_t (&v)[R], int len) {
#pragma unroll
    for (int i = 1; i < R; ++i) {
        if (i < len) {
#pragma unroll
            for (int j = i; j > 0; --j) {
                const bool sw = k[j - 1] > k[j];
                const U lo = sw ? k[j] : k[j - 1];
                const U hi = sw ? k[j - 1] : k[j];
                k[j - 1] = lo;
                k[j] = hi;
                if (PAIRS) {
                    const uint32_t vl = sw ? v[j] : v[j - 1];
                    const uint32_t vh = sw ? v[j - 1] : v[j];
                    v[j - 1] = vl;
                    v[j] = vh;
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Merge rounds of the CTA merge sort: k0/v0 hold sorted runs of w keys, k1/v1
// are scratch of the same size; the run width doubles.  Stable.  Returns 0 if
// the result is in k0/v0, 1 if in k1/v1.  All threads of the CTA must call it.
// ---------------------------------------------------------------------------
template <typename U, bool PAIRS, bool PAD, bool POW2 = false>
__device__ __forceinline__ int smem_merge_rounds(U* k0, U* k1, uint32_t* v0, uint32_t* v1, int len, int w0) {
    // element i of each array lives at ix(i): with PAD, one spare word per 32
    // (the caller sizes the arrays for that), so lanes whose positions are a
    // power of two apart fall in different banks
    auto ix = [](int i) { return PAD ? i + (i >> 5) : i; };
    const int nt = blockDim.x;
    const int chunk = (len + nt - 1) / nt;
    U* ks = k0;
    U* kd = k1;
    uint32_t* vs = v0;
    uint32_t* vd = v1;
    int which = 0;
    for (int w = w0; w < len; w <<= 1) {
        int o = threadIdx.x * chunk;
        const int oend = o + chunk < len ? o + chunk : len;
        while (o < oend) {
            const int pbase = POW2 ? o & -(2 * w) : (o / (2 * w)) * (2 * w);   // (POW2: w is a power of two)
            const int la = (pbase + w < len ? pbase + w : len) - pbase;
            const int lb = (pbase + 2 * w < len ? pbase + 2 * w : len) - pbase - la;
            const int bbase = pbase + la;
            const int k = o - pbase;
            int ia = merge_path<U, int>([&](int i) { return ks[ix(pbase + i)]; }, la,
                                        [&](int i) { return ks[ix(bbase + i)]; }, lb, k);
            int ib = k - ia;
            const int stop = (pbase + la + lb < oend ? pbase + la + lb : oend);
            // head key of each run in a register: one shared load per output
            U ha = ia < la ? ks[ix(pbase + ia)] : (U)0;
            U hb = ib < lb ? ks[ix(bbase + ib)] : (U)0;
            for (; o < stop; ++o) {
                const bool takeB = ia >= la || (ib < lb && hb < ha);
                if (takeB) {
                    kd[ix(o)] = hb;
                    if (PAIRS) vd[ix(o)] = vs[ix(bbase + ib)];
                    ++ib;
                    if (ib < lb) hb = ks[ix(bbase + ib)];
                } else {
                    kd[ix(o)] = ha;
                    if (PAIRS) vd[ix(o)] = vs[ix(pbase + ia)];
                    ++ia;
                    if (ia < la) ha = ks[ix(pbase + ia)];
                }
            }
        }
        __syncthreads();
        U* t = ks; ks = kd; kd = t;
        uint32_t* tv = vs; vs = vd; vd = tv;
        which ^= 1;
    }
    return which;
}

// ---------------------------------------------------------------------------
// CTA merge sort of len <= capacity keys (and values) in shared memory.
// k0/v0 hold the input; k1/v1 are scratch of the same size.  Base runs of
// tins keys are insertion-sorted (one thread per run: in registers up to R
// keys, in shared memory beyond), then merged pairwise, the run
// width doubling.  Stable.  Returns 0 if the result is in k0/v0, 1 if in
// k1/v1.  All threads of the CTA must call it.
// ---------------------------------------------------------------------------
template <typename U, bool PAIRS, int R = reg_run_max<U>(), bool PAD = false>
__device__ int smem_merge_sort(U* k0, U* k1, uint32_t* v0, uint32_t* v1, int len, int tins) {
    auto ix = [](int i) { return PAD ? i + (i >> 5) : i; };   // as in the rounds
    const int nt = blockDim.x;
    const int runs = (len + tins - 1) / tins;
    if (tins <= R) {
        // one run per thread, loaded into registers, sorted, stored back
        // (a thread's run is contiguous in shared memory, so a warp's lanes
        // sit tins words apart; registers keep the exchanges off the banks)
        for (int r = threadIdx.x; r < runs; r += nt) {
            const int lo = r * tins;
            const int m = lo + tins < len ? tins : len - lo;
            U k[R];
            uint32_t v[R];
#pragma unroll
            for (int j = 0; j < R; ++j) {
                k[j] = j < m ? k0[ix(lo + j)] : (U)0;
                v[j] = (PAIRS && j < m) ? v0[ix(lo + j)] : 0u;
            }
            reg_insertion_sort<U, PAIRS, R>(k, v, m);
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (j < m) {
                    k0[ix(lo + j)] = k[j];
                    if (PAIRS) v0[ix(lo + j)] = v[j];
                }
        }
    } else {
        for (int r = threadIdx.x; r < runs; r += nt) {
            const int lo = r * tins;
            const int hi = lo + tins < len ? lo + tins : len;
            for (int i = lo + 1; i < hi; ++i) {
                const U key = k0[ix(i)];
                const uint32_t val = PAIRS ? v0[ix(i)] : 0u;
                int j = i;
                while (j > lo && k0[ix(j - 1)] > key) {   // strictly greater: stable
                    k0[ix(j)] = k0[ix(j - 1)];
                    if (PAIRS) v0[ix(j)] = v0[ix(j - 1)];
                    --j;
                }
                k0[ix(j)] = key;
                if (PAIRS) v0[ix(j)] = val;
            }
        }
    }
    __syncthreads();
    return smem_merge_rounds<U, PAIRS, PAD>(k0, k1, v0, v1, len, tins);
}

// ---------------------------------------------------------------------------
// CTA radix sort (Algorithms 4a/4b in one CTA): stable LSD passes over 8-bit
// digits of k - lo, from k0/v0 through k1/v1, for len <= 32 * COLS keys per
// warp.  passes: digits, from bit first on.  counts: NT / 32 x 256 16-bit
// counters.  Returns 0 if the result is in k0/v0, 1 if in k1/v1.  All threads
// of the CTA must call it.
// ---------------------------------------------------------------------------
template <typename U, bool PAIRS, int NT, int COLS>
__device__ __noinline__ int smem_radix_sort(U* k0, U* k1, uint32_t* v0, uint32_t* v1, int len, U lo, int first,
                                            int passes, uint16_t* counts, uint32_t* scratch) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cols = (len + NT - 1) / NT;   // columns of 32 keys per warp, consecutive in the array
    const int wofs = warp * 32 * cols + lane;
    const uint32_t lt = lanemask_lt();
    uint16_t* const mine = counts + warp * 256;
    for (int p = 0; p < passes; ++p) {
        for (int i = lane; i < 128; i += 32) ((uint32_t*)mine)[i] = 0u;
        __syncwarp();
        U key[COLS];
        uint32_t val[PAIRS ? COLS : 1];
        uint32_t dr[COLS];   // digit | rank << 16
#pragma unroll
        for (int i = 0; i < COLS; ++i) {
            if (i < cols) {
                const int s = wofs + 32 * i;
                const bool have = s < len;
                key[i] = have ? k0[s] : (U)0;
                if (PAIRS) val[PAIRS ? i : 0] = have ? v0[s] : 0u;
                const uint32_t d = digit_of((U)(key[i] - lo), first + 8 * p, 0xFFu);
                uint32_t peers = __ballot_sync(0xffffffffu, have);   // lanes with the same digit
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    const uint32_t m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
                    peers &= (d >> b) & 1u ? m : ~m;
                }
                uint32_t before = 0;
                const int leader = 31 - __clz((int)peers);
                if (have && lane == leader) {
                    before = mine[d];
                    mine[d] = (uint16_t)(before + __popc(peers));
                }
                before = __shfl_sync(0xffffffffu, before, have ? leader : lane);
                dr[i] = d | (before + (uint32_t)__popc(peers & lt)) << 16;
                __syncwarp();
            }
        }
        __syncthreads();
        uint32_t sum = 0, tot;
        if (tid < 256)
            for (int w = 0; w < NW; ++w) sum += counts[w * 256 + tid];
        uint32_t run = block_exclusive_scan<NT>(sum, scratch, &tot);
        if (tid < 256) {
            for (int w = 0; w < NW; ++w) {
                const uint32_t c = counts[w * 256 + tid];
                counts[w * 256 + tid] = (uint16_t)run;
                run += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < COLS; ++i) {
            if (i < cols && wofs + 32 * i < len) {
                const uint32_t at = mine[dr[i] & 0xFFFFu] + (dr[i] >> 16);
                k1[at] = key[i];
                if (PAIRS) v1[at] = val[PAIRS ? i : 0];
            }
        }
        __syncthreads();
        U* t = k0; k0 = k1; k1 = t;
        uint32_t* tv = v0; v0 = v1; v1 = tv;
    }
    return passes & 1;
}

// ---------------------------------------------------------------------------
// Warp bitonic sort of 32*KW keys, ascending.  Lane L holds keys
// [L*KW, (L+1)*KW) of the sequence in k[0..KW) (blocked layout); KW is a power
// of two.  Not stable (used for keys-only sorts, where equal keys are
// identical bit patterns, so the output is the same either way).
// ---------------------------------------------------------------------------
template <typename U>
__device__ __forceinline__ void cmp_swap(U& a, U& b, bool up) {
    const U lo = a < b ? a : b;
    const U hi = a < b ? b : a;
    a = up ? lo : hi;
    b = up ? hi : lo;
}

template <typename U, int KW>
__device__ __forceinline__ void warp_bitonic_sort(U (&k)[KW]) {
    const int lane = threadIdx.x & 31;
    constexpr int N = 32 * KW;
#pragma unroll
    for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= KW) {
                // partner element lives in another lane at the same register
                const int lstride = stride / KW;
#pragma unroll
                for (int r = 0; r < KW; ++r) {
                    const int idx = lane * KW + r;
                    const bool up = ((idx & size) == 0);
                    const U other = __shfl_xor_sync(0xffffffffu, k[r], lstride);
                    const bool lower = (lane & lstride) == 0;   // this lane holds the lower index
                    const bool keep_min = (lower == up);
                    const U mn = k[r] < other ? k[r] : other;
                    const U mx = k[r] < other ? other : k[r];
                    k[r] = keep_min ? mn : mx;
                }
            } else {
#pragma unroll
                for (int r = 0; r < KW; ++r) {
                    if ((r & stride) == 0) {
                        const int idx = lane * KW + r;
                        const bool up = ((idx & size) == 0);
                        cmp_swap(k[r], k[r + stride], up);
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// CTA sort of n keys in k0 (k1: scratch of the same size), keys only, whatever
// their distribution: runs of 32 * KW keys by one warp each, then merge rounds.
// Returns the sorted array, k0 or k1.  The serial merges of a round cost more
// than the bitonic stages that spare it, so the runs are as long as leaves most
// warps one.  2,000 segments of 4,000 Zipf int32 keys, 305 CTAs: 374 us by runs of
// 8 keys, 179 so.
// ---------------------------------------------------------------------------
template <typename U, int KW>
__device__ __noinline__ void warp_sort_runs(U* k, int n) {
    constexpr int RUN = 32 * KW;
    const int lane = threadIdx.x & 31;
    for (int at = (int)(threadIdx.x >> 5) * RUN; at < n; at += (int)(blockDim.x >> 5) * RUN) {
        U x[KW];
#pragma unroll
        for (int r = 0; r < KW; ++r) x[r] = at + r * 32 + lane < n ? k[at + r * 32 + lane] : ~(U)0;
        __syncwarp();
        warp_bitonic_sort<U, KW>(x);
#pragma unroll
        for (int r = 0; r < KW; ++r)
            if (at + lane * KW + r < n) k[at + lane * KW + r] = x[r];
    }
}

template <typename U>
__device__ __noinline__ U* smem_sort_any(U* k0, U* k1, int n) {
    int w;
    if (n <= 512) {
        warp_sort_runs<U, 1>(k0, n);
        w = 32;
    } else if (n <= 2048) {
        warp_sort_runs<U, 4>(k0, n);
        w = 128;
    } else {
        warp_sort_runs<U, 16>(k0, n);
        w = 512;
    }
    __syncthreads();
    return smem_merge_rounds<U, false, false, true>(k0, k1, nullptr, nullptr, n, w) ? k1 : k0;
}

}  // namespace evosort
