// Radix sort of a mid-sized array in one launch (keys, or keys and values;
// 8-bit digits): the LSD passes of Algorithms 4a/4b with the whole array held
// on chip.
//
// Up to a few million keys the chain of kernels (histogram, scan, a pass per
// digit, a copy) is all launches, look-back waits and idle SMs: 1e6 int32 keys
// took 100 us, of which the keys' own traffic is a few.  Here every CTA keeps
// one contiguous chunk in registers, and a cooperative launch makes all CTAs
// resident, so they can meet at barriers over the grid:
//
//   load      each CTA loads its chunk and records, for the whole array, the
//             smallest and largest mapped key, the bits that vary and the
//             order of neighbours;
//   plan      every CTA takes the same decisions K1, K1b and K2 take: input in
//             order or in reverse order is copied, a narrow range is counted
//             by value, a range that needs fewer digits is ranked as key - min,
//             and digits equal in all keys are skipped;
//   pass      ranks its chunk stably (match masks, as the register tile),
//             publishes its 256 digit counts, meets the others, sums the counts
//             of all chunks before its own, and writes its keys to their places
//             in the output: the paper's per-thread histograms and thread-wise
//             offsets, with CTAs as threads.  Every chunk is in registers before
//             the first CTA writes, so one buffer serves all passes, in place or
//             not.
#include "api_internal.h"
#include "fused.cuh"
#include "radix.cuh"

namespace evosort {
namespace {

constexpr int kFusThreads = 1024;
constexpr int kFusWarps = kFusThreads / 32;
constexpr int kFusBins = 256;
constexpr int kFusCount = 8192;   // values of the narrow-range counting sort

// Largest number of keys per thread: what the registers hold beside the ranks.
template <typename U, bool PAIRS>
__host__ __device__ constexpr int fus_kpt() { return sizeof(U) == 4 ? (PAIRS ? 12 : 16) : (PAIRS ? 8 : 12); }

// Control words (64-bit, zeroed by the host): largest complement of a mapped
// key, largest mapped key, bits set in some key, bits clear in some key, order
// flags (bit ORD_*), arrivals at the barriers.
enum : int { FUS_NOTMIN = 0, FUS_MAX = 1, FUS_SET = 2, FUS_CLEAR = 3, FUS_ORDER = 4, FUS_BARRIER = 5, FUS_WORDS = 8 };

struct FusedArgs {
    const void* in;
    void* out;
    const uint32_t* vin;
    uint32_t* vout;
    uint32_t n;
    int cols;                   // keys per thread: the chunk is cols * kFusThreads keys
    KeyMap map;
    unsigned long long* ctl;    // FUS_WORDS
    uint16_t* counts;           // gridDim.x * kFusBins digit counts
    uint32_t* bins;             // kFusCount value counts (keys only)
    PassDesc* desc;             // sizeof(U) + 1 entries, for the profile's records
    uint32_t* status;
    uint32_t limit;             // polls of one barrier
};

template <typename U, bool PAIRS>
constexpr size_t fus_smem() {
    // reorder buffer, warp counters and match masks (or the value bins), tile
    // starts, global starts
    return (size_t)kFusThreads * fus_kpt<U, PAIRS>() * (sizeof(U) + (PAIRS ? 4 : 0)) +
           (size_t)kFusWarps * kFusBins * 4 * 2 + (size_t)kFusBins * 8;
}

// Barrier over the grid; step counts them from 1.  False if it ran out of
// polls (a.limit, as the look-back's waits); every CTA then gives up, here or at
// its next barrier, which the ones that left never reach.  What a barrier
// protects is read only after it was complete, so nothing is read too early.
__device__ __forceinline__ bool fus_barrier(const FusedArgs& a, uint32_t step, int* s_stop) {
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t* const word = (uint32_t*)(a.ctl + FUS_BARRIER);
        __threadfence();
        atomicAdd(word, 1u);
        const uint32_t want = step * gridDim.x;
        uint32_t polls = 0;
        int stop = 0;
        while (ld_relaxed(word) < want) {
            if (++polls > a.limit) {
                atomicOr(a.status, ST_TIMEOUT);
                stop = 1;
                break;
            }
            if (polls > 32u) __nanosleep(64);
        }
        __threadfence();
        *s_stop = stop;
    }
    __syncthreads();
    return *s_stop == 0;
}

template <typename U, bool PAIRS>
__global__ void __launch_bounds__(kFusThreads) radix_fused(const __grid_constant__ FusedArgs a) {
    constexpr int KPT = fus_kpt<U, PAIRS>();
    constexpr int NP = sizeof(U);
    extern __shared__ __align__(16) unsigned char smem[];
    U* s_r = (U*)smem;
    uint32_t* s_rv = (uint32_t*)(smem + (size_t)kFusThreads * KPT * sizeof(U));
    uint32_t* s_wc = (uint32_t*)(smem + (size_t)kFusThreads * KPT * (sizeof(U) + (PAIRS ? 4 : 0)));
    uint32_t* s_wm = s_wc + kFusWarps * kFusBins;
    uint32_t* s_excl = s_wm + kFusWarps * kFusBins;   // first place of a digit in the chunk
    uint32_t* s_to = s_excl + kFusBins;               // global place of the digit's run - s_excl
    __shared__ unsigned long long s_red[4];
    __shared__ uint32_t s_flags, s_w[kFusWarps], s_part[2][8][kFusBins / 2][2];
    __shared__ int s_stop, s_const;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cols = a.cols;
    const uint32_t n = a.n;
    const uint32_t base = blockIdx.x * (uint32_t)(cols * kFusThreads);
    const int valid = (int)min(n - base, (uint32_t)(cols * kFusThreads));
    const int wofs = warp * 32 * cols + lane;   // key i of a lane sits at wofs + 32 * i
    const KeyMap map = a.map;
    const U* in = (const U*)a.in;
    U* out = (U*)a.out;

    // ---- load: keys (and values) into registers, facts about all of them
    U key[KPT];
    uint32_t val[PAIRS ? KPT : 1];
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const int s = wofs + 32 * i;
        if (i < cols && s < valid) {
            key[i] = in[base + s];
            if (PAIRS) val[PAIRS ? i : 0] = a.vin[base + s];
        }
    }
    if (tid < 4) s_red[tid] = 0ull;
    if (tid == 0) s_flags = 0u;
    for (int i = tid; i < kFusWarps * kFusBins; i += kFusThreads) s_wm[i] = 0u;
    if (!PAIRS)
        for (uint32_t i = blockIdx.x * kFusThreads + tid; i < kFusCount; i += gridDim.x * kFusThreads) a.bins[i] = 0u;
    __syncthreads();
    {
        U notmin = 0, mx = 0, set = 0, clear = 0;
        uint32_t flags = 0;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            if (i < cols) {
                const int s = wofs + 32 * i;
                if (s < valid) {
                    key[i] = map_fwd(key[i], map);
                    const U c = ~key[i];
                    notmin = c > notmin ? c : notmin;
                    mx = key[i] > mx ? key[i] : mx;
                    set |= key[i];
                    clear |= c;
                }
                // the next key: the next lane's, or for lane 31 the one in memory
                U next = __shfl_down_sync(0xffffffffu, key[i], 1);
                const bool some = s < valid && base + (uint32_t)s + 1u < n;
                if (some && (lane == 31 || s + 1 >= valid)) next = map_fwd(in[base + s + 1], map);
                if (some) flags |= key[i] > next ? 1u << ORD_DESCENT : (key[i] < next ? 1u << ORD_ASCENT : 1u << ORD_EQUAL);
            }
        }
        unsigned long long r[4] = {notmin, mx, set, clear};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned long long y = __shfl_xor_sync(0xffffffffu, r[q], o);
                r[q] = q < 2 ? (y > r[q] ? y : r[q]) : (r[q] | y);
            }
        }
        flags = __reduce_or_sync(0xffffffffu, flags);
        if (lane == 0) {
            atomicMax(&s_red[0], r[0]);
            atomicMax(&s_red[1], r[1]);
            atomicOr(&s_red[2], r[2]);
            atomicOr(&s_red[3], r[3]);
            if (flags) atomicOr(&s_flags, flags);
        }
    }
    __syncthreads();
    if (tid < 2) atomicMax(&a.ctl[tid], s_red[tid]);
    if (tid >= 2 && tid < 4) atomicOr(&a.ctl[tid], s_red[tid]);
    if (tid == 4) atomicOr(&a.ctl[FUS_ORDER], (unsigned long long)s_flags);
    uint32_t step = 0;
    if (!fus_barrier(a, ++step, &s_stop)) return;

    // ---- plan, the same in every CTA
    const U mn = (U)~(U)a.ctl[FUS_NOTMIN];
    const U span = (U)((U)a.ctl[FUS_MAX] - mn);
    const U vary = (U)a.ctl[FUS_SET] & (U)a.ctl[FUS_CLEAR];
    const uint32_t order = (uint32_t)a.ctl[FUS_ORDER];
    const bool first = blockIdx.x == 0 && tid == 0;
    const bool in_order = !(order >> ORD_DESCENT & 1u);
    const bool reversed = !in_order && !(order >> ORD_ASCENT & 1u) && !(PAIRS && (order >> ORD_EQUAL & 1u));
    if (in_order || reversed) {
        if (first) a.desc[NP].fixup = reversed ? FIX_REVERSE : (a.in == a.out ? FIX_NONE : FIX_IN_TO_OUT);
        if (in_order && a.in == a.out) return;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const int s = wofs + 32 * i;
            if (i < cols && s < valid) {
                const uint32_t to = reversed ? n - 1u - (base + s) : base + s;
                out[to] = map_inv(key[i], map);
                if (PAIRS) a.vout[to] = val[PAIRS ? i : 0];
            }
        }
        return;
    }
    if (!PAIRS && (unsigned long long)span >= 256ull && (unsigned long long)span < (unsigned long long)kFusCount) {
        // narrow range: count by value, write the output from the counts
        uint32_t* s_h = s_wc;   // kFusCount words
        for (int i = tid; i < kFusCount; i += kFusThreads) s_h[i] = 0u;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (i < cols && wofs + 32 * i < valid) atomicAdd(&s_h[(uint32_t)(U)(key[i] - mn)], 1u);
        __syncthreads();
        for (int i = tid; i < kFusCount; i += kFusThreads)
            if (s_h[i]) atomicAdd(&a.bins[i], s_h[i]);
        if (!fus_barrier(a, ++step, &s_stop)) return;
        constexpr int PER = kFusCount / kFusThreads;
        uint32_t c[PER], sum = 0, tot;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            c[j] = a.bins[tid * PER + j];
            sum += c[j];
        }
        uint32_t run = block_exclusive_scan<kFusThreads>(sum, s_wm, &tot);   // (the value bins end before s_wm + 64)
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            s_h[tid * PER + j] = run;
            run += c[j];
        }
        __syncthreads();
        for (int s = tid; s < valid; s += kFusThreads) {
            int lo = 0, hi = kFusCount - 1;   // the last value that starts at or before this place
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_h[mid] <= base + (uint32_t)s)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            out[base + s] = map_inv((U)(mn + (U)lo), map);
        }
        return;
    }
    int varying = 0;
#pragma unroll
    for (int p = 0; p < NP; ++p) varying += ((vary >> (8 * p)) & 0xFFu) != 0;
    const int bits = 64 - __clzll((long long)(unsigned long long)span);   // span > 0: not in order
    const bool rebased = (bits + 7) / 8 < varying;
    const U bias = rebased ? mn : (U)0;
    if (rebased) {
#pragma unroll
        for (int i = 0; i < KPT; ++i) key[i] -= bias;
    }
    const int last = rebased ? (bits + 7) / 8 - 1 : (63 - __clzll((long long)(unsigned long long)vary)) / 8;
    bool loaded = true;   // the chunk is in registers

    for (int p = 0; p <= last; ++p) {
        const int shift = 8 * p;
        if (!rebased && ((vary >> shift) & 0xFFu) == 0) continue;
        if (!loaded) {
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const int s = wofs + 32 * i;
                if (i < cols && s < valid) {
                    key[i] = __ldcg(out + base + s);
                    if (PAIRS) val[PAIRS ? i : 0] = __ldcg(a.vout + base + s);
                }
            }
            loaded = true;
        }
        // ---- stable rank among equal digits of the warp (columns in input
        // order, lanes in order inside a column)
        uint32_t* wc = s_wc + warp * kFusBins;
        uint32_t* wm = s_wm + warp * kFusBins;
        for (int i = lane; i < kFusBins / 4; i += 32) ((uint4*)wc)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (tid == 0) s_const = 0;
        __syncwarp();
        uint32_t rk[(KPT + 1) / 2];
        const uint32_t lt = lanemask_lt();
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            if (i < cols) {   // the same for the whole grid
                const bool have = wofs + 32 * i < valid;
                const uint32_t d = digit_of(key[i], shift, 0xFFu);
                if (have) atomicOr(&wm[d], 1u << lane);
                __syncwarp();
                const uint32_t peers = have ? wm[d] : 1u << lane;
                __syncwarp();
                const int leader = 31 - __clz((int)peers);
                uint32_t o = 0;
                if (have && lane == leader) {
                    o = atomicAdd(&wc[d], (uint32_t)__popc(peers));
                    wm[d] = 0u;
                }
                o = __shfl_sync(0xffffffffu, o, leader) + (uint32_t)__popc(peers & lt);
                rk[i / 2] = i & 1 ? __byte_perm(rk[i / 2], o, 0x5410) : o;
                __syncwarp();
            }
        }
        __syncthreads();
        // ---- the chunk's count of each digit; warp counters -> places in the chunk
        uint32_t cnt = 0;
        if (tid < kFusBins) {
#pragma unroll 8
            for (int w = 0; w < kFusWarps; ++w) cnt += s_wc[w * kFusBins + tid];
            a.counts[blockIdx.x * kFusBins + tid] = (uint16_t)cnt;   // at most 16,384
            uint32_t inc = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) s_w[warp] = inc;
            asm volatile("bar.sync 1, 256;" ::: "memory");
            uint32_t run = inc - cnt;
            for (int w = 0; w < warp; ++w) run += s_w[w];
            s_excl[tid] = run;
#pragma unroll 8
            for (int w = 0; w < kFusWarps; ++w) {
                const uint32_t c = s_wc[w * kFusBins + tid];
                s_wc[w * kFusBins + tid] = run;
                run += c;
            }
        }
        if (!fus_barrier(a, ++step, &s_stop)) return;   // all counts are out, every chunk is in registers
        // ---- global start of this chunk's keys of each digit: eight rows of
        // counts at a time, two digits per thread
        {
            const int pair = tid & (kFusBins / 2 - 1), g = tid / (kFusBins / 2);
            uint32_t t0 = 0, t1 = 0, b0 = 0, b1 = 0;
            const uint32_t* rows = (const uint32_t*)a.counts + pair;
            for (uint32_t r = g; r < gridDim.x; r += 8u) {
                const uint32_t c = __ldcg(rows + r * (kFusBins / 2));
                const uint32_t c0 = c & 0xFFFFu, c1 = c >> 16;
                t0 += c0;
                t1 += c1;
                if (r < blockIdx.x) {
                    b0 += c0;
                    b1 += c1;
                }
            }
            s_part[0][g][pair][0] = t0;
            s_part[0][g][pair][1] = t1;
            s_part[1][g][pair][0] = b0;
            s_part[1][g][pair][1] = b1;
        }
        __syncthreads();
        if (tid < kFusBins) {
            uint32_t tot = 0, before = 0;
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                tot += s_part[0][g][tid >> 1][tid & 1];
                before += s_part[1][g][tid >> 1][tid & 1];
            }
            if (tot == n) s_const = 1;   // one digit holds every key: nothing moves
            uint32_t inc = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) s_w[warp] = inc;
            asm volatile("bar.sync 1, 256;" ::: "memory");
            uint32_t start = inc - tot + before;
            for (int w = 0; w < warp; ++w) start += s_w[w];
            s_to[tid] = start - s_excl[tid];
        }
        __syncthreads();
        const bool same = s_const != 0;
        const bool end = p == last;
        if (same && !end) {   // (the last digit of a range is never equal in all keys unless it was rebased)
            // the next pass ranks what is in the registers; nobody writes the
            // counts before every CTA has read them
            if (!fus_barrier(a, ++step, &s_stop)) return;
            continue;
        }
        if (first) a.desc[p].active = 1;
        // ---- reorder the chunk by digit, then write its runs
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            if (i < cols && wofs + 32 * i < valid) {
                const uint32_t pos = wc[digit_of(key[i], shift, 0xFFu)] + (i & 1 ? rk[i / 2] >> 16 : rk[i / 2] & 0xFFFFu);
                s_r[pos] = key[i];
                if (PAIRS) s_rv[pos] = val[PAIRS ? i : 0];
            }
        }
        __syncthreads();
        for (int s = tid; s < valid; s += kFusThreads) {
            const U k = s_r[s];
            const uint32_t to = s_to[digit_of(k, shift, 0xFFu)] + (uint32_t)s;
            if (to < n) {   // always, unless a barrier gave up
                out[to] = end ? map_inv((U)(k + bias), map) : k;
                if (PAIRS) a.vout[to] = s_rv[s];
            }
        }
        if (end) return;
        if (!fus_barrier(a, ++step, &s_stop)) return;
        loaded = false;
    }
}

template <typename U, bool PAIRS>
cudaError_t launch_fused(FusedArgs& a, int max_grid, cudaStream_t s) {
    static bool configured = false;
    if (!configured) {
        const cudaError_t e = cudaFuncSetAttribute(radix_fused<U, PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)fus_smem<U, PAIRS>());
        if (e != cudaSuccess) return e;
        configured = true;
    }
    a.cols = (int)((a.n + (uint32_t)(max_grid * kFusThreads) - 1u) / (uint32_t)(max_grid * kFusThreads));
    const unsigned grid = (a.n + (uint32_t)(a.cols * kFusThreads) - 1u) / (uint32_t)(a.cols * kFusThreads);
    void* args[] = {(void*)&a};
    return cudaLaunchCooperativeKernel((const void*)radix_fused<U, PAIRS>, dim3(grid), dim3(kFusThreads), args,
                                       fus_smem<U, PAIRS>(), s);
}

}  // namespace

size_t fused_max_keys(int w, bool pairs) {
    const int kpt = w == 4 ? (pairs ? fus_kpt<uint32_t, true>() : fus_kpt<uint32_t, false>())
                           : (pairs ? fus_kpt<uint64_t, true>() : fus_kpt<uint64_t, false>());
    return (size_t)sm_count() * kFusThreads * kpt;
}

size_t fused_ctl_bytes() { return FUS_WORDS * sizeof(unsigned long long); }

cudaError_t launch_radix_fused(int w, const void* in, void* out, const uint32_t* vin, uint32_t* vout, size_t n,
                               const KeyMap& map, unsigned long long* ctl, void* counts, void* bins, PassDesc* desc,
                               uint32_t* status, cudaStream_t s) {
    FusedArgs a;
    a.in = in;
    a.out = out;
    a.vin = vin;
    a.vout = vout;
    a.n = (uint32_t)n;
    a.map = map;
    a.ctl = ctl;
    a.counts = (uint16_t*)counts;
    a.bins = (uint32_t*)bins;
    a.desc = desc;
    a.status = status;
    a.limit = wait_limit();
    const int sms = sm_count();
    if (w == 4) return vout ? launch_fused<uint32_t, true>(a, sms, s) : launch_fused<uint32_t, false>(a, sms, s);
    return vout ? launch_fused<uint64_t, true>(a, sms, s) : launch_fused<uint64_t, false>(a, sms, s);
}

}  // namespace evosort
