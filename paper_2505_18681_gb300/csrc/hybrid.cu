// Partition sort of large arrays of keys (keys only): two unstable partition
// steps by the leading bits, then one sort per bucket on chip.
//
// The LSD passes of Algorithms 4a/4b move every key once per digit that
// varies (eight times for random 64-bit keys) and must be stable, which costs
// match masks and per-warp counters in shared memory.  Going from the most
// significant bits down, each step may place equal digits in any order (equal
// keys are identical bit patterns), and once a bucket fits in shared memory
// its remaining bits are sorted there: every key moves three times, whatever
// its width, and a step ranks a key with one shared atomic.
//
//   K_hs hybrid_sample     one CTA samples kHybSample keys and cuts the key range
//                          into bins: equal stretches where the sample spreads
//                          evenly over them, else bins of equal sampled mass
//                          (4096 cells of the range, light cells joined and
//                          heavy cells split by their next bits).  It also
//                          decides whether the path is tried: not for a
//                          sample in order or in reverse order, for values that
//                          repeat often in the sample, or for a narrow range;
//   K_ha hybrid_count_a    one read of the keys: exact bin counts, exact range;
//   K_hp hybrid_plan       one CTA: where each bin starts, into how many
//                          buckets its keys are cut next, the tiles of the
//                          second step;
//   K_hm hybrid_partition  step A: tiles of the input to their bins (in the
//                          scratch array).  A tile counts its bins with one
//                          shared atomic per key, whose old value is the key's
//                          place, reserves its share of each bin with one
//                          global atomic, reorders in shared memory and writes
//                          runs.  No tile waits for another;
//   K_hb hybrid_count_b    one read: exact counts of every bin's buckets;
//   K_hq hybrid_scan_b     bucket starts; the path is given up here if some
//                          bucket of more than one value is so long that one
//                          CTA would hold up the rest (nothing but scratch was
//                          written);
//   K_hm hybrid_partition  step B: each bin's keys to their buckets (output);
//   K_hg hybrid_groups     cuts the output into runs of whole buckets that fit a
//                          CTA's shared memory;
//   K_hl hybrid_local      sorts each run there (bin_sort.cuh), in place in the
//                          output; a bucket that is longer than that is cut
//                          again by one CTA (cta_sort.cuh);
//   K_hf hybrid_finish     when the path was given up: clears the scratch it
//                          used (it lies in the look-back slots), so that the
//                          radix passes, launched next, find it zeroed.
//
// Every decision is the device's; every kernel returns at once when the path
// is off, and the radix kernels return at once when it was taken.  (One
// cooperative kernel with barriers over the grid in place of the launches was
// slower: 4e7 int64 keys 0.95 against 0.84 ms with its steps inlined, whose
// registers spilled, 1.18 ms with the steps as functions.)
#include <algorithm>
#include <cmath>

#include "api_internal.h"
#include "cta_sort.cuh"
#include "hybrid.cuh"
#include "radix.cuh"

namespace evosort {
namespace {

constexpr int kHybCells = 4096;       // cells of the sampled range
constexpr int kHybCellBits = 12;
constexpr int kHybSample = 8192;      // sampled keys
constexpr int kHybMassMin = 14;       // sampled keys per bin aimed at, at least (about 585 bins)
constexpr int kHybCellShare = 32;     // empty cells that count as much as that
constexpr int kHybBins = 1024;        // most bins of step A, most buckets of one bin
constexpr int kHybRepeat = 24;        // hits of one hash slot of the sample that mean a frequent value
constexpr int kHybThreads = kCtaThreads;
// A bucket that no local sort holds is sorted by one CTA beside the others; up
// to this share of the keys it ends about when they do (one CTA of 304 has a
// three-hundredth of all keys to sort anyway).
constexpr size_t kHybLongShare = 256;
constexpr int kHybLocalWords = kCtaWords;   // words of four bins per thread of the local sort

// Flag of a bucket of one value that no local sort could hold: step B writes
// its keys in their final form.
constexpr uint32_t kHybFinal = 0x80000000u;   // n < 2^31

template <typename U>
__host__ __device__ constexpr int hyb_kpt() { return sizeof(U) == 4 ? 20 : 16; }
template <typename U>
__host__ __device__ constexpr int hyb_tile() { return kHybThreads * hyb_kpt<U>(); }
template <typename U>
__host__ __device__ constexpr int hyb_local_kpt() { return cta_kpt<U>(); }
template <typename U>
__host__ __device__ constexpr int hyb_cap() { return kHybThreads * hyb_local_kpt<U>(); }   // keys of one local sort
// keys per bucket aimed at: small enough that a bucket several times denser
// than its bin's average still fits a local sort, large enough that the tile's
// run in each bucket stays a whole sector or two
template <typename U>
__host__ __device__ constexpr int hyb_target() { return sizeof(U) == 4 ? 2048 : 1024; }
// Stretch of the array whose buckets one local sort takes: what is left of its
// room for a bucket that reaches past the stretch's end.
template <typename U>
__host__ __device__ constexpr int hyb_window() { return hyb_cap<U>() - 1536; }
// The counters that tiles reserve from are hot: thousands of tiles add to the
// same few hundred words, and atomics on one sector are served one after
// another.  Eight of them share a 32-byte sector (so that a warp's atomics are
// four requests), and each sector has a 128-byte line of its own, so that they
// spread over the L2 slices.  1e9 int32 / int64 keys, one step: 3.4 -> 2.7 /
// 5.4 -> 4.0 ms against consecutive words.
__host__ __device__ constexpr uint32_t hyb_spread(uint32_t b) { return (b >> 3) * 32u + (b & 7u); }
// One local sort: keys [start, start + len), all in [lo, lo + width]; (lz,
// mult) cut that range into the sort's bins.
struct __align__(16) HybGroup {
    uint32_t start, len;
    int lz;
    uint32_t mult;
    unsigned long long lo, width;
};

struct HybArgs {
    const void* in;
    void* tmp;
    void* out;
    size_t n;
    KeyMap map;
    uint32_t* ctl;               // HYB_WORDS words (hybrid.cuh)
    int mass;                    // sampled keys per equal stretch aimed at
    uint32_t* lut;               // kHybCells entries (see HybCut)
    unsigned long long* bin_lo;  // smallest and largest key of a bin's cells
    unsigned long long* bin_hi;
    uint32_t* count_a;           // keys per bin
    uint32_t* cursor_a;          // next free place of a bin (hyb_spread)
    uint32_t* base_a;            // kHybBins + 1 bin starts
    uint32_t* off_b;             // kHybBins + 1: first bucket of a bin
    uint32_t* lz_b;              // buckets of a bin: umulhi(norm32(key - bin_lo, lz), mult); bit 8 of
    uint32_t* mult_b;            // lz_b: every bucket is one value
    uint32_t* tile_b;            // kHybBins + 1: first step-B tile of a bin
    void* scratch;               // all of the arrays below, scratch16 16-byte words
    size_t scratch16;
    PassDesc* last;              // the entry after the radix passes
    uint32_t* buckets;           // bucket counts, then starts, then (after step B) ends (hyb_spread)
    struct HybGroup* groups;     // local sorts
    uint32_t longest;            // longest bucket of several values one CTA is left with
    uint32_t max_buckets;        // room of buckets
    uint32_t windows;            // stretches the local sorts are cut from
};

__device__ __forceinline__ bool hyb_on(const uint32_t* ctl) { return ctl[HYB_ON] != 0u && ctl[HYB_FAIL] == 0u; }

// The cut of step A.  A key's position is x = norm32(min(key - lo, width)), 32
// bits over the sampled range; keys below lo or above lo + width go to the
// ends.  Its bin is umulhi(x, bins) (equal stretches) or, through the table of
// the 4096 cells x >> 20, (x >> shift) + offset with the cell's shift (low 5
// bits of its entry: 20, or less where the cell is split) and offset.
// WIDE: 64-bit keys over the whole type (lo 0, lz 0): the position is the high
// word.
template <typename U, bool LIN, bool WIDE>
struct HybCut {
    U lo, width;
    int lz;
    uint32_t bins;
    __device__ __forceinline__ void load(const uint32_t* ctl) {
        lo = (U)(((unsigned long long)ctl[HYB_LO + 1] << 32) | ctl[HYB_LO]);
        width = (U)(((unsigned long long)ctl[HYB_WIDTH + 1] << 32) | ctl[HYB_WIDTH]);
        lz = (int)ctl[HYB_LZ];
        bins = ctl[HYB_BINS];
    }
    __device__ __forceinline__ uint32_t place(U k) const {
        if (WIDE) return (uint32_t)((unsigned long long)k >> 32);
        U d = (k > lo ? k : lo) - lo;
        d = d < width ? d : width;
        return norm32(d, lz);
    }
    __device__ __forceinline__ uint32_t bin(U k, const uint32_t* lut) const {
        const uint32_t x = place(k);
        if (LIN) return __umulhi(x, bins);
        const uint32_t e = lut[x >> (32 - kHybCellBits)];
        return __funnelshift_r(x, 0u, e) + (uint32_t)((int32_t)e >> 5);
    }
};

// Runs f with the variant of the cut (and of the key map: xor alone, or the
// general one of floats) that the control words name.
template <typename U, typename F>
__device__ __forceinline__ void hyb_variant(const uint32_t* ctl, const KeyMap& m, const F& f) {
    const bool lin = ctl[HYB_BINS] != 0u, wide = sizeof(U) == 8 && ctl[HYB_LZ] == 0u;
    const bool plain = m.f == 0 && m.r == 0;
    auto go = [&](auto cut) {
        cut.load(ctl);
        if (plain)
            f(cut, [c = (U)(m.s ^ m.x)](U k) { return (U)(k ^ c); });
        else
            f(cut, [&](U k) { return map_fwd(k, m); });
    };
    if (sizeof(U) == 8 && wide) {
        if (lin) go(HybCut<U, true, sizeof(U) == 8>()); else go(HybCut<U, false, sizeof(U) == 8>());
    } else {
        if (lin) go(HybCut<U, true, false>()); else go(HybCut<U, false, false>());
    }
}

__device__ __forceinline__ uint32_t hash32(unsigned long long k) {
    k *= 0x9E3779B97F4A7C15ull;
    return (uint32_t)(k >> 32);
}

// ---------------------------------------------------------------------------
// K_hs: the sample, by one CTA.
// ---------------------------------------------------------------------------
constexpr size_t hyb_sample_smem() {
    return kHybCells * 4 + kHybCells * 4 + kHybSample * 4 + kHybBins * 8 * 2 + kHybBins * 4;
}

template <typename U>
__global__ void __launch_bounds__(1024) hybrid_sample(HybArgs a) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* s_mass = (uint32_t*)smem;                             // kHybCells
    uint32_t* s_lut = s_mass + kHybCells;                           // kHybCells
    uint32_t* s_hash = s_lut + kHybCells;                           // kHybSample
    unsigned long long* s_lo = (unsigned long long*)(s_hash + kHybSample);
    unsigned long long* s_hi = s_lo + kHybBins;
    uint32_t* s_bin = (uint32_t*)(s_hi + kHybBins);
    __shared__ unsigned long long s_scr[33];
    __shared__ U s_mn[32], s_mx[32];
    constexpr int NT = 1024;
    constexpr int PER = kHybSample / NT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const U* in = (const U*)a.in;
    const size_t stride = a.n / kHybSample;   // n >= kHybSample, checked by the host

    U k[PER];
    U mn = ~(U)0, mx = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const size_t i = (size_t)tid * PER + j;
        k[j] = in[i * stride + (size_t)(((unsigned long long)hash32(i + 1) * stride) >> 32)];   // one in each stretch
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        k[j] = map_fwd(k[j], a.map);
        mn = k[j] < mn ? k[j] : mn;
        mx = k[j] > mx ? k[j] : mx;
    }
    for (int i = tid; i < kHybCells; i += NT) s_mass[i] = 0u;
    for (int i = tid; i < kHybSample; i += NT) s_hash[i] = 0u;
    for (int i = tid; i < kHybBins; i += NT) s_bin[i] = 0u;
    for (int o = 16; o > 0; o >>= 1) {
        const U x = __shfl_xor_sync(0xffffffffu, mn, o), y = __shfl_xor_sync(0xffffffffu, mx, o);
        mn = x < mn ? x : mn;
        mx = y > mx ? y : mx;
    }
    if (lane == 0) {
        s_mn[warp] = mn;
        s_mx[warp] = mx;
    }
    __syncthreads();
    mn = lane < NT / 32 ? s_mn[lane] : ~(U)0;
    mx = lane < NT / 32 ? s_mx[lane] : (U)0;
    for (int o = 16; o > 0; o >>= 1) {
        const U x = __shfl_xor_sync(0xffffffffu, mn, o), y = __shfl_xor_sync(0xffffffffu, mx, o);
        mn = x < mn ? x : mn;
        mx = y > mx ? y : mx;
    }
    const unsigned long long span = (unsigned long long)(U)(mx - mn);
    bool up = false, down = false;   // neighbours in the sample, of one warp
    {
        const U next = __shfl_down_sync(0xffffffffu, k[0], 1);
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const U y = j + 1 < PER ? k[j + 1] : (lane < 31 ? next : k[j]);
            up |= k[j] < y;
            down |= k[j] > y;
        }
    }
    const int any_up = __syncthreads_or(up), any_down = __syncthreads_or(down);
    // a range of under 2^14 values is sorted by counting or in two passes
    if (!any_up || !any_down || (span >> 14) == 0) return;   // HYB_ON stays 0

    // values that hold much of the sample: their slot of a hash table fills.
    // Over more than 24 bits such values end in buckets of several values,
    // which they make too long; up to 24 bits the radix sort needs three
    // passes, which are as fast as this path (1e9 Gaussian int64 keys: 20.8
    // against 22.2 ms) unless many keys leave it after one step as values of
    // their own (Zipf: 17.0 against 15.2 ms).
#pragma unroll
    for (int j = 0; j < PER; ++j) atomicAdd(&s_hash[hash32((unsigned long long)k[j]) >> 19], 1u);
    __syncthreads();
    bool often = false;
    for (int i = tid; i < kHybSample; i += NT) often |= s_hash[i] >= (uint32_t)kHybRepeat;
    if ((__syncthreads_or(often) != 0) == ((span >> 24) != 0)) return;
    if ((span >> 24) == 0 && a.n < kHybridMinNarrow) return;

    // a range that needs the top bit is widened to the whole type, so that the
    // high word of a 64-bit key is its position
    const bool whole = (span >> (8 * sizeof(U) - 1)) != 0;
    HybCut<U, false, false> cut;
    cut.lo = whole ? (U)0 : mn;
    cut.width = whole ? (U)~(U)0 : (U)span;
    cut.lz = __clzll((long long)(unsigned long long)cut.width);
    cut.bins = 0u;
    // bits of x below the smallest key step: a cell is not split further
    const int sbmax = max(0, min(20 - max(0, cut.lz - 32), 10));
#pragma unroll
    for (int j = 0; j < PER; ++j) atomicAdd(&s_mass[cut.place(k[j]) >> 20], 1u);
    __syncthreads();

    // equal stretches: taken when none of them holds much more than its share
    const uint32_t aim = (uint32_t)(kHybSample / a.mass);
#pragma unroll
    for (int j = 0; j < PER; ++j) atomicAdd(&s_bin[__umulhi(cut.place(k[j]), aim)], 1u);
    __syncthreads();
    uint32_t most = 0;
    for (int i = tid; i < kHybBins; i += NT) {
        most = max(most, s_bin[i]);
        s_bin[i] = 0u;
    }
    const bool lin = !__syncthreads_or(most > 2u * (uint32_t)a.mass + 16u);
    if (lin) cut.bins = aim;
    // bins of cells are as fine as the sample allows: a bin of uneven mass is
    // cut evenly in step B
    constexpr uint32_t mass_aim = kHybMassMin;

    // bins of a cell: a heavy cell takes 2^sb bins of its own; light cells
    // share a bin until they hold mass_aim samples, or kHybCellShare cells if
    // they are empty (a bin that is mostly empty range would be cut unevenly
    // in step B).  Scanned together: bins of the heavy cells before (and one
    // each, so that light cells after a heavy one start a new bin), weight of
    // the light cells before.
    constexpr int CPT = kHybCells / NT;
    constexpr uint32_t kShare = mass_aim * kHybCellShare;   // weight of one bin
    static_assert(kHybSample / mass_aim + kHybCells / kHybCellShare + kHybSample / (2 * mass_aim) + 4 <= kHybBins, "bins");
    uint32_t sbs[CPT];
    unsigned long long part = 0;
    auto weight = [&](uint32_t mass, uint32_t sb) {
        return sb ? ((unsigned long long)((1u << (sb & 0xFFu)) + 1u) << 32)
                  : (unsigned long long)(mass * kHybCellShare + mass_aim);
    };
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        const uint32_t mass = s_mass[tid * CPT + j];
        const bool heavy = mass >= 2u * mass_aim;
        int sb = heavy ? 31 - __clz((int)(mass / mass_aim)) : 0;
        if (sb > sbmax) sb = sbmax;
        sbs[j] = heavy ? (uint32_t)sb | 0x100u : 0u;   // 0x100: heavy (sb may be cut to 0)
        part += weight(mass, sbs[j]);
    }
    unsigned long long tot;
    unsigned long long ex = block_exclusive_scan<NT>(part, s_scr, &tot);
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        const uint32_t mass = s_mass[tid * CPT + j];
        const uint32_t light = (uint32_t)ex, hb = (uint32_t)(ex >> 32);
        const uint32_t base = hb + (light + (sbs[j] ? kShare - 1u : 0u)) / kShare;
        s_lut[tid * CPT + j] = base | (sbs[j] & 0xFFu) << 16;
        ex += weight(mass, sbs[j]);
    }
    __syncthreads();

    // key range of each bin.  Equal stretches: from their formula.  Cells: from
    // the first cell that reaches the bin to the last cell that starts at or
    // before it (bins are monotone in the cells).
    for (int b = tid; b < kHybBins; b += NT) {
        bool some = false;
        uint32_t xf = 0, xl = 0;   // first and last position
        int next = kHybCells;      // a bin that no key is sent to lies before this cell
        if (lin) {
            some = (uint32_t)b < aim;
            if (some) {
                xf = part_start((uint32_t)b, aim);
                xl = (uint32_t)b + 1u < aim ? part_start((uint32_t)b + 1u, aim) - 1u : 0xFFFFFFFFu;
            }
        } else {
            int lo = 0, hi = kHybCells;   // first cell whose last bin >= b
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                const uint32_t e = s_lut[mid];
                if ((e & 0xFFFFu) + (1u << (e >> 16)) - 1u >= (uint32_t)b)
                    hi = mid;
                else
                    lo = mid + 1;
            }
            const int first = lo;
            lo = -1;
            hi = kHybCells - 1;           // last cell whose first bin <= b
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if ((s_lut[mid] & 0xFFFFu) <= (uint32_t)b)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            const int last = lo;
            next = first;
            some = first < kHybCells && last >= first;
            if (some) {
                const uint32_t ef = s_lut[first], el = s_lut[last], fb = ef & 0xFFFFu, lb = el & 0xFFFFu;
                xf = ((uint32_t)first << 20) + (((uint32_t)b > fb ? (uint32_t)b - fb : 0u) << (20 - (ef >> 16)));
                const uint32_t sub = min((uint32_t)b - lb, (1u << (el >> 16)) - 1u);
                xl = ((uint32_t)last << 20) + ((sub + 1u) << (20 - (el >> 16))) - 1u;
            }
        }
        unsigned long long off = (unsigned long long)cut.width;
        if (next < kHybCells) off = min(off, denorm32((uint32_t)next << 20, cut.lz));
        unsigned long long blo = (unsigned long long)cut.lo + off, bhi = blo;
        if (some) {
            const unsigned long long dl = denorm32(xf, cut.lz);
            unsigned long long dh = xl == 0xFFFFFFFFu ? (unsigned long long)cut.width : denorm32(xl + 1u, cut.lz) - 1ull;
            if (dh > (unsigned long long)cut.width) dh = (unsigned long long)cut.width;
            blo = (unsigned long long)cut.lo + min(dl, dh);   // (dl > dh: past the largest key, empty)
            bhi = (unsigned long long)cut.lo + dh;
        }
        s_lo[b] = blo;
        s_hi[b] = bhi;
    }
    __syncthreads();
    // the table's entries: shift, and offset of the cell's first bin
    for (int i = tid; i < kHybCells; i += NT) {
        const uint32_t e = s_lut[i], sh = 20u - (e >> 16);
        s_lut[i] = (((e & 0xFFFFu) - (((uint32_t)i << 20) >> sh)) << 5) | sh;
    }
    __syncthreads();

    // no bin of more than one value may hold much more than its share of the
    // sample, no single value a quarter of it (its counters would serialise
    // the atomics); over a narrow range a quarter must be of single values
    bool bad = false;
    uint32_t singles = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t b = lin ? __umulhi(cut.place(k[j]), aim) : cut.bin(k[j], s_lut);
        atomicAdd(&s_bin[b], 1u);
        if (s_lo[b] == s_hi[b]) ++singles;
    }
    singles = __reduce_add_sync(0xffffffffu, singles);
    if (lane == 0) s_mn[warp] = (U)singles;   // (the extents are in registers)
    __syncthreads();
    for (int i = tid; i < kHybBins; i += NT)
        bad |= s_bin[i] > (s_lo[i] != s_hi[i] ? 8u * (lin ? (uint32_t)a.mass : mass_aim) : (uint32_t)kHybSample / 4);
    const uint32_t in_singles = __reduce_add_sync(0xffffffffu, lane < NT / 32 ? (uint32_t)s_mn[lane] : 0u);
    bad |= (span >> 24) == 0 && in_singles < (uint32_t)kHybSample / 4;
    if (__syncthreads_or(bad)) return;   // nothing was written but the control words' zeros
    for (int i = tid; i < kHybCells; i += NT) a.lut[i] = s_lut[i];
    for (int b = tid; b < kHybBins; b += NT) {
        a.bin_lo[b] = s_lo[b];
        a.bin_hi[b] = s_hi[b];
    }
    if (tid == 0) {
        const uint32_t x = norm32(cut.width, cut.lz), e = s_lut[x >> 20];   // the largest position
        a.ctl[HYB_TOP] = lin ? __umulhi(x, aim) : __funnelshift_r(x, 0u, e) + (uint32_t)((int32_t)e >> 5);
        const unsigned long long l = (unsigned long long)cut.lo, w = (unsigned long long)cut.width;
        a.ctl[HYB_LO] = (uint32_t)l;
        a.ctl[HYB_LO + 1] = (uint32_t)(l >> 32);
        a.ctl[HYB_WIDTH] = (uint32_t)w;
        a.ctl[HYB_WIDTH + 1] = (uint32_t)(w >> 32);
        a.ctl[HYB_LZ] = (uint32_t)cut.lz;
        a.ctl[HYB_BINS] = cut.bins;
        a.ctl[HYB_ON] = 1u;
    }
}

// ---------------------------------------------------------------------------
// K_ha: exact counts of the bins, and whether keys lie outside the sampled
// range.
// ---------------------------------------------------------------------------
template <typename U>
__global__ void __launch_bounds__(kHybThreads, 2) hybrid_count_a(HybArgs a) {
    chain_wait();
    if (!hyb_on(a.ctl)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int COLS = 8;   // copies of the counters, lanes spread over them
    uint32_t* s_lut = (uint32_t*)smem;              // kHybCells
    uint32_t* s_cnt = s_lut + kHybCells;            // kHybBins * COLS
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < kHybCells; i += kHybThreads) s_lut[i] = a.lut[i];
    for (int i = tid; i < kHybBins * COLS; i += kHybThreads) s_cnt[i] = 0u;
    __syncthreads();
    hyb_variant<U>(a.ctl, a.map, [&](const auto& cut, const auto& mapped) {
        const U* keys = (const U*)a.in;
        const size_t n = a.n;
        uint32_t* col = s_cnt + (lane & (COLS - 1));
        const U lo = cut.lo, hi = (U)(cut.lo + cut.width);
        bool below = false, above = false;
        auto one = [&](U raw) {
            const U k = mapped(raw);
            below |= k < lo;
            above |= k > hi;
            atomicAdd(&col[cut.bin(k, s_lut) * COLS], 1u);
        };
        constexpr int V = 16 / sizeof(U);
        size_t head = ((16 - ((uintptr_t)keys & 15)) & 15) / sizeof(U);
        if (head > n) head = n;
        const size_t nvec = (n - head) / V;
        const size_t tail0 = head + nvec * V;
        const size_t gtid = (size_t)blockIdx.x * kHybThreads + tid;
        const size_t gthreads = (size_t)gridDim.x * kHybThreads;
        if (gtid < head) one(keys[gtid]);
        if (gtid < n - tail0) one(keys[tail0 + gtid]);
        const uint4* vp = (const uint4*)(keys + head);
        constexpr int kUnroll = 4;
        size_t c0 = gtid;
        for (; c0 + 3 * gthreads < nvec; c0 += gthreads * kUnroll) {
            uint4 q[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) q[u] = __ldcs(vp + c0 + (size_t)u * gthreads);
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                U k[V];
                memcpy(k, &q[u], 16);
#pragma unroll
                for (int j = 0; j < V; ++j) one(k[j]);
            }
        }
        for (; c0 < nvec; c0 += gthreads) {
            const uint4 q = __ldcs(vp + c0);
            U k[V];
            memcpy(k, &q, 16);
#pragma unroll
            for (int j = 0; j < V; ++j) one(k[j]);
        }
        if (__any_sync(0xffffffffu, below) && lane == 0) a.ctl[HYB_BELOW] = 1u;
        if (__any_sync(0xffffffffu, above) && lane == 0) a.ctl[HYB_ABOVE] = 1u;
    });
    __syncthreads();
    for (int b = tid; b < kHybBins; b += kHybThreads) {
        uint32_t s = 0;
        for (int c = 0; c < COLS; ++c) s += s_cnt[b * COLS + ((c + b) & (COLS - 1))];
        if (s) atomicAdd(&a.count_a[b], s);
    }
}

// ---------------------------------------------------------------------------
// K_hp: bin starts, buckets and step-B tiles of each bin.  One CTA.
// ---------------------------------------------------------------------------
template <typename U>
__global__ void __launch_bounds__(kHybThreads) hybrid_plan(HybArgs a) {
    chain_wait();
    if (!hyb_on(a.ctl)) return;
    __shared__ unsigned long long s_scr[kHybThreads / 32 + 1];
    constexpr int PER = kHybBins / kHybThreads;
    uint32_t c[PER], nb[PER], lz[PER], mult[PER];
    unsigned long long keys = 0, two = 0;   // two: tiles << 32 | buckets
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int b = threadIdx.x * PER + j;
        c[j] = a.count_a[b];
        const unsigned long long lo = a.bin_lo[b], hi = a.bin_hi[b], w = hi >= lo ? hi - lo : 0ull;
        uint32_t want = (c[j] + (uint32_t)hyb_target<U>() - 1u) / (uint32_t)hyb_target<U>();
        if (want > (uint32_t)kHybBins) want = (uint32_t)kHybBins;
        int z = 63;
        mult[j] = 0u;
        nb[j] = 1u;
        if (c[j] > 0) nb[j] = cut_range(w, want, &z, &mult[j]);
        lz[j] = (uint32_t)z | (w < (unsigned long long)nb[j] ? 0x100u : 0u);   // 0x100: every bucket is one value
        keys += c[j];
        two += ((unsigned long long)((c[j] + hyb_tile<U>() - 1) / hyb_tile<U>()) << 32) |
               ((nb[j] + 7u) & ~7u);   // whole sectors (hyb_spread)
    }
    unsigned long long tot, tot2;
    unsigned long long base = block_exclusive_scan<kHybThreads, unsigned long long>(keys, s_scr, &tot);
    unsigned long long at = block_exclusive_scan<kHybThreads, unsigned long long>(two, s_scr, &tot2);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int b = threadIdx.x * PER + j;
        a.base_a[b] = (uint32_t)base;
        a.cursor_a[hyb_spread((uint32_t)b)] = (uint32_t)base;
        a.off_b[b] = (uint32_t)at;
        a.tile_b[b] = (uint32_t)(at >> 32);
        a.lz_b[b] = lz[j];
        a.mult_b[b] = mult[j];
        base += c[j];
        at += ((unsigned long long)((c[j] + hyb_tile<U>() - 1) / hyb_tile<U>()) << 32) | ((nb[j] + 7u) & ~7u);
    }
    if (threadIdx.x == 0) {
        a.base_a[kHybBins] = (uint32_t)tot;
        a.off_b[kHybBins] = (uint32_t)tot2;
        a.tile_b[kHybBins] = (uint32_t)(tot2 >> 32);
        // more buckets than the scratch holds (cannot happen by the sizes
        // above), or counts that do not add up: given up
        if ((uint32_t)tot2 > a.max_buckets || tot != (unsigned long long)a.n) a.ctl[HYB_FAIL] = 1u;
    }
}

// ---------------------------------------------------------------------------
// K_hm: one partition step.  A tile is read once into registers and costs
// per key one shared atomic (its old count is the key's place in its bin),
// one read of the bin's first place, one write and one read of the reorder
// buffer and one read of the run's destination.
// ---------------------------------------------------------------------------
template <typename U, bool A>
constexpr size_t hyb_partition_smem() {
    return (size_t)hyb_tile<U>() * sizeof(U) + (size_t)kHybBins * 12 +
           (A ? (size_t)kHybCells * 4 : (size_t)(kHybBins + 1) * 8);
}

// Shared arrays of a partition step.
template <typename U>
struct HybTile {
    U* key;          // reorder buffer
    uint32_t* cnt;   // keys of the tile per bin (zero between tiles)
    uint32_t* at;    // first place of a bin in the tile (| kHybFinal)
    uint32_t* to;    // global place of the bin's run - at
    uint32_t* w;     // warp sums
};

// The keys of a tile, src[0 .. valid), into registers.
template <typename U>
__device__ __forceinline__ void hyb_tile_load(U (&key)[hyb_kpt<U>()], const U* src, int valid) {
    const U* mine = src + threadIdx.x;
    if (valid == hyb_tile<U>()) {
#pragma unroll
        for (int i = 0; i < hyb_kpt<U>(); ++i) key[i] = ld_stream(mine + i * kHybThreads);
    } else {
#pragma unroll
        for (int i = 0; i < hyb_kpt<U>(); ++i)
            key[i] = i * kHybThreads + (int)threadIdx.x < valid ? ld_stream(mine + i * kHybThreads) : (U)0;
    }
}

// One tile: its keys (in registers) to the bins bin_of() names, whose next
// free places are cursor[].  mapped: key map of the load; last: the key map of
// the store for the buckets marked final.  Once the keys are in the reorder
// buffer their registers take the next tile's (next()), whose loads are under
// way while this tile is written.
template <typename U, bool FULL, typename B, typename M, typename L, typename N>
__device__ __forceinline__ void hyb_tile_step(const HybTile<U>& t, U (&key)[hyb_kpt<U>()], U* dst, int valid,
                                              uint32_t n, uint32_t* cursor, const B& bin_of, const M& mapped,
                                              const L& last, const N& next) {
    constexpr int KPT = hyb_kpt<U>();
    constexpr int BPT = 2;   // bins per thread, of the first kHybBins / 2 threads
    static_assert(kHybBins / BPT <= kHybThreads, "bin owners");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool owner = tid < kHybBins / BPT;
    uint32_t rk[(KPT + 1) / 2];   // place in the bin, two 16-bit fields per register (the bin is found again)
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        if (FULL || i * kHybThreads + tid < valid) {
            key[i] = mapped(key[i]);
            const uint32_t r = atomicAdd(&t.cnt[bin_of(key[i])], 1u);
            rk[i / 2] = i & 1 ? __byte_perm(rk[i / 2], r, 0x5410) : r;
        }
    }
    __syncthreads();
    // the tile's share of each bin is reserved with one global atomic, whose
    // answer is not needed before the tile is reordered
    uint32_t c[BPT], g[BPT], sum = 0;
#pragma unroll
    for (int j = 0; j < BPT; ++j) {
        const int b = tid * BPT + j;
        c[j] = owner ? t.cnt[b] : 0u;
        if (owner) t.cnt[b] = 0u;
        g[j] = c[j] ? atomicAdd(&cursor[hyb_spread((uint32_t)b)], c[j]) : 0u;
        sum += c[j];
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) t.w[warp] = inc;
    __syncthreads();
    uint32_t run = inc - sum;
    {
        uint32_t v = lane < kHybThreads / 32 ? t.w[lane] : 0u;
        v = lane < warp ? v : 0u;
        run += __reduce_add_sync(0xffffffffu, v);
    }
    uint32_t first[BPT];
#pragma unroll
    for (int j = 0; j < BPT; ++j) {
        first[j] = run;
        if (owner) t.at[tid * BPT + j] = run;
        run += c[j];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < KPT; ++i)
        if (FULL || i * kHybThreads + tid < valid) t.key[t.at[bin_of(key[i])] + (i & 1 ? rk[i / 2] >> 16 : rk[i / 2] & 0xFFFFu)] = key[i];
    next();
    bool fin = false;
#pragma unroll
    for (int j = 0; j < BPT; ++j) {
        if (owner) t.to[tid * BPT + j] = (g[j] & ~kHybFinal) - first[j];
        fin |= (g[j] & kHybFinal) != 0u;
    }
    const bool any_fin = __syncthreads_or(fin);
    if (any_fin) {   // rare: buckets whose keys leave in their final form
#pragma unroll
        for (int j = 0; j < BPT; ++j)
            if (owner) t.at[tid * BPT + j] = g[j] & kHybFinal;
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const int s = i * kHybThreads + tid;
        if (FULL || s < valid) {
            U k = t.key[s];
            const uint32_t b = bin_of(k);
            const uint32_t to = t.to[b] + (uint32_t)s;
            if (any_fin && t.at[b]) k = last(k);
            if (to < n) dst[to] = k;   // always, unless the counts were inconsistent
        }
    }
    // the next tile writes key, at and to only after two barriers
}

template <typename U>
__global__ void __launch_bounds__(kHybThreads, 2) hybrid_partition_a(HybArgs a) {
    chain_wait();
    if (!hyb_on(a.ctl)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_w[kHybThreads / 32];
    constexpr int TILE = hyb_tile<U>();
    HybTile<U> t;
    t.key = (U*)smem;
    t.cnt = (uint32_t*)(smem + (size_t)TILE * sizeof(U));
    t.at = t.cnt + kHybBins;
    t.to = t.at + kHybBins;
    t.w = s_w;
    uint32_t* s_lut = t.to + kHybBins;
    for (int i = threadIdx.x; i < kHybCells; i += kHybThreads) s_lut[i] = a.lut[i];
    for (int i = threadIdx.x; i < kHybBins; i += kHybThreads) t.cnt[i] = 0u;
    __syncthreads();
    hyb_variant<U>(a.ctl, a.map, [&](const auto& cut, const auto& mapped) {
        auto bin_of = [&](U k) { return cut.bin(k, s_lut); };
        auto same = [](U k) { return k; };
        const uint32_t tiles = (uint32_t)((a.n + TILE - 1) / TILE), full = (uint32_t)(a.n / TILE);
        const U* in = (const U*)a.in;
        auto count = [&](uint32_t i) { return i < full ? TILE : (int)(a.n - (size_t)full * TILE); };
        U key[hyb_kpt<U>()];
        uint32_t i = blockIdx.x;
        if (i < tiles) hyb_tile_load<U>(key, in + (size_t)i * TILE, count(i));
        auto next = [&]() {
            const uint32_t j = i + gridDim.x;
            if (j < tiles) hyb_tile_load<U>(key, in + (size_t)j * TILE, count(j));
        };
        for (; i < full; i += gridDim.x)
            hyb_tile_step<U, true>(t, key, (U*)a.tmp, TILE, (uint32_t)a.n, a.cursor_a, bin_of, mapped, same, next);
        if (i < tiles)
            hyb_tile_step<U, false>(t, key, (U*)a.tmp, count(i), (uint32_t)a.n, a.cursor_a, bin_of, mapped, same, next);
    });
}

// Bucket of a key in its bin; keys outside the sampled range, in the first
// and the last bin, go to the ends.
template <typename U>
struct HybBucket {
    U lo, width;
    int lz;
    uint32_t mult;
    __device__ __forceinline__ uint32_t operator()(U k) const { return __umulhi(norm32((U)(k - lo), lz), mult); }
};
template <typename U>
struct HybEndBucket {
    HybBucket<U> in;
    __device__ __forceinline__ uint32_t operator()(U k) const {
        const U d = (k > in.lo ? k : in.lo) - in.lo;
        return __umulhi(norm32(d < in.width ? d : in.width, in.lz), in.mult);
    }
};
template <typename U>
__device__ __forceinline__ HybBucket<U> hyb_bucket(const HybArgs& a, uint32_t bin) {
    HybBucket<U> b;
    b.lo = (U)a.bin_lo[bin];
    b.width = (U)(a.bin_hi[bin] - a.bin_lo[bin]);
    b.lz = (int)(a.lz_b[bin] & 0xFFu);
    b.mult = a.mult_b[bin];
    return b;
}

template <typename U>
__global__ void __launch_bounds__(kHybThreads, 2) hybrid_partition_b(HybArgs a) {
    chain_wait();
    if (!hyb_on(a.ctl)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_w[kHybThreads / 32];
    constexpr int TILE = hyb_tile<U>();
    HybTile<U> t;
    t.key = (U*)smem;
    t.cnt = (uint32_t*)(smem + (size_t)TILE * sizeof(U));
    t.at = t.cnt + kHybBins;
    t.to = t.at + kHybBins;
    t.w = s_w;
    uint32_t* s_tile = t.to + kHybBins;           // first tile of each bin
    uint32_t* s_base = s_tile + kHybBins + 1;     // start of each bin
    for (int i = threadIdx.x; i <= kHybBins; i += kHybThreads) {
        s_tile[i] = a.tile_b[i];
        s_base[i] = a.base_a[i];
    }
    for (int i = threadIdx.x; i < kHybBins; i += kHybThreads) t.cnt[i] = 0u;
    __syncthreads();
    const bool ends = a.ctl[HYB_BELOW] != 0u || a.ctl[HYB_ABOVE] != 0u;
    const uint32_t tiles = s_tile[kHybBins];
    const KeyMap map = a.map;
    auto same = [](U k) { return k; };
    auto fin = [&](U k) { return map_inv(k, map); };
    U key[hyb_kpt<U>()];
    uint32_t ahead = 0;   // the bin of the tile being loaded: tiles are taken in order, so it only grows
    int loaded = 0;
    auto load = [&](uint32_t i) {
        while (i >= s_tile[ahead + 1]) ++ahead;   // i < s_tile[kHybBins]
        const size_t start = (size_t)s_base[ahead] + (size_t)(i - s_tile[ahead]) * TILE;
        const size_t end = s_base[ahead + 1];
        loaded = end - start < (size_t)TILE ? (int)(end - start) : TILE;
        hyb_tile_load<U>(key, (const U*)a.tmp + start, loaded);
    };
    if (blockIdx.x < tiles) load(blockIdx.x);
    for (uint32_t i = blockIdx.x; i < tiles; i += gridDim.x) {
        const uint32_t bin = ahead;
        const int valid = loaded;
        uint32_t* cursor = a.buckets + hyb_spread(a.off_b[bin]);   // (a multiple of 8)
        const HybBucket<U> b = hyb_bucket<U>(a, bin);
        auto next = [&]() {
            if (i + gridDim.x < tiles) load(i + gridDim.x);
        };
        // (a bin has at most kHybBins buckets; counts of the others stay zero)
        if (valid == TILE && !ends)
            hyb_tile_step<U, true>(t, key, (U*)a.out, valid, (uint32_t)a.n, cursor, b, same, fin, next);
        else
            hyb_tile_step<U, false>(t, key, (U*)a.out, valid, (uint32_t)a.n, cursor, HybEndBucket<U>{b}, same, fin,
                                    next);
    }
}

// ---------------------------------------------------------------------------
// K_hb: counts of every bin's buckets.  Each CTA reads one stretch of the
// partitioned array, bin after bin.
// ---------------------------------------------------------------------------
template <typename U>
__global__ void __launch_bounds__(kHybThreads, 3) hybrid_count_b(HybArgs a) {
    chain_wait();
    if (!hyb_on(a.ctl)) return;
    constexpr int COLS = 4;
    __shared__ uint32_t s_cnt[kHybBins * COLS];
    const int tid = threadIdx.x;
    uint32_t* col = s_cnt + (tid & (COLS - 1));
    const U* keys = (const U*)a.tmp;
    const size_t per = ((a.n + gridDim.x - 1) / gridDim.x + 63) / 64 * 64;
    size_t at = (size_t)blockIdx.x * per;
    const size_t stop = at + per < a.n ? at + per : a.n;
    if (at >= stop) return;
    int lo = 0, hi = kHybBins - 1;   // the bin of the first key: the last one that starts at or before it
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((size_t)a.base_a[mid] <= at)
            lo = mid;
        else
            hi = mid - 1;
    }
    for (int bin = lo; at < stop; ++bin) {
        const size_t end = (size_t)a.base_a[bin + 1] < stop ? (size_t)a.base_a[bin + 1] : stop;
        if (end <= at) continue;
        const uint32_t first = a.off_b[bin], nb = a.off_b[bin + 1] - first;
        if (a.mult_b[bin] == 0u) {   // one bucket
            if (tid == 0) atomicAdd(&a.buckets[hyb_spread(first)], (uint32_t)(end - at));
            at = end;
            continue;
        }
        for (uint32_t i = tid; i < nb * COLS; i += kHybThreads) s_cnt[i] = 0u;
        __syncthreads();
        const HybEndBucket<U> bucket{hyb_bucket<U>(a, (uint32_t)bin)};
        constexpr int kUnroll = 8;
        for (size_t c0 = at + tid; c0 < end; c0 += (size_t)kHybThreads * kUnroll) {
            U k[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                if (c0 + (size_t)u * kHybThreads < end) k[u] = ld_stream(keys + c0 + (size_t)u * kHybThreads);
#pragma unroll
            for (int u = 0; u < kUnroll; ++u)
                if (c0 + (size_t)u * kHybThreads < end)
                    atomicAdd(&col[bucket(k[u]) * COLS], 1u);
        }
        __syncthreads();
        for (uint32_t b = tid; b < nb; b += kHybThreads) {
            uint32_t s = 0;
            for (int c = 0; c < COLS; ++c) s += s_cnt[b * COLS + c];
            if (s) atomicAdd(&a.buckets[hyb_spread(first + b)], s);
        }
        __syncthreads();
        at = end;
    }
}

// ---------------------------------------------------------------------------
// K_hq: bucket counts -> starts, one CTA per bin.
// ---------------------------------------------------------------------------
template <typename U>
__global__ void __launch_bounds__(kHybThreads) hybrid_scan_b(HybArgs a) {
    chain_wait();
    // Other CTAs of this launch may give the path up while this one starts: one
    // thread reads the verdict so far for all of them, or some would leave and
    // the rest wait at the barriers below.
    __shared__ bool s_on;
    if (threadIdx.x == 0) s_on = hyb_on(a.ctl);
    __syncthreads();
    if (!s_on) return;
    __shared__ uint32_t s_scr[kHybThreads / 32 + 1];
    const int bin = blockIdx.x, tid = threadIdx.x;
    constexpr int PER = kHybBins / kHybThreads;
    const uint32_t first = a.off_b[bin], nb = a.off_b[bin + 1] - first;
    // keys outside the sampled range, if there are any, sit in the first
    // bucket of the first bin and the last bucket of the last bin
    const uint32_t top = a.ctl[HYB_TOP];
    const bool low_end = bin == 0 && a.ctl[HYB_BELOW] != 0u;
    const bool high_end = (uint32_t)bin == top && a.ctl[HYB_ABOVE] != 0u;
    const bool one_value = (a.lz_b[bin] & 0x100u) != 0u;
    const uint32_t last = __umulhi(norm32((uint64_t)(a.bin_hi[bin] - a.bin_lo[bin]), (int)(a.lz_b[bin] & 0xFFu)),
                                   a.mult_b[bin]);
    uint32_t c[PER], sum = 0;
    bool bad = false, long_one[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t b = (uint32_t)(tid * PER + j);
        c[j] = b < nb ? a.buckets[hyb_spread(first + b)] : 0u;
        sum += c[j];
        long_one[j] = c[j] > (uint32_t)hyb_cap<U>() && one_value && !(b == 0u && low_end) && !(b == last && high_end);
        bad |= c[j] > a.longest && !long_one[j];
    }
    uint32_t tot;
    uint32_t run = block_exclusive_scan<kHybThreads>(sum, s_scr, &tot) + a.base_a[bin];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t b = (uint32_t)(tid * PER + j);
        if (b < nb) a.buckets[hyb_spread(first + b)] = run | (long_one[j] ? kHybFinal : 0u);
        run += c[j];
    }
    if (tot != a.base_a[bin + 1] - a.base_a[bin]) bad = true;   // counts that do not add up
    if (__syncthreads_or(bad) && tid == 0) a.ctl[HYB_FAIL] = 1u;
}

// ---------------------------------------------------------------------------
// K_hg: the local sorts.  After step B buckets[f] is the end of bucket f.  One
// thread per stretch of hyb_window() keys: the buckets that start in it are
// one group; the last of them, which may reach past the stretch, becomes a
// group of its own if they do not fit together, and is left out if it is one
// long value, which step B wrote in its final form.
// ---------------------------------------------------------------------------
template <typename U>
__global__ void __launch_bounds__(256) hybrid_groups(HybArgs a) {
    chain_wait();
    if (!hyb_on(a.ctl)) return;
    __shared__ uint32_t s_off[kHybBins + 1];
    for (int i = threadIdx.x; i <= kHybBins; i += 256) s_off[i] = a.off_b[i];
    __syncthreads();
    const uint32_t w = blockIdx.x * 256u + threadIdx.x;
    if (w >= a.windows) return;
    const uint32_t nf = s_off[kHybBins], n = (uint32_t)a.n;
    auto end_of = [&](uint32_t f) { return a.buckets[hyb_spread(f)] & ~kHybFinal; };
    // first bucket that starts at or after x
    auto first_from = [&](uint32_t x) {
        if (x == 0u) return 0u;
        uint32_t l = 0, h = nf;
        while (l < h) {
            const uint32_t mid = (l + h) >> 1;
            if (end_of(mid) >= x)
                h = mid;
            else
                l = mid + 1;
        }
        return l + 1u;
    };
    auto bin_of = [&](uint32_t f) {   // the last bin whose first bucket is at most f
        uint32_t l = 0, h = kHybBins - 1;
        while (l < h) {
            const uint32_t mid = (l + h + 1u) >> 1;
            if (s_off[mid] <= f)
                l = mid;
            else
                h = mid - 1u;
        }
        return l;
    };
    // first key of bucket j of a bin (its last key, for buckets past the end)
    auto edge = [&](uint32_t bin, uint32_t j) {
        const unsigned long long lo = a.bin_lo[bin], hi = a.bin_hi[bin];
        const uint32_t mult = a.mult_b[bin];
        if (j == 0u) return lo;
        if (mult == 0u) return hi;
        const unsigned long long x = (((unsigned long long)j << 32) + mult - 1ull) / mult;
        if (x >> 32) return hi;
        return min(hi, lo + denorm32((uint32_t)x, (int)(a.lz_b[bin] & 0xFFu)));
    };
    auto put = [&](uint32_t slot, uint32_t f, uint32_t g, uint32_t s, uint32_t e) {
        HybGroup q = {s, e - s, 63, 0u, 0ull, 0ull};
        if (e > s) {
            // the range of the buckets, to the type's ends where keys outside
            // the sampled range may sit
            const uint32_t bf = bin_of(f), bg = bin_of(g - 1u), top = a.ctl[HYB_TOP];
            unsigned long long lo = edge(bf, f - s_off[bf]), hi = edge(bg, g - s_off[bg]);
            if (g == s_off[bg + 1]) hi = a.bin_hi[bg];
            if (f == 0u && a.ctl[HYB_BELOW] != 0u) lo = 0ull;
            // (the top bin's last bucket; empty ones follow it, to a whole sector)
            const uint32_t last = s_off[top] + __umulhi(norm32((uint64_t)(a.bin_hi[top] - a.bin_lo[top]),
                                                               (int)(a.lz_b[top] & 0xFFu)), a.mult_b[top]);
            if (g > last && a.ctl[HYB_ABOVE] != 0u) hi = (unsigned long long)(U)~(U)0;
            q.lo = lo;
            q.width = hi - lo;
            cut_range(q.width, (uint32_t)(4 * kHybLocalWords * kHybThreads), &q.lz, &q.mult);
        }
        a.groups[slot] = q;
    };
    const uint32_t lo = w * (uint32_t)hyb_window<U>();
    const uint32_t hi = min(n, lo + (uint32_t)hyb_window<U>());
    const uint32_t f0 = first_from(lo), f1 = hi == n ? nf : first_from(hi);
    if (f0 >= f1 || f1 > nf) {   // a bucket that started before reaches past this stretch
        put(w, 0u, 0u, 0u, 0u);
        return;
    }
    const uint32_t s = f0 == 0u ? 0u : end_of(f0 - 1u), m = f1 == 1u ? 0u : end_of(f1 - 2u), e = end_of(f1 - 1u);
    if (a.buckets[hyb_spread(f1 - 1u)] & kHybFinal) {
        put(w, f0, f1 - 1u, s, m);
    } else if (e - s > (uint32_t)hyb_cap<U>()) {
        put(w, f0, f1 - 1u, s, m);
        put(a.windows + atomicAdd(&a.ctl[HYB_MORE], 1u), f1 - 1u, f1, m, e);   // at most one per stretch
    } else {
        put(w, f0, f1, s, e);
    }
}

// ---------------------------------------------------------------------------
// K_hl: local sorts in shared memory, in place in the output.  The next
// group's keys are loaded while this one is sorted and written.
// ---------------------------------------------------------------------------
template <typename U>
__global__ void __launch_bounds__(kHybThreads, 2) hybrid_local(HybArgs a) {
    chain_wait();
    if (!hyb_on(a.ctl)) return;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int KPT = hyb_local_kpt<U>();
    U* k0 = (U*)smem;
    U* k1 = k0 + hyb_cap<U>();
    __shared__ CtaShared<U> s_cta;
    const int tid = threadIdx.x;
    const KeyMap map = a.map;
    const bool plain = map.f == 0 && map.r == 0;   // integers: the key map is one xor
    const U flip = (U)(map.s ^ map.x);
    U* out = (U*)a.out;
    __shared__ HybGroup s_q[2];   // this group's description and the next one's
    const uint32_t more = a.ctl[HYB_MORE], ng = a.windows + more;
    auto group = [&](uint32_t i) {   // the buckets on their own first: the longest are among them
        return (const uint4*)(a.groups + (i < more ? a.windows + i : i - more));
    };
    U key[KPT];
    auto load = [&](const HybGroup& q) {
        const U* mine = out + q.start + tid;
        const uint32_t len = q.len;
        // (every register is written, so none is kept across the sort before)
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            key[i] = (uint32_t)(i * kHybThreads + tid) < len ? ld_stream(mine + i * kHybThreads) : (U)0;
    };
    uint32_t i = blockIdx.x;
    if (i >= ng) return;
    if (tid < 2) ((uint4*)&s_q[0])[tid] = group(i)[tid];
    bin_zero<kHybThreads, kHybLocalWords>(k1);
    __syncthreads();
    load(s_q[0]);
    for (int cur = 0; i < ng; i += gridDim.x, cur ^= 1) {
        if (tid < 2)
            ((uint4*)&s_q[cur ^ 1])[tid] =
                i + gridDim.x < ng ? group(i + gridDim.x)[tid] : make_uint4(0u, 0u, 0u, 0u);
        const HybGroup& q = s_q[cur];
        const uint32_t len = q.len;
        if (len > (uint32_t)hyb_cap<U>()) {
            __syncthreads();
            U* const at = out + q.start;
            cta_split_again<U>(at, (U*)a.tmp + q.start, at, len, GeneralOut<U>(map), smem, s_cta);
            bin_zero<kHybThreads, kHybLocalWords>(k1);
            __syncthreads();
            load(s_q[cur ^ 1]);
        } else if (len > 0) {
            const U* r = block_bin_sort<U, kHybThreads, KPT, kHybLocalWords>(
                key, (int)len, (U)q.lo, q.width, KeyPosition<U>{(U)q.lo, q.lz}, q.mult, k0, k1, s_cta.bin, [&]() { load(s_q[cur ^ 1]); });
            U* const mine = out + q.start + tid;
            const U* const from = r + tid;
            if (plain) {
#pragma unroll
                for (int j = 0; j < KPT; ++j)
                    if ((uint32_t)(j * kHybThreads + tid) < len)
                        st_stream(mine + j * kHybThreads, (U)(from[j * kHybThreads] ^ flip));
            } else {
                for (uint32_t j = tid; j < len; j += kHybThreads) st_stream(out + q.start + j, map_inv(r[j], map));
            }
            if (r == k1) __syncthreads();   // rare: the sorted keys lie where the bins are
            bin_zero<kHybThreads, kHybLocalWords>(k1);
            __syncthreads();
        } else {
            __syncthreads();
            load(s_q[cur ^ 1]);
        }
    }
}

// K_hf: clears the scratch of a path that was given up (it lies in the
// look-back slots the radix passes expect zeroed), as far as it was used.
__global__ void hybrid_finish(HybArgs a) {
    chain_wait();
    if (hyb_on(a.ctl)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.last->hybrid = PART_DONE;   // for the profile's records
        return;
    }
    if (a.ctl[HYB_ON] == 0u) return;   // refused by the sample, which writes nothing then
    if (blockIdx.x == 0 && threadIdx.x == 0) a.last->hybrid = PART_GIVEN_UP;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.scratch16; i += stride)
        ((uint4*)a.scratch)[i] = make_uint4(0u, 0u, 0u, 0u);
}

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

uint32_t hyb_max_buckets(int w, size_t n) {
    const size_t target = w == 4 ? (size_t)hyb_target<uint32_t>() : (size_t)hyb_target<uint64_t>();
    return (uint32_t)(n / target + 10 * kHybBins);   // each bin's share rounded up, to whole sectors
}

template <typename U>
cudaError_t launch_hybrid(const HybArgs& a, int call, cudaStream_t s) {
    static bool configured = false;
    const int count_smem = (kHybCells + kHybBins * 8) * 4;
    if (!configured) {
        struct { const void* f; size_t b; } set[] = {
            {(const void*)hybrid_sample<U>, hyb_sample_smem()},
            {(const void*)hybrid_count_a<U>, (size_t)count_smem},
            {(const void*)hybrid_partition_a<U>, hyb_partition_smem<U, true>()},
            {(const void*)hybrid_partition_b<U>, hyb_partition_smem<U, false>()},
            {(const void*)hybrid_local<U>, cta_smem_bytes<U>()}};
        for (auto& x : set) {
            const cudaError_t e = cudaFuncSetAttribute(x.f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x.b);
            if (e != cudaSuccess) return e;
        }
        configured = true;
    }
    const unsigned two = (unsigned)sm_count() * 2;
    const double keys = (double)a.n * sizeof(U);
    cudaError_t e = cudaSuccess;
    auto step = [&](int pass, double bytes, auto&& launch) {
        ProfScope ps(call, EVOSORT_K_HYBRID, pass, bytes, a.n, s);
        if (e == cudaSuccess) e = launch();
    };
    step(0, 0.0, [&] { return launch_chain(hybrid_sample<U>, 1u, 1024u, hyb_sample_smem(), s, a); });
    step(1, keys, [&] { return launch_chain(hybrid_count_a<U>, two, kHybThreads, count_smem, s, a); });
    step(2, 0.0, [&] { return launch_chain(hybrid_plan<U>, 1u, kHybThreads, 0, s, a); });
    step(3, 2.0 * keys, [&] { return launch_chain(hybrid_partition_a<U>, two, kHybThreads, hyb_partition_smem<U, true>(), s, a); });
    step(4, keys, [&] { return launch_chain(hybrid_count_b<U>, (unsigned)sm_count() * 3, kHybThreads, 0, s, a); });
    step(5, 0.0, [&] { return launch_chain(hybrid_scan_b<U>, (unsigned)kHybBins, kHybThreads, 0, s, a); });
    step(6, 2.0 * keys, [&] { return launch_chain(hybrid_partition_b<U>, two, kHybThreads, hyb_partition_smem<U, false>(), s, a); });
    step(7, 0.0, [&] { return launch_chain(hybrid_groups<U>, (a.windows + 255) / 256, 256, 0, s, a); });
    step(8, 2.0 * keys, [&] { return launch_chain(hybrid_local<U>, two, kHybThreads, cta_smem_bytes<U>(), s, a); });
    step(9, 0.0, [&] { return launch_chain(hybrid_finish, (unsigned)sm_count(), 256, 0, s, a); });
    count_launches(10);
    return e;
}

}  // namespace

static uint32_t hyb_windows(int w, size_t n) {
    const size_t g = w == 4 ? (size_t)hyb_window<uint32_t>() : (size_t)hyb_window<uint64_t>();
    return (uint32_t)((n + g - 1) / g);
}

size_t hybrid_scratch_bytes(int w, size_t n) {
    return up256(kHybCells * 4) + 2 * up256(kHybBins * 8) + 6 * up256((kHybBins + 1) * 4) + up256(kHybBins * 16) +
           up256((size_t)hyb_max_buckets(w, n) * 16) + up256((size_t)hyb_windows(w, n) * 2 * sizeof(HybGroup));
}

cudaError_t launch_hybrid_sort(int w, const void* in, void* out, void* tmp, size_t n, const KeyMap& map, uint32_t* ctl,
                               void* scratch, PassDesc* last, int call, cudaStream_t s) {
    HybArgs a;
    a.max_buckets = hyb_max_buckets(w, n);
    a.last = last;
    a.in = in;
    a.tmp = tmp;
    a.out = out;
    a.n = n;
    a.map = map;
    a.ctl = ctl;
    // as many bins as buckets per bin, so that the runs of a tile are equally
    // long in both steps
    const double target = w == 4 ? hyb_target<uint32_t>() : hyb_target<uint64_t>();
    double bins = std::sqrt((double)n / target);
    bins = bins < 128.0 ? 128.0 : bins;
    a.longest = (uint32_t)std::max((size_t)(w == 4 ? hyb_cap<uint32_t>() : hyb_cap<uint64_t>()), n / kHybLongShare);
    a.mass = std::max(kHybMassMin, (int)(kHybSample / bins));
    char* p = (char*)scratch;
    auto take = [&](size_t bytes) {
        char* q = p;
        p += up256(bytes);
        return q;
    };
    a.lut = (uint32_t*)take(kHybCells * 4);
    a.bin_lo = (unsigned long long*)take(kHybBins * 8);
    a.bin_hi = (unsigned long long*)take(kHybBins * 8);
    uint32_t** arrays[] = {&a.count_a, &a.base_a, &a.off_b, &a.lz_b, &a.mult_b, &a.tile_b};
    for (uint32_t** x : arrays) *x = (uint32_t*)take((kHybBins + 1) * 4);
    a.cursor_a = (uint32_t*)take(kHybBins * 16);
    a.buckets = (uint32_t*)take((size_t)hyb_max_buckets(w, n) * 16);
    a.windows = hyb_windows(w, n);
    a.groups = (HybGroup*)take((size_t)a.windows * 2 * sizeof(HybGroup));
    a.scratch = scratch;
    a.scratch16 = (size_t)(p - (char*)scratch) / 16;
    return w == 4 ? launch_hybrid<uint32_t>(a, call, s) : launch_hybrid<uint64_t>(a, call, s);
}

}  // namespace evosort
