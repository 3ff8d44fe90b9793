// Dispatcher of Algorithm 5 (AdaptivePartitionSort): picks the algorithm and
// its parameters for one call from a table of tuned parameters, keyed by key
// type, size bucket (floor(log2 n)) and a distribution class read off a small
// strided sample of the keys.  The paper keys its parameters on n alone (one
// GA run per size); the class adds what the data itself changes on a GPU:
// which digits are constant, how many lanes of a warp share a digit.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include "evosort.h"
#include "api_internal.h"
#include "common.cuh"

namespace evosort {
namespace {

struct Entry {
    int dt, bucket, cls;
    evosort_params p;
    float ms;
};
std::mutex g_tab_mu;
std::vector<Entry> g_tab;

constexpr int kSample = 4096;

uint64_t host_map(uint64_t u, int dt, bool descending) {
    // order-preserving map of key bits, host copy (same definition as the kernels')
    const int w = dtype_bytes(dt);
    const KeyMap m = key_map_for(dt, descending);
    if (w == 4) {
        const uint32_t x = (uint32_t)u;
        const uint32_t sar = (x & 0x80000000u) ? 0xFFFFFFFFu : 0u;
        return (uint32_t)(((x ^ ((sar & (uint32_t)m.f) | (uint32_t)m.s)) - (uint32_t)m.r) ^ (uint32_t)m.x);
    }
    const uint64_t sar = (u >> 63) ? ~0ull : 0ull;
    return ((u ^ ((sar & m.f) | m.s)) - m.r) ^ m.x;
}

}  // namespace

// What the dispatcher reads off a sample of mapped keys.
struct SampleStats {
    uint64_t vary, least, most;   // bits that vary; smallest and largest key
    // strict rises and falls between neighbours: equal neighbours say nothing
    // about order (90% zeros would otherwise read as both sorted and reverse
    // sorted)
    uint32_t up, down;
    // runs of equal keys once sorted: their number, the longest, the keys in
    // runs of four or more
    uint32_t distinct, longest, often;
    uint32_t topmax;              // keys that share the most common top byte
    uint64_t dict[kDictMax];      // the distinct keys, ascending, if distinct <= kDictMax
};

// Class of the sample of m keys.  With info, the distinct sampled keys when
// there are at most kDictMax of them, and the sample's order (1: no pair falls,
// -1: no pair rises, 0: both happen).
static int class_of(const SampleStats& q, size_t m, int dt, SampleInfo* info) {
    const int w = dtype_bytes(dt);
    if (info) {
        info->dict.clear();
        if (q.distinct <= (uint32_t)kDictMax) info->dict.assign(q.dict, q.dict + q.distinct);
        info->order = q.down == 0 ? 1 : (q.up == 0 ? -1 : 0);
        // (the path's own sample decides in the end; this one only spares the
        // launches and the wait where it is sure to say no)
        const bool wide = info->wide = ((q.most - q.least) >> 24) != 0;
        info->spread = (size_t)q.longest * 4 <= m && (wide ? (size_t)q.longest * 128 <= m : (size_t)q.often * 4 >= m);
    }
    int bits = 0;
    while (bits < 64 && (q.vary >> bits)) ++bits;
    if (q.distinct == 1) return EVOSORT_CLASS_CONSTANT;
    if (q.distinct <= 64) return EVOSORT_CLASS_FEW;          // few values, whatever their order
    const uint32_t moves = q.up + q.down;
    if (q.up >= 0.9 * (double)moves) return EVOSORT_CLASS_SORTED;
    if (q.down >= 0.9 * (double)moves) return EVOSORT_CLASS_REVERSE;
    if (bits <= 16) return EVOSORT_CLASS_NARROW16;
    if (bits <= 4 * w) return EVOSORT_CLASS_NARROW;          // at most half the key bits vary
    if ((size_t)q.topmax * 4 > m) return EVOSORT_CLASS_SKEWED;   // a quarter in one top byte
    return EVOSORT_CLASS_RANDOM;
}

// ---------------------------------------------------------------------------
// K_s: the statistics of a device array's sample, by one CTA: keys i * stride,
// i < m <= kSample, of n.  Equal keys meet in a hash table (twice as many
// slots as keys, linear probing), so that no sort is needed: a slot holds the
// first such key's place + 1, and their number << 16.  The keys of a warp are
// grouped before the table and the byte counts see them, so that frequent
// values do not queue up.  Bound by the latency of the strided reads and of
// its barriers.  It stands in place of a strided copy of the keys to the host
// and a sort there, which cost 30 to 90 us of every call with a table, the most
// on keys that differ much: 300,000 uniform int64 keys 306 -> 154 us (the sort
// included), sorted ones 94 -> 74 us; 9e6 reversed ones 115 -> 109.
// ---------------------------------------------------------------------------
constexpr int kSampleThreads = 1024;
constexpr int kSampleSlots = 2 * kSample;
constexpr int kStatsSlots = 64;   // calls that sample at the same time
__device__ SampleStats g_stats[kStatsSlots];

__device__ __forceinline__ uint32_t sample_hash(uint64_t k) {
    k ^= k >> 32;   // (the multipliers of splitmix64)
    k *= 0xbf58476d1ce4e5b9ull;
    k ^= k >> 27;
    k *= 0x94d049bb133111ebull;
    return (uint32_t)(k >> 40) & (uint32_t)(kSampleSlots - 1);
}

template <typename U>
__device__ __forceinline__ U load_any(const unsigned char* p, bool aligned) {
    if (aligned) return *(const U*)p;
    U x = 0;
    for (int b = 0; b < (int)sizeof(U); ++b) x |= (U)p[b] << (8 * b);
    return x;
}

template <typename U>
__global__ void __launch_bounds__(kSampleThreads) sample_stats(const unsigned char* keys, size_t stride, int m,
                                                               KeyMap map, SampleStats* to, int slot) {
    extern __shared__ __align__(16) unsigned char smem[];
    U* s_key = (U*)smem;                              // kSample
    uint32_t* s_slot = (uint32_t*)(s_key + kSample);  // kSampleSlots
    __shared__ uint32_t s_top[256];
    __shared__ uint32_t s_up, s_down, s_distinct, s_longest, s_often, s_ndict, s_topmax;
    __shared__ unsigned long long s_vary, s_least, s_most;
    __shared__ U s_dict[kDictMax];
    constexpr int PER = kSample / kSampleThreads;
    const int tid = threadIdx.x, lane = tid & 31;
    const bool aligned = (uintptr_t)keys % sizeof(U) == 0;
    U k[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = j * kSampleThreads + tid;
        if (i < m) k[j] = load_any<U>(keys + (size_t)i * stride * sizeof(U), aligned);
    }
    for (int i = tid; i < kSampleSlots; i += kSampleThreads) s_slot[i] = 0u;
    if (tid < 256) s_top[tid] = 0u;
    if (tid == 0) {
        s_up = s_down = s_distinct = s_longest = s_often = s_ndict = s_topmax = 0u;
        s_vary = s_most = 0ull;
        s_least = ~0ull;
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = j * kSampleThreads + tid;
        if (i < m) s_key[i] = k[j] = map_fwd(k[j], map);
    }
    __syncthreads();
    // ---- order, range, varying bits, top bytes, equal keys
    uint32_t up = 0, down = 0;
    unsigned long long vary = 0, least = ~0ull, most = 0;
    const U first = s_key[0];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = j * kSampleThreads + tid;
        const uint32_t here = __ballot_sync(0xffffffffu, i < m);
        if (i < m) {
            const U x = k[j];
            if (i + 1 < m) {
                up += x < s_key[i + 1];
                down += x > s_key[i + 1];
            }
            vary |= (unsigned long long)(U)(x ^ first);
            least = min(least, (unsigned long long)x);
            most = max(most, (unsigned long long)x);
            const uint32_t top = (uint32_t)(x >> (8 * sizeof(U) - 8));
            const uint32_t tp = __match_any_sync(here, top);
            if (lane == __ffs((int)tp) - 1) atomicAdd(&s_top[top], (uint32_t)__popc(tp));
            const uint32_t kp = __match_any_sync(here, x);
            if (lane == __ffs((int)kp) - 1) {
                const uint32_t count = (uint32_t)__popc(kp) << 16;
                uint32_t h = sample_hash((uint64_t)x);
                for (int probe = 0; probe < kSampleSlots; ++probe) {   // (ends: more slots than keys)
                    const uint32_t old = atomicCAS(&s_slot[h], 0u, count | (uint32_t)(i + 1));
                    if (old == 0u) break;
                    if (s_key[(old & 0xFFFFu) - 1u] == x) {
                        atomicAdd(&s_slot[h], count);
                        break;
                    }
                    h = (h + 1u) & (uint32_t)(kSampleSlots - 1);
                }
            }
        }
    }
    up = __reduce_add_sync(0xffffffffu, up);
    down = __reduce_add_sync(0xffffffffu, down);
    const uint32_t vlo = __reduce_or_sync(0xffffffffu, (uint32_t)vary);
    const uint32_t vhi = __reduce_or_sync(0xffffffffu, (uint32_t)(vary >> 32));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        least = min(least, __shfl_xor_sync(0xffffffffu, least, o));
        most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    }
    if (lane == 0) {
        atomicAdd(&s_up, up);
        atomicAdd(&s_down, down);
        atomicOr(&s_vary, (unsigned long long)vhi << 32 | vlo);
        atomicMin(&s_least, least);
        atomicMax(&s_most, most);
    }
    __syncthreads();
    // ---- runs
    uint32_t distinct = 0, longest = 0, often = 0;
    for (int i = tid; i < kSampleSlots; i += kSampleThreads) {
        const uint32_t c = s_slot[i] >> 16;
        distinct += c != 0u;
        longest = max(longest, c);
        if (c >= 4u) often += c;
    }
    distinct = __reduce_add_sync(0xffffffffu, distinct);
    longest = __reduce_max_sync(0xffffffffu, longest);
    often = __reduce_add_sync(0xffffffffu, often);
    const uint32_t top = __reduce_max_sync(0xffffffffu, tid < 256 ? s_top[tid] : 0u);
    if (lane == 0) {
        atomicAdd(&s_distinct, distinct);
        atomicMax(&s_longest, longest);
        atomicAdd(&s_often, often);
        atomicMax(&s_topmax, top);
    }
    __syncthreads();
    SampleStats* const q = to ? to : g_stats + slot;
    const uint32_t nd = s_distinct;
    if (nd <= (uint32_t)kDictMax) {   // the distinct keys, each to its rank
        for (int i = tid; i < kSampleSlots; i += kSampleThreads) {
            const uint32_t f = s_slot[i] & 0xFFFFu;
            if (f) s_dict[atomicAdd(&s_ndict, 1u)] = s_key[f - 1u];   // (nd of them)
        }
        __syncthreads();
        if (tid < (int)nd) {
            const U x = s_dict[tid];
            uint32_t rank = 0;
            for (uint32_t i = 0; i < nd; ++i) rank += s_dict[i] < x;
            q->dict[rank] = (uint64_t)x;
        }
    }
    if (tid == 0) {
        q->vary = s_vary;
        q->least = s_least;
        q->most = s_most;
        q->up = s_up;
        q->down = s_down;
        q->distinct = nd;
        q->longest = s_longest;
        q->often = s_often;
        q->topmax = s_topmax;
    }
}

template <typename U>
static cudaError_t launch_sample(const void* keys, size_t stride, size_t m, KeyMap map, SampleStats* to, int slot,
                                 cudaStream_t s) {
    constexpr int bytes = kSample * (int)sizeof(U) + kSampleSlots * 4;
    static_assert(bytes + 2048 <= 64 * 1024 + 4096, "two CTAs per SM and a little more");
    const cudaError_t e =
        cudaFuncSetAttribute(sample_stats<U>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    sample_stats<U><<<1, kSampleThreads, bytes, s>>>((const unsigned char*)keys, stride, (int)m, map, to, slot);
    count_launches(1);
    return cudaGetLastError();
}

// The statistics of keys i * stride, i < m, of a device array, read back
// (synchronises the stream).  They pass through one of a fixed set of places
// in device memory; a call that finds all of them taken allocates its own.
static cudaError_t sample_device(const void* keys, size_t stride, size_t m, int dt, bool descending, SampleStats* q,
                                 cudaStream_t s) {
    // memory that the GPU cannot read is refused here, before a kernel meets it
    cudaPointerAttributes at{};
    cudaError_t e = cudaPointerGetAttributes(&at, keys);
    if (e == cudaSuccess && at.type == cudaMemoryTypeUnregistered) {
        int dev = 0, pageable = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&pageable, cudaDevAttrPageableMemoryAccess, dev);
        if (e == cudaSuccess && !pageable) e = cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    static std::atomic<uint64_t> taken{0};
    static_assert(kStatsSlots == 64, "one bit each");
    int slot = -1;
    uint64_t t = taken.load();
    while (slot < 0 && ~t) {
        int free = 0;
        while ((t >> free) & 1) ++free;
        if (taken.compare_exchange_weak(t, t | 1ull << free)) slot = free;
    }
    SampleStats* own = nullptr;
    e = slot < 0 ? cudaMallocAsync((void**)&own, sizeof(SampleStats), s) : cudaSuccess;
    const KeyMap map = key_map_for(dt, descending);
    if (e == cudaSuccess)
        e = dtype_bytes(dt) == 4 ? launch_sample<uint32_t>(keys, stride, m, map, own, slot, s)
                                 : launch_sample<uint64_t>(keys, stride, m, map, own, slot, s);
    if (e == cudaSuccess)
        e = own ? cudaMemcpyAsync(q, own, sizeof(*q), cudaMemcpyDeviceToHost, s)
                : cudaMemcpyFromSymbolAsync(q, g_stats, sizeof(*q), (size_t)slot * sizeof(*q), cudaMemcpyDeviceToHost, s);
    const cudaError_t es = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = es;
    if (own) cudaFreeAsync(own, s);
    if (slot >= 0) taken.fetch_and(~(1ull << slot));
    return e;
}

// Class of n keys in host memory, from the same strided sample the device
// path copies (read here directly, no CUDA call).
int classify_host(const void* keys, size_t n, int dt, bool descending) {
    if (n < 2) return EVOSORT_CLASS_CONSTANT;
    const int w = dtype_bytes(dt);
    const size_t m = n < (size_t)kSample ? n : (size_t)kSample;
    const size_t stride = n / m;
    std::vector<uint64_t> raw(m, 0);
    for (size_t i = 0; i < m; ++i) {
        uint64_t u = 0;
        std::memcpy(&u, (const unsigned char*)keys + i * stride * w, w);
        raw[i] = host_map(u, dt, descending);
    }
    SampleStats q{};
    for (size_t i = 0; i + 1 < m; ++i) {
        q.up += raw[i] < raw[i + 1];
        q.down += raw[i] > raw[i + 1];
    }
    uint32_t top[256] = {0};
    for (size_t i = 0; i < m; ++i) {
        q.vary |= raw[i] ^ raw[0];
        top[(raw[i] >> (8 * w - 8)) & 0xFF] += 1;
    }
    q.topmax = *std::max_element(top, top + 256);
    std::sort(raw.begin(), raw.end());
    q.least = raw.front();
    q.most = raw.back();
    for (size_t i = 0; i < m;) {
        size_t j = i + 1;
        while (j < m && raw[j] == raw[i]) ++j;
        if (q.distinct < (uint32_t)kDictMax) q.dict[q.distinct] = raw[i];
        ++q.distinct;
        q.longest = std::max(q.longest, (uint32_t)(j - i));
        if (j - i >= 4) q.often += (uint32_t)(j - i);
        i = j;
    }
    return class_of(q, m, dt, nullptr);
}

// Table entry for (dt, n, cls): the class itself at the nearest size bucket,
// else the random class; false (and *out untouched) when neither is present.
bool table_lookup(int dt, size_t n, int cls, evosort_params* out) {
    int bucket = 0;
    while (bucket < 63 && (n >> (bucket + 1))) ++bucket;
    std::lock_guard<std::mutex> lk(g_tab_mu);
    const Entry* best = nullptr;
    int bestd = 1 << 30;
    for (int pass = 0; pass < (cls == EVOSORT_CLASS_SEGMENTED ? 1 : 2) && !best; ++pass) {
        const int want = pass == 0 ? cls : EVOSORT_CLASS_RANDOM;
        for (const auto& x : g_tab)
            if (x.dt == dt && x.cls == want && std::abs(x.bucket - bucket) < bestd) {
                best = &x;
                bestd = std::abs(x.bucket - bucket);
            }
    }
    if (!best) return false;
    *out = best->p;
    return true;
}

bool table_nonempty() {
    std::lock_guard<std::mutex> lk(g_tab_mu);
    return !g_tab.empty();
}

bool table_has_algo(int dt, int algo) {
    std::lock_guard<std::mutex> lk(g_tab_mu);
    for (const auto& x : g_tab)
        if (x.dt == dt && x.p.algo == algo) return true;
    return false;
}

// Class of keys[0..n) (a device array) from a strided sample, read in the
// order of the sort's direction (synchronises the stream).
evosort_status classify_device(const void* keys, size_t n, int dt, void* stream, bool descending,
                                        int* cls, SampleInfo* info = nullptr) {
    set_error("");
    if (!cls || (n && !keys) || dt < EVOSORT_I32 || dt > EVOSORT_F64) {
        set_error("evosort_classify: bad argument");
        return EVOSORT_ERR_INVALID;
    }
    if (n < 2) {
        *cls = EVOSORT_CLASS_CONSTANT;
        return EVOSORT_OK;
    }
    const size_t m = n < (size_t)kSample ? n : (size_t)kSample;
    SampleStats q;
    const cudaError_t e = sample_device(keys, n / m, m, dt, descending, &q, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        set_error(std::string("evosort_classify: sample: ") + cudaGetErrorString(e));
        return EVOSORT_ERR_CUDA;
    }
    *cls = class_of(q, m, dt, info);
    return EVOSORT_OK;
}

evosort_status plan_for(const void* keys, size_t n, int dt, void* stream, bool descending,
                                 evosort_params* out, int* cls_out, SampleInfo* info) {
    set_error("");
    if (!out) {
        set_error("evosort_plan: null output");
        return EVOSORT_ERR_INVALID;
    }
    evosort_default_params(out);
    out->stream = stream;
    int cls = EVOSORT_CLASS_RANDOM;
    if (table_nonempty() && n >= 2) {
        const evosort_status st = classify_device(keys, n, dt, stream, descending, &cls, info);
        if (st != EVOSORT_OK) return st;
        if (table_lookup(dt, n, cls, out)) out->stream = stream;
        out->descending = descending ? 1 : 0;
    }
    if (cls_out) *cls_out = cls;
    return EVOSORT_OK;
}

}  // namespace evosort

using namespace evosort;

extern "C" {


evosort_status evosort_classify(const void* keys, size_t n, evosort_dtype dt, void* stream, int* cls) {
    return classify_device(keys, n, dt, stream, false, cls);
}

evosort_status evosort_table_set(evosort_dtype dt, int size_bucket, int cls, const evosort_params* p, float ms) {
    if (!p || dt < EVOSORT_I32 || dt > EVOSORT_F64 || size_bucket < 0 || size_bucket > 63 || cls < 0 ||
        cls > EVOSORT_CLASS_SEGMENTED) {
        set_error("evosort_table_set: bad argument");
        return EVOSORT_ERR_INVALID;
    }
    std::lock_guard<std::mutex> lk(g_tab_mu);
    Entry en{dt, size_bucket, cls, *p, ms};
    en.p.stream = nullptr;
    en.p.workspace = nullptr;
    en.p.workspace_bytes = 0;
    for (auto& x : g_tab)
        if (x.dt == dt && x.bucket == size_bucket && x.cls == cls) {
            x = en;
            return EVOSORT_OK;
        }
    g_tab.push_back(en);
    return EVOSORT_OK;
}

void evosort_table_clear(void) {
    std::lock_guard<std::mutex> lk(g_tab_mu);
    g_tab.clear();
}

size_t evosort_table_size(void) {
    std::lock_guard<std::mutex> lk(g_tab_mu);
    return g_tab.size();
}

evosort_status evosort_table_save(const char* path) {
    std::lock_guard<std::mutex> lk(g_tab_mu);
    std::ofstream f(path ? path : "");
    if (!f) {
        set_error("evosort_table_save: cannot open file");
        return EVOSORT_ERR_INVALID;
    }
    f << "# evosort tuned table: dtype size_bucket class algo digit_bits block_size keys_per_thread "
         "rank_mode insertion_threshold seg_block_cap ms [pass_kernel adapt_later adapt_first seg_warp_cap "
         "small_cap seg_giant]\n";
    for (const auto& x : g_tab)
        f << x.dt << ' ' << x.bucket << ' ' << x.cls << ' ' << x.p.algo << ' ' << x.p.digit_bits << ' '
          << x.p.block_size << ' ' << x.p.keys_per_thread << ' ' << x.p.rank_mode << ' '
          << x.p.insertion_threshold << ' ' << x.p.seg_block_cap << ' ' << x.ms << ' ' << x.p.pass_kernel << ' '
          << x.p.adapt_later << ' ' << x.p.adapt_first << ' ' << x.p.seg_warp_cap << ' ' << x.p.small_cap << ' '
          << x.p.seg_giant << '\n';
    return f ? EVOSORT_OK : EVOSORT_ERR_INVALID;
}

evosort_status evosort_table_load(const char* path) {
    std::ifstream f(path ? path : "");
    if (!f) {
        set_error("evosort_table_load: cannot open file");
        return EVOSORT_ERR_INVALID;
    }
    std::string line;
    int lineno = 0;
    while (std::getline(f, line)) {
        ++lineno;
        if (line.empty() || line[0] == '#') continue;
        std::istringstream is(line);
        int dt, bucket, cls;
        evosort_params p;
        evosort_default_params(&p);
        float ms = 0;
        if (!(is >> dt >> bucket >> cls >> p.algo >> p.digit_bits >> p.block_size >> p.keys_per_thread >>
              p.rank_mode >> p.insertion_threshold >> p.seg_block_cap >> ms)) {
            set_error("evosort_table_load: malformed line " + std::to_string(lineno));
            return EVOSORT_ERR_INVALID;
        }
        // optional later columns (0 = default when absent)
        int extra[5] = {0, 0, 0, 0, 0};
        long long giant = 0;
        int got = 0;
        while (got < 5 && (is >> extra[got])) ++got;
        if (got == 5) is >> giant;
        if (!is.eof() && is.fail() && got > 0 && got < 5) {
            set_error("evosort_table_load: malformed optional columns on line " + std::to_string(lineno));
            return EVOSORT_ERR_INVALID;
        }
        p.pass_kernel = extra[0];
        p.adapt_later = extra[1];
        p.adapt_first = extra[2];
        p.seg_warp_cap = extra[3];
        p.small_cap = extra[4];
        p.seg_giant = giant;
        const evosort_status st = evosort_table_set((evosort_dtype)dt, bucket, cls, &p, ms);
        if (st != EVOSORT_OK) return st;
    }
    return EVOSORT_OK;
}

evosort_status evosort_plan(const void* keys, size_t n, evosort_dtype dt, void* stream, evosort_params* out,
                            int* cls_out) {
    return plan_for(keys, n, dt, stream, false, out, cls_out);
}

evosort_status evosort_plan_host(const void* keys, size_t n, evosort_dtype dt, int descending, evosort_params* out,
                                 int* cls_out) {
    set_error("");
    if (!out || (n && !keys) || dt < EVOSORT_I32 || dt > EVOSORT_F64) {
        set_error("evosort_plan_host: bad argument");
        return EVOSORT_ERR_INVALID;
    }
    evosort_default_params(out);
    int cls = EVOSORT_CLASS_RANDOM;
    if (table_nonempty() && n >= 2) {
        cls = classify_host(keys, n, dt, descending != 0);
        table_lookup(dt, n, cls, out);
        out->stream = nullptr;
    }
    out->descending = descending ? 1 : 0;
    if (cls_out) *cls_out = cls;
    return EVOSORT_OK;
}

}  // extern "C"
