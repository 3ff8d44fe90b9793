// Batched segmented sort: many independent arrays of uneven length sorted in
// one persistent launch.  Each segment is sorted with the method its length
// calls for:
//   warp tier   (len < warp cap)     one warp, keys in registers, bitonic
//                                    network across the warp's lanes (warp cap
//                                    32..256, a tuning parameter);
//   block tier  (len <= block cap)   one CTA, keys in shared memory, sorted by
//                                    bins over their range (bin_sort.cuh; floats
//                                    by bins over their values);
//   large tier  (len >  block cap)   one CTA cuts the segment into parts by its
//                                    sampled range, moves the keys there once
//                                    and sorts runs of parts in shared memory
//                                    (cta_sort.cuh; the LSD passes of Algorithms
//                                    4a/4b where two cuts do not separate them);
//   long tier   (len >= 2^31)        the LSD passes with 64-bit counters by one
//                                    CTA (seg_tiers.h), for segments that the
//                                    giant tier did not take;
//   giant tier  (len >= giant)       the device-wide radix sort, one segment at
//                                    a time, before the persistent launch (one
//                                    CTA per segment would leave the rest of the
//                                    GPU idle once the other segments are done).
// K7 seg_count / seg_scan / seg_fill put the segments in a work list, longest
// first (counting sort by floor(log2(len))); K8 seg_sort drains it.  Giant
// segments are the head of that list: the host reads the list's length
// histogram (one small synchronous copy), sorts the head segments with the
// device-wide path and has K8 start after them.
//
// What bounds K8: in the large tier the shared-memory atomics and accesses per
// key of three steps (count, move, bin sort) by two CTAs of 512 threads per SM;
// in the block tier the barriers of one bin sort per segment.  Before, the
// large tier made a stable pass per digit over global memory and the block
// tier merged: 10,000 int32 segments up to 1e6 keys (9.1e8 keys) 17.2 -> 9.3
// ms, 20,000 int64 ones up to 8,000 (2.6e7 keys) 1.80 -> 0.53 ms, 3,000
// float64 ones up to 1e5 (3.5e7 keys) 1.64 -> 0.79 ms.  Keys that neither cuts
// nor bins separate (one value in half of the places, magnitudes of every order,
// a thousand values) are about as fast as then, between 0.75 and 2 times.
#include <algorithm>
#include <vector>

#include "evosort.h"
#include "api_internal.h"
#include "common.cuh"
#include "cta_sort.cuh"
#include "seg_tiers.h"
#include "smem_sort.cuh"

namespace evosort {
namespace {

constexpr int kSB = kCtaThreads;     // threads per CTA
constexpr int kSW = kSB / 32;        // warps per CTA
constexpr int kWKW = 8;              // keys per lane in the warp tier (at most 256 keys)
constexpr int kNB = 48;              // length buckets (floor log2)

struct SegArgs {
    void* keys;
    const uint64_t* off;
    size_t nseg;
    size_t total;
    KeyMap map;
    void* tmp;          // scratch of total keys (large-tier ping-pong)
    uint32_t* hdr;      // [0..kNB) bucket counts, [kNB..2kNB) bucket cursors,
                        // [2kNB] single items, [2kNB+1] warp-tier segments, [2kNB+2] work counter,
                        // [2kNB+3] long-tier segments
    uint32_t* order;    // nseg entries: segment ids, longest first
    uint32_t* status;
    int block_cap;      // keys one CTA sorts in shared memory
    int warp_log2;      // warp tier: len < 2^warp_log2
    uint32_t skip;      // work items sorted before K8 (giant segments)
};

__device__ __forceinline__ int len_bucket(uint64_t len) { return 63 - __clzll((long long)len); }

// A segment is sorted only if it lies inside the array: lo <= hi <= total.
// Any other segment is reported (ST_BAD_OFFSETS) and left out of the work
// list, so no tier ever reads or writes outside [0, total).  total < 2^40 is
// checked on the host, so a valid length always has a bucket below kNB.
__device__ __forceinline__ bool seg_ok(const SegArgs& a, uint64_t lo, uint64_t hi) {
    return lo <= hi && hi <= a.total;
}

// K7a: validate offsets, count segments per length bucket.
__global__ void seg_count(SegArgs a) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && (a.off[0] != 0 || a.off[a.nseg] != a.total)) atomicOr(a.status, ST_BAD_OFFSETS);
    if (i >= a.nseg) return;
    const uint64_t lo = a.off[i], hi = a.off[i + 1];
    if (!seg_ok(a, lo, hi)) {
        atomicOr(a.status, ST_BAD_OFFSETS);
        return;
    }
    const uint64_t len = hi - lo;
    if (len >= 2) atomicAdd(&a.hdr[len_bucket(len)], 1u);
}

// K7b: bucket cursors in descending length order, item counts.
__global__ void seg_scan(SegArgs a) {
    if (threadIdx.x != 0) return;
    uint32_t pos = 0, single = 0, warp = 0, longs = 0;
    for (int b = kNB - 1; b >= 1; --b) {
        a.hdr[kNB + b] = pos;
        pos += a.hdr[b];
        if (b >= a.warp_log2)
            single += a.hdr[b];
        else
            warp += a.hdr[b];
        if (b >= kSegLongLog2) longs += a.hdr[b];
    }
    a.hdr[2 * kNB] = single;
    a.hdr[2 * kNB + 1] = warp;
    a.hdr[2 * kNB + 2] = 0;
    a.hdr[2 * kNB + 3] = longs;
}

// K7c: scatter segment ids into the work list.
__global__ void seg_fill(SegArgs a) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.nseg) return;
    const uint64_t lo = a.off[i], hi = a.off[i + 1];
    if (!seg_ok(a, lo, hi) || hi - lo < 2) return;
    const uint32_t p = atomicAdd(&a.hdr[kNB + len_bucket(hi - lo)], 1u);
    a.order[p] = (uint32_t)i;
}

// ---------------------------------------------------------------------------
// Tiers.
// ---------------------------------------------------------------------------
template <typename U, typename MI, typename MO>
__device__ __forceinline__ void warp_tier(const SegArgs& a, uint64_t lo, int len, const MI& in, const MO& out) {
    const int lane = threadIdx.x & 31;
    U* keys = (U*)a.keys + lo;
    U k[kWKW];
#pragma unroll
    for (int r = 0; r < kWKW; ++r) {
        const int i = lane * kWKW + r;
        k[r] = i < len ? in(keys[i]) : ~(U)0;
    }
    warp_bitonic_sort<U, kWKW>(k);
#pragma unroll
    for (int r = 0; r < kWKW; ++r) {
        const int i = lane * kWKW + r;
        if (i < len) keys[i] = out(k[r]);
    }
}

// One CTA, keys in registers and shared memory: bin sort over the segment's
// own range (bin_sort.cuh).
template <typename U, typename MI, typename MO>
__device__ __forceinline__ void block_tier(const SegArgs& a, unsigned char* smem, CtaShared<U>& sh, uint64_t lo, int len,
                                           const MI& in, const MO& out) {
    U* keys = (U*)a.keys + lo;
    U k[cta_kpt<U>()];
#pragma unroll
    for (int i = 0; i < cta_kpt<U>(); ++i)   // (every register is written)
        k[i] = in(i * kSB + (int)threadIdx.x < len ? keys[i * kSB + threadIdx.x] : (U)0);
    cta_local_sort<U>(k, len, out, smem, sh, [&](int i, U x) { keys[i] = out(x); });
}

template <typename U, typename MI, typename MO>
__global__ void __launch_bounds__(kSB, 2) seg_sort(SegArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_item;
    __shared__ CtaShared<U> sh;
    const MI in(a.map);
    const MO out(a.map);
    const uint32_t single = a.hdr[2 * kNB];
    const uint32_t nwarp = a.hdr[2 * kNB + 1];
    const uint32_t nbatch = (nwarp + kSW - 1) / kSW;
    // the head of the list: sorted by the device-wide path, or left to seg_long
    const uint32_t skip = max(a.skip, a.hdr[2 * kNB + 3]);
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(&a.hdr[2 * kNB + 2], 1u);
        __syncthreads();
        const uint32_t item = s_item;
        __syncthreads();
        if (item >= single + nbatch) break;
        if (item < skip) continue;
        if (item < single) {
            const uint32_t seg = a.order[item];
            const uint64_t lo = a.off[seg], len = a.off[seg + 1] - lo;
            if (len <= (uint64_t)a.block_cap) {
                block_tier<U>(a, smem, sh, lo, (int)len, in, out);
            } else {
                U* keys = (U*)a.keys + lo;
                cta_split_sort<U>(keys, (U*)a.tmp + lo, keys, (uint32_t)len, in, out, smem, sh);
            }
        } else {
            const uint32_t j = (item - single) * kSW + (threadIdx.x >> 5);
            if (j < nwarp) {
                const uint32_t seg = a.order[single + j];
                const uint64_t lo = a.off[seg];
                warp_tier<U>(a, lo, (int)(a.off[seg + 1] - lo), in, out);
            }
        }
    }
}

// Long tier: the head of the work list after the giant segments, one CTA per
// segment.  Launched only for batches that can hold such a segment; a kernel
// of its own, so that the other tiers keep their registers.
template <typename U>
__global__ void __launch_bounds__(kSB) seg_long(SegArgs a) {
    const uint32_t longs = a.hdr[2 * kNB + 3];
    for (uint32_t item = a.skip + blockIdx.x; item < longs; item += gridDim.x) {
        const uint32_t seg = a.order[item];
        const uint64_t lo = a.off[seg];
        const unsigned long long len = a.off[seg + 1] - lo;
        U* keys = (U*)a.keys + lo;
        cta_radix_sort<unsigned long long, false>(keys, (U*)a.tmp + lo, keys, len, GeneralOut<U>(a.map));
    }
}

// (lo, len) of the first `count` work items (the longest segments).
__global__ void seg_head(SegArgs a, uint32_t count, unsigned long long* out) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const uint32_t seg = a.order[i];
    out[2 * i] = a.off[seg];
    out[2 * i + 1] = a.off[seg + 1] - a.off[seg];
}

size_t seg_smem_bytes(int w) { return w == 4 ? cta_smem_bytes<uint32_t>() : cta_smem_bytes<uint64_t>(); }

size_t seg_hdr_bytes() { return 256 * sizeof(uint32_t); }

}  // namespace

size_t segmented_workspace_bytes(size_t total, size_t nseg, int w) {
    return seg_hdr_bytes() + (nseg * 4 + 255) / 256 * 256 + (total * w + 255) / 256 * 256;
}

static int segmented_giant(SegArgs& a, int dt, const Plan& pl, int gb, cudaStream_t s, uint32_t* skip,
                           std::string* err);

int segmented_sort(void* keys, size_t total, const uint64_t* off, size_t nseg, int dt, const Plan& pl, void* ws,
                   size_t ws_bytes, bool caller_ws, cudaStream_t s, std::string* err) {
    const int w = dtype_bytes(dt);
    if (ws_bytes < segmented_workspace_bytes(total, nseg, w)) {
        *err = "workspace too small";
        return EVOSORT_ERR_NOMEM;
    }
    uint32_t* status = status_word(err);
    if (!status) return EVOSORT_ERR_CUDA;
    SegArgs a;
    a.keys = keys;
    a.off = off;
    a.nseg = nseg;
    a.total = total;
    a.map = key_map_for(dt, pl.descending);
    a.hdr = (uint32_t*)ws;
    a.order = (uint32_t*)((char*)ws + seg_hdr_bytes());
    a.tmp = (char*)ws + seg_hdr_bytes() + (nseg * 4 + 255) / 256 * 256;
    a.status = status;
    a.block_cap = pl.seg_block_cap;
    a.warp_log2 = 31 - __builtin_clz((unsigned)pl.seg_warp_cap);
    a.skip = 0;
    const size_t smem = seg_smem_bytes(w);
    const int sms = sm_count();
    cudaError_t e = cudaMemsetAsync(ws, 0, seg_hdr_bytes(), s);
    const unsigned g = (unsigned)((nseg + 255) / 256);
    const int call = prof_call_begin(nullptr, 0, s);
    {
        ProfScope ps(call, EVOSORT_K_SEGMENTED, 0, 0.0, nseg, s);
        if (e == cudaSuccess && g) {
            seg_count<<<g, 256, 0, s>>>(a);
            seg_scan<<<1, 32, 0, s>>>(a);
            seg_fill<<<g, 256, 0, s>>>(a);
            e = cudaGetLastError();
        }
    }
    // giant tier: not while the stream is being captured (the length
    // histogram read would synchronise), nor with a caller workspace (the
    // device-wide path takes its own scratch)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (e == cudaSuccess && pl.seg_giant > 0 && !caller_ws && total >= (size_t)pl.seg_giant)
        e = cudaStreamIsCapturing(s, &cap);
    if (e == cudaSuccess && pl.seg_giant > 0 && !caller_ws && total >= (size_t)pl.seg_giant &&
        cap == cudaStreamCaptureStatusNone) {
        const int gb = 63 - __builtin_clzll((unsigned long long)pl.seg_giant);
        const int rc = segmented_giant(a, dt, pl, gb, s, &a.skip, err);
        if (rc != EVOSORT_OK) return rc;
    }
    {
        ProfScope ps(call, EVOSORT_K_SEGMENTED, 1, 2.0 * total * w, total, s);
        if (e == cudaSuccess) {
            // one kernel per key width and kind of key map
            static int resident[2][2] = {{0, 0}, {0, 0}};
            const int wi = w == 4 ? 0 : 1, fi = dt == EVOSORT_F32 || dt == EVOSORT_F64 ? 1 : 0;
            void (*const kerns[2][2])(SegArgs) = {
                {seg_sort<uint32_t, XorMap<uint32_t>, XorMap<uint32_t>>,
                 seg_sort<uint32_t, FloatIn<uint32_t>, FloatOut<uint32_t>>},
                {seg_sort<uint64_t, XorMap<uint64_t>, XorMap<uint64_t>>,
                 seg_sort<uint64_t, FloatIn<uint64_t>, FloatOut<uint64_t>>}};
            auto kern = kerns[wi][fi];
            if (resident[wi][fi] == 0) {
                e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                int nb = 0;
                if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kSB, smem);
                resident[wi][fi] = nb > 0 ? nb : 1;
            }
            if (e == cudaSuccess) {
                kern<<<(unsigned)(sms * resident[wi][fi]), kSB, smem, s>>>(a);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess && total > kSegCutKeys) {
                void (*const longk)(SegArgs) = w == 4 ? seg_long<uint32_t> : seg_long<uint64_t>;
                e = cudaFuncSetAttribute(longk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                const size_t most = total >> kSegLongLog2;   // such segments
                if (e == cudaSuccess) {
                    longk<<<(unsigned)(most < (size_t)sms ? most : (size_t)sms), kSB, smem, s>>>(a);
                    e = cudaGetLastError();
                    count_launches(1);
                }
            }
        }
    }
    prof_call_end(call, s, nullptr);
    count_launches(4);
    if (e != cudaSuccess) {
        *err = std::string("segmented launch: ") + cudaGetErrorString(e);
        return EVOSORT_ERR_CUDA;
    }
    return EVOSORT_OK;
}

// Giant tier: after K7, count the segments of at least 2^gb keys from the
// length histogram, sort each with the device-wide radix path (scratch from
// the stream-ordered pool, sized for the longest), and return how many head
// items K8 must skip.  Returns 0 items when there are none.
static int segmented_giant(SegArgs& a, int dt, const Plan& pl, int gb, cudaStream_t s, uint32_t* skip,
                           std::string* err) {
    *skip = 0;
    uint32_t hist[kNB];
    cudaError_t e = cudaMemcpyAsync(hist, a.hdr, sizeof(hist), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        *err = std::string("segmented sort: length histogram read: ") + cudaGetErrorString(e);
        return EVOSORT_ERR_CUDA;
    }
    uint32_t k = 0;
    for (int b = gb; b < kNB; ++b) k += hist[b];
    if (k == 0) return EVOSORT_OK;
    std::vector<unsigned long long> head(2 * (size_t)k);
    unsigned long long* d_head = nullptr;
    e = cudaMallocAsync((void**)&d_head, head.size() * sizeof(unsigned long long), s);
    if (e == cudaSuccess) {
        seg_head<<<(k + 255) / 256, 256, 0, s>>>(a, k, d_head);
        count_launches(1);
        e = cudaMemcpyAsync(head.data(), d_head, head.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        cudaFreeAsync(d_head, s);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *err = std::string("segmented sort: giant segment list: ") + cudaGetErrorString(e);
        return EVOSORT_ERR_CUDA;
    }
    const int w = dtype_bytes(dt);
    size_t longest = 0;
    for (uint32_t i = 0; i < k; ++i) longest = std::max<size_t>(longest, head[2 * i + 1]);
    Plan rp;
    default_radix_plan(dt, &rp, longest);
    rp.descending = pl.descending;
    const size_t need = radix_workspace_bytes(longest, w, false, rp);
    void* ws = nullptr;
    e = cudaMallocAsync(&ws, need, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *err = std::string("segmented sort: giant segment scratch: ") + cudaGetErrorString(e);
        return EVOSORT_ERR_NOMEM;
    }
    int rc = EVOSORT_OK;
    for (uint32_t i = 0; i < k && rc == EVOSORT_OK; ++i) {
        void* seg = (char*)a.keys + head[2 * i] * w;
        Plan sp;
        default_radix_plan(dt, &sp, head[2 * i + 1]);
        sp.descending = pl.descending;
        rc = radix_sort(seg, seg, nullptr, nullptr, head[2 * i + 1], dt, sp, ws, need, s, err);
    }
    cudaFreeAsync(ws, s);
    *skip = k;
    return rc;
}

}  // namespace evosort
