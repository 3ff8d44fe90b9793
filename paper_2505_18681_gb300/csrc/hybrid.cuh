// Control words shared by the partition sort (hybrid.cu) and the radix
// kernels that give way to it.
#pragma once

#include "common.cuh"

namespace evosort {

// Words of the control block (zeroed with the radix scratch): the sample's
// decision; set when the path was given up later; the cut of the key range (hybrid.cu): smallest key and width
// (64-bit), leading zeros of the width, number of equal stretches (0: by the
// table of cells), last bin; set when keys lie below or above that
// range; local sorts past one per stretch.
enum : int { HYB_ON = 0, HYB_FAIL = 1, HYB_LO = 4, HYB_WIDTH = 6, HYB_LZ = 8, HYB_BINS = 9, HYB_TOP = 10,
             HYB_BELOW = 11, HYB_ABOVE = 12, HYB_MORE = 13, HYB_WORDS = 16 };

// True once the partition sort has sorted the array (read after its last
// kernel).
__device__ __forceinline__ bool hybrid_done(const uint32_t* ctl) {
    return ctl && ctl[HYB_ON] != 0u && ctl[HYB_FAIL] == 0u;
}

struct PassDesc;
// Scratch of the partition sort; it is cut from the look-back slots.
size_t hybrid_scratch_bytes(int w, size_t n);
// Enqueues the path's kernels: in -> out through tmp (in == out allowed).
// ctl and scratch are zeroed; last: the entry after the radix passes; call: the profile's call number.
cudaError_t launch_hybrid_sort(int w, const void* in, void* out, void* tmp, size_t n, const KeyMap& map, uint32_t* ctl,
                               void* scratch, PassDesc* last, int call, cudaStream_t s);

}  // namespace evosort
