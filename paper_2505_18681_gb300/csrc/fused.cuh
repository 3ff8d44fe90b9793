// Radix sort of a mid-sized array in one launch (fused.cu).
#pragma once

#include "common.cuh"

namespace evosort {

struct PassDesc;
// Most keys the one-launch sort takes.
size_t fused_max_keys(int w, bool pairs);
// Bytes of control words, zeroed before the launch.
size_t fused_ctl_bytes();
// counts: 512 bytes per 1024 keys (rounded up), bins: 32 KB (keys only);
// neither needs to be zeroed.  desc: zeroed pass descriptors of w passes and
// one more, which receive what ran.
cudaError_t launch_radix_fused(int w, const void* in, void* out, const uint32_t* vin, uint32_t* vout, size_t n,
                               const KeyMap& map, unsigned long long* ctl, void* counts, void* bins, PassDesc* desc,
                               uint32_t* status, cudaStream_t s);

}  // namespace evosort
