// Warp reductions shared by the refresh kernels.
#pragma once

#include <cuda_runtime.h>

namespace zo {

// Recursive-halving reduction of R per-lane values across a warp.  Afterwards
// lane l holds the warp sum of element c = l * (R/32) + k (k < R/32) when R >= 32,
// or of element c = l / (32/R) (in p[0]) when R < 32.
template <int R>
__device__ __forceinline__ void warp_reduce_scatter(float (&p)[R], int lane) {
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int o = 16 >> s;
    const int size = R >> s;
    if (size >= 2) {
      const int half = size >> 1;
      const bool upper = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < R / 2; ++i) {
        if (i < half) {
          const float send = upper ? p[i] : p[i + half];
          const float keep = upper ? p[i + half] : p[i];
          p[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
    } else {
      p[0] += __shfl_xor_sync(0xffffffffu, p[0], o);
    }
  }
}

}  // namespace zo
