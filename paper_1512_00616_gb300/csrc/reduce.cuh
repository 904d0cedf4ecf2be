// Warp-level reductions shared by the Krylov kernels.
#pragma once

namespace pp {

template <int CNT, int O, class T>
__device__ __forceinline__ void rs_step(T* v, int lane) {
  if constexpr (O > 0) {
    if constexpr (CNT > 1) {
      constexpr int half = CNT / 2;
      const bool upper = (lane & O) != 0;
#pragma unroll
      for (int t = 0; t < half; ++t) {
        const T send = upper ? v[t] : v[t + half];
        const T keep = upper ? v[t + half] : v[t];
        v[t] = keep + __shfl_xor_sync(0xffffffffu, send, O);
      }
      rs_step<half, O / 2, T>(v, lane);
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], O);
      rs_step<1, O / 2, T>(v, lane);
    }
  }
}

// Warp reduce-scatter of KB (power of two, <= 32) per-lane values: afterwards lane l
// holds the warp sum of value (l >> (5 - log2 KB)) in v[0] (31 shuffles for KB = 32).
template <int KB, class T>
__device__ __forceinline__ void warp_reduce_scatter(T* v, int lane) {
  rs_step<KB, 16, T>(v, lane);
}

template <int KB>
struct ILog2 {
  static constexpr int value = KB >= 32 ? 5 : KB >= 16 ? 4 : KB >= 8 ? 3 : KB >= 4 ? 2 : KB >= 2 ? 1 : 0;
};

}  // namespace pp
