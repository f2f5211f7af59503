// mg_flowstore.cuh -- where a thread keeps its event's colour-flow
// accumulators (JAMPs) while the chunked helicity program runs.
//
// The chunk functions of the largest process update the flows through this
// store: a pattern of amplitudes, summed in a register, is added to (or
// subtracted from) each flow of the pattern at once.  FlowsSmem<R>: the
// thread's column of a [flow][thread] array in shared memory (stride js).
#pragma once

#include "mg_vertices.cuh"

namespace mg {

template <typename R>
struct FlowsSmem {
  cx<R>* p;
  int js;
  template <int N>
  __device__ __forceinline__ void update(const int (&k)[N], const int (&sg)[N], cx<R> v) const {
#pragma unroll
    for (int i = 0; i < N; i++) {
      cx<R>& t = p[k[i] * js];
      t = sg[i] > 0 ? t + v : t - v;
    }
  }
  __device__ __forceinline__ void zero(int n) const {
    for (int c = 0; c < n; c++) p[c * js] = cx<R>{R(0), R(0)};
  }
};

}  // namespace mg
