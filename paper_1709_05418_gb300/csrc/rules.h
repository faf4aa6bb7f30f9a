// rules.h -- index and size rules shared by host code and kernels.  Plain C++, so that a host
// compiler alone can evaluate them over ranges no device buffer of a test would reach.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define RPNN_RULE __host__ __device__ __forceinline__
#else
#define RPNN_RULE inline
#endif

namespace rpnn {

// Offset of shading point i in the lists of positions and directions (three floats a point).
// A render has up to 2^31 - 1 samples, so from i = 715,827,883 on the offset needs 64 bits.
RPNN_RULE int64_t query_at(int64_t i) { return 3 * i; }

}  // namespace rpnn
