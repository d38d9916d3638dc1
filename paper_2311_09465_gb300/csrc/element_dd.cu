// Element operator in double-float (FP64 data): instantiations of element.cuh
#include "element.cuh"

namespace ts {
#define TS_INST_EL_DD(T, N)                                                                     \
  template int launch_element<float2, N>(int, const ElementArgs<float2>&, cudaStream_t);        \
  template int launch_node_prepass<float2, N>(const double*, const uint8_t*, float2*, float2*, \
                                              const float2*, int64_t, cudaStream_t, unsigned*, double*);
TS_FOR_EACH_N(TS_INST_EL_DD, double)
template int launch_gather<float2>(const int32_t*, const int32_t*, const float2*, const uint8_t*, double*, int64_t, int, int,
                                   int, cudaStream_t);
}  // namespace ts
