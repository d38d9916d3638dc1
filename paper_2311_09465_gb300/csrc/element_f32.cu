// Element operator in FP32: instantiations of element.cuh
#include "element.cuh"

namespace ts {
#define TS_INST_EL_F32(T, N)                                                                 \
  template int launch_element<float, N>(int, const ElementArgs<float>&, cudaStream_t);       \
  template int launch_node_prepass<float, N>(const float*, const uint8_t*, float*, float*,  \
                                             const float*, int64_t, cudaStream_t, unsigned*, float*);
TS_FOR_EACH_N(TS_INST_EL_F32, float)
template int launch_gather<float>(const int32_t*, const int32_t*, const float*, const uint8_t*, float*, int64_t, int, int,
                                   int, cudaStream_t);
#define TS_INST_TR_F32(T, N) template int launch_tracer<float, N>(const TracerArgs<float>&, cudaStream_t);
TS_FOR_EACH_N(TS_INST_TR_F32, float)
template int launch_clean<float>(const float*, float*, int64_t, int, cudaStream_t);
}  // namespace ts
