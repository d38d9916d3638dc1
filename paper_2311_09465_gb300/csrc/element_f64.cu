// Tracer in native FP64: instantiations of element.cuh
#include "element.cuh"

namespace ts {
#define TS_INST_TR_F64(T, N)                                                                     \
  template int launch_tracer<double, N>(const TracerArgs<double>&, cudaStream_t);                \
  template int launch_node_prepass<double, N>(const double*, const uint8_t*, double*, double*,   \
                                              const double*, int64_t, cudaStream_t, unsigned*, double*);
TS_FOR_EACH_N(TS_INST_TR_F64, double)
template int launch_gather<double>(const int32_t*, const int32_t*, const double*, const uint8_t*, double*, int64_t, int,
                                   int, int, cudaStream_t);
template int launch_clean<double>(const double*, double*, int64_t, int, cudaStream_t);
}  // namespace ts
