#include "conef_lrgen_codec.cuh"

namespace conef {

template cudaError_t gen_launch_codec<CONEF_C_INT8>(int, int, bool, const DevView &, const int32_t *, int, cudaStream_t, size_t);

}  // namespace conef
