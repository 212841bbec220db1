// The FP32 general z passes of largest stage radix 32 (see gen_z_radix).
#include "mixed_impl.cuh"

namespace demag {
template cudaError_t gen_z_launch<float, 32>(int, float2 *, int, int, int64_t, int64_t, int64_t, int, const float *, int, int,
                                             const float2 *, int, cudaStream_t);
template cudaError_t gen_sp_z_launch<float, 32>(int, float2 *, int, int, int64_t, int64_t, int64_t, int, int, const float *,
                                                int, int, const float2 *, const float2 *, const float2 *, const float2 *,
                                                cudaStream_t);
}  // namespace demag
