// Strip kernels for frames of any pitch and alignment (loader warps in place of TMA;
// float4 and half4 rows through a row buffer, octahedral codes one store per pixel).
#include "nrm_forward_strip.cuh"

namespace nrm {

template const void* strip_kernel<false>(int, bool, int, bool);

}  // namespace nrm
