// Multi-scale strip kernels with half4 output.
#include "nrm_multiscale_strip.cuh"

namespace nrm {

template const void* ms_strip::by_form<NRM_OUT_F16X4>(int, bool, int);

}  // namespace nrm
