// Multi-scale strip kernels with octahedral output.
#include "nrm_multiscale_strip.cuh"

namespace nrm {

template const void* ms_strip::by_form<NRM_OUT_OCT16>(int, bool, int);

}  // namespace nrm
