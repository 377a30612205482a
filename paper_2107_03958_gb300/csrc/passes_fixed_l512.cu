// passes_fixed_l512.cu -- fixed-point FP64 passes, lines of 512 with n = L/2.
#include "passes_fixed_launch.cuh"

namespace wsc {
template conv_status run_fixed<512>(conv_plan_s *, const void *, const void *, void *, int, double, double, double, bool, void *, cudaStream_t);
template conv_status set_attrs_fixed<512>(int);
}  // namespace wsc
