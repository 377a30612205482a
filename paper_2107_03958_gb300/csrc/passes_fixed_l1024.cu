// passes_fixed_l1024.cu -- fixed-point FP64 passes, lines of 1024 with n = L/2.
#include "passes_fixed_launch.cuh"

namespace wsc {
template conv_status run_fixed<1024>(conv_plan_s *, const void *, const void *, void *, int, double, double, double, bool, void *, cudaStream_t);
template conv_status set_attrs_fixed<1024>(int);
}  // namespace wsc
