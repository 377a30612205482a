// passes_fixed_l0.cu -- fixed-point FP64 passes, any other length.
#include "passes_fixed_launch.cuh"

namespace wsc {
template conv_status run_fixed<0>(conv_plan_s *, const void *, const void *, void *, int, double, double, double, bool, void *, cudaStream_t);
template conv_status set_attrs_fixed<0>(int);
}  // namespace wsc
