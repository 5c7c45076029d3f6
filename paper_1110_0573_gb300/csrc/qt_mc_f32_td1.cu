// qt_mc_f32_td1.cu -- mixed-precision instances of the Monte-Carlo kernel for
// one narrow time-dependent term.
#include "qt_mc_dispatch.cuh"

namespace qt {

cudaError_t launch_mc_f32_td1(const McArgs &a, int R, int W, cudaStream_t s) { return dispatch_td_one<float>(a, R, W, s); }

}  // namespace qt
