// Fixed-point x and y transform passes of the FP32-pair spectra.
#include "fxpass.cuh"

namespace vofp {
template void init_fx_attributes<ff>();
template bool fx_xfwd<ff>(vofp_plan*, int, const XArgs&, cudaStream_t);
template bool fx_ypass<ff>(vofp_plan*, const YArgs&, bool, cudaStream_t);
template bool fx_xinv<ff>(vofp_plan*, const XInvArgs&, cudaStream_t);
}  // namespace vofp
