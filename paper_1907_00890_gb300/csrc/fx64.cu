// Fixed-point x and y transform passes of the FP64 spectra.
#include "fxpass.cuh"

namespace vofp {
template void init_fx_attributes<double>();
template bool fx_xfwd<double>(vofp_plan*, int, const XArgs&, cudaStream_t);
template bool fx_ypass<double>(vofp_plan*, const YArgs&, bool, cudaStream_t);
template bool fx_xinv<double>(vofp_plan*, const XInvArgs&, cudaStream_t);
}  // namespace vofp
