// Instantiation of the tuned kernels (dwf_hop2.cuh) for one storage precision
// (DWF_HOP2_STORE) and one group of Ls (DWF_HOP2_GROUP); build.py compiles this file once
// for each of them, in parallel.
#include "dwf_hop2.cuh"

namespace dwf {
namespace hop2 {
using SP = DWF_HOP2_STORE;
template cudaError_t dispatch<SP, DWF_HOP2_GROUP>(const Geom&, const HopLaunch&, cudaStream_t);
template cudaError_t dispatch<SP, DWF_HOP2_GROUP>(const Geom&, const LocalLaunch&, cudaStream_t);
template cudaError_t dispatch<SP, DWF_HOP2_GROUP>(const Geom&, const RUpdateLaunch&, cudaStream_t);
}  // namespace hop2
}  // namespace dwf
