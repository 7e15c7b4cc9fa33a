// Backprojector kernels of geometries whose LORs cross at most 3 slice(s) inside one pixel.
#include "backward.cuh"

namespace spdhg {
template cudaError_t launch_backward_nt<3>(const DevGeom&, int, int, const BwdArgs&, cudaStream_t);
template cudaError_t backward_items_nt<3>(const DevGeom&, int, unsigned short*, unsigned*, const unsigned*, const unsigned*, float4*, int2*, cudaStream_t);
}  // namespace spdhg
