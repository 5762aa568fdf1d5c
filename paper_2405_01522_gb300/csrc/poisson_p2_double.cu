// pass 2 (y/z transforms with the kernel multiply), double
#include "poisson_launch.cuh"

namespace rsx {
template size_t pass2_smem_bytes<double>(const Geom&, bool*);
template size_t pass2_gscratch_bytes<double>(const Geom&, int);
template cudaError_t prepare_pass2<double>(const Geom&, int*);
template cudaError_t launch_pass2<double>(const Geom&, int, Cx<double>*, const Cx<double>*, const double*, double*, int, cudaStream_t);
}  // namespace rsx
