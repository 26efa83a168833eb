// The coarse-cycle cluster of the complex64 cycles (cluster.cuh; a file per
// precision, compiled side by side).
#include "cluster.cuh"

namespace hmg {

template int cluster_size<float>(int);
template bool cluster_layout<float>(std::vector<ClLev<float>>&, int, bool, int, ClArgs<float>&);
template cudaError_t launch_cluster_cycle<float>(const ClArgs<float>&, int, cudaStream_t);
template void launch_cluster_cycle_rag<float>(const std::vector<ClArgs<float>>&, cudaStream_t);

}  // namespace hmg
