// The coarse-cycle cluster of the complex128 cycles (cluster.cuh).
#include "cluster.cuh"

namespace hmg {

template int cluster_size<double>(int);
template bool cluster_layout<double>(std::vector<ClLev<double>>&, int, bool, int, ClArgs<double>&);
template cudaError_t launch_cluster_cycle<double>(const ClArgs<double>&, int, cudaStream_t);
template void launch_cluster_cycle_rag<double>(const std::vector<ClArgs<double>>&, cudaStream_t);

}  // namespace hmg
