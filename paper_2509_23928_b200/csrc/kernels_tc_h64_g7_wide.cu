#include "tc_chain.cuh"

template cudaError_t tc_launch_t<64, 7, false, 2>(const TcMaps&, const TcArgs&, int, cudaStream_t);
template cudaError_t tc_launch_t<64, 7, false, 4>(const TcMaps&, const TcArgs&, int, cudaStream_t);
