#include "tc_chain.cuh"

template cudaError_t tc_launch_t<64, 1, false, 1>(const TcMaps&, const TcArgs&, int, cudaStream_t);
template cudaError_t tc_launch_t<64, 1, true, 1>(const TcMaps&, const TcArgs&, int, cudaStream_t);
