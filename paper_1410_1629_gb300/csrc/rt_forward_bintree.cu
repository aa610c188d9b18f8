// Forward transport on k-d tree grids (the BinTree grid of the SKIRT paper,
// Table 1(d)): the transport engine of rt_transport.cuh instantiated with
// the k-d tree cell walk.
#include "rt_transport.cuh"

// four resident blocks of 256 (64 registers; 4 B of spills) hide more of the
// L2 latency of the node-word loads than three without spills: 350 -> 316 ms
// on the clumpy 2e5-leaf tree
#ifndef RT_BIN_MIN_BLOCKS
#define RT_BIN_MIN_BLOCKS 4
#endif

namespace rtk {

namespace {
__global__ void __launch_bounds__(tr::kBlock, RT_BIN_MIN_BLOCKS) k_forward_bintree(const __grid_constant__ FwdParams P) {
  tr::forward_body<tr::BinGrid>(P);
}
}  // namespace

cudaError_t launch_forward_bintree(const FwdParams& p, int num_sms, cudaStream_t stream) {
  return tr::launch_body<tr::BinGrid, false>(k_forward_bintree, p, num_sms, 0,
                                            stream);
}

}  // namespace rtk
