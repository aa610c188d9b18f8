// Forward transport on octree grids (SKIRT paper, Sect. 2.4): the
// transport engine of rt_transport.cuh instantiated with the octree cell
// walk (ancestor stack per lane in shared memory, top of the tree cached in
// shared memory).
#include "rt_transport.cuh"

// Resident blocks per SM the register allocation aims at: four (64
// registers) fit the shared memory of trees up to depth 10, whose per-lane
// ancestor stacks (dynamic shared memory, depth + 1 entries) take 11 KB of
// the block's 55 KB; deeper trees run three.
#ifndef RT_OCT_MIN_BLOCKS
#define RT_OCT_MIN_BLOCKS 4
#endif

namespace rtk {

namespace {
__global__ void __launch_bounds__(tr::kBlock, RT_OCT_MIN_BLOCKS) k_forward_octree(const __grid_constant__ FwdParams P) {
  tr::forward_body<tr::OctGrid>(P);
}
}  // namespace

cudaError_t launch_forward_octree(const FwdParams& p, int num_sms, cudaStream_t stream) {
  return tr::launch_body<tr::OctGrid, false>(k_forward_octree, p, num_sms, (size_t)tr::kBlock * (size_t)p.oct_levels * sizeof(int),
                                            stream);
}

}  // namespace rtk
