// Forward transport on Voronoi grids (the VoronoiDustGrid of the SKIRT paper,
// Table 1(d) and Sect. 2.4): the transport engine of rt_transport.cuh
// instantiated with the walk across the cells' bisecting planes.
#include "rt_transport.cuh"

// four resident blocks of 256 (64 registers; 16 B of spills): more warps to
// hide the latency of the face-plane loads
#ifndef RT_VOR_MIN_BLOCKS
#define RT_VOR_MIN_BLOCKS 4
#endif

namespace rtk {

namespace {
__global__ void __launch_bounds__(tr::kBlock, RT_VOR_MIN_BLOCKS) k_forward_voronoi(const __grid_constant__ FwdParams P) {
  tr::forward_body<tr::VorGrid>(P);
}
}  // namespace

cudaError_t launch_forward_voronoi(const FwdParams& p, int num_sms, cudaStream_t stream) {
  return tr::launch_body<tr::VorGrid, false>(k_forward_voronoi, p, num_sms, 0,
                                            stream);
}

}  // namespace rtk
