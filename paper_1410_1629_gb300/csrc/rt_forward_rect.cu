// Forward transport on rectilinear grids (cells between arbitrary edges per
// axis; the PowCub grid of the SKIRT paper, Table 1(d)): the transport engine
// of rt_transport.cuh instantiated with the rectilinear cell walk.
#include "rt_transport.cuh"

namespace rtk {

namespace {
__global__ void __launch_bounds__(tr::kBlock, RT_FWD_MIN_BLOCKS) k_forward_rect(const __grid_constant__ FwdParams P) {
  tr::forward_body<tr::RectGrid>(P);
}
}  // namespace

cudaError_t launch_forward_rect(const FwdParams& p, int num_sms, cudaStream_t stream) {
  return tr::launch_body<tr::RectGrid, false>(k_forward_rect, p, num_sms, 0,
                                            stream);
}

}  // namespace rtk
