// Instances of the reverse pass (adj_tile.cuh) for subdomains up to 128 columns wide.
#include "adj_tile.cuh"

namespace ddtv {

cudaError_t launch_adj_tile_32_4(const LocalArgs& a, const AdjArgs& z, int fid, int cl, bool pad, cudaStream_t st) {
  return pad ? launch_adj_tile<32, 4, true, true>(a, z, fid, cl, st) : launch_adj_tile<32, 4, true, false>(a, z, fid, cl, st);
}
cudaError_t prepare_adj_tile_32_4() {
  const cudaError_t e = prepare_adj_tile<32, 4, true, true>();
  return e != cudaSuccess ? e : prepare_adj_tile<32, 4, true, false>();
}

}  // namespace ddtv
