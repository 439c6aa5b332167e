// Instances of the reverse pass (adj_tile.cuh) for subdomains up to 64 columns wide (with
// padding code: subdomains that fill their block run it as well).
#include "adj_tile.cuh"

namespace ddtv {

cudaError_t launch_adj_tile_16_4(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st) {
  return launch_adj_tile<16, 4, true, true>(a, z, fid, cl, st);
}
cudaError_t launch_adj_tile_16_8(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st) {
  return launch_adj_tile<16, 8, false, true>(a, z, fid, cl, st);
}
cudaError_t prepare_adj_tile_16_4() { return prepare_adj_tile<16, 4, true, true>(); }
cudaError_t prepare_adj_tile_16_8() { return prepare_adj_tile<16, 8, false, true>(); }

}  // namespace ddtv
