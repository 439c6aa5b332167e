// Instances of the reverse pass (adj_tile.cuh) for subdomains up to 32 columns wide (with
// padding code: subdomains that fill their block run it as well).
#include "adj_tile.cuh"

namespace ddtv {

cudaError_t launch_adj_tile_8_2(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st) {
  return launch_adj_tile<8, 2, false, true>(a, z, fid, cl, st);
}
cudaError_t launch_adj_tile_8_4(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st) {
  return launch_adj_tile<8, 4, true, true>(a, z, fid, cl, st);
}
cudaError_t prepare_adj_tile_8_2() { return prepare_adj_tile<8, 2, false, true>(); }
cudaError_t prepare_adj_tile_8_4() { return prepare_adj_tile<8, 4, true, true>(); }

}  // namespace ddtv
