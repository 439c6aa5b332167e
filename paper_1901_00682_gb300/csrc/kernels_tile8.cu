// Instances of the micro-tile kernel (fused_tile.cuh) for subdomains up to 32 columns wide.
#include "fused_tile.cuh"

namespace ddtv {

cudaError_t launch_tile_8_2(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<8, 2, false>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_8_2(bool pad, bool chain) { return prepare_tile<8, 2, false>(pad, chain); }

cudaError_t launch_tile_8_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<8, 4, true>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_8_4(bool pad, bool chain) { return prepare_tile<8, 4, true>(pad, chain); }

}  // namespace ddtv
