// Instances of the micro-tile kernel (fused_tile.cuh) for subdomains up to 64 columns wide.
#include "fused_tile.cuh"

namespace ddtv {

cudaError_t launch_tile_16_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<16, 4, true>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_16_4(bool pad, bool chain) { return prepare_tile<16, 4, true>(pad, chain); }

cudaError_t launch_tile_16_8(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<16, 8, false>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_16_8(bool pad, bool chain) { return prepare_tile<16, 8, false>(pad, chain); }
cudaError_t prepare_tile_batch_64() { return prepare_tile_batch<16, 8, 1>(); }
cudaError_t launch_tile_batch_64(const BatchArgs& B, int total_tiles, bool overlap, cudaStream_t st) {
  return launch_tile_batch<16, 8, 1>(B, total_tiles, overlap, st);
}

}  // namespace ddtv
