// Instances of the micro-tile kernel (fused_tile.cuh) for subdomains up to 128 columns wide.
#include "fused_tile.cuh"

namespace ddtv {

cudaError_t launch_tile_32_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<32, 4, true>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_32_4() {
  const cudaError_t e = prepare_tile_batch<32, 4, 8>();
  return e != cudaSuccess ? e : prepare_tile<32, 4, true>();
}
cudaError_t launch_tile_batch_128(const BatchArgs& B, int total_tiles, bool overlap, cudaStream_t st) {
  return launch_tile_batch<32, 4, 8>(B, total_tiles, overlap, st);
}

}  // namespace ddtv
