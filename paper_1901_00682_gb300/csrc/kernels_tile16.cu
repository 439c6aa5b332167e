// Instances of the micro-tile kernel (fused_tile.cuh) for subdomains up to 64 columns wide.
#include "fused_tile.cuh"

namespace ddtv {

namespace {

// Every 64 x 64 subdomain of a batch of images, one CTA each, with its image's fidelity,
// parameters and strips (blockIdx.y = the batch's subdomain).
__global__ void __launch_bounds__(256, 2) k_tile_batch(const BatchArgs B) {
  const int t = blockIdx.y;
  const int img = B.tile_img[t];
  const LocalArgs A = B.args[img];
  const int q = t - B.tile_base[img];
  const int a = q / A.g.NC, b = q - a * A.g.NC;
  const Strips out = B.strips[2 * img + B.write_set];
  switch (B.fid[img]) {
    case FID_L2: tile_solve<16, 8, false, false, FID_L2, false>(A, out, a, b); break;
    case FID_L1: tile_solve<16, 8, false, false, FID_L1, false>(A, out, a, b); break;
    default: tile_solve<16, 8, false, false, FID_SEG, false>(A, out, a, b); break;
  }
}

}  // namespace

cudaError_t launch_tile_16_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<16, 4, true>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_16_4() { return prepare_tile<16, 4, true>(); }

cudaError_t launch_tile_16_8(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<16, 8, false>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_16_8() {
  const cudaError_t e = cudaFuncSetAttribute(k_tile_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)TileLayout<16, 8>::BYTES);
  return e != cudaSuccess ? e : prepare_tile<16, 8, false>();
}

cudaError_t launch_tile_batch_64(const BatchArgs& B, int total_tiles, cudaStream_t st) {
  k_tile_batch<<<dim3(1, total_tiles, 1), TileLayout<16, 8>::NT, TileLayout<16, 8>::BYTES, st>>>(B);
  return cudaGetLastError();
}

}  // namespace ddtv
