// Instances of the micro-tile kernel (fused_tile.cuh) for subdomains up to 128 columns wide.
#include "fused_tile.cuh"

namespace ddtv {

namespace {

template <int FID, bool MASK>
cudaError_t launch_adapt_one(const LocalArgs& a, int cl, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cl * a.g.NC * a.g.NR, 1, 1);
  cfg.blockDim = dim3(128, 1, 1);
  cfg.dynamicSmemBytes = AdaptTileLayout<32, 4>::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (has_interfaces(a.g)) pdl_attr(&attr[cfg.numAttrs++]);
  attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
  attr[cfg.numAttrs].val.clusterDim.x = cl;
  attr[cfg.numAttrs].val.clusterDim.y = 1;
  attr[cfg.numAttrs++].val.clusterDim.z = 1;
  return cudaLaunchKernelEx(&cfg, k_tile_adapt<32, 4, FID, MASK>, a, cl);
}

cudaError_t prepare_adapt() {
  auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AdaptTileLayout<32, 4>::BYTES);
  };
  cudaError_t e;
  if ((e = set(k_tile_adapt<32, 4, FID_L2, false>)) != cudaSuccess) return e;
  if ((e = set(k_tile_adapt<32, 4, FID_L2, true>)) != cudaSuccess) return e;
  if ((e = set(k_tile_adapt<32, 4, FID_L1, false>)) != cudaSuccess) return e;
  if ((e = set(k_tile_adapt<32, 4, FID_L1, true>)) != cudaSuccess) return e;
  return set(k_tile_adapt<32, 4, FID_SEG, false>);
}

}  // namespace

cudaError_t launch_tile_adapt_128(const LocalArgs& a, int fid, cudaStream_t st) {
  const bool m = a.mask != nullptr;
  const int cl = 128 / TileLayout<32, 4>::BAND;
  switch (fid) {
    case FID_L2: return m ? launch_adapt_one<FID_L2, true>(a, cl, st) : launch_adapt_one<FID_L2, false>(a, cl, st);
    case FID_L1: return m ? launch_adapt_one<FID_L1, true>(a, cl, st) : launch_adapt_one<FID_L1, false>(a, cl, st);
    default: return launch_adapt_one<FID_SEG, false>(a, cl, st);
  }
}

cudaError_t launch_tile_32_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return launch_tile<32, 4, true>(a, fid, cl, pad, st);
}
cudaError_t prepare_tile_32_4() {
  cudaError_t e;
  if ((e = prepare_adapt()) != cudaSuccess) return e;
  if ((e = prepare_tile_batch<32, 4, 8>()) != cudaSuccess) return e;
  return prepare_tile<32, 4, true>();
}
cudaError_t launch_tile_batch_128(const BatchArgs& B, int total_tiles, bool overlap, cudaStream_t st) {
  return launch_tile_batch<32, 4, 8>(B, total_tiles, overlap, st);
}

}  // namespace ddtv
