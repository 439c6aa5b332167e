// Instances of the micro-tile kernel (fused_tile.cuh) for subdomains up to 128 columns wide.
#include "fused_tile.cuh"

namespace ddtv {

namespace {

template <int FID, bool MASK>
cudaError_t launch_adapt_one(const LocalArgs& a, int cl, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cl * a.g.NC * a.g.NR, 1, 1);
  cfg.blockDim = dim3(128, 1, 1);
  cfg.dynamicSmemBytes = a.chain ? tile_bytes<32, 4, false, true, true>() : tile_bytes<32, 4, false, true, false>();
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (a.chain || has_interfaces(a.g)) pdl_attr(&attr[cfg.numAttrs++]);
  attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
  attr[cfg.numAttrs].val.clusterDim.x = cl;
  attr[cfg.numAttrs].val.clusterDim.y = 1;
  attr[cfg.numAttrs++].val.clusterDim.z = 1;
  return a.chain ? cudaLaunchKernelEx(&cfg, k_tile_adapt<32, 4, FID, MASK, true>, a, cl)
                 : cudaLaunchKernelEx(&cfg, k_tile_adapt<32, 4, FID, MASK, false>, a, cl);
}

template <bool CHAIN>
cudaError_t prepare_adapt() {
  auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)tile_bytes<32, 4, false, true, CHAIN>());
  };
  cudaError_t e;
  if ((e = set(k_tile_adapt<32, 4, FID_L2, false, CHAIN>)) != cudaSuccess) return e;
  if ((e = set(k_tile_adapt<32, 4, FID_L2, true, CHAIN>)) != cudaSuccess) return e;
  if ((e = set(k_tile_adapt<32, 4, FID_L1, false, CHAIN>)) != cudaSuccess) return e;
  if ((e = set(k_tile_adapt<32, 4, FID_L1, true, CHAIN>)) != cudaSuccess) return e;
  return set(k_tile_adapt<32, 4, FID_SEG, false, CHAIN>);
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
cudaError_t prepare_tile_32_4(bool pad, bool chain) { return prepare_tile<32, 4, true>(pad, chain); }
cudaError_t prepare_tile_batch_128() { return prepare_tile_batch<32, 4, 8>(); }
cudaError_t prepare_tile_adapt_128(bool chain) { return chain ? prepare_adapt<true>() : prepare_adapt<false>(); }
cudaError_t launch_tile_batch_128(const BatchArgs& B, int total_tiles, bool overlap, cudaStream_t st) {
  return launch_tile_batch<32, 4, 8>(B, total_tiles, overlap, st);
}

}  // namespace ddtv
