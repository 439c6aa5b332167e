// Dispatch of the tile-fused reverse pass (adj_tile.cuh): the plan of the forward's
// micro-tile kernel, and the tape it needs.
#include "internal.cuh"

namespace ddtv {

long long adj_alpha_slots_fused(const Grid& g) { return (long long)g.NR * g.NC * 8; }

size_t adj_fused_tape_floats(const Grid& g, int K) {
  TilePlan p;
  if (!tile_plan(g, &p)) return 0;
  return (size_t)g.NR * g.NC * p.cl * 32 * p.nw * kTapeWords * K;
}

cudaError_t adj_fused_prepare(const Grid& g) {
  TilePlan p;
  if (!tile_plan(g, &p)) return cudaErrorInvalidValue;
  if (p.lpr == 8) return p.nw == 2 ? prepare_adj_tile_8_2() : prepare_adj_tile_8_4();
  if (p.lpr == 16) return p.nw == 8 ? prepare_adj_tile_16_8() : prepare_adj_tile_16_4();
  return prepare_adj_tile_32_4();
}

cudaError_t launch_adj_fused(const LocalArgs& a, const AdjArgs& z, int fid, cudaStream_t st) {
  TilePlan p;
  if (!tile_plan(a.g, &p)) return cudaErrorInvalidValue;
  if (p.lpr == 8) return p.nw == 2 ? launch_adj_tile_8_2(a, z, fid, p.cl, st) : launch_adj_tile_8_4(a, z, fid, p.cl, st);
  if (p.lpr == 16)
    return p.nw == 8 ? launch_adj_tile_16_8(a, z, fid, p.cl, st) : launch_adj_tile_16_4(a, z, fid, p.cl, st);
  return launch_adj_tile_32_4(a, z, fid, p.cl, p.pad, st);
}

}  // namespace ddtv
