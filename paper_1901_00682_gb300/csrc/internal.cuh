// Internal declarations shared by the translation units of the dd_tv library.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "pointwise.cuh"

namespace ddtv {

// Image and subdomain grid.  cut_top / cut_bot: the top side of tile row 0 / the
// bottom side of tile row NR-1 lies on an interface with a neighbouring row-block
// shard (its dofs are active, its multipliers and strips sit one line before / after
// the handle's own lines); 0 for a whole image, where those sides are on the image
// boundary.
struct Grid {
  int H, W, NR, NC;
  int cut_top = 0, cut_bot = 0;
};

// Interface strips: the interface values of one torn dual field p~^n.
//   SB (NR-1) x W : bottom side of tile row a (s-side copy of horizontal interface a)
//   ST (NR-1) x W : top side of tile row a+1  (t-side copy)
//   SR (NC-1) x H : right side of tile column b (s-side copy of vertical interface b)
//   SL (NC-1) x H : left side of tile column b+1 (t-side copy)
struct Strips {
  float *SB, *ST, *SR, *SL;
};

// Arguments of one local-solve launch (fused or plain path).
struct LocalArgs {
  Grid g;
  int K;                 // inner iterations
  float tau;             // outer tau (proximal centre phat = p~ -+ tau lambda)
  float c1, c2;          // SEG constants
  const float* f;        // H x W
  const uint8_t* mask;   // H x W or nullptr
  float* u;              // H x W
  float* P1;             // (H + NR) x W torn
  float* P2;             // H x (W + NC) torn
  // the state the micro-tile kernel starts from (u, P1, P2 themselves, or another set of
  // arrays with zeros on the image boundary); the other kernels work in place
  const float *u0, *P10, *P20;
  const float* lamh;     // (NR-1) x W
  const float* lamv;     // (NC-1) x H
  Strips out;            // strips of p~^{n+1} (written at the end)
  // chain != 0 (micro-tile kernel only): the local solve makes the multiplier update itself.
  // Every side keeps its own copy of the multipliers (lam_s: lower / right sides, in the
  // layout of lamh and lamv; lam_t: upper / left sides), which both owners of an interface
  // update with the same operations from the extrapolated strips x_in = 2 p~^n - p~^{n-1}; x_out
  // receives 2 p~^{n+1} - p~^n.  (With a launch of its own the update cost 2 to 3 us per outer
  // iteration.)
  int chain;
  float sigma;
  float *lam_sh, *lam_sv, *lam_th, *lam_tv;
  Strips x_in, x_out;
  const Coef* coef;      // K coefficient sets (device)
  int* err;              // set non-zero by a kernel whose bounded wait ran out
  // adaptive inner stopping (eq. stop_inner1); inner_tol2 = 0 selects K fixed iterations
  double inner_tol2;               // tol^2: stop once sum (dp)^2 < tol^2 sum p^2
  int* inner_used;                 // NR * NC: inner iterations of each tile, last launch
  int* inner_max;                  // running maximum of inner_used
  unsigned long long* inner_work;  // running sum of tile pixels x inner iterations
};

// One set of the full-dimension path's state: u, p and the extrapolated pbar.
struct FullSet {
  float *u, *P1, *P2, *Pb1, *Pb2;  // H x W, (H + 1) x W, H x (W + 1), pbar likewise
};

// Arguments of one launch of full-dimension iterations (constant steps: coef[0]).
struct FullArgs {
  int H, W;
  float c1, c2;
  const float* f;
  const uint8_t* mask;   // or nullptr
  const Coef* coef;
  int* err;
  FullSet in, out;       // distinct arrays
};

// Batch of images solved together (every image partitioned into exact 128 x 128
// subdomains).  Device arrays, one entry per image unless stated otherwise.
struct BatchArgs {
  const LocalArgs* args;   // per-image descriptor (its `out` field is unused)
  const Strips* strips;    // 2 per image: strip sets by parity
  const int* fid;          // fidelity per image
  const int* tile_img;     // per tile of the batch: its image
  const int* tile_base;    // first batch tile of each image
  int write_set;           // strip set receiving p~^{n+1}
};

// Batched multiplier update: per image interface elements in units of 4 edges.
struct BatchIfaceArgs {
  const LocalArgs* args;   // per-image descriptor (geometry, lamh, lamv)
  const Strips* strips;    // 2 per image
  const float* sigma;      // outer sigma per image
  const int* elem_base;    // n_img + 1 prefix sums of (nh + nv) / 4
  int n_img;
  int cur_set;             // strip set holding p~^n
};

// Adjoint fields of the reverse pass (kernels_adjoint.cu).  A* is the adjoint of the
// named forward quantity; AP/AQ/APh live on the torn layout of P1/P2.
struct AdjArgs {
  Grid g;
  int fid;
  float c1, c2;
  const float* f;          // H x W
  const uint8_t* mask;     // H x W or nullptr
  float *Au, *Ad, *Af;     // H x W: u, div pbar (scaled), f
  double* Aal;             // adj_alpha_slots(g) per-block partial sums of the alpha adjoint
  const int4* rowtab;      // H: (tile row, first row, end row) of every pixel row
  const int4* coltab;      // W: (tile column, first column, end column) of every pixel column
  float *AP1, *AP2;        // p
  float *AQ1, *AQ2;        // pbar
  float *APh1, *APh2;      // phat
  float *ALh, *ALv;        // lambda
  Strips APp;              // interface values of p~^{n-1}
  float* tape;             // tile-fused reverse kernel: adj_fused_tape_floats(g, K) floats
  float neg_zero;          // -0.0f (fused_common.cuh round2)
};

// Programmatic dependent launch.  A kernel launched with pdl_attr may start while its
// predecessor in the stream still runs, once every block of that one has called
// pdl_trigger or ended; pdl_wait returns when the predecessor has completed and its
// writes are visible (at once in a kernel launched without the attribute).
//
// The outer iteration is a chain of short kernels: multiplier update, local solves, update,
// ...  Every one of them waits before its first access to what another of them writes; ahead
// of the wait it sets itself up and loads the data (f, the mask, the coefficients), which none
// of them writes.  The wait is also what makes the results of the kernels before the
// predecessor visible: that they have completed is not enough.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

inline void pdl_attr(cudaLaunchAttribute* attr) {
  attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr->val.programmaticStreamSerializationAllowed = 1;
}

// whether a multiplier update precedes the local solves of grid g (otherwise their
// predecessor is the previous local solve itself, whose results they load)
inline bool has_interfaces(const Grid& g) { return g.NR > 1 || g.NC > 1 || g.cut_top || g.cut_bot; }

// ---- kernels_interface.cu
// lambda += sigma ((2 cur_s - prev_s) - (2 cur_t - prev_t)) on every interface edge.
cudaError_t launch_interface(const Grid& g, float sigma, Strips cur, Strips prev, float* lamh, float* lamv,
                             cudaStream_t st);
// s <- interface values of the torn field (P1, P2), t <- those of (R1, R2)
cudaError_t launch_extract_strips(const Grid& g, const float* P1, const float* P2, Strips s, const float* R1,
                                  const float* R2, Strips t, cudaStream_t st);
// P1/P2 <- 0 except the interface values, taken from the strips
cudaError_t launch_scatter_strips(const Grid& g, Strips s, float* P1, float* P2, cudaStream_t st);

// x <- 2 cur - prev (whole strip sets), the extrapolation of launch_interface; lam2 <- [lamh | lamv]
cudaError_t launch_chain_rebuild(int nh, int nv, const float* cur, const float* prev, float* x, const float* lamh,
                                 const float* lamv, float* lam2, cudaStream_t st);

cudaError_t launch_interface_batch(const BatchIfaceArgs& a, int total4, cudaStream_t st);

// ---- kernels_fused.cu
// All tiles of all images of a batch, one launch (BatchArgs.write_set selects the strips);
// tile: the subdomain side, 128 or 64; variant 2 (128 only): the persistent 2 x 4
// micro-tile kernel instead of the micro-tile kernel of fused_tile.cuh.  overlap: a
// multiplier update precedes it in the stream (the batch has interfaces), so it may start
// early.
cudaError_t launch_fused_batch(const BatchArgs& B, int total_tiles, int tile, int variant, bool overlap,
                               cudaStream_t st);
// One outer iteration's local solves, all tiles, fused (returns cudaErrorInvalidValue
// if no fused configuration fits the tile shape).
cudaError_t launch_fused_local(const LocalArgs& a, int fidelity, int variant, cudaStream_t st);
// Whether the local solves should make the multiplier update themselves (LocalArgs.chain).
bool fused_chains(const Grid& g, int variant, int K, double inner_tol2);
// Sets the shared-memory opt-in of the kernels that launch_fused_local (the batch launch) can
// reach on the current device (called at handle creation, outside any stream capture).
cudaError_t fused_prepare(const Grid& g, int variant, int K, double inner_tol2);
cudaError_t fused_prepare_batch(int tile, int variant);
// Whether launch_fused_local(a, ., variant) with a fixed inner count reads a.u0, a.P10, a.P20
// (rather than working in place on a.u, a.P1, a.P2).
bool fused_out_of_place(const Grid& g, int variant);
// Largest tile (rows, cols) the fused kernel supports.
void fused_max_tile(int* rows, int* cols);
// Number of hardware mappings available for 128 x 128 tiles.
int fused_num_variants();

// ---- kernels_fused_mt.cu
// Persistent fused local solver on 2 x 4 micro-tiles (two columns by four rows per
// thread); 128 x 128 tiles with u, f, P1 16-byte aligned (fused_mt_supported).
bool fused_mt_supported(const LocalArgs& a);
cudaError_t launch_fused_mt(const LocalArgs& a, int fidelity, cudaStream_t st);
cudaError_t fused_mt_prepare();
cudaError_t fused_mt_batch_prepare();
// The same kernel over the work list of a batch (every image's arrays 16-byte aligned).
cudaError_t launch_fused_mt_batch(const BatchArgs& B, int total_tiles, cudaStream_t st);

// ---- kernels_fused_mt4.cu
// Persistent fused local solver on 4 x 4 micro-tiles, one warp per thread row, three
// 128-thread CTAs per SM, the state moved by tensor copies; 128 x 128 tiles with 16-byte
// aligned rows (fused_mt4_supported), in place, fixed inner count or (a.inner_tol2 > 0) the
// adaptive stop.  cudaErrorNotSupported if the tensor maps cannot be encoded.
bool fused_mt4_supported(const LocalArgs& a);
cudaError_t launch_fused_mt4(const LocalArgs& a, int fidelity, cudaStream_t st);
cudaError_t fused_mt4_prepare(bool adaptive);

// ---- kernels_tile8.cu, kernels_tile16.cu, kernels_tile32.cu (fused_tile.cuh)
// How the micro-tile kernels cover the subdomains of a grid: lpr lanes per row group (a
// block 4 lpr columns wide), nw warps per CTA (bands of 4 nw (32 / lpr) rows), cl CTAs per
// subdomain; pad: some subdomain does not fill the block.
struct TilePlan {
  int lpr, nw, cl;
  bool pad;
};
// false if a subdomain is larger than 128 x 128
bool tile_plan(const Grid& g, TilePlan* p);
// words of the reverse pass's tape, per thread and inner iteration
constexpr int kTapeWords = 18;

// Warps of the micro-tile kernel per SM: 16 at 128 registers a thread; 12 where padding and the
// multiplier update come together and spill (321 x 481 15.0 us per outer iteration with 16).
constexpr int tile_warps(int nw, bool pad_chain) { return pad_chain && nw <= 4 ? 12 : 16; }

// launch_tile_<lpr>_<nw>
cudaError_t launch_tile_8_2(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st);
cudaError_t launch_tile_8_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st);
cudaError_t launch_tile_16_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st);
cudaError_t launch_tile_16_8(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st);
cudaError_t launch_tile_32_4(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st);
cudaError_t prepare_tile_8_2(bool pad, bool chain);
cudaError_t prepare_tile_8_4(bool pad, bool chain);
cudaError_t prepare_tile_16_4(bool pad, bool chain);
cudaError_t prepare_tile_16_8(bool pad, bool chain);
cudaError_t prepare_tile_32_4(bool pad, bool chain);
cudaError_t prepare_tile_adapt_128(bool chain);
cudaError_t prepare_tile_batch_128();
cudaError_t prepare_tile_batch_64();
// the adaptive inner stop (a.inner_tol2 > 0), every subdomain exactly 128 x 128
cudaError_t launch_tile_adapt_128(const LocalArgs& a, int fid, cudaStream_t st);
// every subdomain of every image of a batch, 64 x 64 or 128 x 128
cudaError_t launch_tile_batch_128(const BatchArgs& B, int total_tiles, bool overlap, cudaStream_t st);
cudaError_t launch_tile_batch_64(const BatchArgs& B, int total_tiles, bool overlap, cudaStream_t st);

// ---- kernels_full.cu
// n <= full_max_steps() full-dimension iterations in one launch, a.in -> a.out (the dofs of
// the image boundary are 0 and not written)
cudaError_t launch_full(const FullArgs& a, int fidelity, int n, cudaStream_t st);
int full_max_steps();
// shared-memory opt-in of the instances of a fidelity (outside any stream capture)
cudaError_t full_prepare(int fidelity);

// ---- kernels_plain.cu
// phat = p~ -+ tau lambda on the interface sides, pbar = p~; full arrays.
cudaError_t launch_plain_phat(const LocalArgs& a, float* Ph1, float* Ph2, float* Pb1, float* Pb2, cudaStream_t st);
// one u-step over the whole torn field (reads pbar)
cudaError_t launch_plain_ustep(const LocalArgs& a, const float* Pb1, const float* Pb2, const Coef* ck, int fidelity,
                               cudaStream_t st);
// one p-step; phat may be nullptr (no proximal term, full-dimension comparator);
// write_strips: also write the interface strips of the new p.
cudaError_t launch_plain_pstep(const LocalArgs& a, const float* Ph1, const float* Ph2, float* Pb1, float* Pb2,
                               const Coef* ck, bool write_strips, cudaStream_t st);

// ---- kernels_reduce.cu
// out[0] = J(u) = alpha F(u) + TV(u); out[1] = dual value of the averaged torn field
// (P1, P2 nullable: then out[1] is not computed).  partials: scratch of
// reduce_partials_count() doubles; counter: one zeroed unsigned int that the kernel
// leaves zeroed.
cudaError_t launch_energy(const Grid& g, int fidelity, float alpha, float c1, float c2, const float* u,
                          const float* f, const uint8_t* mask, const float* P1, const float* P2, double* partials,
                          unsigned int* counter, double* out, cudaStream_t st);
int reduce_partials_count();
// out[0] = sum_j |a_j - b_j|, j < n (float64, deterministic)
cudaError_t launch_row_tv(const float* a, const float* b, int n, double* out, cudaStream_t st);

// ---- kernels_adjoint.cu
// u-step / p-step of the plain path that also record ubar (H x W) and the projection's
// pass bit of every active dof (M1 (H+NR) x W, M2 H x (W+NC); inactive dofs untouched).
// rt / ct: the row and column tables of AdjArgs.
cudaError_t launch_ustep_tape(const LocalArgs& a, const int4* rt, const int4* ct, const float* Pb1, const float* Pb2,
                              const Coef* ck, int fidelity, float* ubar_out, cudaStream_t st);
cudaError_t launch_pstep_tape(const LocalArgs& a, const int4* rt, const int4* ct, const float* Ph1, const float* Ph2,
                              float* Pb1, float* Pb2, const Coef* ck, uint8_t* M1, uint8_t* M2, cudaStream_t st);
// reverse of one inner iteration (two kernels); first / last as in adj_dof
cudaError_t launch_adj_inner(const AdjArgs& r, const Coef* ck, const float* ubar, const uint8_t* M1,
                             const uint8_t* M2, bool first, bool last, cudaStream_t st);
// reverse of the multiplier update and proximal centre of one outer iteration
cudaError_t launch_adj_interface(const AdjArgs& r, float sigma, float tau, cudaStream_t st);
// Af += du^0/df Au
cudaError_t launch_adj_initial(const AdjArgs& r, cudaStream_t st);
// out[0] = sum of x[0..n) (partials: sum_f64_partials_count() doubles; counter zeroed)
cudaError_t launch_sum_f64(const double* x, long long n, double* partials, unsigned int* counter, double* out,
                           cudaStream_t st);
int sum_f64_partials_count();
// number of float64 partial sums the reverse u-kernel keeps for an image grid
long long adj_alpha_slots(const Grid& g);

// ---- kernels_adjoint_fused.cu, kernels_adj_tile8.cu, kernels_adj_tile16.cu,
// kernels_adj_tile32.cu (adj_tile.cuh)
// Recomputation and reverse of one outer iteration's local solves: a = the local solve's
// arguments (state after the multiplier update, not written), z = the adjoint fields (Au,
// AP1/AP2 in: adjoints of u^{n+1}, p~^{n+1}; out: of u^n and of p~^n through the local
// solve; APh1/APh2 out on the subdomain sides; Af +=; Aal += per (tile, CTA) slot).
cudaError_t launch_adj_fused(const LocalArgs& a, const AdjArgs& z, int fidelity, cudaStream_t st);
// floats of the fused reverse kernel's tape (0 if the tile shape is not supported)
size_t adj_fused_tape_floats(const Grid& g, int K);
// shared-memory opt-in of the fused reverse kernels (outside any stream capture)
cudaError_t adj_fused_prepare(const Grid& g);
// alpha partial-sum slots the fused reverse kernel uses
long long adj_alpha_slots_fused(const Grid& g);
// launch_adj_tile_<lpr>_<nw>
cudaError_t launch_adj_tile_8_2(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st);
cudaError_t launch_adj_tile_8_4(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st);
cudaError_t launch_adj_tile_16_4(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st);
cudaError_t launch_adj_tile_16_8(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st);
cudaError_t launch_adj_tile_32_4(const LocalArgs& a, const AdjArgs& z, int fid, int cl, bool pad, cudaStream_t st);
cudaError_t prepare_adj_tile_8_2();
cudaError_t prepare_adj_tile_8_4();
cudaError_t prepare_adj_tile_16_4();
cudaError_t prepare_adj_tile_16_8();
cudaError_t prepare_adj_tile_32_4();

// ---- kernels_misc.cu
// u0 = f (0 on D) for L2/L1, 1/2 for SEG
cudaError_t launch_init_u(const Grid& g, int fidelity, const float* f, const uint8_t* mask, float* u, cudaStream_t st);
// one bounded mbarrier wait that runs out (nothing completes the phase): sets *err,
// writes the device time it took (ns) to *waited_ns
cudaError_t launch_wait_probe(int* err, unsigned long long* waited_ns, cudaStream_t st);
// global field (H+1) x W / H x (W+1) <-> torn field with a 1 x 1 grid (same arrays)
}  // namespace ddtv
