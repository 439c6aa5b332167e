// Fused local solver with cluster barriers: the adaptive inner stop of every subdomain
// shape but exact 128 x 128, and variant 3 of those; and the choice among the fused
// kernels (launch_fused_local).  A fixed inner count runs the micro-tile kernel of
// fused_tile.cuh or, where use_mt4() says so, the persistent one of kernels_fused_mt4.cu.
//
// All inner iterations of one outer iteration of Algorithm 1 for every subdomain in one
// launch (Section 5, local problem eq. local, solved by the
// accelerated primal-dual algorithm with the dual field p as the uniformly convex
// variable; the projection onto the box C of eq. proj_C is fused into the p-step).
//
// Mapping.  One subdomain (tile of mr x mc pixels, mc <= BW, mr <= CL*TR*R) is owned
// by a thread-block cluster of CL CTAs; CTA `rank` owns a band of TR*R tile rows and
// thread (x, y) of it owns pixel column x and the R consecutive band rows y*R ..
// y*R+R-1 (the 32 lanes of a warp are 32 adjacent columns).  Registers hold, per
// pixel: u, the torn dual dofs p1 (top edge) and p2 (left edge), their proximal
// centres h1, h2 and the extrapolation pbar1.  Shared memory holds what neighbours
// read: u (zero-padded on the left), pbar2 (the tile's right side in column mc),
// f (or g), the first-row pbar1 of every thread row, and two halo rows that the
// neighbouring CTAs of the cluster write through distributed shared memory (u of
// the row above the band, pbar1 of the row below it).  The halo of the tile's top
// row and the padding left of column 0 stay zero, so the interface formulas
// D_s u = +u on the top and left sides need no branch; an inactive side (image
// boundary) is kept at 0 by clamping its dofs to [-0, 0].
//
// Synchronisation per inner iteration: two CTA barriers and two phases of the
// cluster barrier.  In each half-step a CTA first computes the row its neighbour
// needs, stores it into the neighbour's halo, arrives on the cluster barrier, then
// computes its other rows; the matching wait comes a half-step later, so the
// cross-SM latency of the cluster barrier hides behind the interior work.  Only
// warps that wrote to a neighbour arrive with release semantics.
#include "internal.cuh"
#include "fused_common.cuh"

namespace ddtv {

namespace {

template <int BW, int R, int TR>
struct SmemLayout {
  static constexpr int BAND = TR * R;
  static constexpr int US = BW + 1;                    // row stride of u (index 0 = zero pad)
  static constexpr int QS = BW + 1;                    // row stride of pbar2 (index mc = right side)
  static constexpr int U = 0;                          // BAND x US   u of the band
  static constexpr int UH = U + BAND * US;             // US          u of the row above the band
  static constexpr int Q2 = UH + US;                   // BAND x QS   pbar2
  static constexpr int Q1 = Q2 + BAND * QS;            // TR x BW     pbar1 of each thread row's first row
  static constexpr int Q1H = Q1 + TR * BW;             // BW          pbar1 of the row below the band
  static constexpr int F = Q1H + BW;                   // BAND x BW   f (or g)
  static constexpr int PR = F + BAND * BW;             // BAND        right-side p
  static constexpr int HR = PR + BAND;                 // BAND        right-side phat
  static constexpr int FLOATS = HR + BAND;
  static constexpr size_t BYTES = sizeof(float) * FLOATS;
};

// ADAPT: adaptive inner stopping (Section 5, eq. stop_inner1).  Every thread sums
// (p^{k+1} - p^k)^2 and (p^{k+1})^2 over the tile dofs it owns, each warp adds its
// threads' sums (float32, fixed shuffle order), one thread adds the warps' sums in
// float64 in a fixed order and stores the CTA's pair into every cluster CTA's slot
// array through DSMEM, and after one more cluster barrier phase one thread of every
// CTA adds the CL pairs in rank order and shares the decision through shared memory:
// all CTAs of the tile take the same decision.  (Float64 work stays with one thread:
// the float64 pipe of this GPU is narrow.)  The u-step's first cluster wait is then
// taken at the end of the previous iteration's p-step instead.
// The local solve of tile (a, b) of the problem A, its interface strips written to out.
template <int BW, int R, int TR, int CL, int FID, bool MASK, bool ADAPT>
__device__ __forceinline__ void fused_tile(const LocalArgs& A, const Strips out, const int a, const int b) {
  using L = SmemLayout<BW, R, TR>;
  constexpr int BAND = L::BAND;
  extern __shared__ float smem[];
  __shared__ double sRed[2 * CL];            // adaptive stop: per-rank (sum dp^2, sum p^2)
  __shared__ double sWarp[2 * (BW * TR / 32)];
  __shared__ int sStop;                      // adaptive stop: the CTA's decision
  float* sU = smem + L::U;
  float* sUh = smem + L::UH;
  float* sQ2 = smem + L::Q2;
  float* sQ1 = smem + L::Q1;
  float* sQ1h = smem + L::Q1H;
  float* sF = smem + L::F;
  float* sPR = smem + L::PR;
  float* sHR = smem + L::HR;

  const Grid g = A.g;
  const int rank = CL > 1 ? (int)blockIdx.x : 0;
  const int r0 = part_start(a, g.H, g.NR), mr = part_start(a + 1, g.H, g.NR) - r0;
  const int c0 = part_start(b, g.W, g.NC), mc = part_start(b + 1, g.W, g.NC) - c0;
  const bool s_top = a > 0 || g.cut_top, s_bot = a + 1 < g.NR || g.cut_bot, s_lft = b > 0, s_rgt = b + 1 < g.NC;
  const int j = threadIdx.x, ty = threadIdx.y;
  const int lr0 = ty * R;            // first band row of this thread
  const int i0 = rank * BAND + lr0;  // first tile row of this thread
  const bool col_ok = j < mc;
  const int W2 = g.W + g.NC;
  const int gj = c0 + j;
  const float tau = A.tau;
  // clamp limits: 0 keeps an image-boundary dof at 0
  const float lim_left = (j == 0 && !s_lft) ? 0.f : 1.f;
  const float lim_top = (i0 == 0 && !s_top) ? 0.f : 1.f;  // applies to r = 0 only
  const int rb = mr - 1 - i0;                              // r of the tile's last row, if in [0, R)
  // the band's last row is read by the CTA below, its first row by the CTA above
  const bool push_down = CL > 1 && ty == TR - 1 && rank + 1 < CL;
  const bool push_up = CL > 1 && ty == 0 && rank > 0;
  uint32_t remote_uh = 0, remote_q1h = 0;
  if (CL > 1) {
    if (push_down) remote_uh = map_rank(smem_addr(sUh + 1 + j), rank + 1);
    if (push_up) remote_q1h = map_rank(smem_addr(sQ1h + j), rank - 1);
  }

  float u[R], p1[R], p2[R], h1[R], h2[R], q1[R];
  uint32_t in_d = 0;
  float pB = 0.f, hB = 0.f, qB = 0.f;  // bottom side of the tile (thread row holding row mr-1)

  // ---- load the tile's state and build the proximal centre
  // The tile's first row sees u = 0 above it.  The other CTAs' halos are written by
  // their neighbours before every read; sQ1h is only read by rows that either have a
  // neighbour below or lie outside the tile (their values are never stored).
  if (rank == 0) {
    if (j == 0) sUh[0] = 0.f;
    sUh[1 + j] = 0.f;
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = i0 + r;
    float uv = 0.f, fv = 0.f, a1 = 0.f, a2 = 0.f, b1 = 0.f, b2 = 0.f;
    if (col_ok && i < mr) {
      const int gi = r0 + i;
      const size_t px = (size_t)gi * g.W + gj;
      uv = A.u[px];
      fv = A.f[px];
      if (FID == FID_SEG) fv = (fv - A.c1) * (fv - A.c1) - (fv - A.c2) * (fv - A.c2);
      if (MASK && A.mask[px]) in_d |= 1u << r;
      a1 = A.P1[(size_t)(gi + a) * g.W + gj];
      a2 = A.P2[(size_t)gi * W2 + gj + b];
      b1 = (i == 0 && s_top) ? phat_t(a1, A.lamh[(ptrdiff_t)(a - 1) * g.W + gj], tau) : a1;
      b2 = (j == 0 && s_lft) ? phat_t(a2, A.lamv[(size_t)(b - 1) * g.H + gi], tau) : a2;
      if (i == mr - 1 && s_bot) {
        pB = A.P1[(size_t)(gi + a + 1) * g.W + gj];
        hB = phat_s(pB, A.lamh[(size_t)a * g.W + gj], tau);
      }
      if (j == mc - 1) {
        float pr = 0.f, hr = 0.f;
        if (s_rgt) {
          pr = A.P2[(size_t)gi * W2 + gj + b + 1];
          hr = phat_s(pr, A.lamv[(size_t)b * g.H + gi], tau);
        }
        sPR[lr0 + r] = pr;
        sHR[lr0 + r] = hr;
        sQ2[(lr0 + r) * L::QS + mc] = pr;
      }
    }
    u[r] = uv;
    p1[r] = a1;
    p2[r] = a2;
    h1[r] = b1;
    h2[r] = b2;
    q1[r] = a1;
    sF[(lr0 + r) * BW + j] = fv;
    sU[(lr0 + r) * L::US] = 0.f;  // left padding (every thread writes the same value)
    if (col_ok) sQ2[(lr0 + r) * L::QS + j] = a2;
  }
  qB = pB;
  sQ1[ty * BW + j] = q1[0];
  if (push_up) st_cluster(remote_q1h, q1[0]);
  __syncthreads();
  if (CL > 1) {
    if (push_up) cluster_arrive<true>(); else cluster_arrive<false>();
  }

  const float4* coef4 = reinterpret_cast<const float4*>(A.coef);

  auto u_px = [&](int r, const Coef& c) {
    const int lr = lr0 + r;
    float below;
    if (r == rb) below = qB;                                 // the tile's bottom side
    else if (r + 1 < R) below = q1[r + 1];
    else if (ty + 1 < TR) below = sQ1[(ty + 1) * BW + j];
    else below = sQ1h[j];                                    // first row of the band below
    const float left = sQ2[lr * L::QS + j];
    const float right = sQ2[lr * L::QS + j + 1];
    const float d = div_px(q1[r], below, left, right);
    u[r] = u_update<FID>(u[r], d, sF[lr * BW + j], MASK && ((in_d >> r) & 1u), c);
    sU[lr * L::US + j + 1] = u[r];
  };

  float sd = 0.f, sp = 0.f;  // adaptive stop: this thread's sums over its tile dofs
  auto res_add = [&](float po, float pn) {
    const float dp = pn - po;
    sd = fmaf(dp, dp, sd);
    sp = fmaf(pn, pn, sp);
  };

  auto p_px = [&](int r, const Coef& c) {
    const int lr = lr0 + r;
    const bool in_tile = ADAPT && col_ok && i0 + r < mr;
    float above;
    if (r > 0) above = u[r - 1];
    else if (ty > 0) above = sU[(lr - 1) * L::US + j + 1];
    else above = sUh[j + 1];                                 // 0 above the tile's first row
    const float o1 = p1[r], o2 = p2[r];
    p_update_lim(p1[r], q1[r], u[r] - above, h1[r], c, r == 0 ? lim_top : 1.f);
    float q2;
    p_update_lim(p2[r], q2, u[r] - sU[lr * L::US + j], h2[r], c, lim_left);
    if (in_tile) {
      res_add(o1, p1[r]);
      res_add(o2, p2[r]);
    }
    if (r == rb && s_bot) {
      const float oB = pB;
      p_update(pB, qB, -u[r], hB, c);
      if (in_tile) res_add(oB, pB);
    }
    if (j == mc - 1 && s_rgt) {
      float pr = sPR[lr], qr;
      const float orr = pr;
      p_update(pr, qr, -u[r], sHR[lr], c);
      if (in_tile) res_add(orr, pr);
      sPR[lr] = pr;
      sQ2[lr * L::QS + mc] = qr;
    }
    if (col_ok) sQ2[lr * L::QS + j] = q2;
  };

  // ---- inner iterations
  int k_run = A.K;
  for (int k = 0; k < A.K; ++k) {
    const float4 ca = __ldg(coef4 + 2 * k), cb = __ldg(coef4 + 2 * k + 1);
    const Coef c{ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
    // u-step: the band's last row first (the CTA below needs it)
    if (CL > 1 && (!ADAPT || k == 0)) cluster_wait();
    u_px(R - 1, c);
    if (push_down) st_cluster(remote_uh, u[R - 1]);
    if (CL > 1) {
      if (push_down) cluster_arrive<true>(); else cluster_arrive<false>();
    }
#pragma unroll
    for (int r = 0; r + 1 < R; ++r) u_px(r, c);
    __syncthreads();
    // p-step: the band's first row first (the CTA above needs its pbar1)
    if (CL > 1) cluster_wait();
    p_px(0, c);
    sQ1[ty * BW + j] = q1[0];
    if (push_up) st_cluster(remote_q1h, q1[0]);
    if (CL > 1) {
      if (push_up) cluster_arrive<true>(); else cluster_arrive<false>();
    }
#pragma unroll
    for (int r = 1; r < R; ++r) p_px(r, c);
    __syncthreads();
    if (ADAPT) {
      // warp sums in float32 (fixed shuffle order), then one thread adds the warps' sums in
      // order in float64
      const int tid = ty * BW + j, lane = tid & 31, wid = tid >> 5;
      float wd = sd, wp = sp;
      sd = sp = 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        wd += __shfl_down_sync(0xffffffffu, wd, o);
        wp += __shfl_down_sync(0xffffffffu, wp, o);
      }
      if (lane == 0) {
        sWarp[2 * wid] = wd;
        sWarp[2 * wid + 1] = wp;
      }
      __syncthreads();
      if (CL > 1) cluster_wait();  // the p-step's cluster phase (halo rows of pbar1)
      if (tid == 0) {
        double td = 0.0, tp = 0.0;
        for (int w = 0; w < BW * TR / 32; ++w) {
          td += sWarp[2 * w];
          tp += sWarp[2 * w + 1];
        }
        if (CL > 1) {
          for (int q = 0; q < CL; ++q) {
            st_cluster_f64(map_rank(smem_addr(sRed + 2 * rank), q), td);
            st_cluster_f64(map_rank(smem_addr(sRed + 2 * rank + 1), q), tp);
          }
        } else {
          sRed[0] = td;
          sRed[1] = tp;
        }
      }
      if (CL > 1) {
        cluster_arrive<true>();
        cluster_wait();
      } else {
        __syncthreads();
      }
      if (tid == 0) {
        double td = 0.0, tp = 0.0;
        for (int q = 0; q < CL; ++q) {
          td += sRed[2 * q];
          tp += sRed[2 * q + 1];
        }
        sStop = (tp == 0.0 || td < A.inner_tol2 * tp) ? 1 : 0;
      }
      __syncthreads();
      if (sStop) {
        k_run = k + 1;
        break;
      }
    }
  }
  if (CL > 1 && !ADAPT) cluster_wait();  // no CTA leaves while a neighbour may still write its halo
  if (ADAPT && rank == 0 && j == 0 && ty == 0) {
    A.inner_used[a * g.NC + b] = k_run;
    atomicMax(A.inner_max, k_run);
    atomicAdd(A.inner_work, (unsigned long long)mr * (unsigned long long)mc * (unsigned long long)k_run);
  }

  // ---- store u^{n+1}, p~^{n+1} and the interface strips
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = i0 + r;
    if (col_ok && i < mr) {
      const int gi = r0 + i;
      A.u[(size_t)gi * g.W + gj] = u[r];
      A.P1[(size_t)(gi + a) * g.W + gj] = p1[r];
      A.P2[(size_t)gi * W2 + gj + b] = p2[r];
      if (i == 0 && s_top) out.ST[(ptrdiff_t)(a - 1) * g.W + gj] = p1[r];
      if (j == 0 && s_lft) out.SL[(size_t)(b - 1) * g.H + gi] = p2[r];
      if (i == mr - 1 && s_bot) {
        A.P1[(size_t)(gi + a + 1) * g.W + gj] = pB;
        out.SB[(size_t)a * g.W + gj] = pB;
      }
      if (j == mc - 1 && s_rgt) {
        const float pr = sPR[lr0 + r];
        A.P2[(size_t)gi * W2 + gj + b + 1] = pr;
        out.SR[(size_t)b * g.H + gi] = pr;
      }
    }
  }
}


template <int BW, int R, int TR, int CL, int FID, bool MASK, bool ADAPT>
__global__ void __launch_bounds__(BW* TR, (BW * TR <= 256 ? 2 : 1)) k_fused(const LocalArgs A) {
  fused_tile<BW, R, TR, CL, FID, MASK, ADAPT>(A, A.out, (int)blockIdx.z, (int)blockIdx.y);
}

// Hardware mappings of exact 128 x 128 subdomains (dd_tv_params.variant):
//   0  the micro-tile kernel of every other shape (fused_tile.cuh), or 1 where that is faster
//   1  persistent 4 x 4 micro-tiles, state moved by tensor copies
//   2  persistent 2 x 4 micro-tiles, 256 threads, 2 CTAs per SM
//   3  the cluster-barrier kernel (one subdomain per cluster)
constexpr int kNumVariants = 4;

template <int BW, int R, int TR, int CL, int FID, bool MASK, bool ADAPT>
cudaError_t launch_one(const LocalArgs& a, cudaStream_t st) {
  using L = SmemLayout<BW, R, TR>;
  // configurations above 48 KB of shared memory need the opt-in attribute, set by
  // fused_prepare() when the handle is created (never during graph capture)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL, a.g.NC, a.g.NR);
  cfg.blockDim = dim3(BW, TR, 1);
  cfg.dynamicSmemBytes = L::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_fused<BW, R, TR, CL, FID, MASK, ADAPT>, a);
}

template <int BW, int R, int TR, int CL, bool ADAPT>
cudaError_t launch_fid(const LocalArgs& a, int fid, cudaStream_t st) {
  const bool m = a.mask != nullptr;
  switch (fid) {
    case FID_L2:
      return m ? launch_one<BW, R, TR, CL, FID_L2, true, ADAPT>(a, st)
               : launch_one<BW, R, TR, CL, FID_L2, false, ADAPT>(a, st);
    case FID_L1:
      return m ? launch_one<BW, R, TR, CL, FID_L1, true, ADAPT>(a, st)
               : launch_one<BW, R, TR, CL, FID_L1, false, ADAPT>(a, st);
    default: return launch_one<BW, R, TR, CL, FID_SEG, false, ADAPT>(a, st);
  }
}

template <int BW, int R, int TR, int CL, int FID, bool MASK, bool ADAPT>
cudaError_t prepare_one() {
  return cudaFuncSetAttribute(k_fused<BW, R, TR, CL, FID, MASK, ADAPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)SmemLayout<BW, R, TR>::BYTES);
}

template <int BW, int R, int TR, int CL, bool ADAPT>
cudaError_t prepare_fid() {
  cudaError_t e;
  if ((e = prepare_one<BW, R, TR, CL, FID_L2, false, ADAPT>()) != cudaSuccess) return e;
  if ((e = prepare_one<BW, R, TR, CL, FID_L2, true, ADAPT>()) != cudaSuccess) return e;
  if ((e = prepare_one<BW, R, TR, CL, FID_L1, false, ADAPT>()) != cudaSuccess) return e;
  if ((e = prepare_one<BW, R, TR, CL, FID_L1, true, ADAPT>()) != cudaSuccess) return e;
  return prepare_one<BW, R, TR, CL, FID_SEG, false, ADAPT>();
}

// The micro-tile kernel (fused_tile.cuh), fixed inner count.
cudaError_t launch_tile_shape(const LocalArgs& a, int fid, cudaStream_t st) {
  TilePlan p;
  if (!tile_plan(a.g, &p)) return cudaErrorInvalidValue;
  if (p.lpr == 8) return p.nw == 2 ? launch_tile_8_2(a, fid, p.cl, p.pad, st) : launch_tile_8_4(a, fid, p.cl, p.pad, st);
  if (p.lpr == 16)
    return p.nw == 8 ? launch_tile_16_8(a, fid, p.cl, p.pad, st) : launch_tile_16_4(a, fid, p.cl, p.pad, st);
  return launch_tile_32_4(a, fid, p.cl, p.pad, st);
}

// size class of the cluster-barrier kernel for a tile shape (up to 32 x 32, 64 x 64 and
// 128 x 128), -1 if none fits
int pick(int mr, int mc) {
  if (mc <= 32 && mr <= 32) return 0;
  if (mc <= 64 && mr <= 64) return 1;
  if (mc <= 128 && mr <= 128) return 2;
  return -1;
}

}  // namespace

// Columns choose the lanes of a row group (a subdomain of mc
// columns in a block of 32, 64 or 128), rows the warps of a CTA and the CTAs of a
// cluster.  Up to 32 x 32 and 64 x 64 one CTA holds the subdomain: no halo leaves the
// SM.  In a cluster of two 32-row CTAs, 64 x 64 subdomains take 256 us per outer
// iteration of 10 inner ones at 4096^2 and 14.1 us at 128^2, in one CTA 217 and 13.0.
// 128 columns run 16-row CTAs in clusters of up to 8: with 32 rows in 8 warps and
// clusters of 4, 4096^2 takes 233 us instead of 215, and 120 x 128 subdomains (2160 x
// 3840) 146 instead of 137.
bool tile_plan(const Grid& g, TilePlan* p) {
  const int mr = (g.H + g.NR - 1) / g.NR, mc = (g.W + g.NC - 1) / g.NC;  // the largest subdomain
  if (mr > 128 || mc > 128) return false;
  p->lpr = mc <= 32 ? 8 : (mc <= 64 ? 16 : 32);
  p->nw = p->lpr == 8 && mr <= 32 ? 2 : (p->lpr == 16 && mr > 32 && mr <= 64 ? 8 : 4);
  const int bw = 4 * p->lpr, band = 4 * p->nw * (32 / p->lpr);
  p->cl = (mr + band - 1) / band;
  p->pad = g.W != bw * g.NC || g.H != p->cl * band * g.NR;
  return true;
}

void fused_max_tile(int* rows, int* cols) {
  *rows = 128;
  *cols = 128;
}

int fused_num_variants() { return kNumVariants; }

namespace {

bool exact_128(const Grid& g) { return g.H == 128 * g.NR && g.W == 128 * g.NC; }

// Whether one wave holds a launch of the micro-tile kernel (on the 148 SMs that take
// clusters).
bool one_wave(const Grid& g, const TilePlan& p) {
  return (long long)g.NR * g.NC * p.cl * p.nw <= 148 * tile_warps(p.nw, p.pad);
}

// The persistent 4 x 4 kernel: variant 1, and the default of launches of several waves with
// few inner iterations.  It has the next subdomain's loads on their way while this one
// iterates, where a CTA of the micro-tile kernel waits for its own; with four CTAs per SM
// instead of three that one iterates faster.  us per outer iteration, persistent / micro-tile:
//
//   state beyond L2     K = 1        2           3            4            10
//   4096 x 4096     80 / 94    93 / 108   111 / 118    127 / 130    231 / 217
//   2560 x 2560     35 / 40    42 / 46     49 / 50      55 / 56
//   ... with a mask 40 / 44    47 / 50     54 / 54      62 / 59
//   state in L2
//   2048 x 2048     22.6 / 24.2  27.2 / 28.4  31.8 / 31.2  35.9 / 35.4
//   ... with a mask 24.4 / 24.7  29.4 / 28.3  34.3 / 32.9
//
// The adaptive stop runs few inner iterations where the tolerance is loose (400 outer
// iterations of at most 10; of them all but the first end after one): 4096 x 4096 1e-3 130 /
// 161, 1e-4 173 / 194, 3e-5 220 / 231, 1e-5 277 / 276, 1e-6 345 / 331; with a mask 1e-4
// 210 / 216, 3e-5 293 / 283; 2048 x 2048 1e-3 37 / 36, 1e-4 48 / 46.
bool use_mt4(const Grid& g, int variant, int K, double inner_tol2, bool masked) {
  TilePlan p;
  if (!exact_128(g) || K > 64 || (g.W + g.NC) % 4 != 0 || !tile_plan(g, &p)) return false;
  if (variant == 1) return inner_tol2 == 0.0;
  if (variant != 0 || one_wave(g, p)) return false;
  // u, f, p1 and p2, read by every launch (67 MB at 2048 x 2048, 105 MB at 2560 x 2560)
  const bool beyond_l2 = 16ll * g.H * g.W > 96ll << 20;
  if (inner_tol2 > 0.0) return beyond_l2 && inner_tol2 >= 2e-5 * 2e-5;
  return K < (beyond_l2 ? (masked ? 3 : 5) : (masked ? 0 : 3));
}

// The adaptive stop in one of the micro-tile kernels: the default of exact 128 x 128
// subdomains.  (W + N_c a multiple of 4 and K <= 64 are no needs of fused_tile.cuh, but its
// residual sums are float32 where those of the cluster-barrier kernel are float64, so a near
// tie could stop a subdomain one iteration apart: every problem keeps the sums it has always
// had.)
bool adapt_in_tile(const Grid& g, int variant, int K) {
  return exact_128(g) && variant == 0 && K <= 64 && (g.W + g.NC) % 4 == 0;
}

}  // namespace

// In the micro-tile kernel and where one wave holds the launch.  The update then saves a
// launch on the chain of latencies: 128 x 128 in 64 x 64 11.4 -> 10.9 us per outer iteration,
// 512 x 512 in 128 x 128 12.7 -> 11.9, 1024 x 1024 18.6 -> 18.1.  With several waves the update of
// the sides costs more instructions than its own launch, which overlaps with the loads: 4096
// x 4096 216 -> 224.
bool fused_chains(const Grid& g, int variant, int K, double inner_tol2) {
  TilePlan p;
  if (!tile_plan(g, &p) || !one_wave(g, p)) return false;
  return inner_tol2 > 0.0 ? adapt_in_tile(g, variant, K) : variant == 0 || !exact_128(g);
}

// Every handle prepares the kernels it can reach and no others: an attribute call per
// kernel instance is most of what creating a small handle costs.
cudaError_t fused_prepare(const Grid& g, int variant, int K, double inner_tol2) {
  TilePlan p;
  if (!tile_plan(g, &p)) return cudaErrorInvalidValue;
  const bool exact128 = exact_128(g), chain = fused_chains(g, variant, K, inner_tol2);
  const bool adaptive = inner_tol2 > 0.0;
  cudaError_t e = cudaSuccess;
  // (whatever a later load brings: without a mask the persistent kernel is taken wherever it
  // is with one)
  if (use_mt4(g, variant, K, inner_tol2, false) && (e = fused_mt4_prepare(adaptive)) != cudaSuccess) return e;
  if (adaptive) {
    if (adapt_in_tile(g, variant, K)) return prepare_tile_adapt_128(chain);
    switch (pick((g.H + g.NR - 1) / g.NR, (g.W + g.NC - 1) / g.NC)) {
      case 0: return prepare_fid<32, 8, 4, 1, true>();
      case 1: return prepare_fid<64, 8, 8, 1, true>();
      default: return prepare_fid<128, 8, 2, 8, true>();
    }
  }
  if (exact128 && variant == 3) return prepare_fid<128, 8, 2, 8, false>();
  if (exact128 && variant == 2 && (e = fused_mt_prepare()) != cudaSuccess) return e;
  if (p.lpr == 8) return p.nw == 2 ? prepare_tile_8_2(p.pad, chain) : prepare_tile_8_4(p.pad, chain);
  if (p.lpr == 16) return p.nw == 8 ? prepare_tile_16_8(p.pad, chain) : prepare_tile_16_4(p.pad, chain);
  return prepare_tile_32_4(p.pad, chain);
}

cudaError_t fused_prepare_batch(int tile, int variant) {
  if (tile == 64) return prepare_tile_batch_64();
  return variant == 2 ? fused_mt_batch_prepare() : prepare_tile_batch_128();
}

cudaError_t launch_fused_batch(const BatchArgs& B, int total_tiles, int tile, int variant, bool overlap,
                               cudaStream_t st) {
  if (tile == 128)
    return variant == 2 ? launch_fused_mt_batch(B, total_tiles, st) : launch_tile_batch_128(B, total_tiles, overlap, st);
  return tile == 64 ? launch_tile_batch_64(B, total_tiles, overlap, st) : cudaErrorInvalidValue;
}

bool fused_out_of_place(const Grid& g, int variant) {  // in the micro-tile kernel
  return variant <= 1 || !exact_128(g);
}

cudaError_t launch_fused_local(const LocalArgs& a, int fid, int variant, cudaStream_t st) {
  // largest tile of the (ragged) partition
  const int mr = (a.g.H + a.g.NR - 1) / a.g.NR, mc = (a.g.W + a.g.NC - 1) / a.g.NC;
  const bool exact128 = exact_128(a.g);  // every tile exactly 128 x 128
  // (only the micro-tile kernel works out of place)
  if (a.u0 == a.u && use_mt4(a.g, variant, a.K, a.inner_tol2, a.mask != nullptr) && fused_mt4_supported(a)) {
    const cudaError_t e = launch_fused_mt4(a, fid, st);
    if (e != cudaErrorNotSupported) return e;
  }
  if (a.inner_tol2 > 0.0) {
    if (adapt_in_tile(a.g, variant, a.K)) return launch_tile_adapt_128(a, fid, st);
    switch (pick(mr, mc)) {
      case 0: return launch_fid<32, 8, 4, 1, true>(a, fid, st);
      case 1: return launch_fid<64, 8, 8, 1, true>(a, fid, st);
      case 2: return launch_fid<128, 8, 2, 8, true>(a, fid, st);
      default: return cudaErrorInvalidValue;
    }
  }
  if (exact128) {
    if (variant == 2 && fused_mt_supported(a)) return launch_fused_mt(a, fid, st);
    if (variant == 3) return launch_fid<128, 8, 2, 8, false>(a, fid, st);
  }
  return launch_tile_shape(a, fid, st);
}

}  // namespace ddtv
