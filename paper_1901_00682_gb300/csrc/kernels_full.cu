// Full-dimension primal-dual iteration (N = 1, the comparator of Section 5), several
// iterations per launch.
//
// One global-memory kernel per half-step streams the whole state through memory at every
// iteration (56 bytes per pixel).  Here a cluster of CTAs holds a block of up to 128 x 128
// pixels on chip, as the micro-tile kernel holds a subdomain (fused_tile.cuh: 4 x 4 pixels
// per thread, packed row pairs, 16-row bands, halo rows by st.async), and runs n
// iterations on it before it writes back.  Blocks overlap: an iteration carries wrong values one row
// and column further in from an edge that is not the image's (p of the first row misses u
// above it, u of the last row the new pbar below it), so after n iterations everything at
// least n rows and columns inside is what the whole image gives, bit for bit, and only that
// is stored.  The launch reads one set of arrays and writes the other, so no block sees
// another's results.
//
// What bounds it: as the local solve, latency and issue slots of the inner loop, times the
// overlap (128 x 128 pixels computed for 108 x 108, or 104, stored at n = 10), and per launch 24 bytes
// read and 20 written per pixel of a block.  n is at most 10: twice as many leave less than
// half of a block to store.  Measured per 10 iterations, before (two launches per iteration)
// and after: 1001 x 1503 218 -> 43 us, 4096 x 4096 2474 -> 306, with a mask 2607 -> 350 (394 with
// a byte load per pixel of the mask); one iteration of 1024 x 1024 17.5 -> 14.4, with a mask 17.5 ->
// 15.7 (17.9 with byte loads), of unaligned rows dd_tv.cu full_half_steps.
#include "fused_tile.cuh"

namespace ddtv {

namespace {

using FL = TileLayout<32, 4>;
constexpr int kBlockSide = FL::BW;

// Blocks along an axis of len pixels: m of them, block q covering [start, start + 128) (or
// the whole axis), storing [from, to).  Starts and bounds are multiples of `al` (4 for the
// columns of an image whose rows are 16-byte aligned, else 1), but for the last start.
struct Axis {
  int len, m, halo, al;
  __host__ __device__ int start(int q) const {
    const int T = (len - kBlockSide + al - 1) / al;
    const int s = m > 1 ? al * (int)((long long)q * T / (m - 1)) : 0;
    return q > 0 && q == m - 1 ? len - kBlockSide : s;
  }
  __host__ __device__ int size() const { return len < kBlockSide ? len : kBlockSide; }
  __host__ __device__ int from(int q) const { return q > 0 ? start(q) + halo : 0; }
  __host__ __device__ int to(int q) const { return q + 1 < m ? start(q + 1) + halo : len; }
};

// n iterations: every interior bound at least n pixels inside both blocks it separates
Axis axis_for(int len, int n, int al) {
  Axis a;
  a.len = len;
  a.al = al;
  a.halo = (n + al - 1) / al * al;
  const int gap = (kBlockSide - a.halo - n) / al;  // largest distance of two starts, in units of al
  a.m = len <= kBlockSide ? 1 : 1 + ((len - kBlockSide + al - 1) / al + gap - 1) / gap;
  return a;
}

template <int FID, bool MASK>
__global__ void __launch_bounds__(FL::NT, 4) k_full(const FullArgs A, const Axis ar, const Axis ac, const int n) {
  constexpr int LPR = FL::LPR, NG = FL::NG, BAND = FL::BAND, BW = FL::BW, NT = FL::NT;
  extern __shared__ __align__(128) float smem[];
  float* sUB = smem + FL::UB;
  float* sQ1 = smem + FL::Q1;
  const uint32_t mbU = smem_addr(smem + FL::MB), mbQ = mbU + 8;
  // a 1-D grid: CTA x % CL of block x / CL, row by row
  const int CL = (ar.size() + BAND - 1) / BAND, rank = (int)(blockIdx.x % (unsigned)CL);
  const int by = (int)(blockIdx.x / (unsigned)CL) / ac.m, bx = (int)(blockIdx.x / (unsigned)CL) - by * ac.m;
  const int W = A.W, W2 = A.W + 1;
  const int c0 = ac.start(bx), mc = ac.size(), r0 = ar.start(by), mr = ar.size();
  const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
  const int j0 = 4 * l, i0 = rank * BAND + 4 * w;
  const bool push_down = w == NG - 1 && rank + 1 < CL, push_up = w == 0 && rank > 0;
  constexpr uint32_t kHaloBytes = 4 * BW;
  float* const myUR = smem + FL::UR + w * FL::SLOT + 4 * (l + 1);
  float* const myQL = smem + FL::QL + w * FL::SLOT + 4 * l;
  float* const myF = smem + FL::F + 4 * tid;
  uint32_t remote_u = 0, remote_q1 = 0, remote_mbU = 0, remote_mbQ = 0;
  if (push_down) {
    remote_u = map_rank(smem_addr(sUB + j0), rank + 1);
    remote_mbU = map_rank(mbU, rank + 1);
  }
  if (push_up) {
    remote_q1 = map_rank(smem_addr(sQ1 + NG * BW + j0), rank - 1);
    remote_mbQ = map_rank(mbQ, rank - 1);
  }
  if (tid == 0) {
    mbar_init(mbU, 1);
    mbar_init(mbQ, 1);
    if (rank > 0) mbar_arrive_expect_tx(mbU, kHaloBytes);
    if (rank + 1 < CL) mbar_arrive_expect_tx(mbQ, kHaloBytes);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  cluster_arrive<true>();  // matched before the first halo is sent: the loads hide the wait
  pdl_trigger();
  pdl_wait();  // the launch before, whose results this one reads

  // clamp limits: 0 on the image boundary
  float lim1[4], lim2[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int gi = r0 + i0 + q, gj = c0 + j0 + q;
    lim1[q] = gi <= 0 || gi >= A.H ? 0.f : 1.f;
    lim2[q] = gj <= 0 || gj >= W ? 0.f : 1.f;
  }
  const Coef co = *A.coef;
  const f32x2 SIG = pk2(co.sig, co.sig), UA = pk2(co.ua, co.ua), UBc = pk2(co.ub, co.ub), PC = pk2(co.pc, co.pc);

  // pairs [column c][e]: rows (e, e + 2) of column j0 + c
  f32x2 U[4][2], P1[4][2], P2[4][2], Q1[4][2], Q2[4][2];
  uint32_t in_d = 0;
  {
    const bool vec = (W & 3) == 0 && (c0 & 3) == 0;
    // the lane's 4 x 4 pixels of every array, all loads in flight before the first is used
    float x[6][4][4];
    const float* const base[6] = {A.f, A.in.u, A.in.P1, A.in.Pb1, A.in.P2, A.in.Pb2};
    const size_t o1 = (size_t)(r0 + i0) * W + c0 + j0, o2 = (size_t)(r0 + i0) * W2 + c0 + j0;
    if (vec && i0 + 3 < mr && j0 + 3 < mc) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int q = 0; q < 4; ++q) load4(base[q] + o1 + (size_t)r * W, x[q][r]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          x[4][r][c] = base[4][o2 + (size_t)r * W2 + c];
          x[5][r][c] = base[5][o2 + (size_t)r * W2 + c];
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int n = i0 + r < mr ? mc - j0 : 0;
#pragma unroll
        for (int q = 0; q < 6; ++q)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            x[q][r][c] = c < n ? base[q][(q < 4 ? o1 + (size_t)r * W : o2 + (size_t)r * W2) + c] : 0.f;
      }
    }
    float qb[4] = {0.f, 0.f, 0.f, 0.f};  // pbar1 of the row below the band (0 below the image)
    if (w == NG - 1) load4(A.in.Pb1 + (size_t)(r0 + i0 + 4) * W + c0 + j0, r0 + i0 + 4 < A.H ? mc - j0 : 0, vec, qb);
    float qr = 0.f;  // pbar2 right of the block (0 right of the image), in the pair order of the slots: rows 0, 2, 1, 3
    const int ro = (l >> 1) + 2 * (l & 1);
    if (l < 4 && mc == BW && c0 + BW < W && i0 + ro < mr) qr = A.in.Pb2[(size_t)(r0 + i0 + ro) * W2 + c0 + BW];
    f32x2 FV[4][2];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        FV[c][e] = pk2(x[0][e][c], x[0][e + 2][c]);
        U[c][e] = pk2(x[1][e][c], x[1][e + 2][c]);
        P1[c][e] = pk2(x[2][e][c], x[2][e + 2][c]);
        Q1[c][e] = pk2(x[3][e][c], x[3][e + 2][c]);
        P2[c][e] = pk2(x[4][e][c], x[4][e + 2][c]);
        Q2[c][e] = pk2(x[5][e][c], x[5][e + 2][c]);
      }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (FID == FID_SEG) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float a = lo2(FV[c][e]), b = hi2(FV[c][e]);
          FV[c][e] = pk2((a - A.c1) * (a - A.c1) - (a - A.c2) * (a - A.c2),
                         (b - A.c1) * (b - A.c1) - (b - A.c2) * (b - A.c2));
        }
      }
      *reinterpret_cast<ulonglong2*>(myF + 4 * NT * c) = make_ulonglong2(FV[c][0], FV[c][1]);
    }
    if (MASK) {  // a word per row where the rows are aligned
      if (vec && i0 + 3 < mr && j0 + 3 < mc) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const uint32_t m = *reinterpret_cast<const uint32_t*>(A.mask + o1 + (size_t)r * W);
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if ((m >> (8 * c)) & 0xffu) in_d |= 1u << (4 * c + r);
        }
      } else {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (i0 + r < mr && j0 + c < mc && A.mask[o1 + (size_t)r * W + c]) in_d |= 1u << (4 * c + r);
      }
    }
    *reinterpret_cast<float4*>(sQ1 + w * BW + j0) = make_float4(lo2(Q1[0][0]), lo2(Q1[1][0]), lo2(Q1[2][0]), lo2(Q1[3][0]));
    *reinterpret_cast<ulonglong2*>(myQL) = make_ulonglong2(Q2[0][0], Q2[0][1]);
    if (w == NG - 1) *reinterpret_cast<float4*>(sQ1 + NG * BW + j0) = make_float4(qb[0], qb[1], qb[2], qb[3]);
    if (w == 0 && rank == 0) *reinterpret_cast<float4*>(sUB + j0) = make_float4(0.f, 0.f, 0.f, 0.f);
    if (l == 0) *reinterpret_cast<float4*>(smem + FL::UR + w * FL::SLOT) = make_float4(0.f, 0.f, 0.f, 0.f);
    if (l < 4) smem[FL::QL + w * FL::SLOT + 4 * LPR + l] = qr;
  }
  __syncthreads();
  bool timed_out = false;
  uint32_t phU = 0, phQ = 0;
  cluster_wait();
  auto wait_u = [&]() {
    if (!mbar_wait(mbU, phU & 1)) timed_out = true;
    ++phU;
    if (l == 0) mbar_arrive_expect_tx(mbU, kHaloBytes);  // arm the next phase
  };
  auto wait_q = [&]() {
    if (!mbar_wait(mbQ, phQ & 1)) timed_out = true;
    ++phQ;
    if (l == 0) mbar_arrive_expect_tx(mbQ, kHaloBytes);
  };

#pragma unroll 2
  for (int k = 0; k < n; ++k) {
    if (push_down && k > 0) wait_q();
    // ---- u-step
    {
      const float4 qb = *reinterpret_cast<const float4*>(sQ1 + (w + 1) * BW + j0);
      const ulonglong2 qn = *reinterpret_cast<const ulonglong2*>(myQL + 4);
      const f32x2 QRn[2] = {qn.x, qn.y};
      const float qbv[4] = {qb.x, qb.y, qb.z, qb.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const ulonglong2 fc = *reinterpret_cast<const ulonglong2*>(myF + 4 * NT * c);
#pragma unroll
        for (int ee = 0; ee < 2; ++ee) {
          const int e = 1 - ee;
          const f32x2 fg = e == 0 ? fc.x : fc.y;
          const f32x2 bt = e == 0 ? sub2(Q1[c][1], Q1[c][0])
                                  : pk2(hi2(Q1[c][0]) - lo2(Q1[c][1]), qbv[c] - hi2(Q1[c][1]));
          const f32x2 right = c < 3 ? Q2[c + 1][e] : QRn[e];
          const f32x2 d = sub2(add2(bt, right), Q2[c][e]);  // div_px
          const f32x2 ub = fma2(SIG, d, U[c][e]);
          const bool dl = MASK && ((in_d >> (4 * c + e)) & 1u), dh = MASK && ((in_d >> (4 * c + e + 2)) & 1u);
          f32x2 un;
          if (FID == FID_L2) {
            un = fma2(UBc, fg, mul2(UA, ub));
            if (MASK) un = pk2(dl ? lo2(ub) : lo2(un), dh ? hi2(ub) : hi2(un));
          } else if (FID == FID_L1) {
            const f32x2 v = sub2(ub, fg);
            un = sub2(ub, pk2(clamp_abs(lo2(v), co.s), clamp_abs(hi2(v), co.s)));
            if (MASK) un = pk2(dl ? lo2(ub) : lo2(un), dh ? hi2(ub) : hi2(un));
          } else {
            un = pk2(prox_ubar<FID>(lo2(ub), lo2(fg), dl, co), prox_ubar<FID>(hi2(ub), hi2(fg), dh, co));
          }
          U[c][e] = un;
        }
      }
      const float4 ul = make_float4(hi2(U[0][1]), hi2(U[1][1]), hi2(U[2][1]), hi2(U[3][1]));
      if (push_down) st_async_v4_f32(remote_u, ul.x, ul.y, ul.z, ul.w, remote_mbU);
      if (w < NG - 1) *reinterpret_cast<float4*>(sUB + (w + 1) * BW + j0) = ul;
      *reinterpret_cast<ulonglong2*>(myUR) = make_ulonglong2(U[3][0], U[3][1]);
    }
    __syncthreads();
    // ---- p-step: theta = 1 and no proximal term, p' = P_C(p + tau0 D u), pbar = p' + (p' - p)
    {
      const ulonglong2 ul = *reinterpret_cast<const ulonglong2*>(myUR - 4);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        {
          const f32x2 tt = fma2(PC, sub2(U[c][1], U[c][0]), P1[c][1]);
          const f32x2 pn = pk2(clamp_abs(lo2(tt), lim1[1]), clamp_abs(hi2(tt), lim1[3]));
          Q1[c][1] = add2(sub2(pn, P1[c][1]), pn);
          P1[c][1] = pn;
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const f32x2 leftu = c > 0 ? U[c - 1][e] : (e == 0 ? ul.x : ul.y);
          const f32x2 tt = fma2(PC, sub2(U[c][e], leftu), P2[c][e]);
          const f32x2 pn = pk2(clamp_abs(lo2(tt), lim2[c]), clamp_abs(hi2(tt), lim2[c]));
          Q2[c][e] = add2(sub2(pn, P2[c][e]), pn);
          P2[c][e] = pn;
        }
      }
      *reinterpret_cast<ulonglong2*>(myQL) = make_ulonglong2(Q2[0][0], Q2[0][1]);
      if (push_up) wait_u();
      const float4 ua = *reinterpret_cast<const float4*>(sUB + w * BW + j0);
      const float uav[4] = {ua.x, ua.y, ua.z, ua.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const f32x2 du = pk2(lo2(U[c][0]) - uav[c], hi2(U[c][0]) - lo2(U[c][1]));
        const f32x2 tt = fma2(PC, du, P1[c][0]);
        const f32x2 pn = pk2(clamp_abs(lo2(tt), lim1[0]), clamp_abs(hi2(tt), lim1[2]));
        Q1[c][0] = add2(sub2(pn, P1[c][0]), pn);
        P1[c][0] = pn;
      }
      const float4 q = make_float4(lo2(Q1[0][0]), lo2(Q1[1][0]), lo2(Q1[2][0]), lo2(Q1[3][0]));
      if (w > 0) *reinterpret_cast<float4*>(sQ1 + w * BW + j0) = q;
      if (push_up) st_async_v4_f32(remote_q1, q.x, q.y, q.z, q.w, remote_mbQ);
    }
    __syncthreads();
  }
  if (push_down) wait_q();  // drain the last pbar1 halo (not read)
  __syncwarp();
  cluster_arrive<false>();  // no CTA leaves while a neighbour may still write into it

  // ---- store what n iterations leave exact
  const int ra = ar.from(by), rb = ar.to(by), ca = ac.from(bx), cb = ac.to(bx);
  const int ja = c0 + j0;
  const bool whole = ja >= ca && ja + 4 <= cb;
  const bool vec = whole && (W & 3) == 0 && (ja & 3) == 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int e = r & 1, h = r >> 1, gi = r0 + i0 + r;
    if (gi < ra || gi >= rb) continue;
    auto put = [&](float* base, int ld, bool v, f32x2 (*X)[2]) {
      float* p = base + (size_t)gi * ld + ja;
      const float x[4] = {half_of(X[0][e], h), half_of(X[1][e], h), half_of(X[2][e], h), half_of(X[3][e], h)};
      if (v) {
        *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (whole || (ja + c >= ca && ja + c < cb)) p[c] = x[c];
      }
    };
    put(A.out.u, W, vec, U);
    put(A.out.P1, W, vec, P1);
    put(A.out.Pb1, W, vec, Q1);
    put(A.out.P2, W2, false, P2);
    put(A.out.Pb2, W2, false, Q2);
  }
  if (timed_out) atomicOr(A.err, 1);
  __syncwarp();
  cluster_wait();
}

template <int FID, bool MASK>
cudaError_t launch_full_one(const FullArgs& a, int n, cudaStream_t st) {
  const Axis ar = axis_for(a.H, n, 1), ac = axis_for(a.W, n, (a.W & 3) == 0 ? 4 : 1);
  const int cl = (ar.size() + FL::BAND - 1) / FL::BAND;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cl * ac.m * ar.m, 1, 1);
  cfg.blockDim = dim3(FL::NT, 1, 1);
  cfg.dynamicSmemBytes = FL::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  pdl_attr(&attr[1]);
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_full<FID, MASK>, a, ar, ac, n);
}

}  // namespace

int full_max_steps() { return 10; }

cudaError_t launch_full(const FullArgs& a, int fid, int n, cudaStream_t st) {
  const bool m = a.mask != nullptr;
  switch (fid) {
    case FID_L2: return m ? launch_full_one<FID_L2, true>(a, n, st) : launch_full_one<FID_L2, false>(a, n, st);
    case FID_L1: return m ? launch_full_one<FID_L1, true>(a, n, st) : launch_full_one<FID_L1, false>(a, n, st);
    default: return launch_full_one<FID_SEG, false>(a, n, st);
  }
}

cudaError_t full_prepare(int fid) {
  cudaError_t e;
  auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FL::BYTES);
  };
  switch (fid) {
    case FID_L2: return (e = set(k_full<FID_L2, false>)) != cudaSuccess ? e : set(k_full<FID_L2, true>);
    case FID_L1: return (e = set(k_full<FID_L1, false>)) != cudaSuccess ? e : set(k_full<FID_L1, true>);
    default: return set(k_full<FID_SEG, false>);
  }
}

}  // namespace ddtv
