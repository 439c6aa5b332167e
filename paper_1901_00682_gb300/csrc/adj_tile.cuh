// Reverse pass of one outer iteration's local solves on the micro-tiles of
// fused_tile.cuh.
//
// One launch recomputes the K inner iterations of every subdomain (tile_solve with ADJ: the
// forward's arithmetic, bit for bit) and records the tape, ubar_k of every pixel and the
// projection's pass bit of every dof, then runs the K reverse iterations of
// kernels_adjoint.cu (same formulas, same operation order) with the adjoint state on chip.
// The state and the adjoints move once per outer iteration.
//
// The reverse iteration has the forward's communication pattern, so it has its mapping too:
// the u-step's adjoint Ad (the adjoint of the divergence) is needed by the row below and
// the column to the right, the p-step's adjoint a_t by the row above and the column to the
// left; rows crossing CTAs travel by st.async on the same two mbarriers, whose phases go on
// counting.  Registers hold the adjoints of u, of p (masked: a_t = [pass] (AP + (1 + theta)
// AQ), formed as soon as AP and AQ are known, is all that the next iteration needs of AP)
// and of pbar; the sums over k (adjoints of phat and f) lie in shared memory in thread
// order, in the forward's places of the proximal centres and one more.  Padding pixels hold
// zero adjoints: those of the first padding column and row are pinned, the others see only
// zeros.
//
// What bounds it: as the forward, latency and issue slots; the tape (18 words per thread and
// iteration) is written and read back within the launch and stays in L2, and the next
// iteration's part of it is copied to shared memory while the current one runs.  Per outer
// iteration of 10 inner ones: 1024 x 1024 80 -> 58 us, 250 x 261 65 -> 33, against a column of
// 8 pixels per thread.
//
// Products are rounded before they are summed (round2), as in the per-step kernels: the
// gradients are theirs bit for bit.
#pragma once

#include "fused_tile.cuh"

namespace ddtv {

namespace {

template <int LPR, int NW>
struct AdjTileLayout {
  using L = TileLayout<LPR, NW>;
  static constexpr int AF = (L::MB + 4 + 3) & ~3;  // adjoint of f, thread order
  static constexpr int TP = AF + 16 * L::NT;       // this iteration's ubar, thread order
  static constexpr int AHB = TP + 16 * L::NT;      // adjoint of phat on the bottom side of a subdomain that fills the block
  static constexpr int TX = AHB + L::BW;           // dL/dalpha terms for the thread of the other row group of a pair
  static constexpr size_t BYTES = sizeof(float) * (TX + 8 * L::NT);
};

// du'/dubar, du'/df, du'/dalpha of u' = prox(ubar) (Section 3 proximity maps); fg is f
// (L2, L1) or g = (f - c1)^2 - (f - c2)^2 (SEG), as in the forward's shared array.
template <int FID>
__device__ __forceinline__ void prox_partials_fg(float ub, float fg, bool in_d, float c1, float c2, const Coef& c,
                                                 float& dub, float& df, float& dal) {
  if (FID == FID_SEG) {
    const float x = fmaf(-c.s, fg, ub);
    const bool pass = x >= 0.0f && x <= 1.0f;
    dub = pass ? 1.0f : 0.0f;
    dal = pass ? -c.sig * fg : 0.0f;
    df = pass ? -c.s * (2.0f * (c2 - c1)) : 0.0f;
    return;
  }
  if (in_d) {
    dub = 1.0f;
    df = 0.0f;
    dal = 0.0f;
    return;
  }
  if (FID == FID_L2) {
    dub = c.ua;
    df = c.ub;
    dal = c.sig * c.ua * c.ua * (fg - ub);
    return;
  }
  const float v = ub - fg;
  const bool pass = fabsf(v) - c.s > 0.0f;
  dub = pass ? 1.0f : 0.0f;
  df = pass ? 0.0f : 1.0f;
  dal = pass ? (v > 0.0f ? -c.sig : c.sig) : 0.0f;
}

// v where the pass bits n (low half) and n + 2 (high half) are set, else 0
__device__ __forceinline__ f32x2 pass2(uint32_t bits, int n, f32x2 v) {
  return pk2((bits >> n) & 1u ? lo2(v) : 0.0f, (bits >> (n + 2)) & 1u ? hi2(v) : 0.0f);
}

// The coefficients of iteration k, as the reverse pass uses them.
__device__ __forceinline__ Coef coef_at(const LocalArgs& A, const float* sCo, bool in_smem, int k) {
  if (!in_smem) return A.coef[k];
  const float* p = sCo + 16 * k;  // each stored twice
  return Coef{p[0], p[2], p[4], p[6], p[8], p[10], p[12], p[14]};
}

// Stores the adjoints of u and p~^n (the sum over all their uses), of phat on the subdomain's
// sides, and adds those of f and alpha.
template <int LPR, int NW, bool PAD>
__device__ __forceinline__ void tile_reverse_store(const Grid& g, const AdjArgs& Z, int a, int b, int tid, int rank, int CL,
                                                   f32x2 (&Au)[4][2], f32x2 (&T1)[4][2], f32x2 (&T2)[4][2], float t_r,
                                                   float h_r, double acc) {
  using L = TileLayout<LPR, NW>;
  using AL = AdjTileLayout<LPR, NW>;
  constexpr int BAND = L::BAND, BW = L::BW, NT = L::NT;
  extern __shared__ __align__(128) float smem[];
  const int r0 = PAD ? part_start(a, g.H, g.NR) : a * CL * BAND, mr = PAD ? part_start(a + 1, g.H, g.NR) - r0 : CL * BAND;
  const int c0 = PAD ? part_start(b, g.W, g.NC) : b * BW, mc = PAD ? part_start(b + 1, g.W, g.NC) - c0 : BW;
  const bool s_top = a > 0 || g.cut_top, s_bot = a + 1 < g.NR || g.cut_bot, s_lft = b > 0, s_rgt = b + 1 < g.NC;
  const int w = tid >> 5, l = tid & 31, G = w * L::RG + l / LPR, j0 = 4 * (l % LPR), i0 = rank * BAND + 4 * G;
  const int W2 = g.W + g.NC;
  const bool fill_c = !PAD || mc == BW, fill_r = !PAD || mr == CL * BAND;
  const bool bottom_lane = fill_r && s_bot && rank == CL - 1 && w == L::kBottomWarp && l < LPR;
  const int rr = tid - L::kRightThread;
  const bool right_lane = fill_c && s_rgt && rr >= 0 && rr < BAND && rank * BAND + rr < mr;
  const float* const myF = smem + L::F + 4 * tid;
  constexpr int kH1 = L::H1 - L::F, kH2 = L::H2 - L::F, kAF = AL::AF - L::F;
  // the adjoint of p~^n = p_0 = pbar_0 = (phat's copy)
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const ulonglong2 h1 = *reinterpret_cast<const ulonglong2*>(myF + kH1 + 4 * NT * c);
    const ulonglong2 h2 = *reinterpret_cast<const ulonglong2*>(myF + kH2 + 4 * NT * c);
    T1[c][0] = add2(T1[c][0], h1.x);
    T1[c][1] = add2(T1[c][1], h1.y);
    T2[c][0] = add2(T2[c][0], h2.x);
    T2[c][1] = add2(T2[c][1], h2.y);
  }
  t_r = t_r + h_r;

  // ---- store: Au, AP (folded), APhat on the subdomain's sides; Af += ; alpha partials
  const bool vec = (g.W & 3) == 0 && (c0 & 3) == 0;
  float af[4][4];  // every load before the first store
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      af[r][c] = i0 + r < mr && c < mc - j0 ? Z.Af[(size_t)(r0 + i0 + r) * g.W + c0 + j0 + c] : 0.f;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int e = r & 1, h = r >> 1, i = i0 + r, gi = r0 + i;
    const int n = i < mr ? mc - j0 : 0;
    const int n1 = (i < mr + (s_bot ? 1 : 0) && (i > 0 || s_top)) ? mc - j0 : 0;
    const size_t px = (size_t)gi * g.W + c0 + j0, e1 = (size_t)(gi + a) * g.W + c0 + j0, e2 = (size_t)gi * W2 + c0 + b + j0;
    store4(Z.Au + px, n, vec, half_of(Au[0][e], h), half_of(Au[1][e], h), half_of(Au[2][e], h), half_of(Au[3][e], h));
    store4(Z.AP1 + e1, n1, vec, half_of(T1[0][e], h), half_of(T1[1][e], h), half_of(T1[2][e], h), half_of(T1[3][e], h));
    const bool side_row = (i == 0 && s_top) || (PAD && i == mr && s_bot);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = j0 + c, q = (r & 1) * 2 + h;  // thread order of the rows: 0, 2, 1, 3
      af[r][c] += myF[kAF + 4 * NT * c + q];
      if (side_row && c < n1) Z.APh1[e1 + c] = myF[kH1 + 4 * NT * c + q];
      if (i < mr && (j < mc || (j == mc && s_rgt)) && (j > 0 || s_lft)) {
        Z.AP2[e2 + c] = half_of(T2[c][e], h);
        if (j == 0 || (PAD && j == mc)) Z.APh2[e2 + c] = myF[kH2 + 4 * NT * c + q];
      }
    }
    store4(Z.Af + px, n, vec, af[r][0], af[r][1], af[r][2], af[r][3]);
  }
  if (right_lane) {
    const size_t e2 = (size_t)(r0 + rank * BAND + rr) * W2 + c0 + BW + b;
    Z.AP2[e2] = t_r;
    Z.APh2[e2] = h_r;
  }
  if (bottom_lane) {
    const size_t e1 = (size_t)(r0 + mr + a) * g.W + c0 + j0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c < mc - j0) {
        Z.AP1[e1 + c] = smem[L::PBS + j0 + c] + smem[AL::AHB + j0 + c];
        Z.APh1[e1 + c] = smem[AL::AHB + j0 + c];
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  double* sw = reinterpret_cast<double*>(smem + L::CO);  // the coefficients are no longer needed
  if (l == 0) sw[w] = acc;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int q = 0; q < NW; ++q) t += sw[q];
    Z.Aal[((size_t)a * g.NC + b) * 8 + rank] += t;
  }
}

template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK>
__device__ __forceinline__ void tile_reverse(const LocalArgs& A, const AdjArgs& Z, const int a, const int b, const int tid,
                                             const int rank, const int CL, const float* tape, const uint32_t in_d,
                                             bool& timed_out) {
  const f32x2 NZ = pk2(Z.neg_zero, Z.neg_zero);
  using L = TileLayout<LPR, NW>;
  using AL = AdjTileLayout<LPR, NW>;
  constexpr int NG = L::NG, BAND = L::BAND, BW = L::BW, NT = L::NT;
  extern __shared__ __align__(128) float smem[];
  float* sUB = smem + L::UB;
  float* sQ1 = smem + L::Q1;
  const float* sCo = smem + L::CO;
  const uint32_t mbU = smem_addr(smem + L::MB), mbQ = mbU + 8;
  const Grid g = A.g;
  const int r0 = PAD ? part_start(a, g.H, g.NR) : a * CL * BAND, mr = PAD ? part_start(a + 1, g.H, g.NR) - r0 : CL * BAND;
  const int c0 = PAD ? part_start(b, g.W, g.NC) : b * BW, mc = PAD ? part_start(b + 1, g.W, g.NC) - c0 : BW;
  const bool s_top = a > 0 || g.cut_top, s_bot = a + 1 < g.NR || g.cut_bot, s_lft = b > 0, s_rgt = b + 1 < g.NC;
  const int w = tid >> 5, l = tid & 31, G = w * L::RG + l / LPR, cl = l % LPR, j0 = 4 * cl, i0 = rank * BAND + 4 * G;
  const int K = A.K, W2 = g.W + g.NC;
  const bool fill_c = !PAD || mc == BW, fill_r = !PAD || mr == CL * BAND;
  const bool last_group = rank == CL - 1 && G == NG - 1;
  const bool push_down = CLU && G == NG - 1 && rank + 1 < CL, push_up = CLU && G == 0 && rank > 0;
  const bool bottom_lane = fill_r && s_bot && rank == CL - 1 && w == L::kBottomWarp && l < LPR;
  const int rr = tid - L::kRightThread;
  const bool right_lane = fill_c && s_rgt && rr >= 0 && rr < BAND && rank * BAND + rr < mr;
  const int r_slot = (rr >> 2) * L::SLOT + 4 * LPR + 2 * (rr & 1) + ((rr >> 1) & 1);
  const bool pad_c = PAD && !fill_c && (mc >> 2) == cl;
  const bool pad_r = PAD && !fill_r && mr >= rank * BAND && ((mr - rank * BAND) >> 2) == G;
  const int cpad = mc & 3, rpad = mr & 3;
  constexpr uint32_t kHaloBytes = 4 * BW;
  float* const myUR = smem + L::UR + G * L::SLOT + 4 * (cl + 1);
  float* const myQL = smem + L::QL + G * L::SLOT + 4 * cl;
  float* const myF = smem + L::F + 4 * tid;
  constexpr int kH1 = L::H1 - L::F, kH2 = L::H2 - L::F, kAF = AL::AF - L::F, kTP = AL::TP - L::F;
  const uint32_t s0 = smem_addr(smem);
  const uint32_t remote = push_down ? map_rank(s0, rank + 1) : (push_up ? map_rank(s0, rank - 1) : 0u);
  const bool coef_smem = K <= L::kMaxSmemCoef;
  // this thread's part of iteration k of the tape: ubar at 4 NT c, pass bits at 16 NT - 3 tid,
  // those of the sides at 17 NT - 3 tid (bit 0: right side; bits 1 .. 4: bottom side)
  const float* tk = tape + (size_t)(K - 1) * kTapeWords * NT + 4 * tid;
  auto bits_of = [&](const float* t, int word) {
    return reinterpret_cast<const uint32_t*>(t)[word * NT - 3 * (int)threadIdx.x];
  };
  uint32_t phU = K, phQ = K;  // phases consumed by the forward
  auto wait_u = [&]() {
    if (!mbar_wait(mbU, phU & 1)) timed_out = true;
    ++phU;
    if (cl == 0) mbar_arrive_expect_tx(mbU, kHaloBytes);
  };
  auto wait_q = [&]() {
    if (!mbar_wait(mbQ, phQ & 1)) timed_out = true;
    ++phQ;
    if (cl == 0) mbar_arrive_expect_tx(mbQ, kHaloBytes);
  };
  auto fetch_tape = [&](const float* t) {  // ubar of this thread's pixels
#pragma unroll
    for (int c = 0; c < 4; ++c) cp_async16(myF + kTP + 4 * NT * c, t + 4 * NT * c);
    cp_async_commit();
  };
  fetch_tape(tk);

  // adjoints: Au of u; T1, T2: a_t of p1, p2; Q1, Q2 of pbar1, pbar2
  f32x2 Au[4][2], T1[4][2], T2[4][2], Q1[4][2], Q2[4][2];
  // dL/dalpha: a compensated float32 sum per column and 8 rows over the K iterations, in the
  // order (7, 0, 1, ..., 6) of the rows, then float64 (the per-column kernels' sums).  The
  // threads of two row groups share 4 columns: each sums 2 of them (the two halves), with
  // the other's 4 rows from shared memory.
  f32x2 acc_s = 0ull, acc_c = 0ull;
  const bool odd = G & 1;
  ulonglong2 own[2];
  float t_r = 0.f, q_r = 0.f, h_r = 0.f;
  {
    const bool vec = (g.W & 3) == 0 && (c0 & 3) == 0;
    const uint32_t bits = bits_of(tk, 16);
    float xu[4][4], x1[4][4], x2[4][4];
    const float* gu = Z.Au + (size_t)(r0 + i0) * g.W + c0 + j0;
    const float* g1 = Z.AP1 + (size_t)(r0 + i0 + a) * g.W + c0 + j0;
    const float* g2 = Z.AP2 + (size_t)(r0 + i0) * W2 + c0 + b + j0;
    if (vec && i0 + 3 < mr && j0 + 3 < mc) {  // all loads in flight together, as the forward's
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        load4(gu + (size_t)r * g.W, xu[r]);
        load4(g1 + (size_t)r * g.W, x1[r]);
#pragma unroll
        for (int c = 0; c < 4; ++c) x2[r][c] = g2[(size_t)r * W2 + c];
      }
    } else {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + r;
        const int n = i < mr ? mc - j0 : 0, n1 = i < mr + (s_bot ? 1 : 0) ? mc - j0 : 0;
        const int n2 = i < mr ? mc + (s_rgt ? 1 : 0) - j0 : 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          xu[r][c] = c < n ? gu[(size_t)r * g.W + c] : 0.f;
          x1[r][c] = c < n1 ? g1[(size_t)r * g.W + c] : 0.f;
          x2[r][c] = c < n2 ? g2[(size_t)r * W2 + c] : 0.f;
        }
      }
    }
    uint32_t xb = 0;
    if (right_lane || bottom_lane) xb = bits_of(tk, 17);
    if (right_lane) t_r = Z.AP2[(size_t)(r0 + rank * BAND + rr) * W2 + c0 + BW + b];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        Au[c][e] = pk2(xu[e][c], xu[e + 2][c]);
        T1[c][e] = pk2(x1[e][c], x1[e + 2][c]);
        T2[c][e] = pk2(x2[e][c], x2[e + 2][c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        T1[c][e] = pass2(bits, 4 * c + e, T1[c][e]);
        T2[c][e] = pass2(bits, 16 + 4 * c + e, T2[c][e]);
        Q1[c][e] = Q2[c][e] = 0ull;
      }
      *reinterpret_cast<ulonglong2*>(myF + kH1 + 4 * NT * c) = make_ulonglong2(0ull, 0ull);
      *reinterpret_cast<ulonglong2*>(myF + kH2 + 4 * NT * c) = make_ulonglong2(0ull, 0ull);
      *reinterpret_cast<ulonglong2*>(myF + kAF + 4 * NT * c) = make_ulonglong2(0ull, 0ull);
    }
    if (!(xb & 1u)) t_r = 0.f;
    *reinterpret_cast<ulonglong2*>(myQL) = make_ulonglong2(T2[0][0], T2[0][1]);
    if (rr >= 0 && rr < BAND) smem[L::QL + r_slot] = t_r;
    if (G > 0) *reinterpret_cast<float4*>(sQ1 + G * BW + j0) = make_float4(lo2(T1[0][0]), lo2(T1[1][0]), lo2(T1[2][0]), lo2(T1[3][0]));
    if (last_group && !(fill_r && s_bot)) *reinterpret_cast<float4*>(sQ1 + NG * BW + j0) = make_float4(0.f, 0.f, 0.f, 0.f);
    if (bottom_lane) {
      float t[4];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        t[c] = c < mc - j0 && ((xb >> (1 + c)) & 1u) ? Z.AP1[(size_t)(r0 + mr + a) * g.W + c0 + j0 + c] : 0.f;
      const float4 tv = make_float4(t[0], t[1], t[2], t[3]);
      *reinterpret_cast<float4*>(smem + L::PBS + j0) = tv;
      *reinterpret_cast<float4*>(sQ1 + NG * BW + j0) = tv;
      *reinterpret_cast<float4*>(smem + L::HBS + j0) = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(smem + AL::AHB + j0) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __syncthreads();
  if (CLU) {
    // the forward's last halos have landed everywhere before the first reverse one is sent
    // (two pushes into one halo buffer must not be in flight at once)
    cluster_arrive<true>();
    cluster_wait();
    if (push_up)
      st_async_v4_f32(remote + 4 * (L::Q1 + NG * BW + j0), lo2(T1[0][0]), lo2(T1[1][0]), lo2(T1[2][0]), lo2(T1[3][0]),
                      remote + 4 * L::MB + 8);
  }

#pragma unroll 1
  for (int k = K - 1; k >= 0; --k) {
    const Coef co = coef_at(A, sCo, coef_smem, k);
    const f32x2 SIG = pk2(co.sig, co.sig), PC = pk2(co.pc, co.pc);
    // pass bits of the next (earlier) iteration; after the last one (k = 0) everything passes
    // with factor 1: AP + AQ, to which the sum of phat's adjoint is added after the loop
    tk -= kTapeWords * NT;
    const uint32_t bn = k > 0 ? bits_of(tk, 16) : ~0u;
    const uint32_t xn = k > 0 && (right_lane || bottom_lane) ? bits_of(tk, 17) : ~0u;
    if (push_down) wait_q();  // a_t of the first row below
    // ---- reverse u-step: Au' = Au - div(pc a_t)
    {
      const float4 qb = *reinterpret_cast<const float4*>(sQ1 + (G + 1) * BW + j0);
      const ulonglong2 qn = *reinterpret_cast<const ulonglong2*>(myQL + 4);
      const float qbv[4] = {qb.x, qb.y, qb.z, qb.w};
      f32x2 left[2] = {round2(PC, T2[0][0], NZ), round2(PC, T2[0][1], NZ)};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const f32x2 x0 = round2(PC, T1[c][0], NZ), x1 = round2(PC, T1[c][1], NZ);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const f32x2 bt = e == 0 ? sub2(x1, x0) : pk2(hi2(x0) - lo2(x1), co.pc * qbv[c] - hi2(x1));
          const f32x2 right = round2(PC, c < 3 ? T2[c + 1][e] : (e == 0 ? qn.x : qn.y), NZ);
          Au[c][e] = sub2(Au[c][e], sub2(add2(bt, right), left[e]));
          left[e] = right;
        }
      }
      if (PAD && pad_c) {
        auto pin = [&](int q) { Au[q][0] = Au[q][1] = 0ull; };
        if (cpad == 0) pin(0);
        else if (cpad == 1) pin(1);
        else if (cpad == 2) pin(2);
        else pin(3);
      }
      if (PAD && pad_r) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (rpad == 0) Au[c][0] = pk2(0.f, hi2(Au[c][0]));
          else if (rpad == 1) Au[c][1] = pk2(0.f, hi2(Au[c][1]));
          else if (rpad == 2) Au[c][0] = pk2(lo2(Au[c][0]), 0.f);
          else Au[c][1] = pk2(lo2(Au[c][1]), 0.f);
        }
      }
      // through the prox: Aubar = du'/dubar Au', Af += du'/df Au', Aalpha += du'/dalpha Au'
      cp_async_wait_all();
      const float cs = co.sig * co.ua * co.ua;
      const f32x2 CS = pk2(cs, cs), UA = pk2(co.ua, co.ua), UBc = pk2(co.ub, co.ub);
      f32x2 TM[4][2];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const ulonglong2 fc = *reinterpret_cast<const ulonglong2*>(myF + 4 * NT * c);
        const ulonglong2 uc = *reinterpret_cast<const ulonglong2*>(myF + kTP + 4 * NT * c);
        ulonglong2 af = *reinterpret_cast<const ulonglong2*>(myF + kAF + 4 * NT * c);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const f32x2 fg = e == 0 ? fc.x : fc.y, ub = e == 0 ? uc.x : uc.y, aun = Au[c][e];
          f32x2 term, daf;
          if (FID == FID_L2 && !MASK) {
            term = round2(round2(CS, sub2(fg, ub), NZ), aun, NZ);
            daf = round2(UBc, aun, NZ);
            Au[c][e] = round2(UA, aun, NZ);
          } else {
            float dub[2], df[2], dal[2];
            prox_partials_fg<FID>(lo2(ub), lo2(fg), MASK && ((in_d >> (4 * c + e)) & 1u), A.c1, A.c2, co, dub[0], df[0], dal[0]);
            prox_partials_fg<FID>(hi2(ub), hi2(fg), MASK && ((in_d >> (4 * c + e + 2)) & 1u), A.c1, A.c2, co, dub[1], df[1],
                                  dal[1]);
            // (a partial of 0 gives 0, whatever its factor)
            term = pk2(dal[0] != 0.f ? dal[0] * lo2(aun) : 0.f, dal[1] != 0.f ? dal[1] * hi2(aun) : 0.f);
            daf = pk2(df[0] != 0.f ? df[0] * lo2(aun) : 0.f, df[1] != 0.f ? df[1] * hi2(aun) : 0.f);
            Au[c][e] = pk2(dub[0] * lo2(aun), dub[1] * hi2(aun));
          }
          if (e == 0) af.x = add2(af.x, daf); else af.y = add2(af.y, daf);
          TM[c][e] = term;
        }
        *reinterpret_cast<ulonglong2*>(myF + kAF + 4 * NT * c) = af;
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        own[q] = odd ? make_ulonglong2(TM[2 + q][0], TM[2 + q][1]) : make_ulonglong2(TM[q][0], TM[q][1]);
        *reinterpret_cast<ulonglong2*>(smem + AL::TX + 4 * (q * NT + tid)) =
            odd ? make_ulonglong2(TM[q][0], TM[q][1]) : make_ulonglong2(TM[2 + q][0], TM[2 + q][1]);
      }
      if (k > 0) fetch_tape(tk);
      // Ad = sigma_k Aubar to the neighbours
      const float4 ul = make_float4(hi2(round2(SIG, Au[0][1], NZ)), hi2(round2(SIG, Au[1][1], NZ)), hi2(round2(SIG, Au[2][1], NZ)),
                                    hi2(round2(SIG, Au[3][1], NZ)));
      if (push_down)
        st_async_v4_f32(remote + 4 * (L::UB + j0), ul.x, ul.y, ul.z, ul.w, remote + 4 * L::MB);
      else if (last_group)
        *reinterpret_cast<float4*>(smem + L::XUB + j0) = ul;
      if (G < NG - 1) *reinterpret_cast<float4*>(sUB + (G + 1) * BW + j0) = ul;
      *reinterpret_cast<ulonglong2*>(myUR) = make_ulonglong2(round2(SIG, Au[3][0], NZ), round2(SIG, Au[3][1], NZ));
    }
    __syncthreads();
    {
      // rows 0 .. 3 are the even group's, 4 .. 7 the odd one's; a quad holds rows 0, 2, 1, 3
      ulonglong2 lo[2], hi[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const ulonglong2 other = *reinterpret_cast<const ulonglong2*>(smem + AL::TX + 4 * (q * NT + (tid ^ LPR)));
        lo[q] = odd ? other : own[q];
        hi[q] = odd ? own[q] : other;
      }
      auto add = [&](int r, float a0, float a1) {
        if (PAD && rank * BAND + 8 * (G >> 1) + r >= mr) return;  // (a zero would move the compensation into the sum)
        const f32x2 y = sub2(pk2(a0, a1), acc_c), t = add2(acc_s, y);
        acc_c = sub2(sub2(t, acc_s), y);
        acc_s = t;
      };
      add(7, hi2(hi[0].y), hi2(hi[1].y));
      add(0, lo2(lo[0].x), lo2(lo[1].x));
      add(1, lo2(lo[0].y), lo2(lo[1].y));
      add(2, hi2(lo[0].x), hi2(lo[1].x));
      add(3, hi2(lo[0].y), hi2(lo[1].y));
      add(4, lo2(hi[0].x), lo2(hi[1].x));
      add(5, lo2(hi[0].y), lo2(hi[1].y));
      add(6, hi2(hi[0].x), hi2(hi[1].x));
    }
    // ---- reverse p-step: AQ' = Ad(above / left) - Ad, AP' = pa a_t - theta AQ, APhat += pb a_t
    const f32x2 PA = pk2(co.pa, co.pa), PB = pk2(co.pb, co.pb), TH = pk2(co.th, co.th);
    const float opn = k > 0 ? 1.0f + coef_at(A, sCo, coef_smem, k - 1).th : 1.0f;
    const f32x2 OPN = pk2(opn, opn);
    auto dof = [&](f32x2& T, f32x2& Q, f32x2 aq, int n) {
      const f32x2 ap = sub2(round2(PA, T, NZ), round2(TH, Q, NZ));
      Q = aq;
      T = pass2(bn, n, add2(ap, round2(OPN, aq, NZ)));
    };
    {
      const ulonglong2 ul = *reinterpret_cast<const ulonglong2*>(myUR - 4);
      f32x2 left[2] = {ul.x, ul.y};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const f32x2 d[2] = {round2(SIG, Au[c][0], NZ), round2(SIG, Au[c][1], NZ)};
        ulonglong2 h1 = *reinterpret_cast<const ulonglong2*>(myF + kH1 + 4 * NT * c);
        ulonglong2 h2 = *reinterpret_cast<const ulonglong2*>(myF + kH2 + 4 * NT * c);
        h1.x = add2(h1.x, round2(PB, T1[c][0], NZ));
        h1.y = add2(h1.y, round2(PB, T1[c][1], NZ));
        h2.x = add2(h2.x, round2(PB, T2[c][0], NZ));
        h2.y = add2(h2.y, round2(PB, T2[c][1], NZ));
        *reinterpret_cast<ulonglong2*>(myF + kH1 + 4 * NT * c) = h1;
        *reinterpret_cast<ulonglong2*>(myF + kH2 + 4 * NT * c) = h2;
        dof(T1[c][1], Q1[c][1], sub2(d[0], d[1]), 4 * c + 1);
        dof(T2[c][0], Q2[c][0], sub2(left[0], d[0]), 16 + 4 * c);
        dof(T2[c][1], Q2[c][1], sub2(left[1], d[1]), 16 + 4 * c + 1);
        left[0] = d[0];
        left[1] = d[1];
      }
      *reinterpret_cast<ulonglong2*>(myQL) = make_ulonglong2(T2[0][0], T2[0][1]);
      if (push_up) wait_u();  // Ad of the last row above
      const float4 ua = *reinterpret_cast<const float4*>(sUB + G * BW + j0);
      const float uav[4] = {ua.x, ua.y, ua.z, ua.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const f32x2 d0 = round2(SIG, Au[c][0], NZ), d1 = round2(SIG, Au[c][1], NZ);
        dof(T1[c][0], Q1[c][0], pk2(uav[c] - lo2(d0), lo2(d1) - hi2(d0)), 4 * c);
      }
      if (k > 0) {
        const float4 q = make_float4(lo2(T1[0][0]), lo2(T1[1][0]), lo2(T1[2][0]), lo2(T1[3][0]));
        if (G > 0) *reinterpret_cast<float4*>(sQ1 + G * BW + j0) = q;
        if (push_up) st_async_v4_f32(remote + 4 * (L::Q1 + NG * BW + j0), q.x, q.y, q.z, q.w, remote + 4 * L::MB + 8);
      }
    }
    auto side = [&](float& t, float& q, float& h, float aq, bool pass) {
      h = h + co.pb * t;
      const float ap = co.pa * t - co.th * q;
      q = aq;
      t = pass ? ap + opn * aq : 0.0f;
    };
    if (right_lane) {
      side(t_r, q_r, h_r, smem[L::UR + r_slot], xn & 1u);
      smem[L::QL + r_slot] = t_r;
    }
    if (bottom_lane) {
      const float4 tv = *reinterpret_cast<const float4*>(smem + L::PBS + j0);
      const float4 qv = *reinterpret_cast<const float4*>(smem + L::HBS + j0);
      const float4 hv = *reinterpret_cast<const float4*>(smem + AL::AHB + j0);
      const float4 dv = *reinterpret_cast<const float4*>(smem + L::XUB + j0);
      float t[4] = {tv.x, tv.y, tv.z, tv.w}, q[4] = {qv.x, qv.y, qv.z, qv.w}, h[4] = {hv.x, hv.y, hv.z, hv.w};
      const float d[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) side(t[c], q[c], h[c], d[c], (xn >> (1 + c)) & 1u);
      const float4 tn = make_float4(t[0], t[1], t[2], t[3]);
      *reinterpret_cast<float4*>(smem + L::PBS + j0) = tn;
      *reinterpret_cast<float4*>(smem + L::HBS + j0) = make_float4(q[0], q[1], q[2], q[3]);
      *reinterpret_cast<float4*>(smem + AL::AHB + j0) = make_float4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<float4*>(sQ1 + NG * BW + j0) = tn;
    }
    __syncthreads();
  }
  if (CLU) {
    __syncwarp();
    cluster_arrive<false>();  // no CTA leaves while a neighbour may still write into it
  }

  // the geometry again rather than in registers through the loop
  int tid2, a2 = a, b2 = b;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid2));
  asm volatile("" : "+r"(a2), "+r"(b2));
  const double acc = ((double)lo2(acc_s) - (double)lo2(acc_c)) + ((double)hi2(acc_s) - (double)hi2(acc_c));
  tile_reverse_store<LPR, NW, PAD>(A.g, Z, a2, b2, tid2, rank, CL, Au, T1, T2, t_r, h_r, acc);
}

// CTAs of up to 4 warps run 12 warps per SM: the reverse loop does not fit the forward's 128
// registers (with 16 warps, forward and backward of 250 x 261 take 2610 us instead of 2340, of two
// 1024 x 1024 3840 instead of 3600).  Those of 8 warps (64 x 64 subdomains) run two per SM at 128
// registers, with 136 to 220 bytes of spills per thread: at the 168 of the others only one would
// fit.
template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK>
__global__ void __launch_bounds__(32 * NW, NW <= 4 ? 12 / NW : 2) k_adj_tile(const LocalArgs A, const AdjArgs Z, const int cl) {
  const unsigned t = CLU ? blockIdx.x / (unsigned)cl : blockIdx.x, rank = CLU ? blockIdx.x - t * (unsigned)cl : 0u;
  const unsigned a = t / (unsigned)A.g.NC;
  tile_solve<LPR, NW, CLU, PAD, FID, MASK, false, true>(A, A.out, (int)a, (int)(t - a * (unsigned)A.g.NC), (int)rank,
                                                 CLU ? cl : 1, &Z);
}

template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK>
cudaError_t launch_adj_tile_one(const LocalArgs& a, const AdjArgs& z, int cl, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(CLU ? cl : 1) * a.g.NC * a.g.NR, 1, 1);
  cfg.blockDim = dim3(32 * NW, 1, 1);
  cfg.dynamicSmemBytes = AdjTileLayout<LPR, NW>::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (has_interfaces(a.g)) pdl_attr(&attr[cfg.numAttrs++]);
  if (CLU) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cl;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  return cudaLaunchKernelEx(&cfg, k_adj_tile<LPR, NW, CLU, PAD, FID, MASK>, a, z, cl);
}

template <int LPR, int NW, bool CLU, bool PAD>
cudaError_t launch_adj_tile(const LocalArgs& a, const AdjArgs& z, int fid, int cl, cudaStream_t st) {
  const bool m = a.mask != nullptr;
  switch (fid) {
    case FID_L2:
      return m ? launch_adj_tile_one<LPR, NW, CLU, PAD, FID_L2, true>(a, z, cl, st)
               : launch_adj_tile_one<LPR, NW, CLU, PAD, FID_L2, false>(a, z, cl, st);
    case FID_L1:
      return m ? launch_adj_tile_one<LPR, NW, CLU, PAD, FID_L1, true>(a, z, cl, st)
               : launch_adj_tile_one<LPR, NW, CLU, PAD, FID_L1, false>(a, z, cl, st);
    default: return launch_adj_tile_one<LPR, NW, CLU, PAD, FID_SEG, false>(a, z, cl, st);
  }
}

template <int LPR, int NW, bool CLU, bool PAD>
cudaError_t prepare_adj_tile() {
  auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AdjTileLayout<LPR, NW>::BYTES);
  };
  cudaError_t e;
  if ((e = set(k_adj_tile<LPR, NW, CLU, PAD, FID_L2, false>)) != cudaSuccess) return e;
  if ((e = set(k_adj_tile<LPR, NW, CLU, PAD, FID_L2, true>)) != cudaSuccess) return e;
  if ((e = set(k_adj_tile<LPR, NW, CLU, PAD, FID_L1, false>)) != cudaSuccess) return e;
  if ((e = set(k_adj_tile<LPR, NW, CLU, PAD, FID_L1, true>)) != cudaSuccess) return e;
  return set(k_adj_tile<LPR, NW, CLU, PAD, FID_SEG, false>);
}

}  // namespace
}  // namespace ddtv
