// Fused local solver on 4 x 4 micro-tiles for subdomains of any shape up to 128 x 128.
//
// What bounds the local solve is latency and issue slots, not memory: a subdomain
// lives on chip for its whole inner loop, so the time of an inner iteration is the
// length of its dependency chain (two barriers, the shared-memory exchange) and the
// instructions its warps issue in between.  Holding 16 pixels per thread puts most
// neighbours in registers, lets the arithmetic run on packed float32 pairs and leaves
// one 16-byte exchange per edge and 16 pixels.
//
// Mapping.  LPR lanes hold a row group: 4 rows of 4 LPR columns (LPR = 8, 16, 32 for
// subdomains up to 32, 64, 128 columns wide), so a warp holds 32 / LPR row groups and a
// CTA of NW warps a band of BAND = 4 NW (32 / LPR) rows.  A subdomain is one CTA, or a
// cluster of the fewest CTAs whose bands cover its rows; halo rows then travel with
// st.async counted on mbarriers (bounded waits), as in kernels_fused_mt.cu.  Registers
// hold u, the dual dofs p1 (top edge) and p2 (left edge) and their extrapolations; f and
// the proximal centres, read once per inner iteration by the thread that owns them, wait
// in shared memory in the owner's order, which keeps a thread within 128 registers and
// four 128-thread CTAs on an SM.
//
// Shapes.  A subdomain smaller than the block of pixels its threads cover is padded on
// the right and at the bottom.  u is pinned to 0 in the first padding column and row, so
// the dof on the left edge of that column is the subdomain's right side (D_s u = -u of
// the last column) and the dof on the top edge of that row its bottom side, updated as
// any other dof; what lies further out is never read by a pixel of the subdomain.  (The
// lane that holds the column or row branches on its place in the micro-tile; as selects the
// pinning cost half as many instructions again as the iteration.)  Where
// the subdomain fills the block (no padding) the sides are updated by lanes of other
// warps.  A side on the image boundary is kept at 0 by
// clamping its dofs to [-0, 0].
//
// Measured per outer iteration of 10 inner ones, multiplier update included, against
// the kernels it replaced (the cluster-barrier kernel, a column of 8 pixels per thread;
// for exact 128 x 128 subdomains the persistent clusters of kernels_fused_mt4.cu with
// three CTAs per SM): 1080 x 1920 in 120 x 128 subdomains 106 -> 41 us, 2160 x 3840
// 446 -> 139, 2999 x 3001 in 125 x 125/126 473 -> 161, 4096 x 4096 in 64 x 64 571 -> 214 and in
// 32 x 32 526 -> 197, 512 x 512 in 32 x 32 19.6 -> 8.3, 128 x 128 in 64 x 64 22.1 -> 10.8, 321 x
// 481 in 107 x 120/121 26.2 -> 13.9; in 128 x 128 subdomains 512 x 512 14.4 -> 11.8, 1024 x 1024
// 22.8 -> 18.1, 4096 x 4096 230 -> 217 (K = 10; where the persistent kernel is the faster
// one, use_mt4() in kernels_fused.cu), a batch of 64 images (168 Mpixel) 2730 -> 2320; with
// the adaptive stop, 1024 x 1024 and 18.7 inner iterations on average, 54 -> 43.
//
// Every value is computed with the operations of the scalar iteration in its order
// (pointwise.cuh), so the results are those of the plain path bit for bit.
#pragma once

#include "fused_common.cuh"
#include "internal.cuh"

namespace ddtv {

namespace {

template <int LPR_, int NW_>
struct TileLayout {
  static constexpr int LPR = LPR_, NW = NW_;
  static constexpr int RG = 32 / LPR;               // row groups per warp
  static constexpr int NG = NW * RG;                // row groups per CTA
  static constexpr int BAND = 4 * NG, BW = 4 * LPR, NT = 32 * NW;
  static constexpr int SLOT = 4 * (LPR + 1);        // a row group's UR / QL slots
  static constexpr int kMaxSmemCoef = 64;
  static constexpr int UB = 0;                      // (NG + 1) x BW: row 0 = u above the band, G + 1 = last row of group G
  static constexpr int Q1 = UB + (NG + 1) * BW;     // (NG + 1) x BW: row G = pbar1 of group G's first row, NG = below
  static constexpr int UR = Q1 + (NG + 1) * BW;     // NG x SLOT: slot 0 = 0 (left of the tile), cl + 1 = u of lane cl's right column
  static constexpr int QL = UR + NG * SLOT;         // NG x SLOT: slot cl = pbar2 of lane cl's left edge, LPR = the right side
  static constexpr int F = QL + NG * SLOT;          // 4 x NT x 4: f (or g), thread order
  static constexpr int H1 = F + 16 * NT;            // proximal centres, thread order
  static constexpr int H2 = H1 + 16 * NT;
  static constexpr int CO = H2 + 16 * NT;           // kMaxSmemCoef x 16: the coefficients, each twice
  static constexpr int PBS = CO + 16 * kMaxSmemCoef;  // p of the bottom side of a subdomain that fills the block
  static constexpr int HBS = PBS + BW;              // its proximal centre
  static constexpr int XUB = HBS + BW;              // u of the subdomain's last row, for that side
  static constexpr int MB = XUB + BW;               // two mbarriers
  static constexpr size_t BYTES = sizeof(float) * MB + 16;
  static constexpr int kRightThread = 32;           // threads kRightThread + i update the right side of band row i
  static constexpr int kBottomWarp = NW > 2 ? 2 : 0;
  static_assert(Q1 % 4 == 0 && UR % 4 == 0 && QL % 4 == 0 && F % 4 == 0 && CO % 4 == 0 && PBS % 4 == 0 && MB % 2 == 0,
                "16-byte alignment of the vector accesses");
  static_assert(kRightThread + BAND <= NT, "a thread per right-side dof");
};

// Shared memory with an inpainting domain D, behind the layout above: a word per pixel, thread
// order.  f is taken as 0 on D, where the prox is the identity; then L1, ubar - P(ubar - f),
// is it with the difference times 0, and L2, ua ubar + ub f, with ua replaced by 1: the
// words are the factor 0 or 1, or the mask that keeps ua.
constexpr bool use_mask_words(bool clu, bool mask, bool adj, bool adapt) { return clu && mask && !adj && !adapt; }

template <int LPR, int NW>
struct MaskTileLayout {
  using L = TileLayout<LPR, NW>;
  static constexpr int DM = (L::MB + 4 + 3) & ~3;
  static constexpr size_t BYTES = sizeof(float) * (DM + 16 * L::NT);
};

// Shared memory of the adaptive inner stop, behind the layout above.
template <int LPR, int NW>
struct AdaptTileLayout {
  using L = TileLayout<LPR, NW>;
  static constexpr int kMaxCL = 8;
  static constexpr int OU = (L::MB + 4 + 3) & ~3;    // u of the iteration before, thread order
  static constexpr int PS = OU + 16 * L::NT;         // every thread's residual sums
  static constexpr int RED = PS + 4 * L::NT;         // two buffers (parity of the phase) of a pair per CTA
  static constexpr int STOP = RED + 2 * 2 * kMaxCL;  // the CTA's decision
  static constexpr int MBR = STOP + 2;               // two mbarriers, one per parity
  static constexpr size_t BYTES = sizeof(float) * MBR + 16;
  static constexpr int kReduceWarp = NW - 1;         // adds the CTA's residual sums and sends them
  static constexpr int kDecideWarp = 1;              // takes the stop decision
  static_assert(RED % 2 == 0 && MBR % 2 == 0, "8-byte alignment of the pairs and mbarriers");
};

// Shared memory of the multiplier update (CHAIN), behind whichever of the above the instance
// has.  (What an instance does not need it does not ask for: four CTAs past 164 KB or 196 KB
// leave the L1 cache less, 4096 x 4096 with a mask 240 -> 265 us.)
template <int LPR, int NW, bool WORDS, bool ADAPT>
struct ChainTileLayout {
  using L = TileLayout<LPR, NW>;
  static constexpr size_t kBefore = ADAPT   ? AdaptTileLayout<LPR, NW>::BYTES
                                    : WORDS ? MaskTileLayout<LPR, NW>::BYTES
                                            : L::BYTES;
  static constexpr int OT = (int)((kBefore / sizeof(float) + 3) & ~(size_t)3);  // p~^n on the upper and lower side (BW each),
  static constexpr int OL = OT + 2 * L::BW;    // ... on the left and right side, of the band's rows (BAND each)
  static constexpr int LT = OL + 2 * L::BAND;  // the new multipliers of the upper and lower side (BW each)
  static constexpr int LL = LT + 2 * L::BW;    // ... of the left and right side (BAND each)
  static constexpr size_t BYTES = sizeof(float) * (LL + 2 * L::BAND);
};

// shared memory of an instance of the forward kernel
template <int LPR, int NW, bool WORDS, bool ADAPT, bool CHAIN>
constexpr size_t tile_bytes() {
  return CHAIN ? ChainTileLayout<LPR, NW, WORDS, ADAPT>::BYTES : ChainTileLayout<LPR, NW, WORDS, ADAPT>::kBefore;
}

// four consecutive floats (16-byte aligned)
__device__ __forceinline__ void load4(const float* p, float* v) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  v[0] = x.x;
  v[1] = x.y;
  v[2] = x.z;
  v[3] = x.w;
}

// four consecutive floats of a row, the first n valid (n <= 0: none), the rest 0
__device__ __forceinline__ void load4(const float* p, int n, bool vec, float* v) {
  if (vec && n >= 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
    return;
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = c < n ? p[c] : 0.f;
}

__device__ __forceinline__ void store4(float* p, int n, bool vec, float a, float b, float c, float d) {
  if (vec && n >= 4) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
    return;
  }
  if (n > 0) p[0] = a;
  if (n > 1) p[1] = b;
  if (n > 2) p[2] = c;
  if (n > 3) p[3] = d;
}

__device__ __forceinline__ float half_of(f32x2 v, int h) { return h ? hi2(v) : lo2(v); }

// Stores the subdomain's u, p1, p2 and sides.
template <int LPR, int NW, bool PAD, bool CHAIN, class CH>
__device__ __forceinline__ void tile_store(const LocalArgs& A, const Strips& out, int a, int b, int tid, int CL, int rank,
                                           const f32x2 (&U)[4][2], const f32x2 (&P1)[4][2], const f32x2 (&P2)[4][2],
                                           float pr_s) {
  using L = TileLayout<LPR, NW>;
  constexpr int BAND = L::BAND, BW = L::BW;
  extern __shared__ __align__(128) float smem[];
  const Grid g = A.g;
  const int r0 = PAD ? part_start(a, g.H, g.NR) : a * CL * BAND, mr = PAD ? part_start(a + 1, g.H, g.NR) - r0 : CL * BAND;
  const int c0 = PAD ? part_start(b, g.W, g.NC) : b * BW, mc = PAD ? part_start(b + 1, g.W, g.NC) - c0 : BW;
  const bool s_top = a > 0 || g.cut_top, s_bot = a + 1 < g.NR || g.cut_bot, s_lft = b > 0, s_rgt = b + 1 < g.NC;
  const bool fill_c = !PAD || mc == BW, fill_r = !PAD || mr == CL * BAND;
  const int w = tid >> 5, l = tid & 31, G = w * L::RG + l / LPR, j0 = 4 * (l % LPR), i0 = rank * BAND + 4 * G;
  const int W2 = g.W + g.NC;
  const int rr = tid - L::kRightThread;
  const bool right_lane = fill_c && s_rgt && rr >= 0 && rr < BAND && rank * BAND + rr < mr;
  const bool bottom_lane = fill_r && s_bot && rank == CL - 1 && w == L::kBottomWarp && l < LPR;
  const bool vec = (g.W & 3) == 0 && (c0 & 3) == 0;
  // the strips of a set start at multiples of the interface edges, not of 4 floats
  const bool vec_t = vec && (reinterpret_cast<uintptr_t>(out.ST) & 15) == 0;
  const bool vec_b = vec && (reinterpret_cast<uintptr_t>(out.SB) & 15) == 0;
  if (CHAIN) {  // 2 p~^{n+1} - p~^n of the sides and their multipliers
    const Strips& x = A.x_out;
    const float *oldt = smem + CH::OT + j0, *oldl = smem + CH::OL + 4 * G;
    const float *lamt = smem + CH::LT + j0, *laml = smem + CH::LL + 4 * G;
    if (i0 == 0 && s_top) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < mc - j0) {
          const ptrdiff_t e = (ptrdiff_t)(a - 1) * g.W + c0 + j0 + c;
          x.ST[e] = fmaf(2.0f, lo2(P1[c][0]), -oldt[c]);
          A.lam_th[e] = lamt[c];
        }
    }
    const bool pad_bot = PAD && s_bot && !fill_r && mr >= i0 && mr < i0 + 4;
    if (pad_bot || bottom_lane) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int r = mr - i0;
        const f32x2 v = r & 1 ? P1[c][1] : P1[c][0];
        const float pn = pad_bot ? (r >> 1 ? hi2(v) : lo2(v)) : smem[L::PBS + j0 + c];
        const ptrdiff_t e = (ptrdiff_t)a * g.W + c0 + j0 + c;
        if (c < mc - j0) {
          x.SB[e] = fmaf(2.0f, pn, -oldt[BW + c]);
          A.lam_sh[e] = lamt[BW + c];
        }
      }
    }
    if (j0 == 0 && s_lft) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (i0 + r < mr) {
          const ptrdiff_t e = (ptrdiff_t)(b - 1) * g.H + r0 + i0 + r;
          x.SL[e] = fmaf(2.0f, half_of(P2[0][r & 1], r >> 1), -oldl[r]);
          A.lam_tv[e] = laml[r];
        }
    }
    if (PAD && s_rgt && !fill_c && mc >= j0 && mc < j0 + 4) {
      const int q = mc - j0;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const f32x2 v = q == 0 ? P2[0][r & 1] : (q == 1 ? P2[1][r & 1] : (q == 2 ? P2[2][r & 1] : P2[3][r & 1]));
        const ptrdiff_t e = (ptrdiff_t)b * g.H + r0 + i0 + r;
        if (i0 + r < mr) {
          x.SR[e] = fmaf(2.0f, half_of(v, r >> 1), -oldl[BAND + r]);
          A.lam_sv[e] = laml[BAND + r];
        }
      }
    }
    if (right_lane) {
      const ptrdiff_t e = (ptrdiff_t)b * g.H + r0 + rank * BAND + rr;
      x.SR[e] = fmaf(2.0f, pr_s, -smem[CH::OL + BAND + rr]);
      A.lam_sv[e] = smem[CH::LL + BAND + rr];
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int e = r & 1, h = r >> 1, i = i0 + r, gi = r0 + i;
    const int n = i < mr ? mc - j0 : 0;
    const int n1 = i < mr + (s_bot ? 1 : 0) ? mc - j0 : 0;
    const int n2 = i < mr ? mc + (s_rgt ? 1 : 0) - j0 : 0;
    store4(A.u + (size_t)gi * g.W + c0 + j0, n, vec, half_of(U[0][e], h), half_of(U[1][e], h), half_of(U[2][e], h),
           half_of(U[3][e], h));
    const float q0 = half_of(P1[0][e], h), q1 = half_of(P1[1][e], h), q2 = half_of(P1[2][e], h), q3 = half_of(P1[3][e], h);
    store4(A.P1 + (size_t)(gi + a) * g.W + c0 + j0, n1, vec, q0, q1, q2, q3);
    if (r == 0 && i == 0 && s_top) store4(out.ST + (ptrdiff_t)(a - 1) * g.W + c0 + j0, n1, vec_t, q0, q1, q2, q3);
    if (PAD && i == mr && s_bot) store4(out.SB + (size_t)a * g.W + c0 + j0, n1, vec_b, q0, q1, q2, q3);
    store4(A.P2 + (size_t)gi * W2 + c0 + b + j0, n2, false, half_of(P2[0][e], h), half_of(P2[1][e], h),
           half_of(P2[2][e], h), half_of(P2[3][e], h));
    if (j0 == 0 && s_lft && i < mr) out.SL[(size_t)(b - 1) * g.H + gi] = half_of(P2[0][e], h);
    if (PAD && s_rgt && i < mr) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (j0 + c == mc) out.SR[(size_t)b * g.H + gi] = half_of(P2[c][e], h);
    }
  }
  if (right_lane) {
    const int gi = r0 + rank * BAND + rr;
    A.P2[(size_t)gi * W2 + c0 + BW + b] = pr_s;
    out.SR[(size_t)b * g.H + gi] = pr_s;
  }
  if (bottom_lane) {
    const float4 v = *reinterpret_cast<const float4*>(smem + L::PBS + j0);
    store4(A.P1 + (size_t)(r0 + mr + a) * g.W + c0 + j0, mc - j0, vec, v.x, v.y, v.z, v.w);
    store4(out.SB + (size_t)a * g.W + c0 + j0, mc - j0, vec_b, v.x, v.y, v.z, v.w);
  }
}

// all bits set if -1 <= x <= 1 (not for NaN), else 0
__device__ __forceinline__ uint32_t in_box(float x) {
  uint32_t m;
  asm("set.le.u32.f32 %0, %1, 0f3F800000;" : "=r"(m) : "f"(fabsf(x)));
  return m;
}

// Reverse of the K iterations whose tape lies at `tape` (adj_tile.cuh).
template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK>
__device__ __forceinline__ void tile_reverse(const LocalArgs& A, const AdjArgs& Z, const int a, const int b, const int tid,
                                             const int rank, const int CL, const float* tape, const uint32_t in_d,
                                             bool& timed_out);

// The local solve of subdomain (a, b) of the problem A, its interface strips written to
// out, by CTA rank of CL.  CLU: the subdomain is a cluster (else one CTA: rank 0 of 1).
// PAD: the subdomain may be smaller than the block (false: every subdomain fills it).
// ADJ: record the tape (Z->tape) and run the reverse pass instead of the store.
//
// ADAPT: adaptive inner stopping (Section 5, eq. stop_inner1).  Every thread sums (p^{k+1} -
// p^k)^2 and (p^{k+1})^2 over its dofs in the p-step of iteration k (packed float32 pairs) and
// leaves the sums in shared memory.  At the start of iteration k + 1 one warp adds the CTA's
// sums (float32, fixed order) and sends the CTA's pair with st.async to slot `rank` of every
// CTA of the cluster, counted on one of two mbarriers (by the parity of the phase, so that a
// phase is always consumed everywhere before its barrier is armed again).  Before the
// barrier between the u-step and the p-step of iteration k + 1, one warp per CTA waits for the
// pairs and adds them in a fixed tree: every CTA takes the same decision without a cluster
// barrier.  On "stop" the u-step of iteration k + 1 is undone (each iteration first copies u
// to shared memory), its u halo is drained and the p-step is skipped: the solve keeps k + 1
// inner iterations, as the rule prescribes.
//
// CHAIN: the multiplier update is made here as the state is loaded (LocalArgs.chain).
template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK, bool CHAIN = false, bool ADJ = false,
          bool ADAPT = false>
__device__ __forceinline__ void tile_solve(const LocalArgs& A, const Strips out, const int a, const int b,
                                           const int rank, const int CL, const AdjArgs* Z = nullptr) {
  using L = TileLayout<LPR, NW>;
  constexpr int NG = L::NG, BAND = L::BAND, BW = L::BW, NT = L::NT;
  extern __shared__ __align__(128) float smem[];
  float* sUB = smem + L::UB;
  float* sQ1 = smem + L::Q1;
  float* sCo = smem + L::CO;
  const uint32_t mbU = smem_addr(smem + L::MB), mbQ = mbU + 8;
  using AD = AdaptTileLayout<LPR, NW>;
  const uint32_t mbR = smem_addr(smem + AD::MBR);
  static_assert(!ADAPT || (CLU && !PAD && !ADJ && NW > 2), "the adaptive stop: clusters of full blocks");
  // D as words in shared memory in clusters (4096 x 4096 in 128 x 128, L1: 246 -> 239 us), as bits
  // where other arrays need the room and in single CTAs (1024 x 768 in 64 x 64: 20.4 us, with
  // words 22.2: registers)
  constexpr bool kWords = use_mask_words(CLU, MASK, ADJ, ADAPT), kBits = MASK && !kWords;
  constexpr int kDM = MaskTileLayout<LPR, NW>::DM - L::F;
  using CH = ChainTileLayout<LPR, NW, kWords, ADAPT>;

  const Grid g = A.g;
  const int r0 = PAD ? part_start(a, g.H, g.NR) : a * CL * BAND, mr = PAD ? part_start(a + 1, g.H, g.NR) - r0 : CL * BAND;
  const int c0 = PAD ? part_start(b, g.W, g.NC) : b * BW, mc = PAD ? part_start(b + 1, g.W, g.NC) - c0 : BW;
  const bool s_top = a > 0 || g.cut_top, s_bot = a + 1 < g.NR || g.cut_bot, s_lft = b > 0, s_rgt = b + 1 < g.NC;
  const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
  const int G = w * L::RG + l / LPR, cl = l % LPR;  // row group, lane of the group
  const int j0 = 4 * cl;                            // first column in the subdomain
  const int i0 = rank * BAND + 4 * G;               // first row in the subdomain
  const int K = A.K;
  const int W2 = g.W + g.NC;
  const float tau = A.tau;
  const bool fill_c = !PAD || mc == BW, fill_r = !PAD || mr == CL * BAND;  // no padding column / row
  const bool last_group = rank == CL - 1 && G == NG - 1;
  const bool push_down = CLU && G == NG - 1 && rank + 1 < CL;  // u of the band's last row
  const bool push_up = CLU && G == 0 && rank > 0;              // pbar1 of the band's first row
  const bool bottom_lane = fill_r && s_bot && rank == CL - 1 && w == L::kBottomWarp && l < LPR;
  const int rr = tid - L::kRightThread;                        // band row whose right side this thread updates
  const bool right_lane = fill_c && s_rgt && rr >= 0 && rr < BAND && rank * BAND + rr < mr;
  const int r_slot = (rr >> 2) * L::SLOT + 4 * LPR + 2 * (rr & 1) + ((rr >> 1) & 1);
  constexpr uint32_t kHaloBytes = 4 * BW;
  float* const myUR = smem + L::UR + G * L::SLOT + 4 * (cl + 1);
  float* const myQL = smem + L::QL + G * L::SLOT + 4 * cl;
  float* const myF = smem + L::F + 4 * tid;  // column c at + c * 4 NT; the proximal centres likewise
  constexpr int kH1 = L::H1 - L::F, kH2 = L::H2 - L::F;
  // the neighbour's shared memory: every array lies where it does here
  const uint32_t s0 = smem_addr(smem);
  const uint32_t remote = push_down ? map_rank(s0, rank + 1) : (push_up ? map_rank(s0, rank - 1) : 0u);
  pdl_trigger();
  if (CLU) {
    if (tid == 0) {
      mbar_init(mbU, 1);
      mbar_init(mbQ, 1);
      // the first phases, armed before any neighbour may complete them
      if (rank > 0) mbar_arrive_expect_tx(mbU, kHaloBytes);
      if (rank + 1 < CL) mbar_arrive_expect_tx(mbQ, kHaloBytes);
      if (ADAPT) {
        for (int q = 0; q < 2; ++q) {
          mbar_init(mbR + 8 * q, 1);
          mbar_arrive_expect_tx(mbR + 8 * q, 8 * CL);
        }
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    cluster_arrive<true>();  // matched before the first halo is sent: the loads hide the wait
  }
  // the first padding column and row, if this lane holds them
  const bool pad_c = PAD && !fill_c && (mc >> 2) == cl;
  const bool pad_r = PAD && !fill_r && mr >= rank * BAND && ((mr - rank * BAND) >> 2) == G;
  const int cpad = mc & 3, rpad = mr & 3;  // where in the lane's 4 x 4 pixels
  // clamp limits of the dofs of the lane's first row / column: 0 on an image-boundary side
  const float lim_top = (i0 == 0 && !s_top) || (pad_r && rpad == 0 && !s_bot) ? 0.f : 1.f;
  const float lim_left = (j0 == 0 && !s_lft) || (pad_c && cpad == 0 && !s_rgt) ? 0.f : 1.f;

  // pairs [column c][e]: rows (e, e + 2) of column j0 + c
  f32x2 U[4][2], P1[4][2], P2[4][2], Q1[4][2], Q2[4][2];
  uint32_t in_d = 0;  // bit 4c + r: pixel (row r, column j0 + c) lies in the inpainting domain
  float pr_s = 0.f, hr_s = 0.f;

  // ---- load the state, build the proximal centre.  Every load is in flight before the first
  // is used: one latency, not one per array (the loads were 3.8 of 16 us per subdomain).
  const bool coef_smem = K <= L::kMaxSmemCoef;
  if (coef_smem)
    for (int q = tid; q < 16 * K; q += NT)
      cp_async4(sCo + q, reinterpret_cast<const float*>(A.coef) + (q >> 4) * 8 + ((q & 15) >> 1));
  cp_async_commit();
  {
    const bool vec = (g.W & 3) == 0 && (c0 & 3) == 0;
    float h1[4][4], h2[4][4], fv[4][4];
    float u[4][4], p1[4][4], p2[4][4];
    const float* gu = A.u0 + (size_t)(r0 + i0) * g.W + c0 + j0;
    const float* gf = A.f + (size_t)(r0 + i0) * g.W + c0 + j0;
    const float* g1 = A.P10 + (size_t)(r0 + i0 + a) * g.W + c0 + j0;
    const float* g2 = A.P20 + (size_t)(r0 + i0) * W2 + c0 + b + j0;
    const uint8_t* gm = MASK ? A.mask + (size_t)(r0 + i0) * g.W + c0 + j0 : nullptr;
    uint32_t mb[4] = {0, 0, 0, 0};  // mask bytes of the lane's rows
    const bool whole = vec && i0 + 3 < mr && j0 + 3 < mc;
    auto data = [&](int r) {  // f and the mask of a row
      if (whole) {
        load4(gf + (size_t)r * g.W, fv[r]);
        if (MASK) mb[r] = *reinterpret_cast<const uint32_t*>(gm + (size_t)r * g.W);
      } else {
        const int n = i0 + r < mr ? mc - j0 : 0;  // pixels of this lane's row
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          fv[r][c] = c < n ? gf[(size_t)r * g.W + c] : 0.f;
          if (MASK && c < n) mb[r] |= (uint32_t)gm[(size_t)r * g.W + c] << (8 * c);
        }
      }
    };
    auto state = [&](int r) {
      if (whole) {
        load4(gu + (size_t)r * g.W, u[r]);
        load4(g1 + (size_t)r * g.W, p1[r]);
#pragma unroll
        for (int c = 0; c < 4; ++c) p2[r][c] = g2[(size_t)r * W2 + c];
      } else {
        const int i = i0 + r;
        const int n = i < mr ? mc - j0 : 0;
        const int n1 = i < mr + (s_bot ? 1 : 0) ? mc - j0 : 0;             // p1 dofs (row mr: the bottom side)
        const int n2 = i < mr ? mc + (s_rgt ? 1 : 0) - j0 : 0;             // p2 dofs (column mc: the right side)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          u[r][c] = c < n ? gu[(size_t)r * g.W + c] : 0.f;
          p1[r][c] = c < n1 ? g1[(size_t)r * g.W + c] : 0.f;
          p2[r][c] = c < n2 ? g2[(size_t)r * W2 + c] : 0.f;
        }
      }
    };
    // the data, which no launch of the loop writes, before the previous launch has ended; the state
    // and the multipliers after.  (Branches around all rows, so that the loads of a row do not wait
    // for another's.)
    if (whole) {
#pragma unroll
      for (int r = 0; r < 4; ++r) data(r);
    } else {
#pragma unroll
      for (int r = 0; r < 4; ++r) data(r);
    }
    pdl_wait();
    if (whole) {
#pragma unroll
      for (int r = 0; r < 4; ++r) state(r);
    } else {
#pragma unroll
      for (int r = 0; r < 4; ++r) state(r);
    }
    // pbar1 of the row below the band: the next CTA's first row (its halo of later
    // iterations), the bottom side of a subdomain that fills the block, or 0
    const int ib = rank * BAND + BAND;
    const int nb = G == NG - 1 && ib < mr + (s_bot ? 1 : 0) ? mc - j0 : 0;
    const bool bottom_fill = last_group && fill_r && s_bot;
    float qb[4], lb[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) qb[c] = c < nb ? A.P10[(size_t)(r0 + ib + a) * g.W + c0 + j0 + c] : 0.f;
    if (right_lane) pr_s = A.P20[(size_t)(r0 + rank * BAND + rr) * W2 + c0 + BW + b];

    // the multipliers of the sides this lane holds
    const bool top = i0 == 0 && s_top, left = j0 == 0 && s_lft, bot = pad_r && s_bot, rgt = pad_c && s_rgt;
    const bool low = bot || bottom_fill;
    float lt[4], ll[4], lr[4], l_r = 0.f;
    const ptrdiff_t et = (ptrdiff_t)(a - 1) * g.W + c0 + j0, eb = (ptrdiff_t)a * g.W + c0 + j0;
    const ptrdiff_t el = (ptrdiff_t)(b - 1) * g.H + r0 + i0, er = (ptrdiff_t)b * g.H + r0 + i0;
    const ptrdiff_t es = (ptrdiff_t)b * g.H + r0 + rank * BAND + rr;
    if (!CHAIN) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        lt[c] = top && c < mc - j0 ? A.lamh[et + c] : 0.f;
        lb[c] = low && c < mc - j0 ? A.lamh[eb + c] : 0.f;
        ll[c] = left && i0 + c < mr ? A.lamv[el + c] : 0.f;
        lr[c] = rgt && i0 + c < mr ? A.lamv[er + c] : 0.f;
      }
      if (right_lane) l_r = A.lamv[es];
    } else {
      // lambda + sigma (x_s - x_t), on this side's copy (kernels_interface.cu lam_step); branches,
      // so that the warps without a side skip it
      auto step = [&](const float* lam, const float* xs, const float* xt, ptrdiff_t e, int n, float* v, float* keep) {
        float l0[4], s0[4], t0[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          l0[c] = c < n ? lam[e + c] : 0.f;
          s0[c] = c < n ? xs[e + c] : 0.f;
          t0[c] = c < n ? xt[e + c] : 0.f;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = fmaf(A.sigma, s0[c] - t0[c], l0[c]);
        *reinterpret_cast<float4*>(keep) = make_float4(v[0], v[1], v[2], v[3]);
      };
      // (stored to global memory at the end: a store in flight here holds up the first release
      // operation of the loop, 4096 x 4096 343 us per outer iteration instead of 223)
#pragma unroll
      for (int c = 0; c < 4; ++c) lt[c] = lb[c] = ll[c] = lr[c] = 0.f;
      if (top) step(A.lam_th, A.x_in.SB, A.x_in.ST, et, mc - j0, lt, smem + CH::LT + j0);
      if (low) step(A.lam_sh, A.x_in.SB, A.x_in.ST, eb, mc - j0, lb, smem + CH::LT + BW + j0);
      if (left) step(A.lam_tv, A.x_in.SR, A.x_in.SL, el, mr - i0, ll, smem + CH::LL + 4 * G);
      if (PAD && rgt) step(A.lam_sv, A.x_in.SR, A.x_in.SL, er, mr - i0, lr, smem + CH::LL + BAND + 4 * G);
      if (right_lane) {
        l_r = fmaf(A.sigma, A.x_in.SR[es] - A.x_in.SL[es], A.lam_sv[es]);
        smem[CH::LL + BAND + rr] = l_r;
      }
    }
    if (right_lane) hr_s = phat_s(pr_s, l_r, tau);

#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        h1[r][c] = p1[r][c];
        h2[r][c] = p2[r][c];
        if (r == 0 && top) h1[r][c] = phat_t(p1[r][c], lt[c], tau);
        if (PAD && bot && rpad == r) h1[r][c] = phat_s(p1[r][c], lb[c], tau);
        if (c == 0 && left) h2[r][c] = phat_t(p2[r][c], ll[r], tau);
        if (PAD && rgt && cpad == c) h2[r][c] = phat_s(p2[r][c], lr[r], tau);
        if (FID == FID_SEG) fv[r][c] = (fv[r][c] - A.c1) * (fv[r][c] - A.c1) - (fv[r][c] - A.c2) * (fv[r][c] - A.c2);
        const bool d = MASK && ((mb[r] >> (8 * c)) & 0xffu);
        if (kBits && d) in_d |= 1u << (4 * c + r);
        if (kWords && d) fv[r][c] = 0.f;
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        U[c][e] = pk2(u[e][c], u[e + 2][c]);
        Q1[c][e] = P1[c][e] = pk2(p1[e][c], p1[e + 2][c]);
        Q2[c][e] = P2[c][e] = pk2(p2[e][c], p2[e + 2][c]);
      }
      *reinterpret_cast<float4*>(myF + 4 * NT * c) = make_float4(fv[0][c], fv[2][c], fv[1][c], fv[3][c]);
      if (kWords) {
        float m[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const bool d = (mb[r] >> (8 * c)) & 0xffu;
          m[r] = FID == FID_L1 ? (d ? 0.f : 1.f) : __uint_as_float(d ? 0u : ~0u);
        }
        *reinterpret_cast<float4*>(myF + kDM + 4 * NT * c) = make_float4(m[0], m[2], m[1], m[3]);
      }
      *reinterpret_cast<float4*>(myF + kH1 + 4 * NT * c) = make_float4(h1[0][c], h1[2][c], h1[1][c], h1[3][c]);
      *reinterpret_cast<float4*>(myF + kH2 + 4 * NT * c) = make_float4(h2[0][c], h2[2][c], h2[1][c], h2[3][c]);
    }
    if (CHAIN) {  // p~^n of the sides, for their extrapolation at the end
      if (top) *reinterpret_cast<float4*>(smem + CH::OT + j0) = make_float4(p1[0][0], p1[0][1], p1[0][2], p1[0][3]);
      if (bottom_fill) *reinterpret_cast<float4*>(smem + CH::OT + BW + j0) = make_float4(qb[0], qb[1], qb[2], qb[3]);
      if (left) *reinterpret_cast<float4*>(smem + CH::OL + 4 * G) = make_float4(p2[0][0], p2[1][0], p2[2][0], p2[3][0]);
      if (PAD && bot) {
        auto put = [&](int r) { *reinterpret_cast<float4*>(smem + CH::OT + BW + j0) = make_float4(p1[r][0], p1[r][1], p1[r][2], p1[r][3]); };
        if (rpad == 0) put(0);
        else if (rpad == 1) put(1);
        else if (rpad == 2) put(2);
        else put(3);
      }
      if (PAD && rgt) {
        auto put = [&](int c) { *reinterpret_cast<float4*>(smem + CH::OL + BAND + 4 * G) = make_float4(p2[0][c], p2[1][c], p2[2][c], p2[3][c]); };
        if (cpad == 0) put(0);
        else if (cpad == 1) put(1);
        else if (cpad == 2) put(2);
        else put(3);
      }
      if (right_lane) smem[CH::OL + BAND + rr] = pr_s;
    }
    *reinterpret_cast<float4*>(sQ1 + G * BW + j0) = make_float4(p1[0][0], p1[0][1], p1[0][2], p1[0][3]);
    *reinterpret_cast<ulonglong2*>(myQL) = make_ulonglong2(P2[0][0], P2[0][1]);
    if (G == NG - 1) {
      *reinterpret_cast<float4*>(sQ1 + NG * BW + j0) = make_float4(qb[0], qb[1], qb[2], qb[3]);
      if (bottom_fill) {
        *reinterpret_cast<float4*>(smem + L::PBS + j0) = make_float4(qb[0], qb[1], qb[2], qb[3]);
        *reinterpret_cast<float4*>(smem + L::HBS + j0) =
            make_float4(phat_s(qb[0], lb[0], tau), phat_s(qb[1], lb[1], tau), phat_s(qb[2], lb[2], tau),
                        phat_s(qb[3], lb[3], tau));
      }
    }
    if (G == 0 && rank == 0) *reinterpret_cast<float4*>(sUB + j0) = make_float4(0.f, 0.f, 0.f, 0.f);  // u above the tile
    if (cl == 0) *reinterpret_cast<float4*>(smem + L::UR + G * L::SLOT) = make_float4(0.f, 0.f, 0.f, 0.f);  // u left of it
    // the slot right of the last lane: the right side of a subdomain that fills the block, else 0
    if (rr >= 0 && rr < BAND) smem[L::QL + r_slot] = pr_s;
  }
  cp_async_wait_all();
  __syncthreads();
  bool timed_out = false;
  uint32_t phU = 0, phQ = 0;  // index of the next phase of mbU / mbQ this thread waits for
  if (CLU) cluster_wait();  // every CTA's barriers are initialised and armed
  auto wait_u = [&]() {
    if (!mbar_wait(mbU, phU & 1)) timed_out = true;
    ++phU;
    if (cl == 0) mbar_arrive_expect_tx(mbU, kHaloBytes);  // arm the next phase
  };
  auto wait_q = [&]() {
    if (!mbar_wait(mbQ, phQ & 1)) timed_out = true;
    ++phQ;
    if (cl == 0) mbar_arrive_expect_tx(mbQ, kHaloBytes);
  };
  // tape of one CTA, per iteration: 16 NT words of ubar in thread order, NT words of pass bits
  // (bit 4c + r: the p1 dof of row r, column c; bit 16 + 4c + r: p2), NT of the sides that
  // other lanes update; `live`: the bits of active dofs
  float* tape = nullptr;
  uint32_t live = 0;
  if (ADJ) {
    tape = Z->tape + ((size_t)(a * g.NC + b) * CL + rank) * kTapeWords * K * NT;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int i = i0 + (q & 3), j = j0 + (q >> 2);
      if (i < mr + (s_bot ? 1 : 0) && (i > 0 || s_top) && j < mc) live |= 1u << q;
      if (i < mr && j < mc + (s_rgt ? 1 : 0) && (j > 0 || s_lft)) live |= 1u << (16 + q);
    }
  }
  // Two iterations per trip save the moves of the new dual values; with padding or a mask
  // the doubled code no longer fits the registers and the instruction cache (per outer
  // iteration, 2160 x 3840 in 120 x 128 subdomains: 144 us unrolled, 138 not; 4096 x 4096 in
  // 64 x 64: 207 and 219, with a mask 248 and 229).
  int k_run = K;  // inner iterations kept (ADAPT; < K: u of the last u-step undone)
#pragma unroll(PAD || MASK || ADJ || ADAPT ? 1 : 2)
  for (int k = 0; k < K; ++k) {
    // this thread's sums of (p^{k+1} - p^k)^2 and (p^{k+1})^2
    f32x2 SD = 0ull, SP = 0ull;
    auto residual = [&](f32x2 pn, f32x2 po) {
      if (ADAPT) {
        const f32x2 d = sub2(pn, po);
        SD = fma2(d, d, SD);
        SP = fma2(pn, pn, SP);
      }
    };
    if (ADAPT && k > 0) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        *reinterpret_cast<ulonglong2*>(smem + AD::OU + 4 * (NT * c + tid)) = make_ulonglong2(U[c][0], U[c][1]);
      if (w == AD::kReduceWarp) {
        // the CTA's residual sums of iteration k - 1 to every CTA of the cluster
        f32x2 D = 0ull, P = 0ull;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
          const float4 r = *reinterpret_cast<const float4*>(smem + AD::PS + 4 * (l + 32 * q));
          D = add2(D, pk2(r.x, r.y));
          P = add2(P, pk2(r.z, r.w));
        }
        f32x2 v = pk2(lo2(D) + hi2(D), lo2(P) + hi2(P));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = add2(v, __shfl_xor_sync(0xffffffffu, v, o));
        const uint32_t par = (k - 1) & 1;
        if (l < CL)  // lane l to CTA l, slot rank
          st_async_v2(map_rank(s0 + 4 * (AD::RED + 2 * AD::kMaxCL * par + 2 * rank), l), lo2(v), hi2(v),
                      map_rank(mbR + 8 * par, l));
      }
    }
    // (the coefficients of each half-step are loaded when it begins: registers)
    f32x2 SIG, UA, UBc, SS;
    if (coef_smem) {
      const ulonglong2 cf0 = *reinterpret_cast<const ulonglong2*>(sCo + 16 * k);
      const ulonglong2 cf1 = *reinterpret_cast<const ulonglong2*>(sCo + 16 * k + 4);
      SIG = cf0.x, UA = cf0.y, UBc = cf1.x, SS = cf1.y;
    } else {
      const float4 ca = __ldg(reinterpret_cast<const float4*>(A.coef) + 2 * k);
      SIG = pk2(ca.x, ca.x), UA = pk2(ca.y, ca.y), UBc = pk2(ca.z, ca.z), SS = pk2(ca.w, ca.w);
    }
    const Coef cu{lo2(SIG), lo2(UA), lo2(UBc), lo2(SS), 0.f, 0.f, 0.f, 0.f};
    if (push_down && k > 0) wait_q();  // pbar1 halo of iteration k - 1
    // ---- u-step: pair e = 1 (holding the group's last row) first
    {
      const float4 qb = *reinterpret_cast<const float4*>(sQ1 + (G + 1) * BW + j0);  // pbar1 of the row below
      const ulonglong2 qn = *reinterpret_cast<const ulonglong2*>(myQL + 4);         // left edge of the lane to the right
      const f32x2 QRn[2] = {qn.x, qn.y};
      const float qbv[4] = {qb.x, qb.y, qb.z, qb.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const ulonglong2 fc = *reinterpret_cast<const ulonglong2*>(myF + 4 * NT * c);
        ulonglong2 dm = make_ulonglong2(0ull, 0ull);
        if (kWords) dm = *reinterpret_cast<const ulonglong2*>(myF + kDM + 4 * NT * c);
        f32x2 ubar[2];
#pragma unroll
        for (int ee = 0; ee < 2; ++ee) {
          const int e = 1 - ee;
          const f32x2 fg = e == 0 ? fc.x : fc.y;
          // bottom - top: for e = 1 the rows below (2, 4) straddle pair 0 and the group below
          const f32x2 bt = e == 0 ? sub2(Q1[c][1], Q1[c][0])
                                  : pk2(hi2(Q1[c][0]) - lo2(Q1[c][1]), qbv[c] - hi2(Q1[c][1]));
          const f32x2 right = c < 3 ? Q2[c + 1][e] : QRn[e];
          const f32x2 d = sub2(add2(bt, right), Q2[c][e]);  // div_px
          const f32x2 ub = fma2(SIG, d, U[c][e]);
          ubar[e] = ub;
          const bool dl = kBits && ((in_d >> (4 * c + e)) & 1u), dh = kBits && ((in_d >> (4 * c + e + 2)) & 1u);
          const f32x2 de = e == 0 ? dm.x : dm.y;
          f32x2 un;
          if (FID == FID_L2) {
            f32x2 ua = UA;
            if (kWords) ua = (UA & de) | (0x3f8000003f800000ull & ~de);
            un = fma2(UBc, fg, mul2(ua, ub));
            if (kBits) un = pk2(dl ? lo2(ub) : lo2(un), dh ? hi2(ub) : hi2(un));
          } else if (FID == FID_L1) {  // ubar - P_[-s,s](ubar - f)
            f32x2 v = sub2(ub, fg);
            if (kWords) v = mul2(v, de);
            un = sub2(ub, pk2(clamp_abs(lo2(v), cu.s), clamp_abs(hi2(v), cu.s)));
            if (kBits) un = pk2(dl ? lo2(ub) : lo2(un), dh ? hi2(ub) : hi2(un));
          } else {
            un = pk2(prox_ubar<FID>(lo2(ub), lo2(fg), dl, cu), prox_ubar<FID>(hi2(ub), hi2(fg), dh, cu));
          }
          U[c][e] = un;
        }
        if (ADJ)
          *reinterpret_cast<ulonglong2*>(tape + (size_t)k * kTapeWords * NT + 4 * NT * c + 4 * tid) =
              make_ulonglong2(ubar[0], ubar[1]);
      }
      // u of the first padding column and row: 0 where the side is an interface (D_s u =
      // -u), u of the pixel before it where it is the image boundary (D_s u = 0: the dof
      // stays 0; in the lane's first column or row the clamp limit does that)
      if (PAD && pad_c) {
        auto pin = [&](int q) {
#pragma unroll
          for (int e = 0; e < 2; ++e) U[q][e] = s_rgt || q == 0 ? 0ull : U[q > 0 ? q - 1 : 0][e];
        };
        if (cpad == 0) pin(0);
        else if (cpad == 1) pin(1);
        else if (cpad == 2) pin(2);
        else pin(3);
      }
      if (PAD && pad_r) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (rpad == 0) U[c][0] = pk2(0.f, hi2(U[c][0]));
          else if (rpad == 1) U[c][1] = pk2(s_bot ? 0.f : lo2(U[c][0]), hi2(U[c][1]));
          else if (rpad == 2) U[c][0] = pk2(lo2(U[c][0]), s_bot ? 0.f : lo2(U[c][1]));
          else U[c][1] = pk2(lo2(U[c][1]), s_bot ? 0.f : hi2(U[c][0]));
        }
      }
      const float4 ul = make_float4(hi2(U[0][1]), hi2(U[1][1]), hi2(U[2][1]), hi2(U[3][1]));
      if (push_down)
        st_async_v4_f32(remote + 4 * (L::UB + j0), ul.x, ul.y, ul.z, ul.w, remote + 4 * L::MB);
      else if (last_group)
        *reinterpret_cast<float4*>(smem + L::XUB + j0) = ul;  // for the bottom side's update
      if (G < NG - 1) *reinterpret_cast<float4*>(sUB + (G + 1) * BW + j0) = ul;
      *reinterpret_cast<ulonglong2*>(myUR) = make_ulonglong2(U[3][0], U[3][1]);
    }
    if (ADAPT && k > 0 && w == AD::kDecideWarp) {  // on iteration k - 1
      const uint32_t par = (k - 1) & 1;
      if (!mbar_wait(mbR + 8 * par, ((k - 1) >> 1) & 1)) timed_out = true;
      f32x2 v = l < CL ? *reinterpret_cast<const f32x2*>(smem + AD::RED + 2 * AD::kMaxCL * par + 2 * l) : 0ull;
#pragma unroll
      for (int o = AD::kMaxCL / 2; o > 0; o >>= 1) v = add2(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (l == 0) {
        mbar_arrive_expect_tx(mbR + 8 * par, 8 * CL);  // the barrier's next phase
        const float td = lo2(v), tp = hi2(v);
        *reinterpret_cast<int*>(smem + AD::STOP) = (timed_out || tp == 0.f || td < (float)A.inner_tol2 * tp) ? 1 : 0;
      }
    }
    __syncthreads();
    if (ADAPT && k > 0 && *reinterpret_cast<const int*>(smem + AD::STOP)) {
      // keep iterations 0 .. k - 1; the u halo this u-step sent is drained
      k_run = k;
      if (push_up) wait_u();
      break;
    }
    f32x2 PA, PC, PB, TH;
    if (coef_smem) {
      const ulonglong2 cf2 = *reinterpret_cast<const ulonglong2*>(sCo + 16 * k + 8);
      const ulonglong2 cf3 = *reinterpret_cast<const ulonglong2*>(sCo + 16 * k + 12);
      PA = cf2.x, PC = cf2.y, PB = cf3.x, TH = cf3.y;
    } else {
      const float4 cb = __ldg(reinterpret_cast<const float4*>(A.coef) + 2 * k + 1);
      PA = pk2(cb.x, cb.x), PC = pk2(cb.y, cb.y), PB = pk2(cb.z, cb.z), TH = pk2(cb.w, cb.w);
    }
    const Coef co{0.f, 0.f, 0.f, 0.f, lo2(PA), lo2(PC), lo2(PB), lo2(TH)};
    uint32_t bits = 0;
    auto record = [&](f32x2 t, int n) {  // pass bits n (low half) and n + 2 (high half)
      if (ADJ) bits |= (in_box(lo2(t)) & (1u << n)) | (in_box(hi2(t)) & (4u << n));
    };
    // ---- p-step: first the dofs that need no row above the group (in the first group that
    // row is the halo from the CTA above), then the first row's pbar1 and its push upwards
    {
      const ulonglong2 ul = *reinterpret_cast<const ulonglong2*>(myUR - 4);  // right column of the lane to the left
      f32x2 H0[4];  // the proximal centres of rows (0, 2), for the second part
      auto p1_odd = [&](int c, f32x2 h) {  // rows (1, 3)
        const f32x2 tt = fma2(PC, sub2(U[c][1], U[c][0]), fma2(PA, P1[c][1], mul2(PB, h)));  // p_target
        record(tt, 4 * c + 1);
        const f32x2 pn = pk2(clamp_abs(lo2(tt), 1.f), clamp_abs(hi2(tt), 1.f));
        Q1[c][1] = fma2(TH, sub2(pn, P1[c][1]), pn);
        residual(pn, P1[c][1]);
        P1[c][1] = pn;
      };
      auto p2_dof = [&](int c, int e, f32x2 h) {
        const f32x2 leftu = c > 0 ? U[c > 0 ? c - 1 : 0][e] : (e == 0 ? ul.x : ul.y);
        const f32x2 tt = fma2(PC, sub2(U[c][e], leftu), fma2(PA, P2[c][e], mul2(PB, h)));
        record(tt, 16 + 4 * c + e);
        const float ll = c == 0 ? lim_left : 1.f;
        const f32x2 pn = pk2(clamp_abs(lo2(tt), ll), clamp_abs(hi2(tt), ll));
        Q2[c][e] = fma2(TH, sub2(pn, P2[c][e]), pn);
        residual(pn, P2[c][e]);
        P2[c][e] = pn;
      };
      if (!ADAPT) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const ulonglong2 h1 = *reinterpret_cast<const ulonglong2*>(myF + kH1 + 4 * NT * c);
          const ulonglong2 h2 = *reinterpret_cast<const ulonglong2*>(myF + kH2 + 4 * NT * c);
          H0[c] = mul2(PB, h1.x);
          p1_odd(c, h1.y);
          p2_dof(c, 0, h2.x);
          p2_dof(c, 1, h2.y);
        }
      } else {  // the order in which the residuals are summed
#pragma unroll
        for (int c = 0; c < 4; ++c) p2_dof(c, 0, *reinterpret_cast<const f32x2*>(myF + kH2 + 4 * NT * c));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const ulonglong2 h1 = *reinterpret_cast<const ulonglong2*>(myF + kH1 + 4 * NT * c);
          H0[c] = mul2(PB, h1.x);
          p1_odd(c, h1.y);
          p2_dof(c, 1, *reinterpret_cast<const f32x2*>(myF + kH2 + 4 * NT * c + 2));
        }
      }
      *reinterpret_cast<ulonglong2*>(myQL) = make_ulonglong2(Q2[0][0], Q2[0][1]);
      if (push_up) wait_u();  // u halo of iteration k
      const float4 ua = *reinterpret_cast<const float4*>(sUB + G * BW + j0);  // u of the row above
      const float uav[4] = {ua.x, ua.y, ua.z, ua.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        // rows (0, 2): the rows above (-1, 1) straddle the group above and pair 1
        const f32x2 du = pk2(lo2(U[c][0]) - uav[c], hi2(U[c][0]) - lo2(U[c][1]));
        const f32x2 tt = fma2(PC, du, fma2(PA, P1[c][0], H0[c]));
        record(tt, 4 * c);
        const f32x2 pn = pk2(clamp_abs(lo2(tt), lim_top), clamp_abs(hi2(tt), 1.f));
        Q1[c][0] = fma2(TH, sub2(pn, P1[c][0]), pn);
        residual(pn, P1[c][0]);
        P1[c][0] = pn;
      }
      const float4 q = make_float4(lo2(Q1[0][0]), lo2(Q1[1][0]), lo2(Q1[2][0]), lo2(Q1[3][0]));
      if (G > 0) *reinterpret_cast<float4*>(sQ1 + G * BW + j0) = q;
      if (push_up) st_async_v4_f32(remote + 4 * (L::Q1 + NG * BW + j0), q.x, q.y, q.z, q.w, remote + 4 * L::MB + 8);
    }
    uint32_t* const tapeM =
        ADJ ? reinterpret_cast<uint32_t*>(tape) + (size_t)k * kTapeWords * NT + 16 * NT + tid : nullptr;
    if (ADJ) *tapeM = bits & live;
    uint32_t xbits = 0;
    if (right_lane) {  // Du = -u of the last column ((-pc) u = pc (-u) exactly)
      const float tt = fmaf(-co.pc, smem[L::UR + r_slot], fmaf(co.pa, pr_s, co.pb * hr_s));
      if (ADJ) xbits |= in_box(tt) & 1u;
      const float pn = clamp_abs(tt, 1.f);
      smem[L::QL + r_slot] = fmaf(co.th, pn - pr_s, pn);
      residual(pk2(pn, 0.f), pk2(pr_s, 0.f));
      pr_s = pn;
    }
    if (bottom_lane) {  // Du = -u of the last row
      const float4 pv = *reinterpret_cast<const float4*>(smem + L::PBS + j0);
      const float4 hv = *reinterpret_cast<const float4*>(smem + L::HBS + j0);
      const float4 uv = *reinterpret_cast<const float4*>(smem + L::XUB + j0);
      float pB[4] = {pv.x, pv.y, pv.z, pv.w}, qB[4];
      const float hB[4] = {hv.x, hv.y, hv.z, hv.w}, uB[4] = {uv.x, uv.y, uv.z, uv.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (ADJ) xbits |= in_box(p_target(pB[c], -uB[c], hB[c], co)) & (2u << c);
        const float po = pB[c];
        p_update(pB[c], qB[c], -uB[c], hB[c], co);
        residual(pk2(pB[c], 0.f), pk2(po, 0.f));
      }
      *reinterpret_cast<float4*>(smem + L::PBS + j0) = make_float4(pB[0], pB[1], pB[2], pB[3]);
      *reinterpret_cast<float4*>(sQ1 + NG * BW + j0) = make_float4(qB[0], qB[1], qB[2], qB[3]);
    }
    if (ADJ && (right_lane || bottom_lane)) tapeM[NT] = xbits;
    if (ADAPT && k + 1 < K)  // added up at the start of iteration k + 1
      *reinterpret_cast<float4*>(smem + AD::PS + 4 * tid) = make_float4(lo2(SD), hi2(SD), lo2(SP), hi2(SP));
    __syncthreads();
  }
  const bool stopped = ADAPT && k_run < K;
  if (CLU && push_down && !stopped) wait_q();  // drain the last pbar1 halo (not read)
  if (stopped) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(smem + AD::OU + 4 * (NT * c + tid));
      U[c][0] = v.x;
      U[c][1] = v.y;
    }
  }
  if (ADAPT && rank == 0 && tid == 0) {
    A.inner_used[a * g.NC + b] = k_run;
    atomicMax(A.inner_max, k_run);
    atomicAdd(A.inner_work, (unsigned long long)mr * (unsigned long long)mc * (unsigned long long)k_run);
  }
  if constexpr (ADJ) {
    int tid2, a2 = a, b2 = b;  // the geometry again rather than in registers, as below
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid2));
    asm volatile("" : "+r"(a2), "+r"(b2));
    tile_reverse<LPR, NW, CLU, PAD, FID, MASK>(A, *Z, a2, b2, tid2, rank, CL, tape, in_d, timed_out);
    if (CLU) {
      if (timed_out) atomicOr(A.err, 1);
      __syncwarp();
      cluster_wait();
    }
    return;
  }
  if (CLU) {
    __syncwarp();
    cluster_arrive<false>();  // no CTA leaves while a neighbour may still write into it; the
                              // stores below hide the wait
  }

  // ---- store u^{n+1}, p~^{n+1} and the interface strips.  The geometry is worked out again
  // rather than kept in registers through the loop (the asm hides that it is the same).
  int tid2 = tid, a2 = a, b2 = b;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid2));
  asm volatile("" : "+r"(a2), "+r"(b2));
  tile_store<LPR, NW, PAD, CHAIN, CH>(A, out, a2, b2, tid2, CL, rank, U, P1, P2, pr_s);
  if (CLU) {
    if (timed_out) atomicOr(A.err, 1);
    __syncwarp();
    cluster_wait();
  }
}

template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK, bool CHAIN>
__global__ void __launch_bounds__(32 * NW, tile_warps(NW, PAD && CHAIN) / NW) k_tile(const LocalArgs A, const int cl) {
  // block x = CTA x % cl of subdomain x / cl (a 1-D grid: any number of subdomains)
  const unsigned t = CLU ? blockIdx.x / (unsigned)cl : blockIdx.x, rank = CLU ? blockIdx.x - t * (unsigned)cl : 0u;
  const unsigned a = t / (unsigned)A.g.NC;
  tile_solve<LPR, NW, CLU, PAD, FID, MASK, CHAIN>(A, A.out, (int)a, (int)(t - a * (unsigned)A.g.NC), (int)rank, CLU ? cl : 1);
}

// adaptive inner stop, subdomains that fill their block
template <int LPR, int NW, int FID, bool MASK, bool CHAIN>
__global__ void __launch_bounds__(32 * NW, 16 / NW) k_tile_adapt(const LocalArgs A, const int cl) {
  const unsigned t = blockIdx.x / (unsigned)cl, rank = blockIdx.x - t * (unsigned)cl, a = t / (unsigned)A.g.NC;
  tile_solve<LPR, NW, true, false, FID, MASK, CHAIN, false, true>(A, A.out, (int)a, (int)(t - a * (unsigned)A.g.NC), (int)rank, cl);
}

template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK>
cudaError_t prepare_tile_one(bool chain) {
  constexpr bool words = use_mask_words(CLU, MASK, false, false);
  auto set = [](auto kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  const cudaError_t e = set(k_tile<LPR, NW, CLU, PAD, FID, MASK, false>, tile_bytes<LPR, NW, words, false, false>());
  return e != cudaSuccess || !chain
             ? e
             : set(k_tile<LPR, NW, CLU, PAD, FID, MASK, true>, tile_bytes<LPR, NW, words, false, true>());
}

template <int LPR, int NW, bool CLU, bool PAD>
cudaError_t prepare_tile_fid(bool chain) {
  cudaError_t e;
  if ((e = prepare_tile_one<LPR, NW, CLU, PAD, FID_L2, false>(chain)) != cudaSuccess) return e;
  if ((e = prepare_tile_one<LPR, NW, CLU, PAD, FID_L2, true>(chain)) != cudaSuccess) return e;
  if ((e = prepare_tile_one<LPR, NW, CLU, PAD, FID_L1, false>(chain)) != cudaSuccess) return e;
  if ((e = prepare_tile_one<LPR, NW, CLU, PAD, FID_L1, true>(chain)) != cudaSuccess) return e;
  return prepare_tile_one<LPR, NW, CLU, PAD, FID_SEG, false>(chain);
}

// the instances a grid with or without padding reaches, the chained ones if asked for
template <int LPR, int NW, bool CLU>
cudaError_t prepare_tile(bool pad, bool chain) {
  return pad ? prepare_tile_fid<LPR, NW, CLU, true>(chain) : prepare_tile_fid<LPR, NW, CLU, false>(chain);
}

template <int LPR, int NW, bool CLU, bool PAD, int FID, bool MASK>
cudaError_t launch_tile_one(const LocalArgs& a, int cl, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(CLU ? cl : 1) * a.g.NC * a.g.NR, 1, 1);
  cfg.blockDim = dim3(32 * NW, 1, 1);
  constexpr bool words = use_mask_words(CLU, MASK, false, false);
  cfg.dynamicSmemBytes = a.chain ? tile_bytes<LPR, NW, words, false, true>() : tile_bytes<LPR, NW, words, false, false>();
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (a.chain || has_interfaces(a.g)) pdl_attr(&attr[cfg.numAttrs++]);
  if (CLU) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cl;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  return a.chain ? cudaLaunchKernelEx(&cfg, k_tile<LPR, NW, CLU, PAD, FID, MASK, true>, a, cl)
                 : cudaLaunchKernelEx(&cfg, k_tile<LPR, NW, CLU, PAD, FID, MASK, false>, a, cl);
}

template <int LPR, int NW, bool CLU, bool PAD>
cudaError_t launch_tile_fid(const LocalArgs& a, int fid, int cl, cudaStream_t st) {
  const bool m = a.mask != nullptr;
  switch (fid) {
    case FID_L2:
      return m ? launch_tile_one<LPR, NW, CLU, PAD, FID_L2, true>(a, cl, st)
               : launch_tile_one<LPR, NW, CLU, PAD, FID_L2, false>(a, cl, st);
    case FID_L1:
      return m ? launch_tile_one<LPR, NW, CLU, PAD, FID_L1, true>(a, cl, st)
               : launch_tile_one<LPR, NW, CLU, PAD, FID_L1, false>(a, cl, st);
    default: return launch_tile_one<LPR, NW, CLU, PAD, FID_SEG, false>(a, cl, st);
  }
}

template <int LPR, int NW, bool CLU>
cudaError_t launch_tile(const LocalArgs& a, int fid, int cl, bool pad, cudaStream_t st) {
  return pad ? launch_tile_fid<LPR, NW, CLU, true>(a, fid, cl, st) : launch_tile_fid<LPR, NW, CLU, false>(a, fid, cl, st);
}

// Every subdomain of a batch of images (all of them fill their block), CL CTAs each, with
// its image's fidelity, parameters and strips.
template <int LPR, int NW, int CL>
__global__ void __launch_bounds__(32 * NW, 16 / NW) k_tile_batch(const BatchArgs B) {
  const int t = (int)blockIdx.x / CL, rank = (int)blockIdx.x % CL;
  const int img = B.tile_img[t];
  const LocalArgs A = B.args[img];
  const int q = t - B.tile_base[img];
  const int a = q / A.g.NC, b = q - a * A.g.NC;
  const Strips out = B.strips[2 * img + B.write_set];
  switch (B.fid[img]) {
    case FID_L2: tile_solve<LPR, NW, (CL > 1), false, FID_L2, false>(A, out, a, b, rank, CL); break;
    case FID_L1: tile_solve<LPR, NW, (CL > 1), false, FID_L1, false>(A, out, a, b, rank, CL); break;
    default: tile_solve<LPR, NW, (CL > 1), false, FID_SEG, false>(A, out, a, b, rank, CL); break;
  }
}

template <int LPR, int NW, int CL>
cudaError_t prepare_tile_batch() {
  return cudaFuncSetAttribute(k_tile_batch<LPR, NW, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)TileLayout<LPR, NW>::BYTES);
}

template <int LPR, int NW, int CL>
cudaError_t launch_tile_batch(const BatchArgs& B, int total_tiles, bool overlap, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL * total_tiles, 1, 1);
  cfg.blockDim = dim3(32 * NW, 1, 1);
  cfg.dynamicSmemBytes = TileLayout<LPR, NW>::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (overlap) pdl_attr(&attr[cfg.numAttrs++]);
  if (CL > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = CL;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  return cudaLaunchKernelEx(&cfg, k_tile_batch<LPR, NW, CL>, B);
}

}  // namespace
}  // namespace ddtv
