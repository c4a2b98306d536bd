// gwl_fused.cuh -- the mixed likelihood of a small group of rows on one CTA:
// coefficients, bin sums and combination with nothing passed through global
// memory.
//
// A CTA of eight warps owns up to 32 rows of theta.  Its warps first play the
// parts of the float-float prologue (eight parts instead of the four of
// k_prologue, so that no warp's dependent chain holds two elementary
// functions in a row where they are independent), while the table rows of the
// first windows are being copied into shared memory; then all threads form
// the anchor terms of the rows' 32-bin blocks, one (row, block) per thread;
// then warps take (row, window) items, longest rows first, and sum them with
// the lane and block order of k_window, so that every FP32 sum has the bits
// that k_window gives; then the windows' sums are added in window order and
// combined in FP64, one row per thread.
//
// Against the separate clearing, prologue and bin-loop kernels this takes out
// two launches with the waits between them, the coefficient records' way
// through L2, the global claim counters with their ~1 us round trips, two
// thirds of the anchor work (a short row has 10-19 blocks, and k_window gives
// each row's blocks a whole warp) and, by the folded warp reduction below,
// half of the reduction's instructions.
#pragma once

#include "gwl_bins.cuh"
#include "gwl_ff.cuh"

namespace gwl {

constexpr int kFusedRows = 32;  // rows per CTA at most (one per lane in the prologue)

// Anchor record of a (row, block): the anchor terms of the detectors, then a
// flag (nonzero: the block takes the FP32 delta), in 8- or 16-byte units.
__host__ __device__ constexpr int anchor_rec_floats(int ndet) { return ndet == 1 ? 2 : ndet <= 3 ? 4 : 8; }

// Where the parts of a CTA's dynamic shared memory begin (floats).
struct FusedLayout {
  int anchor;   // anchor rows of the staged windows (the table rows begin at 0)
  int cal;      // calibration rows
  int rec;      // anchor records [R][blocks]
  int part;     // FP32 sums [R][windows][S NDET]
  int total;
};

__host__ __device__ inline FusedLayout fused_layout(int ndet, int cal_row, int CH, int nwc, int R) {
  FusedLayout l;
  const int bins = CH * nwc, blocks = (CH + kAnchor - 1) / kAnchor * nwc;
  l.anchor = blocks * block_floats(ndet);
  l.cal = l.anchor + blocks * kAnchorRowFloats;
  l.rec = l.cal + (cal_row ? (bins + 2) * cal_row : 0);  // calibration rows are staged in pairs
  l.rec = (l.rec + 3) & ~3;
  l.part = l.rec + R * blocks * anchor_rec_floats(ndet);
  l.total = l.part + R * nwc * (cal_row ? 3 : 2) * ndet;
  return l;
}

// One event's tables and launch shape, as the group's code needs them.
struct FusedArgs {
  SegInfo seg;
  const float* tab;     // blocked table (FP32-delta bins)
  const float* low;     // blocked low parts, read in place by the blocks with float-float deltas
  const float* anchor;  // anchor rows
  int CH;               // bins per window (a multiple of 32)
  int nwc;              // windows staged together
  float df;
  // calibration model (instances with CAL only)
  const float* cal;
  int cal_row;
  int cal_par;          // first calibration parameter of a row
  int nn;
  const float* calQ;
  int* status;
  unsigned long long* ffc;  // diagnostic counter of float-float-delta blocks, or null
};

// The context's tables and window as such arguments, and a group's dynamic
// shared memory (gwl_fused.cu).
FusedArgs fused_args(const gwl_ctx* c, int nwc);
size_t fused_bytes(const gwl_ctx* c, int nwc, int R);

// The group's warps are the first NW of the CTA's (8 or 16; the coefficients
// use eight, the bin sums all); other warps of the CTA take no part, so the
// group has a barrier of its own.
template <int NW>
__device__ __forceinline__ void group_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * NW) : "memory");
}

// Static shared memory of a group.
template <int NDET, bool CAL, int NW>
struct FusedSmem {
  static constexpr int NS = (CAL ? 3 : 2) * NDET;  // sums per row
  FF lmc[kFusedRows], leta[kFusedRows], eta[kFusedRows], amp[kFusedRows];
  FF phi[6][kFusedRows];
  FF sky[4][kFusedRows], ori[3][kFusedRows];
  FF P[2 * NDET][kFusedRows], ang[2][kFusedRows], hterm[NDET][kFusedRows];
  double Kr[NDET][kFusedRows], Ki[NDET][kFusedRows];
  double acc[NS][kFusedRows];  // sums over the window groups before the last one
  PropMixed pm[kFusedRows];
  int ncut[kFusedRows], flag[kFusedRows];
  int order[kFusedRows];  // rows by descending cut
  int next, maxcut, fail;
  alignas(8) uint64_t bar;
  alignas(16) float4 nodes[CAL ? NW * NDET * kMaxCalNodes : 1];
};

// One thread: the table rows (and anchor and calibration rows) of windows
// [w0, w0 + nwc) into shared memory, completing on the group's barrier.
template <int NDET, bool CAL>
__device__ __forceinline__ void fused_stage(const FusedArgs& a, const FusedLayout& L, float* dyn, int w0,
                                            uint64_t* bar) {
  const int64_t j0 = (int64_t)w0 * a.CH;
  int64_t j1 = j0 + (int64_t)a.nwc * a.CH;
  if (j1 > a.seg.M) j1 = a.seg.M;
  const int n = (int)(j1 - j0), nb = (n + kAnchor - 1) / kAnchor;
  const uint32_t bytes = (uint32_t)nb * (uint32_t)(block_floats(NDET) * 4);
  const uint32_t abytes = (uint32_t)nb * (uint32_t)(kAnchorRowFloats * 4);
  const uint32_t cbytes = CAL ? (uint32_t)((n + 1) & ~1) * (uint32_t)a.cal_row * 4u : 0u;
  mbar_arrive_expect_tx(bar, bytes + abytes + cbytes);
  bulk_g2s(dyn, a.tab + j0 / kAnchor * block_floats(NDET), bytes, bar);
  bulk_g2s(dyn + L.anchor, a.anchor + (j0 / kAnchor) * kAnchorRowFloats, abytes, bar);
  if constexpr (CAL) bulk_g2s(dyn + L.cal, a.cal + j0 * a.cal_row, cbytes, bar);
}

// The quadratics in eta of the PN coefficients (pn_coeffs in gwl_device.cuh),
// a + b eta + c eta^2, summed in that order: of p4, gamma, p6, and the three of
// p7 (its non-spinning part, its chi_s and its delta chi_a factors).
constexpr int kPnP4 = 0, kPnGam = 1, kPnP6 = 2, kPnP7 = 3, kPnP7s = 4, kPnP7a = 5;
static __constant__ FF kPnQuad[6][3] = {
    {ffc(3058673.0 / 1016064.0), ffc(5429.0 / 1008.0), ffc(617.0 / 144.0)},
    {ffc(732985.0 / 2268.0), ffc(-(24260.0 / 81.0)), ffc(-(340.0 / 9.0))},
    {ffc(11583231236531.0 / 4694215680.0 - (640.0 / 3.0) * kPi * kPi - (6848.0 / 21.0) * kGammaE),
     ffc(-15737765635.0 / 3048192.0 + (2255.0 / 12.0) * kPi * kPi), ffc(76055.0 / 1728.0)},
    {ffc(77096675.0 / 254016.0), ffc(378515.0 / 1512.0), ffc(-(74045.0 / 756.0))},
    {ffc(-25150083775.0 / 3048192.0), ffc(10566655595.0 / 762048.0), ffc(-(1042165.0 / 3024.0))},
    {ffc(-25150083775.0 / 3048192.0), ffc(26804935.0 / 6048.0), ffc(-(1985.0 / 48.0))}};
static __device__ __noinline__ FF pn_quad(FF eta, FF eta2, int k) {
  return (kPnQuad[k][0] + eta * kPnQuad[k][1]) + eta2 * kPnQuad[k][2];
}
// eta = q / (1 + q)^2 and delta = (1 - q) / (1 + q).
static __device__ __noinline__ FF pn_eta(FF q) {
  const FF opq = q + 1.0;
  return q / (opq * opq);
}
static __device__ __noinline__ FF pn_delta(FF q) { return (1.0 - q) / (q + 1.0); }

// The coefficients of rows 0 .. R-1, th(k, lane) giving parameter k of the
// lane's row and out(lane) whether the row is refused whatever its parameters
// (both called only for lanes below R): the arithmetic of prologue_rows_ff,
// operation by operation, on the first eight warps, no chain longer than it
// must be.  K_d and the <h|h> terms are left to fused_amplitudes.  Ends with a
// barrier after which pm, ncut, flag and maxcut are in place; warp 7 then sorts
// the rows, without a barrier after it.
//   part 0: ln(pi Mc T_sun); c_m           part 4: dec, H prefetch; response and delay of detector 0
//   part 1: PN orders 2-4; amplitude       part 5: psi, PN order 5; ... of detector 1
//   part 2: ln eta; K's phase angle        part 6: iota, checks; ... of detector 2
//   part 3: ra, PN order 6; cut            part 7: PN order 7; ... of detector 3
// What bounds it is the fetching of its code (each warp runs straight-line code
// once per launch or step), so the elementary functions, the division and the
// quadratics are out of line.
template <int NDET, bool CAL, int NW, class Th, class Out>
__device__ __forceinline__ void fused_coeffs(const SegInfo& s, int R, FusedSmem<NDET, CAL, NW>& sm, Th th, Out out) {
  const int part = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool valid = lane < R;
  // ---- phase 1
  if (part == 0) {
    const double mc = valid ? th(0) : 10.0;
    sm.lmc[lane] = log(ff_from(mc) * (kPi * kTsun));
  } else if (part == 2) {
    const FF eta = pn_eta(ff_from(valid ? th(1) : 0.5));
    sm.eta[lane] = eta;
    sm.leta[lane] = log(eta);
    sm.order[lane] = lane;
  } else if (part < 8) {
    if (part >= 3 && part < 7) {  // the sine and cosine of one angle
      const double x = valid ? (part == 3 ? th(7) : part == 4 ? th(8) : part == 5 ? th(6) : th(5)) : 0.0;
      FF f = ff_from(x);
      if (part == 3) f = f - s.gmst;
      FF sn, cs;
      sincos(f, &sn, &cs);
      FF* o = part == 3 ? &sm.sky[0][lane] : part == 4 ? &sm.sky[2][lane] : part == 5 ? &sm.ori[0][lane] : nullptr;
      if (part < 6) {
        o[0] = sn;
        o[kFusedRows] = cs;
      } else {
        sm.ori[2][lane] = cs;
      }
    }
    if (part == 4) {
      if (valid) prefetch_cut_H(s, th(0), th(1));
    } else if (part == 6) {
      double x[11];
#pragma unroll
      for (int k = 0; k < 11; ++k) x[k] = valid ? th(k) : 1.0;
      sm.flag[lane] = valid && physical_bits(x) && !out(lane) ? 0 : 1;
    } else {  // parts 1, 3, 5, 7: the PN coefficients, as pn_coeffs forms them
      const FF q = ff_from(valid ? th(1) : 0.5), chi1 = ff_from(valid ? th(2) : 0.0),
               chi2 = ff_from(valid ? th(3) : 0.0);
      const FF eta = pn_eta(q), eta2 = eta * eta;
      if (part == 1) {
        const FF x1 = 1.0 / (q + 1.0), x2 = q * x1;
        const FF beta = ((113.0 / 12.0) * x1 * x1 + 6.25 * eta) * chi1 + ((113.0 / 12.0) * x2 * x2 + 6.25 * eta) * chi2;
        sm.phi[0][lane] = (743.0 / 336.0 + (11.0 / 4.0) * eta) * (20.0 / 9.0);
        sm.phi[1][lane] = 4.0 * beta - 16.0 * kPi;
        sm.phi[2][lane] = pn_quad(eta, eta2, kPnP4) * 10.0 - (10.0 * 79.0 / 8.0) * eta * chi1 * chi2;
      } else {
        const FF delta = pn_delta(q), chis = (chi1 + chi2) * 0.5, chia = (chi1 - chi2) * 0.5;
        if (part == 5) {
          const FF gam = pn_quad(eta, eta2, kPnGam) * chis + ((140.0 / 9.0) * eta + 732985.0 / 2268.0) * delta * chia;
          sm.phi[3][lane] = kPi * (38645.0 / 756.0 - (65.0 / 9.0) * eta) - gam;
        } else if (part == 3) {
          sm.phi[4][lane] = pn_quad(eta, eta2, kPnP6) - (127825.0 / 1296.0) * eta2 * eta +
                            kPi * ((2270.0 / 3.0) * delta * chia + ((2270.0 / 3.0) - 520.0 * eta) * chis);
        } else {
          sm.phi[5][lane] = kPi * pn_quad(eta, eta2, kPnP7) +
                            (pn_quad(eta, eta2, kPnP7s) + (5345.0 / 36.0) * eta2 * eta) * chis +
                            delta * pn_quad(eta, eta2, kPnP7a) * chia;
        }
      }
    }
  }
  group_sync<NW>();
  // ---- phase 2
  if (part == 0) {
    Scale<FF> S;
    S.la = sm.lmc[lane] - 0.6 * sm.leta[lane];
    S.a13 = exp(S.la * (1.0 / 3.0));
    S.amp = ff(0.0f);
    PNCoeffs<FF> P;
    P.eta = sm.eta[lane];
    P.p2 = sm.phi[0][lane];
    P.p3 = sm.phi[1][lane];
    P.p4 = sm.phi[2][lane];
    P.p5c = sm.phi[3][lane];
    P.p6c = sm.phi[4][lane];
    P.p7 = sm.phi[5][lane];
    FF c[kNBasis], ccyc;
    basis_coeffs(P, S, c, ccyc);
    const bool ok = sm.flag[lane] == 0;
#pragma unroll
    for (int m = 0; m < kNBasis; ++m) {
      sm.pm[lane].ch[m] = ok ? c[m].hi : 0.0f;
      sm.pm[lane].cl[m] = ok ? c[m].lo : 0.0f;
    }
  } else if (part == 1) {
    const double dl = valid ? th(4) : 100.0;
    sm.amp[lane] = exp((sm.lmc[lane] - kLnPi) * (5.0 / 6.0)) * s.amp_c_ff / ff_from(dl);
  } else if (part == 2) {
    // the same constant-phase cycles as basis_coeffs forms in part 0
    const double phic = valid ? th(10) : 0.0;
    const FF la = sm.lmc[lane] - 0.6 * sm.leta[lane];
    const FF ccyc = const_cycles(cycles_pref(sm.eta[lane]), sm.phi[3][lane], la);
    FF sa, ca;
    sincos(ff_from(phic) + 0.25 * kPi - (2.0 * kPi) * frac_near(ccyc), &sa, &ca);
    sm.ang[0][lane] = sa;
    sm.ang[1][lane] = ca;
  } else if (part == 3) {
    const FF la = sm.lmc[lane] - 0.6 * sm.leta[lane];
    const FF a13 = exp(la * (1.0 / 3.0));
    int ncut = 0;
    if (sm.flag[lane] == 0) {
      ncut = (int)s.M;
      if (s.fcut_mode == 0) ncut = count_bins_le(s, ff_to_double(1.0 / (kSix32 * (a13 * a13 * a13))));
    }
    sm.ncut[lane] = ncut;
    const int nm = __reduce_max_sync(0xffffffffu, ncut);
    if (lane == 0) sm.maxcut = nm;
  } else if (part - 4 < NDET) {
    const int d = part - 4;
    const bool ok = sm.flag[lane] == 0;
    Sky<FF> k;
    k.sl = sm.sky[0][lane];
    k.cl = sm.sky[1][lane];
    k.sd = sm.sky[2][lane];
    k.cd = sm.sky[3][lane];
    const FF tau = delay_vc(ff_from(valid ? th(9) : 0.0), k, s.vtx_c_ff[d]);
    sm.pm[lane].th[d] = ok ? tau.hi : 0.0f;
    sm.pm[lane].tl[d] = ok ? tau.lo : 0.0f;
    FF Pr, Pi;
    response(k, sm.ori[0][lane], sm.ori[1][lane], sm.ori[2][lane], s.geom_ff[d], Pr, Pi);
    sm.P[2 * d][lane] = Pr;
    sm.P[2 * d + 1][lane] = Pi;
  }
  group_sync<NW>();
  // rows by descending cut, where warps take more than one row
  if (part == 7 && R > NW) {
    const int n = valid ? sm.ncut[lane] : -1;
    int rank = 0;
#pragma unroll 4
    for (int l = 0; l < 32; ++l) {
      const int m = __shfl_sync(0xffffffffu, n, l);
      rank += (m > n || (m == n && l < lane)) ? 1 : 0;
    }
    sm.order[rank] = lane;
  }
}

// K_d and the <h|h> term of detector d, one row per lane (one warp; after
// fused_coeffs).
template <int NDET, bool CAL, int NW>
__device__ __forceinline__ void fused_amplitudes(const SegInfo& s, FusedSmem<NDET, CAL, NW>& sm, int d, int lane) {
  const int ncut = sm.ncut[lane];
  const double H = ncut > 0 ? s.H[(int64_t)d * s.M + ncut - 1] : 0.0;
  const FF amp = sm.amp[lane], Pr = sm.P[2 * d][lane], Pi = sm.P[2 * d + 1][lane];
  const FF sa = sm.ang[0][lane], ca = sm.ang[1][lane];
  const FF kr = amp * (Pr * ca - Pi * sa), ki = amp * (Pr * sa + Pi * ca);
  sm.Kr[d][lane] = ff_to_double(kr);
  sm.Ki[d][lane] = ff_to_double(ki);
  sm.hterm[d][lane] = (kr * kr + ki * ki) * ff_from(H);
}

// The anchor record of a (row, block): the row's anchor terms at the block's
// anchor row ra, and whether the block takes the FP32 delta.
template <int NDET>
__device__ __forceinline__ void anchor_record(const PropMixed& P, const float* __restrict__ ra, float* __restrict__ o) {
  float ch[kNBasis], cl[kNBasis], th[NDET], tl[NDET], an[NDET];
#pragma unroll
  for (int m = 0; m < kNBasis; ++m) {
    ch[m] = P.ch[m];
    cl[m] = P.cl[m];
  }
#pragma unroll
  for (int d = 0; d < NDET; ++d) {
    th[d] = P.th[d];
    tl[d] = P.tl[d];
  }
  const bool fast = anchor_terms<NDET>(ra, ch, cl, th, tl, an);
#pragma unroll
  for (int d = 0; d < NDET; ++d) o[d] = an[d];
  o[NDET] = fast ? 1.0f : 0.0f;
}

// Warp sums of n FP32 values per lane with the tree of an xor butterfly over
// 16, 8, 4, 2, 1: at each level a lane keeps one half of its values and hands
// the other half to its partner, so that value v is added up by the lanes
// whose upper lane bits spell v, with the same operand pairs, hence the same
// bits, as the butterfly of every value on every lane (n <= 16; 9 shuffles
// instead of 30 for six values).  The result of value v is returned on lanes
// [v W, v W + W), W = 32 / P, P the power of two at or above n.
template <int N>
struct FoldP {
  static constexpr int P = N <= 2 ? 2 : N <= 4 ? 4 : N <= 8 ? 8 : 16;
  static constexpr int W = 32 / P;
};
template <int N>
__device__ __forceinline__ float warp_fold(const float (&v)[N], int lane) {
  constexpr int P = FoldP<N>::P;
  float t[P];
#pragma unroll
  for (int k = 0; k < P; ++k) t[k] = k < N ? v[k] : 0.0f;
  int off = 16;
#pragma unroll
  for (int h = P / 2; h >= 1; h >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const float send = up ? t[k] : t[k + h];
      const float keep = up ? t[k + h] : t[k];
      t[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (; off >= 1; off >>= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], off);
  return t[0];
}

// The part of a row's coefficients that its bins use, and its running sums.
template <int NDET>
struct RowState {
  float ch[kNBasis], dtl[NDET];
  float U[NDET], V[NDET], X[NDET];
  __device__ __forceinline__ void start(const PropMixed& P, float df, int lane) {
#pragma unroll
    for (int q = 0; q < kNBasis / 4; ++q)
      *reinterpret_cast<float4*>(&ch[4 * q]) = reinterpret_cast<const float4*>(P.ch)[q];
    const float lane_df = (float)lane * df;
#pragma unroll
    for (int d = 0; d < NDET; ++d) {
      dtl[d] = __fmul_rn(P.th[d], lane_df);
      U[d] = V[d] = X[d] = 0.0f;
    }
  }
  // The lane's anchor terms of the block with anchor record rec; whether the block takes the FP32 delta.
  __device__ __forceinline__ bool record(const float* __restrict__ rec, float (&ad)[NDET]) const {
    constexpr int AR = anchor_rec_floats(NDET);
    float r[AR];
    if constexpr (AR == 2) {
      *reinterpret_cast<float2*>(r) = *reinterpret_cast<const float2*>(rec);
    } else {
#pragma unroll
      for (int q = 0; q < AR / 4; ++q)
        *reinterpret_cast<float4*>(&r[4 * q]) = *reinterpret_cast<const float4*>(rec + 4 * q);
    }
#pragma unroll
    for (int d = 0; d < NDET; ++d) ad[d] = __fadd_rn(r[d], dtl[d]);
    return r[NDET] != 0.0f;
  }
};

// FP32 sums of one row over blocks [b, bend) of its bins [jl, jl + n) of the
// staged windows (jl a multiple of 32, in bins from the first staged one; j0
// that one's index in the segment): the blocks in order, lanes over a block's
// bins, as anchored_sums_cal.  cal: the staged windows' calibration rows.  A:
// the segment's low parts (low), df, cal_row and ffc.
template <int NDET, bool CAL, class A>
__device__ __forceinline__ void fused_row_blocks(const A& a, const float* __restrict__ dyn, const float* __restrict__ cal,
                                                 const PropMixed& P, RowState<NDET>& R, const float* __restrict__ rec,
                                                 int j0, int jl, int n, int b, int bend, int lane,
                                                 const float4* __restrict__ nodes) {
  constexpr int RX = 4 * ((kNBasis + 2 * NDET + 3) / 4);
  constexpr int LO = kNBasis + 2 * NDET, RXF = 4 * ((LO + kNBasis + 3) / 4);
  constexpr int AR = anchor_rec_floats(NDET);
  constexpr int BF = block_floats(NDET);
  const float* row = dyn + (jl / kAnchor + b) * BF + 4 * lane;
  const float* crow = CAL ? cal + (jl + b * kAnchor + lane) * a.cal_row : nullptr;
  const int cstep = CAL ? kAnchor * a.cal_row : 0;
  CalBin<NDET, float> cb0, cb1;
  while (b < bend) {
    float ad0[NDET], ad1[NDET];
    bool f0 = R.record(rec + AR * b, ad0);
    while (f0 && b + 2 <= bend && (b + 2) * kAnchor <= n && R.record(rec + AR * (b + 1), ad1)) {
      // two complete blocks with FP32 deltas, in straight-line code so that their chains interleave; a loop of
      // its own, with the next pair's first record read at its end (against one loop over pairs and single
      // blocks: 8 s, every row in all 13 windows, 8192 rows 210 -> 203 us; 16 s BNS, 2 detectors 349 -> 330)
      float v0[RX], v1[RX];
#pragma unroll
      for (int k = 0; k < RX / 4; ++k) {
        *reinterpret_cast<float4*>(&v0[4 * k]) = reinterpret_cast<const float4*>(row)[kAnchor * k];
        *reinterpret_cast<float4*>(&v1[4 * k]) = reinterpret_cast<const float4*>(row + BF)[kAnchor * k];
      }
      if constexpr (CAL) {
        cal_eval<NDET>(crow, nodes, cb0);
        cal_eval<NDET>(crow + cstep, nodes, cb1);
      }
      bin_anchor<NDET, CAL>(v0, R.ch, ad0, R.U, R.V, cb0, R.X);
      bin_anchor<NDET, CAL>(v1, R.ch, ad1, R.U, R.V, cb1, R.X);
      b += 2;
      row += 2 * BF;
      if (CAL) crow += 2 * cstep;
      if (b >= bend) return;
      f0 = R.record(rec + AR * b, ad0);
    }
    if (b * kAnchor + lane < n) {  // lanes past the cut sit out
      if constexpr (CAL) cal_eval<NDET>(crow, nodes, cb0);
      float v[RX];
#pragma unroll
      for (int k = 0; k < RX / 4; ++k)
        *reinterpret_cast<float4*>(&v[4 * k]) = reinterpret_cast<const float4*>(row)[kAnchor * k];
      if (f0) {
        bin_anchor<NDET, CAL>(v, R.ch, ad0, R.U, R.V, cb0, R.X);
      } else {
        if (a.ffc && lane == 0) atomicAdd(a.ffc, 1ull);
        float x[RXF], cl[kNBasis], lo[kNBasis];
#pragma unroll
        for (int q = 0; q < kNBasis / 4; ++q)
          *reinterpret_cast<float4*>(&cl[4 * q]) = reinterpret_cast<const float4*>(P.cl)[q];
        const float4* low = reinterpret_cast<const float4*>(a.low + (int64_t)((j0 + jl) / kAnchor + b) * kLowFloats) + lane;
#pragma unroll
        for (int k = 0; k < kLowUnits; ++k) *reinterpret_cast<float4*>(&lo[4 * k]) = __ldg(low + kAnchor * k);
#pragma unroll
        for (int k = 0; k < RXF; ++k) x[k] = k < LO ? v[k] : k < LO + kNBasis ? lo[k - LO] : 0.0f;
        bin_anchor_exact<NDET, CAL>(x, R.ch, cl, ad0, R.U, R.V, cb0, R.X);
      }
    }
    b += 1;
    row += BF;
    if (CAL) crow += cstep;
  }
}

// All blocks of a row's bins [jl, jl + n).
template <int NDET, bool CAL, class A>
__device__ __forceinline__ void fused_row_sums(const A& a, const float* __restrict__ dyn, const float* __restrict__ cal,
                                               const PropMixed& P, const float* __restrict__ rec, int j0, int jl, int n,
                                               int lane, const float4* __restrict__ nodes, RowState<NDET>& R) {
  R.start(P, a.df, lane);
  fused_row_blocks<NDET, CAL>(a, dyn, cal, P, R, rec, j0, jl, n, 0, (n + kAnchor - 1) / kAnchor, lane, nodes);
}

// The sums of NR rows over the first n[k] bins of a staged window by one warp,
// without calibration: blocks that are complete and take the FP32 delta for
// every row read the table once for all of them, the others row by row, so
// that each row's blocks keep their order.  rec[k]: row k's anchor records.
template <int NDET, int NR, class A>
__device__ __forceinline__ void fused_shared_sums(const A& a, const float* __restrict__ dyn,
                                                  const PropMixed* (&P)[NR], const float* (&rec)[NR], int j0, int (&n)[NR],
                                                  int lane, RowState<NDET> (&R)[NR]) {
  constexpr int RX = 4 * ((kNBasis + 2 * NDET + 3) / 4), AR = anchor_rec_floats(NDET), BF = block_floats(NDET);
  int full = n[0] / kAnchor, end = 0;  // blocks complete in every row; blocks of the longest row
#pragma unroll
  for (int k = 0; k < NR; ++k) {
    R[k].start(*P[k], a.df, lane);
    full = n[k] / kAnchor < full ? n[k] / kAnchor : full;
    const int e = (n[k] + kAnchor - 1) / kAnchor;
    end = e > end ? e : end;
  }
  int b = 0;
  while (b < end) {
    const float* row = dyn + b * BF + 4 * lane;
    for (; b < full; ++b, row += BF) {
      float ad[NR][NDET];
      bool fast = true;
#pragma unroll
      for (int k = 0; k < NR; ++k) fast &= R[k].record(rec[k] + AR * b, ad[k]);
      if (!fast) break;
      float v[RX];
#pragma unroll
      for (int k = 0; k < RX / 4; ++k)
        *reinterpret_cast<float4*>(&v[4 * k]) = reinterpret_cast<const float4*>(row)[kAnchor * k];
      CalBin<NDET, float> none;
#pragma unroll
      for (int k = 0; k < NR; ++k) bin_anchor<NDET, false>(v, R[k].ch, ad[k], R[k].U, R[k].V, none, R[k].X);
    }
    int e = b;  // up to the next block that all rows share, or to the end
    for (; e < full; ++e) {
      bool fast = true;
#pragma unroll
      for (int k = 0; k < NR; ++k) fast &= rec[k][AR * e + NDET] != 0.0f;
      if (fast) break;
    }
    if (e >= full) e = end;
    if (b == e) break;
#pragma unroll 1
    for (int k = 0; k < NR; ++k) {  // row 0, then the rows move up: one copy of the code
      const int ek = (n[0] + kAnchor - 1) / kAnchor;
      fused_row_blocks<NDET, false>(a, dyn, nullptr, *P[0], R[0], rec[0], j0, 0, n[0], b, e < ek ? e : ek, lane, nullptr);
      const PropMixed* p0 = P[0];
      const float* rec0 = rec[0];
      const int n0 = n[0];
      const RowState<NDET> R0 = R[0];
#pragma unroll
      for (int q = 0; q + 1 < NR; ++q) {
        P[q] = P[q + 1];
        rec[q] = rec[q + 1];
        n[q] = n[q + 1];
        R[q] = R[q + 1];
      }
      P[NR - 1] = p0;
      rec[NR - 1] = rec0;
      n[NR - 1] = n0;
      R[NR - 1] = R0;
    }
    b = e;
  }
}

// Bin sums of the group's rows (all its threads; fused_coeffs before it): the
// windows in groups of nwc, each staged unless it is in place, its anchor
// records, its items.  The first items are the detectors' amplitudes, the
// others (row, window) pairs.  The windows' sums of every group but the last
// are added to sm.acc in window order; the last group's are left in place for
// fused_combine.  st: the group that shared memory holds.  crow(r): the
// calibration parameters of row r.  Ends without a barrier after the last
// items; returns false when a bounded wait ran out (the same on every thread).
struct FusedStage {
  int w0 = 0;             // first window of the group in shared memory
  bool pending = true;    // its copy is in flight (the caller has started the first one)
  uint32_t parity = 0;    // the barrier's phase
};

template <int NDET, bool CAL, int NW, class Crow>
__device__ __forceinline__ bool fused_bins(const FusedArgs& a, const FusedLayout& L, float* dyn, int R,
                                           FusedSmem<NDET, CAL, NW>& sm, FusedStage& st, Crow crow) {
  constexpr int NS = FusedSmem<NDET, CAL, NW>::NS, AR = anchor_rec_floats(NDET);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int gbins = a.CH * a.nwc, gblk = (a.CH + kAnchor - 1) / kAnchor * a.nwc;
  const int maxcut = sm.maxcut;
  for (int w0 = 0; (int64_t)w0 * a.CH < maxcut; w0 += a.nwc) {
    const int j0 = w0 * a.CH;
    const int top = maxcut - j0 < gbins ? maxcut - j0 : gbins;  // the longest row's bins in this group
    if (st.w0 != w0 || st.pending) {
      if (st.w0 != w0) {  // (a pending copy is always group 0's, the first one taken)
        if (t == 0) {
          fence_proxy_async_smem();
          fused_stage<NDET, CAL>(a, L, dyn, w0, &sm.bar);
        }
        st.w0 = w0;
      }
      if (!mbar_wait_bounded(&sm.bar, st.parity, a.status)) sm.fail = 1;
      st.parity ^= 1u;
      st.pending = false;
    }
    // anchor records, blocks of a row on neighbouring threads
    const int nb = (top + kAnchor - 1) / kAnchor;
    for (int i = t; i < R * nb; i += 32 * NW) {
      const int r = i / nb, b = i - r * nb;
      if (j0 + b * kAnchor < sm.ncut[r])
        anchor_record<NDET>(sm.pm[r], dyn + L.anchor + b * kAnchorRowFloats, dyn + L.rec + (r * gblk + b) * AR);
    }
    if (t == 0) sm.next = 0;
    group_sync<NW>();
    if (sm.fail) return false;
    const int nwa = (top + a.CH - 1) / a.CH;  // windows of the group that hold bins
    const int nk = w0 == 0 ? NDET : 0;
    while (true) {
      int item = 0;
      if (lane == 0) item = atomicAdd(&sm.next, 1);
      item = __shfl_sync(0xffffffffu, item, 0) - nk;
      if (item >= R * nwa) break;
      if (item < 0) {
        fused_amplitudes<NDET, CAL, NW>(a.seg, sm, item + nk, lane);
        continue;
      }
      const int wl = item / R, r = sm.order[item - wl * R];
      const int jl = wl * a.CH;
      int n = sm.ncut[r] - j0 - jl;
      if (n <= 0) continue;
      if (n > a.CH) n = a.CH;
      float4* nodes = sm.nodes + (CAL ? warp * NDET * kMaxCalNodes : 0);
      if constexpr (CAL) cal_nodes_fill<NDET, true>(crow(r), a.nn, a.calQ, lane, nodes);
      float v[NS];
      RowState<NDET> rs;
      fused_row_sums<NDET, CAL>(a, dyn, dyn + L.cal, sm.pm[r], dyn + L.rec + (r * gblk + jl / kAnchor) * AR, j0, jl, n, lane,
                                nodes, rs);
#pragma unroll
      for (int d = 0; d < NDET; ++d) {
        v[2 * d] = rs.U[d];
        v[2 * d + 1] = rs.V[d];
        if constexpr (CAL) v[2 * NDET + d] = rs.X[d];
      }
      const float s = warp_fold<NS>(v, lane);
      constexpr int W = FoldP<NS>::W;
      if (lane % W == 0 && lane / W < NS) dyn[L.part + (r * a.nwc + wl) * NS + lane / W] = s;
    }
    if (j0 + gbins < maxcut) {  // another group follows: its sums go on top of these
      group_sync<NW>();
      for (int i = t; i < R * NS; i += 32 * NW) {
        const int r = i / NS, k = i - r * NS;
        const int left = sm.ncut[r] - j0;
        double x = w0 == 0 ? 0.0 : sm.acc[k][r];
        for (int wl = 0; wl < nwa && wl * a.CH < left; ++wl) x += (double)dyn[L.part + (r * a.nwc + wl) * NS + k];
        sm.acc[k][r] = x;
      }
      group_sync<NW>();
    }
  }
  return true;
}

// lnL of row r from the sums (one thread; a barrier after fused_bins): -inf for
// an unphysical row, 0 without an in-band bin.
template <int NDET, bool CAL, int NW>
__device__ __forceinline__ double fused_combine(const FusedArgs& a, const FusedLayout& L, const float* __restrict__ dyn,
                                                const FusedSmem<NDET, CAL, NW>& sm, int r) {
  constexpr int NS = FusedSmem<NDET, CAL, NW>::NS;
  const int ncut = sm.ncut[r];
  if (sm.flag[r]) return -INFINITY;
  if (ncut <= 0) return 0.0;
  const int gbins = a.CH * a.nwc;
  const int j0 = (sm.maxcut - 1) / gbins * gbins;  // the last group's first bin
  const float* part = dyn + L.part + r * a.nwc * NS;
  const bool one = ncut <= a.CH;  // the row's only window
  auto sum = [&](int k) {
    if (one) return (double)part[k];
    double x = j0 > 0 ? sm.acc[k][r] : 0.0;
#pragma unroll 1
    for (int wl = 0; wl < a.nwc && j0 + wl * a.CH < ncut; ++wl) x += (double)part[wl * NS + k];
    return x;
  };
  FF hh = ff(0.0f);
  double acc = 0.0;
#pragma unroll
  for (int d = 0; d < NDET; ++d) {
    hh = hh + sm.hterm[d][r];
    const double kr = sm.Kr[d][r], ki = sm.Ki[d][r];
    const double U = sum(2 * d), V = sum(2 * d + 1);
    // the fused multiply-adds that flush_pending's expressions compile to
    acc = __dadd_rn(acc, __fma_rn(kr, U, -__dmul_rn(ki, V)));
    if constexpr (CAL) acc = __fma_rn(-0.5 * __fma_rn(kr, kr, __dmul_rn(ki, ki)), sum(2 * NDET + d), acc);
  }
  return acc - 0.5 * ff_to_double(hh);
}

}  // namespace gwl
