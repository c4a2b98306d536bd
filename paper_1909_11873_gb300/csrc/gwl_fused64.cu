// gwl_fused64.cu -- the FP64 likelihood in one kernel: each CTA takes a group of
// rows from parameters to lnL, as gwl_fused.cuh does for the mixed path.
//
// GB300 issues an FP64 warp instruction about every 16 cycles per SM whatever
// its active lanes, so the FP64 path is bound by how evenly that pipe is kept
// busy over the SMs.  In the separate kernels the bin loop's warps race for
// rows: with about a thousand rows the SMs that pass the prologue's wait first
// take 16 each and others none, and a row's windows follow one another.  Here
// every SM gets the same number of rows, and a row is cut into pieces of 128
// bins that the warps of a CTA, or of a cluster of CTAs, share.  The arithmetic per row and bin is that
// of prologue_rows and bin_f64; the FP64 sums are added in another order: a
// piece's four blocks of 32 bins lane by lane, a fixed fold of the lanes, then
// the pieces in bin order.  However the work is split, that order stays, so a
// row's lnL has the same bits in every batch.
//
// Measured back to back (us a call, 8 s BBH, 3 detectors, one kernel against
// three, 384-bin windows), at 1 / 32 / 150 / 250 / 1021 / 2000 / 8192 rows:
// 15.6 / 17.3 / 29.7 / 45.2 / 114.7 / 209.6 / 725 against 65.6 / 76.6 / 139 / 157
// / 201 / 218 / 727; rows over the whole band (8 s BNS), 1 / 64 / 250 / 1000:
// 45.1 / 145 / 510 / 1655 against 79.9 / 205 / 510 / 1638.
#include <cmath>

#include "gwl_bins.cuh"

namespace gwl {

constexpr int kRows64 = 32;  // rows per CTA at most (one per lane in the prologue)
constexpr int kPiece = 128;  // bins per piece

struct Fused64Args {
  SegInfo seg;
  const double* tab;  // FP64 rows
  int row_elems;      // doubles per row
  int np;             // pieces a CTA stages together
  int lc;             // log2 of C, the CTAs per group of rows (a cluster)
  int keep;           // pieces whose sums a CTA holds (np, or all of its own where C > 1)
  int team;           // warps that share an item: 1, 2 or 4
  int* status;
};

template <int NDET>
struct Smem64 {
  static constexpr int NS = 2 * NDET;
  double lmc[kRows64], leta[kRows64], amp[kRows64];
  double eta[kRows64], phi[6][kRows64];
  double sky[4][kRows64], ori[3][kRows64];
  double P[2 * NDET][kRows64], ang[2][kRows64], hterm[NDET][kRows64];
  double Kr[NDET][kRows64], Ki[NDET][kRows64];
  double acc[NS][kRows64];
  PropF64 pf[kRows64];
  int ncut[kRows64], flag[kRows64];
  int next, maxcut, fail;
  int item[4][2];
  alignas(8) uint64_t bar;
};

// The coefficients of the group's rows, eight parts (gwl_fused.cuh's).
template <int NDET>
__device__ __forceinline__ void coeffs64(const SegInfo& s, int R, Smem64<NDET>& sm, const double* __restrict__ row) {
  const int part = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool valid = lane < R;
  auto th = [&](int k, double other) {
    return !valid ? other : s.param_pos[k] >= 0 ? row[s.param_pos[k]] : s.fixed[k];
  };
  // ---- phase 1
  if (part == 0) {
    sm.lmc[lane] = ::log(th(0, 10.0) * (kPi * kTsun));
  } else if (part == 1) {
    const PNCoeffs<double> P = pn_coeffs(th(1, 0.5), th(2, 0.0), th(3, 0.0));
    sm.eta[lane] = P.eta;
    sm.phi[0][lane] = P.p2;
    sm.phi[1][lane] = P.p3;
    sm.phi[2][lane] = P.p4;
    sm.phi[3][lane] = P.p5c;
    sm.phi[4][lane] = P.p6c;
    sm.phi[5][lane] = P.p7;
  } else if (part == 2) {
    const double q = th(1, 0.5), opq = q + 1.0;
    sm.leta[lane] = ::log(q / (opq * opq));
  } else if (part < 7) {
    double x = part == 3 ? th(7, 0.0) - s.gmst : part == 4 ? th(8, 0.0) : part == 5 ? th(6, 0.0) : th(5, 0.0);
    double sn, cs;
    ::sincos(x, &sn, &cs);
    double* o = part == 3 ? &sm.sky[0][lane] : part == 4 ? &sm.sky[2][lane] : &sm.ori[0][lane];
    if (part < 6) {
      o[0] = sn;
      o[kRows64] = cs;
    } else {
      sm.ori[2][lane] = cs;
    }
  } else {
    double x[11];
#pragma unroll
    for (int k = 0; k < 11; ++k) x[k] = th(k, 1.0);
    const bool ok = valid && physical_bits(x);
    sm.flag[lane] = ok ? 0 : 1;
    if (ok) prefetch_cut_H(s, x[0], x[1]);
  }
  __syncthreads();
  // ---- phase 2
  if (part == 0) {
    Scale<double> S;
    S.la = sm.lmc[lane] - 0.6 * sm.leta[lane];
    S.a13 = ::exp(S.la * (1.0 / 3.0));
    S.amp = 0.0;
    PNCoeffs<double> P;
    P.eta = sm.eta[lane];
    P.p2 = sm.phi[0][lane];
    P.p3 = sm.phi[1][lane];
    P.p4 = sm.phi[2][lane];
    P.p5c = sm.phi[3][lane];
    P.p6c = sm.phi[4][lane];
    P.p7 = sm.phi[5][lane];
    double c[kNBasis], ccyc;
    basis_coeffs(P, S, c, ccyc);
#pragma unroll
    for (int m = 0; m < kNBasis; ++m) sm.pf[lane].c[m] = c[m];
  } else if (part == 1) {
    sm.amp[lane] = ::exp((sm.lmc[lane] - kLnPi) * (5.0 / 6.0)) * (kAmpConst * kC / kMpc * s.amp_scale) / th(4, 100.0);
  } else if (part == 2) {
    const double la = sm.lmc[lane] - 0.6 * sm.leta[lane];
    double sa, ca;
    k_angle(th(10, 0.0), const_cycles(cycles_pref(sm.eta[lane]), sm.phi[3][lane], la), sa, ca);
    sm.ang[0][lane] = sa;
    sm.ang[1][lane] = ca;
  } else if (part == 3) {
    const double a13 = ::exp((sm.lmc[lane] - 0.6 * sm.leta[lane]) * (1.0 / 3.0));
    int ncut = 0;
    if (sm.flag[lane] == 0) {
      ncut = (int)s.M;
      if (s.fcut_mode == 0) ncut = count_bins_le(s, 1.0 / (kSix32 * a13 * a13 * a13));
    }
    sm.ncut[lane] = ncut;
    const int nm = __reduce_max_sync(0xffffffffu, ncut);
    if (lane == 0) sm.maxcut = nm;
  } else if (part - 4 < NDET) {
    const int d = part - 4;
    Sky<double> k;
    k.sl = sm.sky[0][lane];
    k.cl = sm.sky[1][lane];
    k.sd = sm.sky[2][lane];
    k.cd = sm.sky[3][lane];
    sm.pf[lane].tau[d] = delay(th(9, 0.0), k, s.geom + 9 * d);
    double Pr, Pi;
    response(k, sm.ori[0][lane], sm.ori[1][lane], sm.ori[2][lane], s.geom + 9 * d, Pr, Pi);
    sm.P[2 * d][lane] = Pr;
    sm.P[2 * d + 1][lane] = Pi;
  }
  __syncthreads();
}

// warp_fold (gwl_fused.cuh) on doubles (at most eight values): value v's warp sum
// on lanes [v W, v W + W), W = 32 / P, P the power of two at or above the count.
template <int N>
struct Fold64 {
  static constexpr int P = N <= 2 ? 2 : N <= 4 ? 4 : 8;
  static constexpr int W = 32 / P;
};
template <int N>
__device__ __forceinline__ double warp_fold64(const double (&v)[N], int lane) {
  static_assert(N <= 8, "at most eight sums");
  constexpr int P = Fold64<N>::P;
  double t[P];
#pragma unroll
  for (int k = 0; k < P; ++k) t[k] = k < N ? v[k] : 0.0;
  int off = 16;
#pragma unroll
  for (int h = P / 2; h >= 1; h >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const double send = up ? t[k] : t[k + h];
      const double keep = up ? t[k + h] : t[k];
      t[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (; off >= 1; off >>= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], off);
  return t[0];
}

// The U and V of detector d with one bin's sine and cosine, as bin_f64 adds them.
__device__ __forceinline__ void add_bin64(double gr, double gi, double sn, double cs, double& U, double& V) {
  U = fma(gr, cs, fma(gi, sn, U));
  V = fma(gi, cs, fma(-gr, sn, V));
}

// Barrier of team q, of n threads.
__device__ __forceinline__ void team_sync(int q, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + q), "r"(n) : "memory");
}

// A double in the shared memory of the cluster's CTA `rank`, at this CTA's address p.
__device__ __forceinline__ double cluster_load(const double* p, uint32_t rank) {
  uint32_t ra;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ra) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.aligned;\n barrier.cluster.wait.aligned;" ::: "memory");
}

// K_d and the <h|h> term of detector d, one row per lane (one warp).
template <int NDET>
__device__ __forceinline__ void amplitudes64(const SegInfo& s, Smem64<NDET>& sm, int d, int lane) {
  const int nc = sm.ncut[lane];
  const double H = nc > 0 ? s.H[(int64_t)d * s.M + nc - 1] : 0.0;
  const double amp = sm.amp[lane], Pr = sm.P[2 * d][lane], Pi = sm.P[2 * d + 1][lane];
  const double sa = sm.ang[0][lane], ca = sm.ang[1][lane];
  sm.Kr[d][lane] = amp * (Pr * ca - Pi * sa);
  sm.Ki[d][lane] = amp * (Pr * sa + Pi * ca);
  sm.hterm[d][lane] = amp * amp * (Pr * Pr + Pi * Pi) * H;
}

// A cluster of C CTAs takes the same R rows: every CTA forms their coefficients
// and sums every C-th piece of the bins, the first CTA adds the pieces' sums (from
// the CTAs' shared memory) and writes lnL.
//
// An item is a (row, piece) on one warp or, with few rows, on a team of two or
// four: a block takes a lone warp 3.5 us, nearly all of it in the phase and its
// sine and cosine.  A team's warps form those of two blocks or one each, and
// then, each for its detectors, add the four blocks' terms in the order in which
// one warp would.
template <int NDET>
__global__ void __launch_bounds__(256, 1) k_fused64(const __grid_constant__ Fused64Args a,
                                                    const double* __restrict__ theta, int64_t B, int R,
                                                    double* __restrict__ lnl) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ Smem64<NDET> sm;
  constexpr int NS = Smem64<NDET>::NS;
  double* rows = reinterpret_cast<double*>(smem_raw);  // [np][piece] rows of this CTA's pieces
  double* part = rows + (int64_t)a.np * kPiece * a.row_elems;  // [R][keep][NS]
  const int t = threadIdx.x, lane = t & 31, team = a.team;
  const int group = (t >> 5) / team, tw = (t >> 5) % team;
  double* trig = part + R * a.keep * NS + group * (4 * NS * 32);  // (teams) [4 blocks][sine, cosine][32] of this one
  const int C = 1 << a.lc, rank = (int)blockIdx.x & (C - 1);
  // this CTA's pieces p0 + C i (i < count), one thread
  auto stage = [&](int64_t p0, int count) {
    uint32_t bytes = 0;
    for (int pass = 0; pass < 2; ++pass) {
      for (int i = 0; i < count; ++i) {
        const int64_t j0 = (p0 + (int64_t)C * i) * kPiece;
        const int64_t n = a.seg.M - j0 < kPiece ? a.seg.M - j0 : kPiece;
        if (n <= 0) break;
        const uint32_t nb = (uint32_t)n * (uint32_t)a.row_elems * 8u;
        if (pass == 0) bytes += nb;
        else bulk_g2s(rows + (int64_t)i * kPiece * a.row_elems, a.tab + j0 * a.row_elems, nb, &sm.bar);
      }
      if (pass == 0) mbar_arrive_expect_tx(&sm.bar, bytes);
    }
  };
  cudaTriggerProgrammaticLaunchCompletion();
  if (t == 0) {
    sm.fail = 0;
    mbar_init(&sm.bar, 1);
    fence_mbar_init();
    stage(rank, a.np);
  }
  cudaGridDependencySynchronize();  // theta's writer and lnl's earlier users are done
  const int64_t row0 = (int64_t)(blockIdx.x >> a.lc) * R;
  const int n = B - row0 < R ? (int)(B - row0) : R;
  coeffs64<NDET>(a.seg, n, sm, theta + (row0 + lane) * a.seg.stride);
  const int maxcut = sm.maxcut;
  const int all = (maxcut + kPiece - 1) / kPiece;  // pieces of the longest row
  uint32_t parity = 0;
  bool pending = true;
  int turn = 0;  // (teams) which of sm.item's slots is next
  for (int p0 = rank; p0 - rank < all; p0 += C * a.np) {
    // own pieces that hold bins (none where the rows end before this rank's first one)
    const int np = p0 < all ? min(a.np, (all - p0 + C - 1) / C) : 0;
    if (p0 != rank && np > 0 && t == 0) {
      fence_proxy_async_smem();
      stage(p0, np);
    }
    if (t == 0) sm.next = 0;
    if (p0 == rank || np > 0) {
      if (!mbar_wait_bounded(&sm.bar, parity, a.status)) sm.fail = 1;
      parity ^= 1u;
      pending = false;
    }
    __syncthreads();
    if (sm.fail) break;  // (every thread: the barriers below are still met)
    const int s0 = C > 1 ? (p0 - rank) >> a.lc : 0;  // where the first piece's sums go
    // all rows' first pieces first: the last ones are the longest rows'
    if (team > 1) {
      const int nk = p0 == 0 ? 1 : 0;  // the first CTA's first item is the detectors' amplitudes
      while (true) {
        if (tw == 0 && lane == 0) sm.item[group][turn] = atomicAdd(&sm.next, 1);
        team_sync(group, 32 * team);  // (and every warp of the team is done with the last item's trig)
        const int item = sm.item[group][turn] - nk;
        turn ^= 1;
        if (item >= n * np) break;
        if (item < 0) {
          for (int d = tw; d < NDET; d += team) amplitudes64<NDET>(a.seg, sm, d, lane);
          continue;
        }
        const int pc = item / n, r = item - pc * n;
        const int nb = sm.ncut[r] - (p0 + C * pc) * kPiece;  // the piece's bins below the row's cut, or more
        if (nb <= 0) continue;
        const double* pr = rows + (int64_t)pc * kPiece * a.row_elems;
        double c[kNBasis], tau[NDET];
#pragma unroll
        for (int m = 0; m < kNBasis; ++m) c[m] = sm.pf[r].c[m];
#pragma unroll
        for (int d = 0; d < NDET; ++d) tau[d] = sm.pf[r].tau[d];
        for (int b = tw; b < kPiece / 32 && 32 * b + lane < nb; b += team) {
          double x[RowD<NDET>::n], sn[NDET], cs[NDET];
          load_row<NDET>(pr + (int64_t)(32 * b + lane) * a.row_elems, x);
          phase_f64<NDET>(x, c, tau, sn, cs);
#pragma unroll
          for (int d = 0; d < NDET; ++d) {
            trig[(b * NS + 2 * d) * 32 + lane] = sn[d];
            trig[(b * NS + 2 * d + 1) * 32 + lane] = cs[d];
          }
        }
        team_sync(group, 32 * team);
        for (int d = tw; d < NDET; d += team) {
          double v[2] = {0.0, 0.0};
#pragma unroll
          for (int b = 0; b < kPiece / 32; ++b)
            if (32 * b + lane < nb) {
              const double* g = pr + (int64_t)(32 * b + lane) * a.row_elems + 9 + 2 * d;
              add_bin64(g[0], g[1], trig[(b * NS + 2 * d) * 32 + lane], trig[(b * NS + 2 * d + 1) * 32 + lane], v[0], v[1]);
            }
          const double sum = warp_fold64<2>(v, lane);
          if (lane % 16 == 0) part[(r * a.keep + s0 + pc) * NS + 2 * d + lane / 16] = sum;
        }
      }
    } else {
      const int nk = p0 == 0 ? NDET : 0;  // the first CTA's first items are the detectors' amplitudes
      while (true) {
        int item = 0;
        if (lane == 0) item = atomicAdd(&sm.next, 1);
        item = __shfl_sync(0xffffffffu, item, 0) - nk;
        if (item >= n * np) break;
        if (item < 0) {
          amplitudes64<NDET>(a.seg, sm, item + nk, lane);
          continue;
        }
        const int pc = item / n, r = item - pc * n;
        int nb = sm.ncut[r] - (p0 + C * pc) * kPiece;  // the piece's bins below the row's cut
        if (nb <= 0) continue;
        if (nb > kPiece) nb = kPiece;
        double c[kNBasis], tau[NDET], U[NDET], V[NDET], v[NS];
#pragma unroll
        for (int m = 0; m < kNBasis; ++m) c[m] = sm.pf[r].c[m];
#pragma unroll
        for (int d = 0; d < NDET; ++d) {
          tau[d] = sm.pf[r].tau[d];
          U[d] = V[d] = 0.0;
        }
        const double* pr = rows + (int64_t)pc * kPiece * a.row_elems;
        for (int j = lane; j < nb; j += 32) {
          double x[RowD<NDET>::n];
          load_row<NDET>(pr + (int64_t)j * a.row_elems, x);
          bin_f64<NDET>(x, c, tau, U, V);
        }
#pragma unroll
        for (int d = 0; d < NDET; ++d) {
          v[2 * d] = U[d];
          v[2 * d + 1] = V[d];
        }
        const double sum = warp_fold64<NS>(v, lane);
        constexpr int W = Fold64<NS>::W;
        if (lane % W == 0 && lane / W < NS) part[(r * a.keep + s0 + pc) * NS + lane / W] = sum;
      }
    }
    __syncthreads();
    if (C == 1) {  // the pieces' sums in bin order (one thread per row and sum)
      for (int i = t; i < n * NS; i += 256) {
        const int r = i / NS, k = i - r * NS;
        double x = p0 == 0 ? 0.0 : sm.acc[k][r];
#pragma unroll 1
        for (int pc = 0; pc < np && (p0 + pc) * kPiece < sm.ncut[r]; ++pc) x += part[(r * a.keep + pc) * NS + k];
        sm.acc[k][r] = x;
      }
      __syncthreads();
    }
  }
  if (pending) mbar_wait_bounded(&sm.bar, parity, a.status);  // no copy may outlive the CTA
  if (C > 1) {
    cluster_sync();  // every CTA's sums are in place
    if (rank == 0) {  // the same order, each CTA's pieces from its shared memory
      for (int i = t; i < n * NS; i += 256) {
        const int r = i / NS, k = i - r * NS, m = (sm.ncut[r] + kPiece - 1) / kPiece;
        double x = 0.0;
        for (int p = 0; p < m; p += 8) {
          double v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            v[u] = p + u < m ? cluster_load(&part[(r * a.keep + ((p + u) >> a.lc)) * NS + k], (uint32_t)((p + u) & (C - 1)))
                             : 0.0;
#pragma unroll
          for (int u = 0; u < 8; ++u) x += v[u];
        }
        sm.acc[k][r] = x;
      }
    }
  }
  __syncthreads();
  if (rank == 0 && t < n) {
    double l = -INFINITY;
    if (!sm.flag[t]) {
      l = 0.0;
      if (sm.ncut[t] > 0) {
        double hh = 0.0;
#pragma unroll
        for (int d = 0; d < NDET; ++d) {
          hh += sm.hterm[d][t];
          l += sm.Kr[d][t] * sm.acc[2 * d][t] - sm.Ki[d][t] * sm.acc[2 * d + 1][t];
        }
        l -= 0.5 * hh;
      }
    }
    lnl[row0 + t] = l;
  }
  if (C > 1) cluster_sync();  // the sums have been read before any CTA leaves
}

// ---------------------------------------------------------------- host side
template <int NDET>
static size_t room64() {
  return 227 * 1024 - sizeof(Smem64<NDET>) - 256;
}

// Whether gwl_loglike takes this form for a batch of B, and its launch shape.
//
// Rows are dealt out evenly, one CTA per SM.  C CTAs may share a group of R rows
// (a cluster): of C = 1, 2, 4 and 8 the one with the fewest rows per SM, R / C, is
// taken, the smallest C among equals, so that neither a handful of rows nor a batch
// just above the number of SMs leaves SMs idle (160 rows on 152 SMs: 5 rows on 4
// CTAs each instead of 2 on every second SM).  Clusters of more CTAs than a row has
// pieces leave CTAs idle, so C stays below twice the pieces of a row in the middle of
// the mass prior (8 s BBH, 3 pieces: 100 rows 29.4 us on single CTAs, 39.6 on clusters
// of eight; 16 rows 16.0 on clusters of four, 30.1 of eight; 8 s BNS, 63 pieces: 100
// rows 234 us on clusters of eight, 271 on single CTAs).
//
// An item is a (row, piece); few rows have fewer items than the SM has warps, and then
// four warps share one up to 1.5 rows per SM, two up to 3 (one row, 8 s BBH: 15.7 us,
// 32.9 with a warp per item; 380 rows: 54.0 us, 54.7 with teams of four, 56.0 without).
// Segments of more than kMaxBins64 bins keep the separate kernels, whose (row, window)
// tasks spread over the whole chip (us here against there: 16 s BNS, 2 detectors, 250
// rows 696 / 625, 1216 rows 2610 / 2654; 32 s BNS, 3 detectors, 1300 rows 8495 / 8019;
// where rows use a small part of their bins the one kernel would win: 16 s BBH, 3
// detectors, 250 rows 80 / 201, 2000 rows 399 / 411).
constexpr int64_t kMaxBins64 = 8192;

bool fused64_used(const gwl_ctx* c, int64_t B) {
  if (c->opt.precision != GWL_FP64 || c->n_cal_nodes || B <= 0) return false;
  return c->M <= kMaxBins64;
}

template <int NDET>
static cudaError_t run_fused64(gwl_ctx* c, const double* theta, int64_t B, double* lnl, cudaStream_t st) {
  const int64_t sms = c->num_sms;
  const int64_t waves = (B + sms * kRows64 - 1) / (sms * kRows64);
  int64_t R = (B + sms * waves - 1) / (sms * waves);
  int lc = 0;
  const int64_t mid = (c->mid_cut + kPiece - 1) / kPiece;  // pieces of a row in the middle of the prior
  if (waves == 1)
    for (int k = 1; k <= 3 && 1 << k < 2 * mid; ++k) {
      // clusters resident together: one per TPC (two SMs); four of four or two of eight in a GPC of 18-20 SMs
      const int64_t groups = k == 1 ? sms / 2 : k == 2 ? sms * 4 / 19 : sms * 2 / 19;
      const int64_t r = (B + groups - 1) / groups;
      if (r <= kRows64 && r << lc < R << k) {
        R = r;
        lc = k;
      }
    }
  const int C = 1 << lc;
  const int grid = (int)((B + R - 1) / R) * C;
  Fused64Args a;
  a.seg = c->seg;
  a.tab = c->d_tab_f64;
  a.row_elems = c->row_doubles;
  a.lc = lc;
  a.team = 2 * R <= 3 * C ? 4 : R <= 3 * C ? 2 : 1;
  // the pieces that fit beside their sums (of one staging or, in a cluster, of all) and the teams' sines and cosines
  constexpr int NS = 2 * NDET;
  const int64_t own = ((c->M + kPiece - 1) / kPiece + C - 1) / C;
  const size_t per_row = sizeof(double) * (size_t)R * NS, rows = sizeof(double) * (size_t)kPiece * a.row_elems;
  const size_t fixed = (a.team > 1 ? sizeof(double) * (8 / a.team) * 4 * NS * 32 : 0) + (C > 1 ? per_row * own : 0);
  const size_t per_piece = rows + (C > 1 ? 0 : per_row);
  const int64_t fit = (int64_t)((room64<NDET>() - fixed) / per_piece);
  a.np = (int)(fit < own ? fit : own);
  a.keep = C > 1 ? (int)own : a.np;
  a.status = c->d_status;
  const size_t smem = fixed + (size_t)a.np * per_piece;
  cudaError_t e = raise_smem_limit((const void*)k_fused64<NDET>, c->device, smem);
  if (e != cudaSuccess) return e;
  ProfScope ps(c, GWL_KERNEL_BINS, st);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = C;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, k_fused64<NDET>, a, theta, B, (int)R, lnl);
  c->launches++;
  return e;
}

cudaError_t launch_fused64(gwl_ctx* c, const double* theta, int64_t B, double* lnl, cudaStream_t st) {
  switch (c->n_det) {
    case 1: return run_fused64<1>(c, theta, B, lnl, st);
    case 2: return run_fused64<2>(c, theta, B, lnl, st);
    case 3: return run_fused64<3>(c, theta, B, lnl, st);
    default: return run_fused64<4>(c, theta, B, lnl, st);
  }
}

}  // namespace gwl
