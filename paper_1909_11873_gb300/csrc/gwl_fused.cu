// gwl_fused.cu -- the mixed likelihood in one kernel (gwl_fused.cuh): each CTA
// takes a group of rows from parameters to lnL.
//
// What bounds it: the dependent float-pair chains of the coefficients (latency,
// about half of the kernel) and then the issue of the bin sums, of which the
// hardware sine and cosine are the largest pipe.  Measured back to back on the
// 8 s, 3-detector batch of 8192 rows (704-bin windows): 17.9 us a call against
// 32.1-33.3 us with the clearing, prologue and bin-loop kernels; with the
// calibration model, 4096 rows: 21.1 against 35.4 us; 4 s, 1 detector, 1000
// rows: 11.7 against 24.7 us; one row: 8.6 against 18.8 us.
#include "gwl_fused.cuh"

namespace gwl {

template <int NDET, bool CAL>
__global__ void __launch_bounds__(256, 2) k_fused(const __grid_constant__ FusedArgs a, const double* __restrict__ theta,
                                                  int64_t B, int R, double* __restrict__ lnl) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  constexpr int NW = 8;
  __shared__ FusedSmem<NDET, CAL, NW> sm;
  float* dyn = reinterpret_cast<float*>(smem_raw);
  const FusedLayout L = fused_layout(NDET, CAL ? a.cal_row : 0, a.CH, a.nwc, R);
  // the next call's kernel may become resident as CTAs leave; it stages its
  // table rows and waits for this grid before it reads anything else
  cudaTriggerProgrammaticLaunchCompletion();
  if (threadIdx.x == 0) {
    sm.fail = 0;
    mbar_init(&sm.bar, 1);
    fence_mbar_init();
    fused_stage<NDET, CAL>(a, L, dyn, 0, &sm.bar);
  }
  cudaGridDependencySynchronize();  // theta's writer and lnl's earlier users are done
  const int64_t row0 = (int64_t)blockIdx.x * R;
  const int n = B - row0 < R ? (int)(B - row0) : R;
  const int lane = threadIdx.x & 31;
  const double* row = theta + (row0 + lane) * a.seg.stride;
  fused_coeffs<NDET, CAL, NW>(a.seg, n, sm,
                          [&](int k) { return a.seg.param_pos[k] >= 0 ? row[a.seg.param_pos[k]] : a.seg.fixed[k]; },
                          [](int) { return false; });
  FusedStage st;
  if (!fused_bins<NDET, CAL, NW>(a, L, dyn, n, sm, st,
                             [&](int r) { return theta + (row0 + r) * a.seg.stride + a.cal_par; }))
    return;
  if (st.pending) mbar_wait_bounded(&sm.bar, st.parity, a.status);  // no copy may outlive the CTA
  __syncthreads();
  if (threadIdx.x < n) lnl[row0 + threadIdx.x] = fused_combine<NDET, CAL, NW>(a, L, dyn, sm, threadIdx.x);
}

// ---------------------------------------------------------------- host side
int lnl_window(const gwl_ctx* c) { return c->window > c->M ? (int)c->M : c->window; }

size_t fused_bytes(const gwl_ctx* c, int nwc, int R) {
  return sizeof(float) * (size_t)fused_layout(c->n_det, c->n_cal_nodes ? c->row_cal_f : 0, lnl_window(c), nwc, R).total;
}

int fused_window_count(const gwl_ctx* c) {
  const int CH = lnl_window(c);
  return (int)((c->M + CH - 1) / CH);
}

// Windows of R rows' groups that fit `room` bytes of dynamic shared memory (0: none).
int fused_windows(const gwl_ctx* c, int R, size_t room) {
  const int nw = fused_window_count(c);
  if ((lnl_window(c) % kAnchor && nw > 1) || fused_bytes(c, 1, R) > room) return 0;
  int w = 1;
  while (w < nw && fused_bytes(c, w + 1, R) <= room) ++w;
  return w;
}

// Static shared memory of the kernel.
template <int NDET>
static size_t static_of(bool cal) {
  return cal ? sizeof(FusedSmem<NDET, true, 8>) : sizeof(FusedSmem<NDET, false, 8>);
}
static size_t fused_static(const gwl_ctx* c) {
  const bool cal = c->n_cal_nodes > 0;
  switch (c->n_det) {
    case 1: return static_of<1>(cal);
    case 2: return static_of<2>(cal);
    case 3: return static_of<3>(cal);
    default: return static_of<4>(cal);
  }
}
constexpr size_t kSmemPerSm = 228 * 1024;  // 1 KB of it goes to each resident CTA's system part

// Groups of nwc windows that a row in the middle of the mass prior has.
int fused_groups(const gwl_ctx* c, int nwc) {
  const int64_t nw = (c->mid_cut + lnl_window(c) - 1) / lnl_window(c);
  return (int)((nw + nwc - 1) / nwc);
}

// Whether the one-kernel form is the faster one for R rows per CTA, per_sm CTAs
// per SM, nwc windows staged together.
//
// A CTA walks through its rows' windows by itself, a group of nwc after another,
// while the separate bin loop spreads (row, window) pairs over the whole chip.
// Up to four groups (three with the calibration model) the one kernel wins at
// any batch.  Beyond, each group costs 4-6 us of staging and barriers, which have
// to be shared by enough (row, window) items: a CTA with fewer of them than warps
// leaves the others idle.  How many are enough depends on the other side: it is
// slow where its windows leave room for one CTA per SM, and fast in small batches,
// which leave the one-kernel form SMs without a row.  The lines below are drawn
// through 760 calls timed both ways (1-4 detectors, 4 to 128 s, 256- to 1344-bin
// windows, 1 to 6000 rows, with and without calibration), among them, in us a
// call, one kernel against three:
//   8 s BBH, 3 detectors, 1 group               B = 1 / 400 / 1216 / 4096: 9 / 10 / 11 / 14 against 17 / 19 / 21 / 27
//   8 s, every row in all 13 windows, 3 groups  B = 1 / 400 / 1216 / 4096: 20 / 32 / 50 / 109 against 28 / 59 / 84 / 177
//   16 s BNS, 2 detectors, 640-bin windows      B = 1 / 400 / 1217 / 4096: 33 / 48 / 98 / 192 against 33 / 70 / 115 / 278
//   16 s BNS, 2 detectors, 1280-bin windows     B = 1 / 400 / 1217 / 4096: 38 / 52 / 94 / 182 against 29 / 55 / 93 / 223
//   32 s BNS, 3 detectors, 1280-bin windows     B = 1 / 152 / 400 / 1216: 89 / 91 / 103 / 171 against 36 / 89 / 129 / 273
//   32 s BNS, 3 detectors, 640-bin windows      B = 1 / 400 / 1217 / 2400: 63 / 105 / 211 / 251 against 47 / 114 / 213 / 364
//   16 s BNS, calibrated, 640-bin windows       B = 1 / 400 / 1216 / 1600 / 2400: 68 / 109 / 179 / 251 / 278
//                                                                      against 37 / 97 / 184 / 228 / 317
static bool fused_pays(const gwl_ctx* c, int64_t B, int per_sm, int R, int nwc) {
  const bool cal = c->n_cal_nodes > 0;
  const int G = fused_groups(c, nwc);
  if (G <= (cal ? 3 : 4)) return true;
  const int items = R * nwc, rounds = (items + 7) / 8;  // of the eight warps
  // whether two CTAs of k_window fit an SM: its window, and its own arrays
  const size_t window = (size_t)lnl_window(c) * lnl_row_bytes(c) +
                        (size_t)(lnl_window(c) / kAnchor) * kAnchorRowFloats * sizeof(float);
  const bool two = window + 2304 + (cal ? 3328 : 1024) * c->n_det + 1024 <= kSmemPerSm / 2;
  // (a few calibrated rows, one window at a time, would be 1.3-1.9 times faster in three kernels up to six groups too)
  if (!two) return per_sm == 2 || items >= (cal && nwc == 1 ? 6 : 4) || (cal && G <= 6 && nwc == 1);
  if (per_sm == 2) return cal ? items >= 17 || (items >= 7 && 10 * items >= 64 * rounds) : items >= 6 || G <= 16;
  if (cal)
    return 4 * B >= c->num_sms &&
           ((G <= 5 && items >= 3) || (items >= 8 && 20 * items >= 152 * rounds) || (items >= 20 && 10 * items >= 64 * rounds));
  return items >= (B >= c->num_sms ? 3 : 2 * B >= c->num_sms ? 5 : 6);
}

// The launch shape of the fused kernel for a batch of B: CTAs, rows per CTA and
// windows staged together; false where it does not fit.  Up to a row for each warp
// (B <= 8 SMs) one CTA per SM, with all its shared memory for windows; past that
// two CTAs per SM, in whole waves of at most 32 rows each.  Small batches on segments
// of more than 32 windows always go to the separate kernels.
static bool fused_fits(const gwl_ctx* c, int64_t B, int* grid, int* rows, int* nwc, int* per_sm) {
  if (c->opt.precision != GWL_MIXED || B <= 0) return false;
  *per_sm = B <= 8 * (int64_t)c->num_sms ? 1 : 2;
  if (fused_window_count(c) > 32 && *per_sm == 1) return false;
  const int64_t slots = *per_sm * (int64_t)c->num_sms;
  const int64_t waves = (B + slots * kFusedRows - 1) / (slots * kFusedRows);
  const int64_t R = (B + slots * waves - 1) / (slots * waves);
  const int64_t G = (B + R - 1) / R;
  const int w = fused_windows(c, (int)R, (*per_sm == 1 ? 227 * 1024 : kSmemPerSm / 2 - 1024) - fused_static(c) - 128);
  if (w == 0) return false;
  *grid = (int)G;
  *rows = (int)R;
  *nwc = w;
  return true;
}

// The same, false too where the separate kernels are the faster ones.  (Of the
// batches that are not the lane layout's: with GWL_BINS_AUTO, the default, those
// are the ones below 2048 rows, and calibrated ones; from 2048 rows on the
// one-kernel form runs with GWL_BINS_WARP, which the autotuner sets where it is
// the faster one.)
bool fused_shape(const gwl_ctx* c, int64_t B, int* grid, int* rows, int* nwc) {
  int per_sm;
  return fused_fits(c, B, grid, rows, nwc, &per_sm) && fused_pays(c, B, per_sm, *rows, *nwc);
}

// Whether gwl_loglike takes the fused kernel for a batch of B.
bool fused_used(const gwl_ctx* c, int64_t B) {
  int grid, rows, nwc;
  return !lanes_seg(c, B) && fused_shape(c, B, &grid, &rows, &nwc);
}

// Whether it could (a walk of n chains has a line of its own).
bool fused_possible(const gwl_ctx* c, int64_t n) {
  int grid, rows, nwc, per_sm;
  return !lanes_seg(c, n) && fused_fits(c, n, &grid, &rows, &nwc, &per_sm);
}

FusedArgs fused_args(const gwl_ctx* c, int nwc) {
  FusedArgs a;
  a.seg = c->seg;
  a.tab = c->d_tab_block;
  a.low = c->d_tab_low;
  a.anchor = c->d_anchor;
  a.CH = lnl_window(c);
  a.nwc = nwc;
  a.df = (float)c->df;
  a.cal = c->d_cal_f;
  a.cal_row = c->row_cal_f;
  a.cal_par = c->opt.n_dim;
  a.nn = c->n_cal_nodes;
  a.calQ = c->d_calQ_f;
  a.status = c->d_status;
  a.ffc = c->count_ff ? c->d_ffc : nullptr;
  return a;
}

template <int NDET, bool CAL>
static cudaError_t run_fused(gwl_ctx* c, const double* theta, int64_t B, double* lnl, int grid, int rows, int nwc,
                             cudaStream_t st) {
  const FusedArgs a = fused_args(c, nwc);
  const size_t smem = fused_bytes(c, nwc, rows);
  cudaError_t e = raise_smem_limit((const void*)k_fused<NDET, CAL>, c->device, smem);
  if (e != cudaSuccess) return e;
  ProfScope ps(c, GWL_KERNEL_BINS, st);
  e = launch_pdl(k_fused<NDET, CAL>, dim3(grid), dim3(256), smem, st, a, theta, B, rows, lnl);
  c->launches++;
  return e;
}

cudaError_t launch_fused(gwl_ctx* c, const double* theta, int64_t B, double* lnl, int grid, int rows, int nwc,
                         cudaStream_t st) {
  const bool cal = c->n_cal_nodes > 0;
  switch (c->n_det) {
    case 1: return cal ? run_fused<1, true>(c, theta, B, lnl, grid, rows, nwc, st)
                       : run_fused<1, false>(c, theta, B, lnl, grid, rows, nwc, st);
    case 2: return cal ? run_fused<2, true>(c, theta, B, lnl, grid, rows, nwc, st)
                       : run_fused<2, false>(c, theta, B, lnl, grid, rows, nwc, st);
    case 3: return cal ? run_fused<3, true>(c, theta, B, lnl, grid, rows, nwc, st)
                       : run_fused<3, false>(c, theta, B, lnl, grid, rows, nwc, st);
    default: return cal ? run_fused<4, true>(c, theta, B, lnl, grid, rows, nwc, st)
                        : run_fused<4, false>(c, theta, B, lnl, grid, rows, nwc, st);
  }
}

// The one-kernel form wherever it fits, the faster one or not.
cudaError_t launch_fused_possible(gwl_ctx* c, const double* theta, int64_t B, double* lnl, cudaStream_t st) {
  int grid, rows, nwc, per_sm;
  if (!fused_fits(c, B, &grid, &rows, &nwc, &per_sm)) return cudaErrorInvalidValue;
  return launch_fused(c, theta, B, lnl, grid, rows, nwc, st);
}

}  // namespace gwl
