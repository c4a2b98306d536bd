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

// The launch shape of the fused kernel for a batch of B: CTAs, rows per CTA and
// windows staged together; false where the separate kernels run.
//
// Up to a row for each warp (B <= 8 SMs) one CTA per SM, with all its shared
// memory for windows; past that two CTAs per SM, in whole waves of at most 32
// rows each.  A CTA walks through its rows' windows by itself, while the
// separate bin loop spreads (row, window) pairs over the whole chip, so the
// line is drawn by the number of windows (us per call, 640-bin windows, one
// kernel against three):
//   8 s BBH, 3 detectors (one window in use)   B = 1 / 250 / 1900 / 8192 / 20000:
//     8.6 / 10.4 / 12.2 / 19.6 / 48.2 against 16.6 / 19.2 / 22.4 / 33.7 / 58.0
//   8 s, every row in all 13 windows           B = 1 / 250 / 1900 / 8192:
//     21.1 / 26.0 / 65.2 / 203 against 26.6 / 39.4 / 97.5 / 291
//   16 s BNS, 2 detectors, 26 windows          B = 1 / 250 / 1900 / 8192:
//     34.1 / 43.8 / 112 / 330 against 33.2 / 50.4 / 139 / 476
//   32 s BNS, 3 detectors, 51 windows          B = 1 / 64 / 250 / 1900:
//     59.4 / 61.7 / 73.7 / 243 against 48.4 / 57.5 / 82.1 / 278
//   128 s BNS, 406 windows                     B = 64 / 1000 / 1900 / 4000:
//     327 / 1014 / 1492 / 2720 against 248 / 895 / 1529 / 3109
// so segments of up to 32 windows take it at any batch, longer ones where the
// batch gives every warp of two CTAs per SM a row.
bool fused_shape(const gwl_ctx* c, int64_t B, int* grid, int* rows, int* nwc) {
  if (c->opt.precision != GWL_MIXED || B <= 0) return false;
  if (fused_window_count(c) > 32 && B <= 8 * (int64_t)c->num_sms) return false;
  const int per_sm = B <= 8 * (int64_t)c->num_sms ? 1 : 2;
  const int64_t slots = per_sm * (int64_t)c->num_sms;
  const int64_t waves = (B + slots * kFusedRows - 1) / (slots * kFusedRows);
  const int64_t R = (B + slots * waves - 1) / (slots * waves);
  const int64_t G = (B + R - 1) / R;
  const int w = fused_windows(c, (int)R, (per_sm == 1 ? 227 * 1024 : kSmemPerSm / 2 - 1024) - fused_static(c) - 128);
  if (w == 0) return false;
  *grid = (int)G;
  *rows = (int)R;
  *nwc = w;
  return true;
}

// Whether gwl_loglike takes the fused kernel for a batch of B.
bool fused_used(const gwl_ctx* c, int64_t B) {
  int grid, rows, nwc;
  return !lanes_seg(c, B) && fused_shape(c, B, &grid, &rows, &nwc);
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

}  // namespace gwl
