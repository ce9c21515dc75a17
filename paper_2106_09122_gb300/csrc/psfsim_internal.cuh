// Internal declarations shared by the psfsim CUDA translation units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/psfsim.h"

#define PSFSIM_MAX_RADII 256
#define PSFSIM_FRAC_BITS 40  // fixed-point fraction bits of the rotation coordinates
#define PSFSIM_THETA_BINS 16 // angle bins per radial bracket when ordering columns
// Column-ordering buckets: (bracket, angle bin) for valid columns, one more for zero columns.
static inline __host__ __device__ int psfsim_num_buckets(int n_r) { return (n_r - 1) * PSFSIM_THETA_BINS + 1; }

// Per-column geometry, computed once per build on the device (FP64, Sec. 2):
// radial bracket k (-1: beyond the last radius, zero column), the two lerp
// weights, and cos/sin of the polar angle as fixed-point integers
// round(v * 2^PSFSIM_FRAC_BITS).  Exact integer arithmetic on these makes
// theta = 0 the identity and quarter turns exact permutations.
struct ColGeom {
  int k;
  int bin;        // polar-angle bin (0..PSFSIM_THETA_BINS-1), for column ordering only
  float w0, w1;  // weights of L[k] and L[k+1]
  long long C, Sn;
};
static_assert(sizeof(ColGeom) == 32, "ColGeom layout");

struct psfsim_plan {
  int storage, interp, n, n_r;
  int64_t M, K, ld;
  int N;          // scene side for grid builds, 0 for point builds
  bool quadrant;  // FUSED: columns are the x > 0, y > 0 quadrant of the N x N grid
  int64_t Kg;     // columns with geometry tables (K, or K/4 for the quadrant)
  int64_t K_valid;  // FUSED: columns inside the last radius (host copy, read back at build)
  double S;
  const float *d_lib;
  double radii[PSFSIM_MAX_RADII];
  char *ws;
  size_t ws_bytes;
  int64_t a_off, lo_off, scale_off, geom_off, order_off, bstart_off, pts_off, status_off, libmax_off, plib_off,
      cols_off, mtorder_off;
  char *pix;  // split storage, during the build: pair entries and pixel order of the pixel-wise build (NULL: another build)
  int device, num_sms;
  bool live;            // products skip the zero columns listed in the workspace (live.cu)
  int64_t live_cols;    // FP32 storage: columns the products read (all of them when !live)
  int k_tiles;          // split storage: 64-column k-tiles the products read (ld / 64 when !live)
  bool short_runs;      // split storage: at most 2.5 k-tiles on average between skipped ones
  int64_t dead_groups;  // split storage: 32-column groups in none of them
  int fit_ks;           // column splits of the fit-gradient forward, fixed at first use (0: not yet)
  CUtensorMap lib_map;  // 3D tensor map over the library for TMA staging
};

// Workspace layout for a given shape; returns total bytes.
struct WsLayout {
  int64_t ld, a_off, lo_off, scale_off, geom_off, order_off, bstart_off, pts_off, status_off, libmax_off, plib_off,
      cols_off, mtorder_off, total;  // total: what a build needs
  int64_t pix_off, total_pix;      // ... and with the pixel-wise split build's tables (total, -1 where it has none)
};
WsLayout psfsim_layout(int n, int64_t K, int storage, int n_r);
// FUSED storage's copy of the library: one 32-byte pair entry per bracket
// pair and padded pixel, plus a zero entry; psfsim_launch_pair_library also
// writes the column table (fused.cu).
int64_t psfsim_pair_library_bytes(int n, int n_r);
// ... and its column table: the generators' (angle-sorted) columns, with
// their starting coordinates, steps and weights, padded to whole k-tiles.
int64_t psfsim_fused_columns_bytes(int64_t K);
// ... and its M-tile order (the image's 8 x 16 pixel tiles, nearest the centre first).
int64_t psfsim_fused_mtile_order_bytes(int n);
cudaError_t psfsim_launch_pair_library(psfsim_plan *h, cudaStream_t st);
cudaError_t psfsim_launch_pair_entries(const float *lib, int n, int n_r, float *entries, int num_sms, cudaStream_t st);
// Extra workspace of the pixel-wise dense split build of an even grid (0: it does not apply; split_build.cu).
int64_t psfsim_pixel_build_bytes(int n, int64_t K, int storage, int n_r);

// Live (not identically zero) columns of a dense plan on a scene grid: counted
// on the host, listed in the workspace by the build (live.cu).
void psfsim_live_count(psfsim_plan *h);
cudaError_t psfsim_launch_live_table(psfsim_plan *h, cudaStream_t st);

// Kernel launchers (return cudaError_t of the launch).
cudaError_t psfsim_launch_build(psfsim_plan *h, cudaStream_t st);
cudaError_t psfsim_launch_forward_fp32(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                       bool skip_zeros, cudaStream_t st);
size_t psfsim_forward_fp32_scratch(const psfsim_plan *h, int B);
cudaError_t psfsim_launch_adjoint_fp32(const psfsim_plan *h, const float *g, int B, float *gx,
                                       cudaStream_t st);
// y[b, i] = sum_ks part[(ks * B + b) * ld + i], fixed order.
cudaError_t psfsim_launch_reduce_partials(const float *part, int KS, int B, int64_t ld, int64_t M, float *y,
                                          cudaStream_t st);
// Split-BF16 and BF16 storage: build, tensor-core forward and adjoint.  A product's
// scratch is reported monotone in the batch; the launchers check it against what
// the call takes, before they enqueue anything (kScratchTooSmall), so that a call is
// planned once.
constexpr cudaError_t kScratchTooSmall = cudaErrorMemoryValueTooLarge;
cudaError_t psfsim_launch_split_build(psfsim_plan *h, cudaStream_t st);
size_t psfsim_forward_tc_scratch(const psfsim_plan *h, int B);  // compact storage: of B rotated scenes
size_t psfsim_tc_taken(const psfsim_plan *h, int B, bool adjoint);  // the call's own launches
int psfsim_tc_run(const psfsim_plan *h, int B, bool adjoint);       // most k-tiles that one unit adds up
cudaError_t psfsim_launch_forward_tc(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                     size_t scratch_bytes, cudaStream_t st);
cudaError_t psfsim_launch_forward_tc_sym(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                         size_t scratch_bytes, cudaStream_t st);
// Images from the partial images of rotated scenes (sym.cu): rotated scene
// q = 4 b + m is slot q % per of block q / per, whose partials are
// part[KS][cap][rows]; y[b][i] = sum_m sum_ks part at P^-m(i).
struct SymSum {
  const float *part[16];  // the caller's scratch: several splits are added in place
  int cap[16], KS[16];
  int per, n;
  int64_t rows;
};
cudaError_t psfsim_launch_sym_sum(SymSum S, int B, float *y, cudaStream_t st);
// Adjoint of split and BF16 storage, dense or compact, on the tensor cores.
size_t psfsim_adjoint_tc_scratch(const psfsim_plan *h, int B);  // compact storage: of B turned residuals
cudaError_t psfsim_launch_adjoint_tc(const psfsim_plan *h, const float *g, int B, float *gx, void *scratch,
                                     size_t scratch_bytes, cudaStream_t st);
// ... of one residual where (nearly) every column is read, on CUDA cores (split_adjoint.cu).
bool psfsim_adjoint_one_better(const psfsim_plan *h);
size_t psfsim_adjoint_one_scratch(const psfsim_plan *h);
cudaError_t psfsim_launch_adjoint_one(const psfsim_plan *h, const float *g, float *gx, void *scratch, cudaStream_t st);
// Test hook: a tensor-core forward of one job, or of the wide form, on one CTA with
// every wait bounded by wait_ns and load number stall_it never issued.
bool psfsim_forward_tc_one_launch(const psfsim_plan *h, int B);
cudaError_t psfsim_launch_forward_tc_stall(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                           size_t scratch_bytes, uint64_t wait_ns, int64_t stall_it, cudaStream_t st);
// Multi-job persistent tensor-core forward (several split-BF16 plans, one launch).
int psfsim_multi_validate(const psfsim_job_t *jobs, int njobs);
size_t psfsim_forward_multi_scratch(const psfsim_job_t *jobs, int njobs, const psfsim_tuning_t *tune);
cudaError_t psfsim_launch_forward_multi(const psfsim_job_t *jobs, int njobs, const psfsim_tuning_t *tune,
                                        void *scratch, size_t scratch_bytes, cudaStream_t st);
// FP32 forward products (column-major A, gemv.cu): partial images part[KS][B][ld].
struct FwdCols {
  const float *A;
  int64_t ld;
  const float *x;     // [B][K] scenes (or whole scenes whose rotations are the batch, see order)
  int64_t K;          // scene pixels
  const int *live;    // columns read, ascending (NULL: all)
  int64_t L;          // how many
  const int *dead;    // the other columns: zero in A, but a non-finite scene value there makes the image NaN
  int64_t D;
  const int *order;   // compact storage: quadrant pixel of every column; scene b / 4 turned b % 4 times is slot b
  int N;
  int B;
  float *part;
};
int psfsim_gemv_max_splits(int64_t ld, int64_t K, int num_sms);  // sizes the caller's scratch
cudaError_t psfsim_launch_gemv_partials(const FwdCols &P, int max_splits, int num_sms, bool skip_zeros, int *KS,
                                        cudaStream_t st);
// FP32 adjoint products: gx[b][column] = sum_i A[i, column] g[b][i].
struct AdjCols {
  const float *A;
  int64_t ld, M;
  const float *g;     // [B][M]
  float *gx;          // [B][K]
  int64_t K;
  const int *live;    // columns read, ascending (NULL: all)
  int64_t L;
  const int *dead;    // the other columns: zero, or NaN for a residual that is not finite everywhere
  int64_t D;
  int B;
};
cudaError_t psfsim_launch_adjoint_cols(const AdjCols &P, int num_sms, cudaStream_t st);
// FP32 storage compacted by the quarter-turn symmetry and zero columns.
size_t psfsim_forward_sym_scratch(const psfsim_plan *h, int B);
cudaError_t psfsim_launch_forward_sym(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                      cudaStream_t st);
size_t psfsim_adjoint_sym_scratch(const psfsim_plan *h, int B);
cudaError_t psfsim_launch_adjoint_sym(const psfsim_plan *h, const float *g, int B, float *gx, void *scratch,
                                      cudaStream_t st);
// Fused (A regenerated on chip) forward.
size_t psfsim_forward_fused_scratch(const psfsim_plan *h, int B);
cudaError_t psfsim_launch_forward_fused(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                        cudaStream_t st);
// Test hook: the fused forward of <= 32 scenes on one CTA with every wait
// bounded by wait_ns and the x load of k-tile number stall_load never issued.
cudaError_t psfsim_launch_forward_fused_stall(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                              uint64_t wait_ns, int64_t stall_load, cudaStream_t st);

static inline int64_t psfsim_round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

// Columns stored in A: the quadrant's valid columns for the compacted storages.
static inline int64_t psfsim_cols(const psfsim_plan *h) { return h->quadrant ? h->K_valid : h->K; }

// Split-BF16 storage compacted by the quarter-turn symmetry (sym.cu).
size_t psfsim_forward_split_sym_scratch(const psfsim_plan *h, int B);
cudaError_t psfsim_launch_forward_split_sym(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                            size_t scratch_bytes, cudaStream_t st);

// Launch configuration with programmatic stream serialization: the kernel may
// be scheduled while the previous kernel in the stream finishes; it calls
// griddep_wait before touching that kernel's results.
inline cudaLaunchConfig_t psfsim_pdl_config(dim3 grid, int threads, cudaStream_t st, cudaLaunchAttribute (&attr)[1]) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Fit gradient on FP32_SYM storage (the compact quadrant matrix), three
// launches; the C-ABI calls in fit_gradient.cu dispatch here.
struct RingParams;
size_t psfsim_sym_gradient_scratch(psfsim_plan *h);
cudaError_t psfsim_sym_forward_loss(psfsim_plan *h, const RingParams &P, const float *d, double sigma, float *z,
                                    float *y, float *r, void *scratch, cudaStream_t st);
cudaError_t psfsim_sym_adjoint_chain(psfsim_plan *h, const float *r, float *gz, double *out, void *scratch,
                                     cudaStream_t st);
