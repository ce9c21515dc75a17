// FP32 storage compacted by two exact structures of A (PSFSIM_FP32_SYM):
//   * columns of scene pixels beyond the last library radius are zero
//     (nothing is stored for them);
//   * quarter-turn symmetry: with fixed-point rotation coordinates the column
//     of scene pixel R(j) = (-y, x) is bit-exactly the column of pixel j with
//     the image turned by a quarter (P), so only the x > 0, y > 0 quadrant
//     Q0 of an even N x N scene is stored.
// Forward:  S = sum_{m=0..3} P^m (A_Q0 X^(m)),  X^(m)_t = x_{R^m(j_t)};
// adjoint:  (A^T g)_{R^m(j_t)} = (A_Q0^T (g o P^m))_t.
// Both reuse the FP32 GEMV kernels on the compact matrix (K_valid columns)
// with the four rotations as a batch of four; the forward gathers them itself,
// and permutation kernels carry the symmetry on the image side.  Results equal the dense FP32 path up to
// the order of the FP32 sums.
#include "psfsim_internal.cuh"

namespace {

__device__ __forceinline__ void rotate_pixel(int N, int m, int &ix, int &iy) {
  for (int r = 0; r < m; ++r) {  // R(ix, iy) = (N-1-iy, ix): (x, y) -> (-y, x)
    const int nx = N - 1 - iy;
    iy = ix;
    ix = nx;
  }
}

// P^m of an image pixel: (p, q) -> (q, n-1-p), applied m times.
__device__ __forceinline__ int64_t perm_pixel(int n, int m, int64_t i) {
  int p = (int)(i / n), q = (int)(i % n);
  for (int r = 0; r < m; ++r) {
    const int np = q;
    q = n - 1 - p;
    p = np;
  }
  return (int64_t)p * n + q;
}

// y[b][i] = sum_m sum_ks part_m[ks][P^-m(i)] (fixed order), one 32 x 32 pixel
// block of an image per CTA: the quarter and three-quarter turns are read along
// their own rows and transposed through shared memory, so every access is a run
// of 32 pixels, and k-splits and rotations are added in one pass over the
// partial images.  Bound by reading them; a thread has the 8 loads of its two
// pixels in flight (one pixel of 1024 threads and two dependent rounds of
// loads: 58 us for 256 rotated images of 256 x 256, 39 now; a copy per job
// and a gather through the permutations took 154).
constexpr int kSumThreads = 512;
__global__ void __launch_bounds__(kSumThreads) sym_sum_kernel(const __grid_constant__ SymSum S, float *__restrict__ y) {
  __shared__ float t1[32][33], t3[32][33];
  constexpr int kRows = kSumThreads / 32, kPer = 32 / kRows;
  const int n = S.n, b = blockIdx.z;
  const int P0 = blockIdx.y * 32, Q0 = blockIdx.x * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int blk = 4 * b / S.per, slot = 4 * b % S.per;  // a scene's four rotations share a block
  const int64_t step = (int64_t)S.cap[blk] * S.rows;
  const float *v = S.part[blk] + (int64_t)slot * S.rows;
  float acc[kPer][4] = {};
#pragma unroll 4
  for (int ks = 0; ks < S.KS[blk]; ++ks, v += step) {
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int r = ty + e * kRows;
      if (Q0 + r < n && P0 + tx < n) {  // P^-1(p, q) = (n-1-q, p), P^-3(p, q) = (q, n-1-p)
        acc[e][1] += v[S.rows + (int64_t)(n - 1 - Q0 - r) * n + P0 + tx];
        acc[e][3] += v[3 * S.rows + (int64_t)(Q0 + r) * n + n - 1 - P0 - tx];
      }
      if (P0 + r < n && Q0 + tx < n) {
        acc[e][0] += v[(int64_t)(P0 + r) * n + Q0 + tx];
        acc[e][2] += v[2 * S.rows + (int64_t)(n - 1 - P0 - r) * n + n - 1 - Q0 - tx];
      }
    }
  }
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    t1[ty + e * kRows][tx] = acc[e][1];
    t3[ty + e * kRows][tx] = acc[e][3];
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    const int r = ty + e * kRows, p = P0 + r, q = Q0 + tx;
    if (p < n && q < n) y[((int64_t)b * n + p) * n + q] = ((acc[e][0] + t1[tx][r]) + acc[e][2]) + t3[tx][r];
  }
}

// gp[(b*4 + m) * M + i] = g[b][P^m(i)]; and gx (nz values) = 0, for the scene
// pixels without a column.
__global__ void sym_gperm(const float *__restrict__ g, int B, int n, float *__restrict__ gp, float *__restrict__ gx,
                          int64_t nz) {
  const int64_t M = (int64_t)n * n;
  const int64_t total = (int64_t)B * 4 * M;
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t idx = first; idx < total; idx += stride) {
    const int bm = (int)(idx / M);
    const int64_t i = idx % M;
    gp[idx] = g[(int64_t)(bm >> 2) * M + perm_pixel(n, bm & 3, i)];
  }
  for (int64_t j = first; j < nz; j += stride) gx[j] = 0.f;
}

// gx[b][R^m(order[t])] = gc[(b*4 + m) * Kv + t]; every other scene pixel is zero.
__global__ void sym_scatter(const float *__restrict__ gc, int B, int N, int64_t Kv, const int *__restrict__ order,
                            float *__restrict__ gx) {
  const int H = N / 2;
  const int64_t total = (int64_t)B * 4 * Kv;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int bm = (int)(idx / Kv);
    const int64_t t = idx % Kv;
    const int j0 = order[t];
    int ix = H + j0 % H, iy = H + j0 / H;
    rotate_pixel(N, bm & 3, ix, iy);
    gx[(int64_t)(bm >> 2) * N * N + (int64_t)iy * N + ix] = gc[idx];
  }
}

unsigned grid_for(int64_t total, int num_sms) {
  const int64_t g = (total + 255) / 256;
  const int64_t cap = (int64_t)num_sms * 16;
  return (unsigned)(g < 1 ? 1 : (g < cap ? g : cap));
}

// K-splits for the compact GEMV: partial sums kept well below the bytes of the
// compact A (at least 64 columns per split).
int sym_splits(const psfsim_plan *h) {
  const int ks = psfsim_gemv_max_splits(h->ld, h->K_valid, h->num_sms);
  const int64_t cap = h->K_valid / 64 > 0 ? h->K_valid / 64 : 1;
  return ks < cap ? ks : (int)cap;
}

}  // namespace

// Several k-splits are added first, in place, by the reduction (reduce.cuh): 28
// splits of one image's four rotations (16 CTAs here) took 60 us in this kernel's
// own loop, which keeps at most two.
cudaError_t psfsim_launch_sym_sum(SymSum S, int B, float *y, cudaStream_t st) {
  for (int blk = 0; blk * S.per < 4 * B; ++blk)
    if (S.KS[blk] > 2) {
      float *part = const_cast<float *>(S.part[blk]);
      const cudaError_t e = psfsim_launch_reduce_partials(part, S.KS[blk], S.cap[blk], S.rows, S.rows, part, st);
      if (e != cudaSuccess) return e;
      S.KS[blk] = 1;
    }
  const unsigned t = (unsigned)((S.n + 31) / 32);
  sym_sum_kernel<<<dim3(t, t, (unsigned)B), kSumThreads, 0, st>>>(S, y);
  return cudaGetLastError();
}

size_t psfsim_forward_sym_scratch(const psfsim_plan *h, int B) {
  return (size_t)sym_splits(h) * 4 * B * h->ld * 4;
}

// Two launches: the product over the four rotations of every scene, gathered
// by the product itself, and the sum over splits and rotations.
cudaError_t psfsim_launch_forward_sym(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                      cudaStream_t st) {
  if (h->K_valid == 0) return cudaMemsetAsync(y, 0, (size_t)B * h->M * 4, st);
  FwdCols P = {};
  P.A = reinterpret_cast<const float *>(h->ws + h->a_off);
  P.ld = h->ld;
  P.x = x;
  P.K = h->K;
  P.L = h->K_valid;
  P.order = reinterpret_cast<const int *>(h->ws + h->order_off);
  P.N = h->N;
  P.B = 4 * B;
  P.part = static_cast<float *>(scratch);
  int KS = 1;
  const cudaError_t e = psfsim_launch_gemv_partials(P, sym_splits(h), h->num_sms, false, &KS, st);
  if (e != cudaSuccess) return e;
  SymSum S = {};
  S.part[0] = P.part;
  S.cap[0] = P.B;
  S.KS[0] = KS;
  S.per = P.B;
  S.rows = h->ld;
  S.n = h->n;
  return psfsim_launch_sym_sum(S, B, y, st);
}

size_t psfsim_adjoint_sym_scratch(const psfsim_plan *h, int B) {
  return (size_t)psfsim_round_up((int64_t)4 * B * h->M * 4, 256) + (size_t)4 * B * h->K_valid * 4;
}

cudaError_t psfsim_launch_adjoint_sym(const psfsim_plan *h, const float *g, int B, float *gx, void *scratch,
                                      cudaStream_t st) {
  const int *order = reinterpret_cast<const int *>(h->ws + h->order_off);
  const float *A = reinterpret_cast<const float *>(h->ws + h->a_off);
  float *gp = static_cast<float *>(scratch);
  float *gc = reinterpret_cast<float *>(static_cast<char *>(scratch) + psfsim_round_up((int64_t)4 * B * h->M * 4, 256));
  if (h->K_valid == 0) return cudaMemsetAsync(gx, 0, (size_t)B * h->K * 4, st);
  cudaError_t e;
  sym_gperm<<<grid_for((int64_t)4 * B * h->M, h->num_sms), 256, 0, st>>>(g, B, h->n, gp, gx, (int64_t)B * h->K);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  AdjCols P = {};
  P.A = A;
  P.ld = h->ld;
  P.M = h->M;
  P.g = gp;
  P.gx = gc;
  P.K = P.L = h->K_valid;
  P.B = 4 * B;
  if ((e = psfsim_launch_adjoint_cols(P, h->num_sms, st)) != cudaSuccess) return e;
  sym_scatter<<<grid_for((int64_t)4 * B * h->K_valid, h->num_sms), 256, 0, st>>>(gc, B, h->N, h->K_valid, order, gx);
  return cudaGetLastError();
}

// ---- split-BF16 storage with the same compaction (PSFSIM_SPLIT_BF16_SYM) ----
// Forward: the four rotated scenes of every scene run as a batch of 4B through
// the tcgen05 product over the compact columns (its scene split gathers them),
// and the 4B partial images are summed through the inverse quarter turns.  The
// adjoint is tc_gemm.cu's, over the four turns of every residual.

size_t psfsim_forward_split_sym_scratch(const psfsim_plan *h, int B) { return psfsim_forward_tc_scratch(h, 4 * B); }

cudaError_t psfsim_launch_forward_split_sym(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                            size_t scratch_bytes, cudaStream_t st) {
  return psfsim_launch_forward_tc_sym(h, x, B, y, scratch, scratch_bytes, st);
}
