// Adjoint A^T g of one residual on split-BF16 or BF16 storage whose columns are
// (nearly) all read: gx[j] = sigma_j sum_i (hi_ij + lo_ij) g_i (lo = 0 for BF16).
// Each thread owns 8 consecutive columns (one 16-byte load of hi, and of lo, per
// row); the rows are split KS ways into partial sums in caller scratch, reduced in
// a fixed order (deterministic).  It streams A at HBM rate with two short launches,
// where the tensor-core form (tc_gemm.cu) has three and its tiles' latency, but it
// reads dead columns too.  One residual, this form / tensor cores, BF16: 48^2 images
// on 160^2 pixels, all live 27 / 38 us, 128^2 on 128^2 all live 87 / 101, 85 % of the
// k-tiles 87 / 87, 72 % 87 / 75; 256^2 on 128^2 314 / 348; split 128^2 161 / 172.
#include <cuda_bf16.h>

#include "psfsim_internal.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kColsPerCta = kThreads * 8;

__device__ __forceinline__ uint4 ld_stream16(const void *p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Row i's 8 columns from element `off`: hi + lo (kLo) or hi alone.
template <bool kLo>
__device__ __forceinline__ void load8(const __nv_bfloat16 *hi, const __nv_bfloat16 *lo, int64_t off, float (&a)[8]) {
  const uint4 h = ld_stream16(hi + off), l = kLo ? ld_stream16(lo + off) : make_uint4(0, 0, 0, 0);
  const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    a[2 * t] = __uint_as_float(hw[t] << 16) + __uint_as_float(lw[t] << 16);
    a[2 * t + 1] = __uint_as_float(hw[t] & 0xFFFF0000u) + __uint_as_float(lw[t] & 0xFFFF0000u);
  }
}

template <bool kLo>
__global__ void __launch_bounds__(kThreads) adj_one_kernel(const __nv_bfloat16 *__restrict__ hi,
                                                           const __nv_bfloat16 *__restrict__ lo,
                                                           const float *__restrict__ scale, int64_t ld, int64_t M,
                                                           const float *__restrict__ g, float *__restrict__ part) {
  const int64_t j = (int64_t)blockIdx.x * kColsPerCta + 8 * threadIdx.x;
  const int KS = gridDim.y, ks = blockIdx.y;
  if (j >= ld) return;
  const int64_t i0 = M * ks / KS, i1 = M * (ks + 1) / KS;
  float acc[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) acc[t] = 0.f;
  int64_t i = i0;
  for (; i + 2 <= i1; i += 2) {
    float a0[8], a1[8];
    load8<kLo>(hi, lo, i * ld + j, a0);
    load8<kLo>(hi, lo, (i + 1) * ld + j, a1);
    const float g0 = __ldg(g + i), g1 = __ldg(g + i + 1);
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[t] = fmaf(a1[t], g1, fmaf(a0[t], g0, acc[t]));
  }
  if (i < i1) {
    float a0[8];
    load8<kLo>(hi, lo, i * ld + j, a0);
    const float g0 = __ldg(g + i);
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[t] = fmaf(a0[t], g0, acc[t]);
  }
  float *out = part + (int64_t)ks * ld + j;
#pragma unroll
  for (int t = 0; t < 8; ++t) acc[t] *= scale[j + t];
  *reinterpret_cast<float4 *>(out) = make_float4(acc[0], acc[1], acc[2], acc[3]);
  *reinterpret_cast<float4 *>(out + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
}

// Eight CTAs an SM over the column blocks, at least 8 rows each.
int splits(const psfsim_plan *h) {
  const int64_t blocks = (h->ld + kColsPerCta - 1) / kColsPerCta, most = h->M / 8 > 0 ? h->M / 8 : 1;
  const int64_t ks = (int64_t)h->num_sms * 8 / blocks;
  return (int)(ks < 1 ? 1 : ks < most ? ks : most);
}

}  // namespace

// Where it is the faster one: dense storage of at least 8192 columns (fewer leave it
// hundreds of splits to sum) whose bytes exceed those of the k-tiles read by less than
// what the tensor-core form loses on them, 4.5 % and 30 MB (its extra launch and
// start-up, some 5 us).
bool psfsim_adjoint_one_better(const psfsim_plan *h) {
  if (h->quadrant || h->K < 8192) return false;
  const double row = h->lo_off >= 0 ? 4.0 : 2.0, rows = (double)h->M;
  return rows * row * (double)h->ld < 1.045 * rows * row * 64.0 * (double)h->k_tiles + 30e6;
}

size_t psfsim_adjoint_one_scratch(const psfsim_plan *h) { return (size_t)splits(h) * (size_t)h->ld * 4; }

cudaError_t psfsim_launch_adjoint_one(const psfsim_plan *h, const float *g, float *gx, void *scratch, cudaStream_t st) {
  const int KS = splits(h);
  float *part = static_cast<float *>(scratch);
  const __nv_bfloat16 *hi = reinterpret_cast<const __nv_bfloat16 *>(h->ws + h->a_off);
  const float *scale = reinterpret_cast<const float *>(h->ws + h->scale_off);
  const dim3 grid((unsigned)((h->ld + kColsPerCta - 1) / kColsPerCta), (unsigned)KS);
  if (h->lo_off >= 0)
    adj_one_kernel<true><<<grid, kThreads, 0, st>>>(hi, reinterpret_cast<const __nv_bfloat16 *>(h->ws + h->lo_off), scale,
                                                    h->ld, h->M, g, part);
  else
    adj_one_kernel<false><<<grid, kThreads, 0, st>>>(hi, nullptr, scale, h->ld, h->M, g, part);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return psfsim_launch_reduce_partials(part, KS, 1, h->ld, h->K, gx, st);
}
