// Device building blocks of the FP32 products with a stored A (column-major,
// each PSF contiguous), shared by the plain forward/adjoint kernels (gemv.cu)
// and the fit-gradient kernels (fit_gradient.cu, fit_sym.cu).  Both directions
// stream A once from HBM with 128-bit loads that bypass L1.
#pragma once

#include <stdint.h>

namespace psfsim_gemv {

__device__ __forceinline__ float4 ld_stream4(const float *p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}

// As ld_stream4, or zeros where !take (predicated: no branch around the load).
__device__ __forceinline__ float4 ld_stream4_if(const float *p, bool take) {
  float4 v;
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "mov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\tmov.f32 %2, 0f00000000;\n\tmov.f32 %3, 0f00000000;\n\t"
      "@q ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=&f"(v.x), "=&f"(v.y), "=&f"(v.z), "=&f"(v.w)
      : "l"(p), "r"((int)take));
  return v;
}

constexpr int kFwdThreads = 256;
constexpr int kRowsPerCta = kFwdThreads * 4;

// acc[b][e] = sum_{j0 <= j < j1} A[r + e, j] x[b kXStride + j - j0] for the
// thread's 4 rows, the range's scene values in shared memory.
template <int BB, int kXStride>
__device__ __forceinline__ void fwd_accumulate(const float *__restrict__ A, int64_t ld, const float *__restrict__ x,
                                               int64_t r, int64_t j0, int64_t j1, float (&acc)[BB][4]) {
#pragma unroll
  for (int b = 0; b < BB; ++b) acc[b][0] = acc[b][1] = acc[b][2] = acc[b][3] = 0.f;
  const float *a = A + j0 * ld + r;
  auto xval = [&](int b, int64_t j) -> float { return x[b * kXStride + (j - j0)]; };
  int64_t j = j0;
  for (; j + 4 <= j1; j += 4, a += 4 * ld) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = ld_stream4(a + u * ld);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int b = 0; b < BB; ++b) {
        const float xv = xval(b, j + u);
        acc[b][0] = fmaf(v[u].x, xv, acc[b][0]);
        acc[b][1] = fmaf(v[u].y, xv, acc[b][1]);
        acc[b][2] = fmaf(v[u].z, xv, acc[b][2]);
        acc[b][3] = fmaf(v[u].w, xv, acc[b][3]);
      }
    }
  }
  for (; j < j1; ++j, a += ld) {
    const float4 v = ld_stream4(a);
#pragma unroll
    for (int b = 0; b < BB; ++b) {
      const float xv = xval(b, j);
      acc[b][0] = fmaf(v.x, xv, acc[b][0]);
      acc[b][1] = fmaf(v.y, xv, acc[b][1]);
      acc[b][2] = fmaf(v.z, xv, acc[b][2]);
      acc[b][3] = fmaf(v.w, xv, acc[b][3]);
    }
  }
}

// acc[e] = sum_c A[r + e, js[c]] xs[c] for the thread's 4 rows over n listed
// columns, columns and values in shared memory.  The columns are added 16 at a
// time, so that no chain of roundings is longer than 16 + n / 16: some 140 columns
// a CTA in the 128^2 fit workload, whose image errs 0.73e-7 against 64 bits (the
// compact plan's single chains: 0.94e-7) at the same time; the loop waits for memory.
__device__ __forceinline__ void fwd_accumulate_list(const float *__restrict__ A, int64_t ld, const int *js,
                                                    const float *xs, int n, int64_t r, float (&acc)[4]) {
  acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
  const float *a = A + r;
  for (int c0 = 0; c0 < n; c0 += 16) {
    const int c1 = c0 + 16 < n ? c0 + 16 : n;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    auto add = [&](const float4 &v, float x) {
      s[0] = fmaf(v.x, x, s[0]);
      s[1] = fmaf(v.y, x, s[1]);
      s[2] = fmaf(v.z, x, s[2]);
      s[3] = fmaf(v.w, x, s[3]);
    };
    int c = c0;
    for (; c + 4 <= c1; c += 4) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = ld_stream4(a + (int64_t)js[c + u] * ld);
#pragma unroll
      for (int u = 0; u < 4; ++u) add(v[u], xs[c + u]);
    }
    for (; c < c1; ++c) add(ld_stream4(a + (int64_t)js[c] * ld), xs[c]);
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[e] += s[e];
  }
}

constexpr int kAdjThreads = 256;
constexpr int kStashCols = 128;

}  // namespace psfsim_gemv
