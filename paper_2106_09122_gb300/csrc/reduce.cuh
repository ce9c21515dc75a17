// Sum of an image's k-split partials in a fixed order, by a CTA of 256 threads.
//   KS <= 8   a thread adds all partials of its 4 rows, its loads all in flight
//             (a CTA: 1024 rows);
//   KS > 8    a CTA covers 128 rows, its 8 warps take ks = warp, warp + 8, ...
//             and combine through shared memory.
// Bound by reading the partials.  With the second form alone, 6 of 8 warps had
// nothing to load at two splits: 64 images of 256 x 256 took 40 us over the
// same product without a split.
#pragma once

#include <stdint.h>

constexpr int kRedSerial = 8;

inline int64_t reduce_ctas(int KS, int64_t M) {
  const int64_t per = KS <= kRedSerial ? 1024 : 128;
  return (M + per - 1) / per;
}

// out[0 .. M) = sum_ks p[ks step + 0 .. rows), rows >= M a multiple of 4 and p, step
// 16-byte aligned.  out may be p itself with M = rows: a thread's rows are read
// before they are written, by itself or before a barrier.  red: shared memory.
__device__ __forceinline__ void reduce_partials(const float *p, int64_t step, int KS, int64_t rows, int64_t M,
                                                float *out, float4 (*red)[32]) {
  const bool serial = KS <= kRedSerial;
  const int c4 = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int64_t r = ((int64_t)blockIdx.x * (serial ? 256 : 32) + (serial ? threadIdx.x : c4)) * 4;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (serial) {
    if (r >= M) return;
    float4 v[kRedSerial];
#pragma unroll
    for (int k = 0; k < kRedSerial; ++k)
      if (k < KS) v[k] = *reinterpret_cast<const float4 *>(p + k * step + r);
#pragma unroll
    for (int k = 0; k < kRedSerial; ++k)
      if (k < KS) {
        s.x += v[k].x; s.y += v[k].y; s.z += v[k].z; s.w += v[k].w;
      }
  } else {
    if (r < rows) {
#pragma unroll 4
      for (int ks = grp; ks < KS; ks += 8) {
        const float4 v = *reinterpret_cast<const float4 *>(p + ks * step + r);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
      }
    }
    red[grp][c4] = s;
    __syncthreads();
    if (grp != 0 || r >= M) return;
    s = red[0][c4];
#pragma unroll
    for (int k = 1; k < 8; ++k) {
      const float4 v = red[k][c4];
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
  }
  if (r + 4 <= M && (reinterpret_cast<uintptr_t>(out + r) & 15) == 0) {
    *reinterpret_cast<float4 *>(out + r) = s;
    return;
  }
  out[r] = s.x;
  if (r + 1 < M) out[r + 1] = s.y;
  if (r + 2 < M) out[r + 2] = s.z;
  if (r + 3 < M) out[r + 3] = s.w;
}
