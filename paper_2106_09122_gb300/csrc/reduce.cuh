// Sum of an image's k-split partials in a fixed order, by CTAs of 256 threads.
//   serial    a thread adds all partials of its 4 rows, four loads in flight, each
//             four added to each other first (a CTA: 1024 rows);
//   by warps  a CTA covers 128 rows, its 8 warps take ks = warp, warp + 8, ... and
//             combine through shared memory.
// Bound by reading the partials.  By warps alone, warps without a partial, many
// short CTAs and a barrier each cost more than that: 64 images of 65536 pixels from
// 2 partials 22.6 us, serial 8.3 (KS = 8: 39.0 / 24.7, 20: 71.7 / 52.5, 76 at 16
// images: 51.1 / 48.6).  With few rows and many partials the loads come one after
// another: one image of 16384 pixels from 76 partials 4.2 us by warps, 8.2 serial.
// From 2^18 rows on (images together) serial is never slower; below, four partials
// are one round of loads either way.  Two kernels: one holding both forms kept the
// registers of the larger (12 partials of 8 x 16384: 6.0 -> 7.4 us).
#pragma once

#include <stdint.h>

inline bool reduce_serial(int KS, int64_t rows) { return KS <= 4 || rows >= (1 << 18); }

inline int64_t reduce_ctas(bool serial, int64_t M) {
  const int64_t per = serial ? 1024 : 128;
  return (M + per - 1) / per;
}

// out[0 .. M) = sum_ks p[ks step + 0 .. rows), rows >= M a multiple of 4 and p, step
// 16-byte aligned.  out may be p itself with M = rows: a thread's rows are read
// before they are written, by itself or before a barrier.
template <bool kSerial>
__device__ __forceinline__ void reduce_partials(const float *p, int64_t step, int KS, int64_t rows, int64_t M,
                                                float *out) {
  const int c4 = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int64_t r = ((int64_t)blockIdx.x * (kSerial ? 256 : 32) + (kSerial ? (int)threadIdx.x : c4)) * 4;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [](float4 &a, const float4 &b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; };
  if (kSerial) {
    if (r >= M) return;
    p += r;
    for (int k0 = 0; k0 < KS; k0 += 4, p += 4 * step) {
      float4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        v[k] = k0 + k < KS ? *reinterpret_cast<const float4 *>(p + k * step) : make_float4(0.f, 0.f, 0.f, 0.f);
      add(v[0], v[1]);
      add(v[0], v[2]);
      add(v[0], v[3]);
      add(s, v[0]);
    }
  } else {
    __shared__ float4 red[8][32];
    if (r < rows) {
#pragma unroll 4
      for (int ks = grp; ks < KS; ks += 8) add(s, *reinterpret_cast<const float4 *>(p + ks * step + r));
    }
    red[grp][c4] = s;
    __syncthreads();
    if (grp != 0 || r >= M) return;
    s = red[0][c4];
#pragma unroll
    for (int k = 1; k < 8; ++k) add(s, red[k][c4]);
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
