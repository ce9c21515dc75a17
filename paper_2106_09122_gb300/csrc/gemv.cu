// Products with a stored FP32 A (column-major, each PSF contiguous):
//   forward  S = A Z   (Eq. 6): row-parallel, split over columns, partials in
//            caller scratch, then a fixed-order reduction (deterministic);
//   adjoint  A^T g:            contiguous column ranges per CTA, rows split
//            across the CTA, fixed-order reduction.
#include "gemv_device.cuh"
#include "psfsim_internal.cuh"
#include "reduce.cuh"

using namespace psfsim_gemv;

namespace {

// Forward partials: CTA (tile, ks) adds the ks-th share of the columns for 1024
// rows and BB scenes, part[(ks B + b0 + b) ld + r].  Bound by reading A once
// (B <= 16 scenes a pass; the FMAs of 16 take as long):
//   * only live columns are read (live.cu; 44 % of them at 12 of 16 lambda/D),
//     and with kFilter only those that are non-zero in some scene of the pass;
//   * a share is every KS-th group of four columns, so a filtered scene's flux
//     spreads evenly without a list made beforehand;
//   * the share's scene values go through shared memory, 256 columns at a
//     time, as BB contiguous floats a column: one 16-byte broadcast load
//     serves four scenes.  Read from global memory per thread, a group of 8
//     scenes ran at half the rate of one.
// 11 scenes of the 128^2 plan: 660 us in passes of 8, 2 and 1 over all columns,
// 95 us in one pass over the live ones (HBM floor 70).
constexpr int kChunkCols = kFwdThreads;
constexpr int kShare = 4;

__host__ __device__ constexpr int fwd_min_ctas(int BB) { return BB == 1 ? 6 : BB == 4 ? 4 : BB == 8 ? 3 : 2; }

template <int BB, bool kFilter, bool kSym>
__global__ void __launch_bounds__(kFwdThreads, fwd_min_ctas(BB)) fwd_cols_kernel(const FwdCols P, int b0, int nb) {
  __shared__ __align__(16) float xs[kChunkCols * BB];
  __shared__ int js[kChunkCols];
  __shared__ int used[kFwdThreads / 32];
  __shared__ unsigned bad;  // scenes with a non-finite value at a column that is not read
  const int64_t r = (int64_t)blockIdx.x * kRowsPerCta + 4 * threadIdx.x;
  const int KS = gridDim.y, ks = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int U = BB <= 4 ? 4 : 8;  // columns in flight per thread
  float acc[BB][4];
#pragma unroll
  for (int b = 0; b < BB; ++b) acc[b][0] = acc[b][1] = acc[b][2] = acc[b][3] = 0.f;
  if (threadIdx.x == 0) bad = 0u;
  if (!kSym && P.dead) {
    __syncthreads();
    for (int64_t e = ks + (int64_t)KS * threadIdx.x; e < P.D; e += (int64_t)KS * kFwdThreads) {
      const float *xj = P.x + (int64_t)b0 * P.K + P.dead[e];
      for (int b = 0; b < nb; ++b)
        if (!isfinite(xj[(int64_t)b * P.K])) atomicOr(&bad, 1u << b);
    }
  }
  const float *A = P.A + r;
  auto add = [&](const float4 &v, const float *xc) {
#pragma unroll
    for (int b = 0; b < BB; ++b) {
      acc[b][0] = fmaf(v.x, xc[b], acc[b][0]);
      acc[b][1] = fmaf(v.y, xc[b], acc[b][1]);
      acc[b][2] = fmaf(v.z, xc[b], acc[b][2]);
      acc[b][3] = fmaf(v.w, xc[b], acc[b][3]);
    }
  };
  auto values = [&](int c, float (&xc)[BB]) {
    if (BB == 1) {
      xc[0] = xs[c];
    } else {
#pragma unroll
      for (int b = 0; b < BB; b += 4) {
        const float4 q = *reinterpret_cast<const float4 *>(xs + c * BB + b);
        xc[b] = q.x;
        xc[b + 1 < BB ? b + 1 : 0] = q.y;
        xc[b + 2 < BB ? b + 2 : 0] = q.z;
        xc[b + 3 < BB ? b + 3 : 0] = q.w;
      }
    }
  };
  const int64_t groups = (P.L + kShare - 1) / kShare;
  for (int64_t base = 0; ks + KS * (base / kShare) < groups; base += kChunkCols) {
    const int64_t i = (ks + KS * ((base + threadIdx.x) / kShare)) * kShare + threadIdx.x % kShare;
    float xv[BB];
    int j = 0;
    bool take = i < P.L;
    if (take) {
      j = !kSym && P.live ? P.live[i] : (int)i;
      bool any = false;
#pragma unroll
      for (int b = 0; b < BB; ++b) {
        xv[b] = 0.f;
        if (b < nb) {
          if (kSym) {
            const int H = P.N / 2, j0 = P.order[i], q = b0 + b;
            int ix = H + j0 % H, iy = H + j0 / H;
            for (int k = 0; k < (q & 3); ++k) {  // R(ix, iy) = (N-1-iy, ix)
              const int nx = P.N - 1 - iy;
              iy = ix;
              ix = nx;
            }
            xv[b] = P.x[(int64_t)(q >> 2) * P.N * P.N + (int64_t)iy * P.N + ix];
          } else {
            xv[b] = P.x[(int64_t)(b0 + b) * P.K + j];
          }
          any = any || xv[b] != 0.f;
        }
      }
      if (kFilter) take = any;
    }
    // slots: the columns taken, in order (without the filter they fill the front anyway)
    const unsigned votes = __ballot_sync(0xffffffffu, take);
    __syncthreads();  // the chunk before is consumed
    if (lane == 0) used[warp] = __popc(votes);
    __syncthreads();
    int slot = __popc(votes & ((1u << lane) - 1u)), count = 0;
#pragma unroll
    for (int w = 0; w < kFwdThreads / 32; ++w) {
      if (w < warp) slot += used[w];
      count += used[w];
    }
    if (take) {
      js[slot] = j;
#pragma unroll
      for (int b = 0; b < BB; ++b) xs[slot * BB + b] = xv[b];
    }
    __syncthreads();
    if (r < P.ld) {
      int c = 0;
      for (; c + U <= count; c += U) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = ld_stream4(A + (int64_t)js[c + u] * P.ld);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          float xc[BB];
          values(c + u, xc);
          add(v[u], xc);
        }
      }
      for (; c < count; ++c) {
        const float4 v = ld_stream4(A + (int64_t)js[c] * P.ld);
        float xc[BB];
        values(c, xc);
        add(v, xc);
      }
    }
  }
  if (!kSym && P.dead) __syncthreads();
  if (r >= P.ld) return;
#pragma unroll
  for (int b = 0; b < BB; ++b) {
    if (b >= nb) break;
    const float z = !kSym && P.dead && (bad >> b & 1u) ? __int_as_float(0x7fffffff) : 0.f;
    *reinterpret_cast<float4 *>(P.part + ((int64_t)ks * P.B + b0 + b) * P.ld + r) =
        make_float4(acc[b][0] + z, acc[b][1] + z, acc[b][2] + z, acc[b][3] + z);
  }
}

// y[b, i] = sum_ks part[ks, b, i] (reduce.cuh).  y may be part itself with M = ld.
template <bool kSerial>
__global__ void __launch_bounds__(256) fwd_reduce_kernel(const float *part, int KS, int B, int64_t ld, int64_t M,
                                                         float *y) {
  const int b = blockIdx.y;
  reduce_partials<kSerial>(part + (int64_t)b * ld, (int64_t)B * ld, KS, ld, M, y + (int64_t)b * M);
}

// One residual: gx[j] = sum_i A[i, j] g[i] for the CTA's contiguous range of the
// live columns; the CTA's 256 threads split the rows (float4 strided), reduce in
// registers, then across warps through a double-buffered shared array.  Fixed
// assignment and order: deterministic.  The columns that are not read get zero,
// or NaN when some residual value is not finite (0 x inf), which the first
// column's pass over g finds out.
template <bool kVec>
__global__ void __launch_bounds__(kAdjThreads) adj_kernel(const AdjCols P, int b0) {
  __shared__ float red[2][kAdjThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t0 = P.L * blockIdx.x / gridDim.x, t1 = P.L * (blockIdx.x + 1) / gridDim.x;
  const float *g = P.g + (int64_t)b0 * P.M;
  float *gx = P.gx + (int64_t)b0 * P.K;
  int parity = 0;
  float zero = 0.f;  // 0, or NaN from this thread's rows
  for (int64_t t = t0; t < t1; ++t, parity ^= 1) {
    const int64_t j = P.live ? P.live[t] : t;
    const float *col = P.A + j * P.ld;
    const bool probe = P.dead && t == t0;
    float acc = 0.f;
    auto add = [&](const float4 &v, const float4 &gv) {
      acc = fmaf(v.x, gv.x, acc);
      acc = fmaf(v.y, gv.y, acc);
      acc = fmaf(v.z, gv.z, acc);
      acc = fmaf(v.w, gv.w, acc);
      if (probe) zero += 0.f * gv.x + 0.f * gv.y + 0.f * gv.z + 0.f * gv.w;
    };
    if (kVec) {
      const int64_t M4 = P.M >> 2;
      const float4 *g4 = reinterpret_cast<const float4 *>(g);
      int64_t i4 = threadIdx.x;
      constexpr int T = kAdjThreads;
      for (; i4 + 3 * T < M4; i4 += 4 * T) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = ld_stream4(col + 4 * (i4 + T * u));
#pragma unroll
        for (int u = 0; u < 4; ++u) add(v[u], __ldg(g4 + i4 + T * u));
      }
      for (; i4 < M4; i4 += T) add(ld_stream4(col + 4 * i4), __ldg(g4 + i4));
    } else {
      for (int64_t i = threadIdx.x; i < P.M; i += kAdjThreads) {
        const float gi = __ldg(g + i);
        acc = fmaf(__ldg(col + i), gi, acc);
        if (probe) zero += 0.f * gi;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) red[parity][warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      float s = red[parity][0];
#pragma unroll
      for (int w = 1; w < kAdjThreads / 32; ++w) s += red[parity][w];
      gx[j] = s;
    }
  }
  if (!P.dead) return;
  if (t0 == t1)  // no column of its own to look at g with
    for (int64_t i = threadIdx.x; i < P.M; i += kAdjThreads) zero += 0.f * g[i];
  const bool bad = __syncthreads_or(zero != 0.f);
  const int64_t d0 = P.D * blockIdx.x / gridDim.x, d1 = P.D * (blockIdx.x + 1) / gridDim.x;
  for (int64_t e = d0 + threadIdx.x; e < d1; e += kAdjThreads) gx[P.dead[e]] = bad ? __int_as_float(0x7fffffff) : 0.f;
}

// 2, 4 or 8 residuals and few columns: a CTA per column, the threads splitting the
// rows, every residual read from L2 once per column.  Where the batched kernel below
// has a CTA for two columns, its tiles of rows come one after another and that is what
// it takes.  8 residuals, this form / batched: 128^2 on 452 columns 14 / 21 us, on 608
// 15 / 21, 640 26 / 28, 1000 29 / 29; 160^2 on 452 21 / 32; a call of 64 on 64^2, 452
// columns 50 / 66.  A thread adds 16 products by themselves before its sum (the same
// time; 64 registers, four CTAs an SM).
template <int BB, bool kVec>
__global__ void __launch_bounds__(kAdjThreads) adj_few_kernel(const AdjCols P, int b0) {
  __shared__ float red[2][kAdjThreads / 32][BB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t0 = P.L * blockIdx.x / gridDim.x, t1 = P.L * (blockIdx.x + 1) / gridDim.x;
  const float *g = P.g + (int64_t)b0 * P.M;
  int parity = 0;
  for (int64_t t = t0; t < t1; ++t, parity ^= 1) {
    const int64_t j = P.live ? P.live[t] : t;
    const float *col = P.A + j * P.ld;
    float acc[BB];
#pragma unroll
    for (int b = 0; b < BB; ++b) acc[b] = 0.f;
    if (kVec) {
      const int64_t M4 = P.M >> 2;
      int64_t i4 = threadIdx.x;
      constexpr int T = kAdjThreads;
      auto add = [&](const float4 &v, int64_t at, float (&s)[BB]) {
#pragma unroll
        for (int b = 0; b < BB; ++b) {
          const float4 gv = __ldg(reinterpret_cast<const float4 *>(g + (int64_t)b * P.M) + at);
          s[b] = fmaf(v.x, gv.x, s[b]);
          s[b] = fmaf(v.y, gv.y, s[b]);
          s[b] = fmaf(v.z, gv.z, s[b]);
          s[b] = fmaf(v.w, gv.w, s[b]);
        }
      };
      for (; i4 + 3 * T < M4; i4 += 4 * T) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = ld_stream4(col + 4 * (i4 + T * u));
        float s[BB];
#pragma unroll
        for (int b = 0; b < BB; ++b) s[b] = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u) add(v[u], i4 + T * u, s);
#pragma unroll
        for (int b = 0; b < BB; ++b) acc[b] += s[b];
      }
      for (; i4 < M4; i4 += T) add(ld_stream4(col + 4 * i4), i4, acc);
    } else {
      for (int64_t i = threadIdx.x; i < P.M; i += kAdjThreads) {
        const float v = __ldg(col + i);
#pragma unroll
        for (int b = 0; b < BB; ++b) acc[b] = fmaf(v, __ldg(g + (int64_t)b * P.M + i), acc[b]);
      }
    }
#pragma unroll
    for (int b = 0; b < BB; ++b) {
      float s = acc[b];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) red[parity][warp][b] = s;
    }
    __syncthreads();
    if (threadIdx.x < BB) {
      float s = red[parity][0][threadIdx.x];
#pragma unroll
      for (int w = 1; w < kAdjThreads / 32; ++w) s += red[parity][w][threadIdx.x];
      P.gx[(int64_t)(b0 + threadIdx.x) * P.K + j] = s;
    }
  }
}

// Several residuals: a CTA owns a contiguous range of the live columns (at most
// kAdjCols at a time) and walks the rows in tiles of 2048, eight rows a thread,
// with the tile's BB residuals in registers, two columns in hand at once.  Their
// 2 BB sums are halved across the warp's lanes until each group of lanes holds
// one, which it adds to its place in shared memory.  Bound by reading A once per
// BB residuals, then by issue: the more rows a thread has, the less the exchange
// of its sums weighs (with four rows a thread and 32 sums it took as long as the
// FMAs, 122 us for 8 residuals of the 128^2 plan; 102 now).  Reading the residuals from
// L2 per column instead moved eight times A's bytes: 320 us.
constexpr int kAdjCols = 64;
__host__ __device__ constexpr int adj_min_ctas(int BB) { return BB == 8 ? 2 : 3; }

template <int BB>
__global__ void __launch_bounds__(kAdjThreads, adj_min_ctas(BB)) adj_batch_kernel(const AdjCols P, int b0, int nb) {
  constexpr int R = 2;                        // row quads a thread holds
  constexpr int kTile = 4 * R * kAdjThreads;  // rows per tile
  constexpr int S = 2 * BB, kLanes = 32 / S;  // sums in hand; lanes that end with the same one
  __shared__ float red[kAdjThreads / 32][kAdjCols * BB];
  __shared__ int js[kAdjCols];
  __shared__ unsigned bad;  // residuals with a non-finite value
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t0 = P.L * blockIdx.x / gridDim.x, t1 = P.L * (blockIdx.x + 1) / gridDim.x;
  const bool vec = P.M % 4 == 0 && (reinterpret_cast<uintptr_t>(P.g) & 15) == 0;
  if (threadIdx.x == 0) bad = 0u;
  unsigned mine = 0u;
  bool probe = P.dead != nullptr;
  for (int64_t p0 = t0; p0 < t1 || probe; p0 += kAdjCols) {
    const int cols = (int)(t1 - p0 < kAdjCols ? t1 - p0 : kAdjCols);
    if ((int)threadIdx.x < cols) js[threadIdx.x] = P.live ? P.live[p0 + threadIdx.x] : (int)(p0 + threadIdx.x);
    __syncthreads();
    // The thread's row quad h of a tile is r0 + 1024 h + 4 threadIdx.x.  A's
    // padding rows are zero and allocated up to ld, a multiple of 32.
    auto load_a = [&](int64_t r0, int q, float4 (&v)[2][R]) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const bool take = q + c < cols;
        const float *col = P.A + (int64_t)js[take ? q + c : 0] * P.ld + 4 * threadIdx.x;
#pragma unroll
        for (int h = 0; h < R; ++h) {
          const int64_t r = r0 + h * 4 * kAdjThreads;
          v[c][h] = ld_stream4_if(col + r, take && r + 4 * threadIdx.x < P.M);
        }
      }
    };
    float4 v[2][R], gv[BB][R];
    if (cols > 0) load_a(0, 0, v);
    for (int64_t r0 = 0; r0 < P.M; r0 += kTile) {
#pragma unroll
      for (int h = 0; h < R; ++h) {
        const int64_t r = r0 + h * 4 * kAdjThreads + 4 * threadIdx.x;
#pragma unroll
        for (int b = 0; b < BB; ++b) {
          gv[b][h] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (b < nb && r < P.M) {
            const float *gb = P.g + (int64_t)(b0 + b) * P.M + r;
            if (vec) {
              gv[b][h] = __ldg(reinterpret_cast<const float4 *>(gb));
            } else {
              gv[b][h].x = gb[0];
              if (r + 1 < P.M) gv[b][h].y = gb[1];
              if (r + 2 < P.M) gv[b][h].z = gb[2];
              if (r + 3 < P.M) gv[b][h].w = gb[3];
            }
          }
        }
      }
      if (probe)
#pragma unroll
        for (int b = 0; b < BB; ++b)
#pragma unroll
          for (int h = 0; h < R; ++h)
            if (!(isfinite(gv[b][h].x) && isfinite(gv[b][h].y) && isfinite(gv[b][h].z) && isfinite(gv[b][h].w)))
              mine |= 1u << b;
      for (int q = 0; q < cols; q += 2) {
        float s[S];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int b = 0; b < BB; ++b) {
            float t = 0.f;
#pragma unroll
            for (int h = 0; h < R; ++h) {
              t = fmaf(v[c][h].x, gv[b][h].x, t);
              t = fmaf(v[c][h].y, gv[b][h].y, t);
              t = fmaf(v[c][h].z, gv[b][h].z, t);
              t = fmaf(v[c][h].w, gv[b][h].w, t);
            }
            s[c * BB + b] = t;
          }
        // The next columns load while these sums are exchanged.
        if (q + 2 < cols)
          load_a(r0, q + 2, v);
        else if (r0 + kTile < P.M)
          load_a(r0 + kTile, 0, v);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const int o = 16 >> k, n = S >> (k + 1);
          if (n > 0) {  // a lane keeps the half of its sums that its bit o names
#pragma unroll
            for (int i = 0; i < BB; ++i)
              if (i < n) {
                const bool up = lane & o;
                const float keep = up ? s[i + n] : s[i], give = up ? s[i] : s[i + n];
                s[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
              }
          } else {
            s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
          }
        }
        if (lane % kLanes == 0) {  // sum lane / kLanes: column q + sum / BB, residual sum % BB
          float *slot = &red[warp][q * BB + lane / kLanes];
          *slot = r0 == 0 ? s[0] : *slot + s[0];
        }
      }
    }
    __syncthreads();
    for (int o = threadIdx.x; o < cols * BB; o += kAdjThreads) {
      const int b = o % BB;
      float s = red[0][o];
#pragma unroll
      for (int w = 1; w < kAdjThreads / 32; ++w) s += red[w][o];
      if (b < nb) P.gx[(int64_t)(b0 + b) * P.K + js[o / BB]] = s;
    }
    probe = false;
    __syncthreads();
  }
  if (!P.dead) return;
  if (mine) atomicOr(&bad, mine);
  __syncthreads();
  const int64_t d0 = P.D * blockIdx.x / gridDim.x, d1 = P.D * (blockIdx.x + 1) / gridDim.x;
  for (int64_t e = d0 + threadIdx.x; e < d1; e += kAdjThreads)
    for (int b = 0; b < nb; ++b)
      P.gx[(int64_t)(b0 + b) * P.K + P.dead[e]] = bad >> b & 1u ? __int_as_float(0x7fffffff) : 0.f;
}

// One pass: nb scenes from b0 with KS splits.
cudaError_t fwd_pass(const FwdCols &P, int BB, int b0, int nb, int KS, bool filter, cudaStream_t st) {
  const dim3 grid((unsigned)((P.ld + kRowsPerCta - 1) / kRowsPerCta), (unsigned)KS);
  auto go = [&](auto kern) {
    kern<<<grid, kFwdThreads, 0, st>>>(P, b0, nb);
    return cudaGetLastError();
  };
#define PSFSIM_FWD(n)                                                                                          \
  (P.order ? go(fwd_cols_kernel<n, false, true>)                                                               \
           : filter ? go(fwd_cols_kernel<n, true, false>) : go(fwd_cols_kernel<n, false, false>))
  switch (BB) {
    case 1: return filter ? go(fwd_cols_kernel<1, true, false>) : go(fwd_cols_kernel<1, false, false>);
    case 4: return PSFSIM_FWD(4);
    case 8: return PSFSIM_FWD(8);
    case 12: return PSFSIM_FWD(12);
    default: return PSFSIM_FWD(16);
  }
#undef PSFSIM_FWD
}

FwdCols fwd_cols(const psfsim_plan *h, const float *x, int B, float *part) {
  const int *list = reinterpret_cast<const int *>(h->ws + h->order_off);
  FwdCols P;
  P.A = reinterpret_cast<const float *>(h->ws + h->a_off);
  P.ld = h->ld;
  P.x = x;
  P.K = h->K;
  P.live = h->live ? list : nullptr;
  P.L = h->live_cols;
  P.dead = h->live ? list + h->live_cols : nullptr;
  P.D = h->K - h->live_cols;
  P.order = nullptr;
  P.N = h->N;
  P.B = B;
  P.part = part;
  return P;
}

}  // namespace

// Column splits the scratch of a forward allows: eight CTAs an SM over the row
// tiles, at least 8 columns each.
int psfsim_gemv_max_splits(int64_t ld, int64_t K, int num_sms) {
  const int64_t row_blocks = (ld + kRowsPerCta - 1) / kRowsPerCta;
  int64_t ks = (int64_t)num_sms * 8 / row_blocks;
  ks = ks < 1 ? 1 : ks;
  const int64_t max_ks = K / 8 > 0 ? K / 8 : 1;
  return (int)(ks < max_ks ? ks : max_ks);
}

// Passes of at most 16 scenes, evenly filled, with whole waves of resident CTAs.
cudaError_t psfsim_launch_gemv_partials(const FwdCols &P, int max_splits, int num_sms, bool skip_zeros, int *KS_out,
                                        cudaStream_t st) {
  const int passes = (P.B + 15) / 16, per0 = (P.B + passes - 1) / passes;
  const int per = P.order ? (per0 + 3) / 4 * 4 : per0;  // a scene's rotations stay together
  const int BB = per == 1 ? 1 : (per + 3) / 4 * 4;
  const int64_t row_blocks = (P.ld + kRowsPerCta - 1) / kRowsPerCta;
  int64_t KS = (int64_t)num_sms * fwd_min_ctas(BB) / row_blocks;
  const int64_t max_ks = P.L / 8 > 0 ? P.L / 8 : 1;
  KS = KS < 1 ? 1 : KS;
  // A thread adds its share's columns one after another, and 12 or 16 scenes leave
  // few CTAs: where that chain is long, whole waves of shorter shares.  Image of 16
  // scenes against 64 bits, one wave / now: 256^2 of 128^2 4.5e-7 / 1.4e-7, 160^2
  // 2.2e-7 / 1.3e-7, 128^2 1.21e-7 / 0.89e-7; time 452 / 466, 252 / 261 and 114 / 121
  // us (11 scenes: 93 / 95).  Shorter chains gain nothing that the longer sum over
  // splits does not lose.  Sub-sums of 8 columns or sums folded into shared memory
  // every 64 cost 8 to 13 % at all sizes.
  const int64_t chain = P.L / KS, waves = chain > 320 && chain <= 512 ? 2 : (chain + 511) / 512;
  const int64_t most = max_splits / KS > 1 ? max_splits / KS : 1;
  KS *= waves < 1 ? 1 : waves < most ? waves : most;
  KS = KS < max_ks ? KS : max_ks;
  KS = KS < max_splits ? KS : max_splits;
  *KS_out = (int)KS;
  for (int b0 = 0; b0 < P.B; b0 += per) {
    const cudaError_t e = fwd_pass(P, BB, b0, P.B - b0 < per ? P.B - b0 : per, (int)KS, skip_zeros, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// One residual at a time, or passes of 2 to 8.  The form for few columns takes those of
// a compact plan or of field points (dense grids also have their dead columns to fill,
// for which every CTA would look through the residuals) where each has a CTA resident
// at once, four an SM.  Passes of 2 and 4 also between 6 and 8 columns an SM, two rounds
// of it where the batched form's CTAs, three an SM, have more than a pair each: 4
// residuals of 128^2 on 1000 columns 20 / 25 us, 160^2 on 1200 30 / 38; between 4 and 6
// both take the same.  Passes of 3, 5, 6 or 7 never do: that form would make two of them.
cudaError_t psfsim_launch_adjoint_cols(const AdjCols &P, int num_sms, cudaStream_t st) {
  const bool vec = (P.M % 4 == 0) && ((reinterpret_cast<uintptr_t>(P.g) & 15) == 0);
  auto grid_of = [](int64_t n) { return (unsigned)(n < 1 ? 1 : n); };
  for (int b0 = 0, nb; b0 < P.B; b0 += nb) {
    const int left = P.B - b0;
    if (left == 1) {
      nb = 1;
      auto kern = vec ? adj_kernel<true> : adj_kernel<false>;
      int per_sm = 1;
      const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kAdjThreads, 0);
      if (e != cudaSuccess) return e;
      const int64_t grid = (int64_t)num_sms * (per_sm < 1 ? 1 : per_sm);
      kern<<<grid_of(grid < P.L ? grid : P.L), kAdjThreads, 0, st>>>(P, b0);
    } else if (!P.dead && (left >= 8 || left == 4 || left == 2) &&
               (P.L <= 4ll * num_sms || (left < 8 && P.L > 6ll * num_sms && P.L <= 8ll * num_sms))) {
      nb = left >= 8 ? 8 : left;
      auto kern = nb == 8   ? (vec ? adj_few_kernel<8, true> : adj_few_kernel<8, false>)
                  : nb == 4 ? (vec ? adj_few_kernel<4, true> : adj_few_kernel<4, false>)
                            : (vec ? adj_few_kernel<2, true> : adj_few_kernel<2, false>);
      kern<<<grid_of(P.L), kAdjThreads, 0, st>>>(P, b0);
    } else {
      const int passes = (left + 7) / 8;
      nb = (left + passes - 1) / passes;
      const int per_sm = adj_min_ctas(nb <= 4 ? 4 : 8);
      auto kern = nb <= 4 ? adj_batch_kernel<4> : adj_batch_kernel<8>;
      const int64_t grid = (P.L + 1) / 2, most = (int64_t)per_sm * num_sms;
      kern<<<grid_of(grid < most ? grid : most), kAdjThreads, 0, st>>>(P, b0, nb);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t psfsim_forward_fp32_scratch(const psfsim_plan *h, int B) {
  return (size_t)psfsim_gemv_max_splits(h->ld, h->K, h->num_sms) * (size_t)B * (size_t)h->ld * 4;
}

// skip_zeros: only the columns of scene pixels that are non-zero in some scene
// of a pass.  Without zeros the columns, their shares and so the bits are those
// of the dense forward.
cudaError_t psfsim_launch_forward_fp32(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                       bool skip_zeros, cudaStream_t st) {
  float *part = reinterpret_cast<float *>(scratch);
  int KS = 1;
  const cudaError_t e = psfsim_launch_gemv_partials(fwd_cols(h, x, B, part),
                                                    psfsim_gemv_max_splits(h->ld, h->K, h->num_sms), h->num_sms,
                                                    skip_zeros, &KS, st);
  if (e != cudaSuccess) return e;
  return psfsim_launch_reduce_partials(part, KS, B, h->ld, h->M, y, st);
}

cudaError_t psfsim_launch_reduce_partials(const float *part, int KS, int B, int64_t ld, int64_t M, float *y,
                                          cudaStream_t st) {
  const bool serial = reduce_serial(KS, (int64_t)B * M);
  const dim3 grid((unsigned)reduce_ctas(serial, M), (unsigned)B);
  if (serial)
    fwd_reduce_kernel<true><<<grid, 256, 0, st>>>(part, KS, B, ld, M, y);
  else
    fwd_reduce_kernel<false><<<grid, 256, 0, st>>>(part, KS, B, ld, M, y);
  return cudaGetLastError();
}

cudaError_t psfsim_launch_adjoint_fp32(const psfsim_plan *h, const float *g, int B, float *gx, cudaStream_t st) {
  const int *list = reinterpret_cast<const int *>(h->ws + h->order_off);
  AdjCols P;
  P.A = reinterpret_cast<const float *>(h->ws + h->a_off);
  P.ld = h->ld;
  P.M = h->M;
  P.g = g;
  P.gx = gx;
  P.K = h->K;
  P.live = h->live ? list : nullptr;
  P.L = h->live_cols;
  P.dead = h->live ? list + h->live_cols : nullptr;
  P.D = h->K - h->live_cols;
  P.B = B;
  return psfsim_launch_adjoint_cols(P, h->num_sms, st);
}
