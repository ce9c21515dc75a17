// Split-BF16 and BF16 storage of A for the tensor-core path.
//
// A_ij (the same lerp + bilinear-rotation element as the FP32 build, Sec. 2)
// is stored as sigma_j (hi_ij + lo_ij): sigma_j is the smallest power of two
// >= max(max|L_k|, max|L_{k+1}|) over the column's radial bracket (an exact
// bound on |A_ij|, since the lerp and bilinear weights are convex), hi =
// RN_bf16(A_ij / sigma_j), lo = RN_bf16(A_ij / sigma_j - hi); BF16 storage
// keeps hi alone.  hi and lo are row-major [rows][ld] (each image pixel's row
// contiguous along the scene pixels: K-major for the MMA), ld = K rounded up
// to 64, rows = M rounded up to 128; padding is zero.
#include <cuda_bf16.h>

#include <cmath>

#include "live.cuh"
#include "psfsim_internal.cuh"

namespace {

constexpr int kTileRows = 128;
constexpr int kTileCols = 64;

// libmax[k] = max |L_k|, from zero: the CTAs of row blockIdx.y = k share its
// pixels (one CTA a PSF took 35 us for 60 PSFs of 256 x 256).  The maximum of
// non-negative floats is that of their bits; NaN is passed over, as by fmaxf.
constexpr int kMaxParts = 8;
__global__ void __launch_bounds__(256) libmax_kernel(const float *lib, int64_t M, float *libmax) {
  const float *L = lib + (int64_t)blockIdx.y * M;
  float m = 0.f;
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x)
    m = fmaxf(m, fabsf(L[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned *>(libmax) + blockIdx.y, __float_as_uint(m));
}

__device__ __forceinline__ float pow2_at_least(float m) {
  if (!(m > 0.f)) return 1.f;
  int e;
  const float f = frexpf(m, &e);  // m = f 2^e, f in [0.5, 1)
  return f == 0.5f ? m : ldexpf(1.f, e);
}

struct SplitParams {
  int n;
  int64_t K, ld, M, rows;
  const ColGeom *geom;
  const int *order;  // compacted storage: column j is geometry entry order[j] (else null: entry j)
  const float *lib;
  const float *libmax;
  __nv_bfloat16 *hi;
  __nv_bfloat16 *lo;  // null for BF16 storage
  float *scale;
};

__device__ __forceinline__ float element(const float *L0, const float *L1, int n, long long a2, long long b2,
                                         float w0, float w1) {
  constexpr int kShift = PSFSIM_FRAC_BITS + 1;
  const int q0 = (int)(a2 >> kShift);
  const int p0 = (int)(b2 >> kShift);
  if (q0 < -1 || q0 > n - 1 || p0 < -1 || p0 > n - 1) return 0.f;
  const unsigned fa = (unsigned)((unsigned long long)a2 >> (kShift - 32));
  const unsigned fb = (unsigned)((unsigned long long)b2 >> (kShift - 32));
  constexpr float kInv32 = 2.3283064365386963e-10f;
  const float wa1 = __uint2float_rn(fa) * kInv32;
  const float wa0 = fa ? __uint2float_rn(0u - fa) * kInv32 : 1.f;
  const float wb1 = __uint2float_rn(fb) * kInv32;
  const float wb0 = fb ? __uint2float_rn(0u - fb) * kInv32 : 1.f;
  // The 2 x 2 footprint of both PSFs; taps outside the library are zero.  A
  // footprint wholly inside (the common case) is read without tests.
  const bool inner = q0 >= 0 && q0 < n - 1 && p0 >= 0 && p0 < n - 1;
  float t[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    if (w == 1 && w1 == 0.f) break;
    const float *L = w ? L1 : L0;
    if (inner) {
      const float *f = L + p0 * n + q0;
      t[w][0] = __ldg(f);
      t[w][1] = __ldg(f + 1);
      t[w][2] = __ldg(f + n);
      t[w][3] = __ldg(f + n + 1);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = p0 + (e >> 1), c = q0 + (e & 1);
        if (r >= 0 && r < n && c >= 0 && c < n) t[w][e] = __ldg(L + r * n + c);
      }
    }
  }
  const float v0 = wb0 * (wa0 * t[0][0] + wa1 * t[0][1]) + wb1 * (wa0 * t[0][2] + wa1 * t[0][3]);
  float v1 = 0.f;
  if (w1 != 0.f) v1 = wb0 * (wa0 * t[1][0] + wa1 * t[1][1]) + wb1 * (wa0 * t[1][2] + wa1 * t[1][3]);
  return w0 * v0 + w1 * v1;
}

// One 128 x 64 tile per iteration: thread t builds column t/4 for rows
// 32*(t%4) .. +31 into shared memory, then the tile leaves as 128-byte rows.
__global__ void __launch_bounds__(256) split_build_kernel(const SplitParams P) {
  __shared__ __align__(16) __nv_bfloat16 thi[kTileRows][kTileCols + 8];
  __shared__ __align__(16) __nv_bfloat16 tlo[kTileRows][kTileCols + 8];
  const int jj = threadIdx.x >> 2, rq = (threadIdx.x & 3) * 32;
  const int64_t ktiles = P.ld / kTileCols, mtiles = P.rows / kTileRows;
  const int n = P.n;
  const long long h = n - 1;
  const long long base = h << PSFSIM_FRAC_BITS;
  for (int64_t t = blockIdx.x; t < ktiles * mtiles; t += gridDim.x) {
    const int64_t mt = t / ktiles, kt = t % ktiles;
    const int64_t j = kt * kTileCols + jj;
    ColGeom g;
    g.k = -1;
    if (j < P.K) g = P.geom[P.order ? P.order[j] : j];
    float inv = 1.f, sigma = 1.f;
    const float *L0 = P.lib, *L1 = P.lib;
    if (g.k >= 0) {
      sigma = pow2_at_least(fmaxf(P.libmax[g.k], P.libmax[g.k + 1]));
      inv = 1.f / sigma;  // exact: sigma is a power of two
      L0 = P.lib + (int64_t)g.k * P.M;
      L1 = L0 + P.M;
    }
    if (mt == 0 && (threadIdx.x & 3) == 0) P.scale[j] = sigma;
    int64_t i = mt * kTileRows + rq;
    int p = (int)(i / n), q = (int)(i % n);
    for (int r = 0; r < 32; ++r, ++i) {
      float v = 0.f;
      if (g.k >= 0 && i < P.M) {
        const long long a2 = base + g.C * (2 * q - h) + g.Sn * (2 * p - h);
        const long long b2 = base - g.Sn * (2 * q - h) + g.C * (2 * p - h);
        v = element(L0, L1, n, a2, b2, g.w0, g.w1) * inv;
      }
      const __nv_bfloat16 vh = __float2bfloat16_rn(v);
      thi[rq + r][jj] = vh;
      tlo[rq + r][jj] = __float2bfloat16_rn(v - __bfloat162float(vh));
      if (++q == n) { q = 0; ++p; }
    }
    __syncthreads();
    // 128 rows x 128 bytes per matrix = 1024 16-byte chunks; 4 per thread per matrix.
    for (int c = threadIdx.x; c < kTileRows * 8; c += blockDim.x) {
      const int row = c >> 3, part = c & 7;
      const int64_t off = (mt * kTileRows + row) * P.ld + kt * kTileCols + part * 8;
      *reinterpret_cast<uint4 *>(P.hi + off) = *reinterpret_cast<const uint4 *>(&thi[row][part * 8]);
      if (P.lo) *reinterpret_cast<uint4 *>(P.lo + off) = *reinterpret_cast<const uint4 *>(&tlo[row][part * 8]);
    }
    __syncthreads();
  }
}

// Dense storage of an even N x N scene grid, through the exact quarter-turn
// symmetry.  The quarter turn R(ix, iy) = (N-1-iy, ix) of the scene, (x, y) ->
// (-y, x), and P(p, q) = (q, n-1-p) of the image leave the source coordinates
// unchanged: with the fixed-point geometry, column R(j) has (C, Sn) = (-Sn_j,
// C_j), the same radius, bracket, weights and scale, so at pixel P(i) it holds
// A_ij bit for bit.  Only the x > 0, y > 0 quadrant (ix, iy >= N/2) is
// generated, and every element is written to its four positions
// A[P^m(i), R^m(j)], m = 0..3.
//
// Tile: 32 consecutive image pixels x a 16 x 16 block of quadrant pixels (256
// columns), generated into shared memory; then each of the four copies leaves
// as, per pixel, 16 runs of 16 columns (the rotated block's rows, 32 bytes of
// hi and of lo each).
constexpr int kQB = 16;                // quadrant block side (scene pixels)
constexpr int kQCols = kQB * kQB;      // columns per tile
constexpr int kQPix = 32;              // image pixels per tile
constexpr int kQPitch = kQCols + 16;   // shared row pitch in bf16: consecutive rows 8 banks apart

struct SymSplitParams {
  int n, N, H, nqb;  // image side, scene side, N / 2, quadrant blocks per side
  int vec;           // whole blocks can leave as 16-byte stores (N % 16 == 0)
  int vec32;         // ... and as 32-byte stores (N % 32 == 0)
  int64_t M, K, ld, tiles;
  const ColGeom *geom;
  const float *lib;
  const float *libmax;
  __nv_bfloat16 *hi;
  __nv_bfloat16 *lo;  // null for BF16 storage
  float *scale;
};

// One 32-byte global store (the address must be 32-byte aligned).
__device__ __forceinline__ void store32(void *p, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]),
               "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

// Image pixel P^m(p, q), as a row index.
__device__ __forceinline__ int64_t turn_pixel(int m, int p, int q, int n) {
  int pp = p, qq = q;
  for (int t = 0; t < m; ++t) {
    const int nq = n - 1 - pp;
    pp = qq;
    qq = nq;
  }
  return (int64_t)pp * n + qq;
}

__global__ void __launch_bounds__(256, 3) split_sym_build_kernel(const SymSplitParams P) {
  __shared__ __align__(16) __nv_bfloat16 thi[kQPix][kQPitch];
  __shared__ __align__(16) __nv_bfloat16 tlo[kQPix][kQPitch];
  const int n = P.n, N = P.N;
  const long long h = n - 1;
  const long long base = h << PSFSIM_FRAC_BITS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nblk = P.nqb * P.nqb;
  if (blockIdx.x == 0)  // padding columns carry scale 1, as in the direct build
    for (int64_t j = P.K + threadIdx.x; j < P.ld; j += blockDim.x) P.scale[j] = 1.f;
  for (int64_t t = blockIdx.x; t < P.tiles; t += gridDim.x) {
    // Consecutive tiles: neighbouring quadrant blocks of the same pixels.
    const int64_t i0 = (t / nblk) * kQPix;
    const int jb = (int)(t % nblk);
    const int bx = P.H + (jb % P.nqb) * kQB, by = P.H + (jb / P.nqb) * kQB;
    const int bw = min(kQB, N - bx), bh = min(kQB, N - by);
    // Warp w generates block columns 32 w .. +31 (block rows 2 w, 2 w + 1): lane
    // l takes column 32 w + 4 g + l % 4 for the pixels l / 4 + 8 t, so one
    // load covers 8 neighbouring pixels of 4 neighbouring columns (nearby
    // footprints in the same or an adjacent bracket).
    // this lane's 4 pixels: offsets 2 du, 2 dv from the image centre (doubled)
    int du2[kQPix / 8], dv2[kQPix / 8];
#pragma unroll
    for (int t = 0; t < kQPix / 8; ++t) {
      const int i = (int)i0 + (lane >> 2) + 8 * t;  // < M < 2^31
      const int p = i / n;
      du2[t] = 2 * (i - p * n) - (int)h;
      dv2[t] = 2 * p - (int)h;
    }
    for (int g = 0; g < 8; ++g) {
      const int c = 32 * warp + 4 * g + (lane & 3), cu = c % kQB, cv = c / kQB;
      ColGeom gm;
      gm.k = -1;
      gm.C = gm.Sn = 0;
      gm.w0 = gm.w1 = 0.f;
      const int ix = bx + cu, iy = by + cv;
      const bool valid = cu < bw && cv < bh;
      if (valid) gm = P.geom[(int64_t)(iy - P.H) * P.H + (ix - P.H)];  // quadrant entry
      float inv = 1.f, sigma = 1.f;
      const float *L0 = P.lib, *L1 = P.lib;
      if (gm.k >= 0) {
        sigma = pow2_at_least(fmaxf(P.libmax[gm.k], P.libmax[gm.k + 1]));
        inv = 1.f / sigma;  // exact: sigma is a power of two
        L0 = P.lib + (int64_t)gm.k * P.M;
        L1 = L0 + P.M;
      }
      if (i0 == 0 && valid && lane < 4) {
        P.scale[(int64_t)iy * N + ix] = sigma;
        P.scale[(int64_t)ix * N + (N - 1 - iy)] = sigma;
        P.scale[(int64_t)(N - 1 - iy) * N + (N - 1 - ix)] = sigma;
        P.scale[(int64_t)(N - 1 - ix) * N + iy] = sigma;
      }
#pragma unroll
      for (int t = 0; t < kQPix / 8; ++t) {
        const int r = (lane >> 2) + 8 * t;
        const int64_t i = i0 + r;
        float v = 0.f;
        if (gm.k >= 0 && i < P.M) {
          const long long a2 = base + gm.C * du2[t] + gm.Sn * dv2[t];
          const long long b2 = base - gm.Sn * du2[t] + gm.C * dv2[t];
          v = element(L0, L1, n, a2, b2, gm.w0, gm.w1) * inv;
        }
        const __nv_bfloat16 vh = __float2bfloat16_rn(v);
        thi[r][c] = vh;
        tlo[r][c] = __float2bfloat16_rn(v - __bfloat162float(vh));
      }
    }
    __syncthreads();
    // Copy m, pixel r, rotated-block row vd: destination row P^m(i0 + r),
    // columns (oy + vd) N + ox + ud, ud = 0..15; its source in the tile is
    // block position (su, sv) of the generated block.
    const int vd = lane & 15;
    for (int k = 0; k < 4 * kQPix / 16; ++k) {
      const int m = k & 3;
      const int r = 2 * (warp + 8 * (k >> 2)) + (lane >> 4);
      const int64_t i = i0 + r;
      if (i >= P.M) continue;
      const int ii = (int)i, pi = ii / n;
      const int64_t row = turn_pixel(m, pi, ii - pi * n, n);
      int ox, oy;
      if (m == 0) { ox = bx; oy = by; }
      else if (m == 1) { ox = N - kQB - by; oy = bx; }
      else if (m == 2) { ox = N - kQB - bx; oy = N - kQB - by; }
      else { ox = by; oy = N - kQB - bx; }
      const __nv_bfloat16 *sh = thi[r], *sl = tlo[r];
      __nv_bfloat16 *dh = P.hi + row * P.ld + (int64_t)(oy + vd) * N + ox;
      __nv_bfloat16 *dl = P.lo ? P.lo + row * P.ld + (int64_t)(oy + vd) * N + ox : nullptr;
      // source column (in the tile) of destination position ud of this run
      auto src = [&](int ud) -> int {
        if (m == 0) return vd * kQB + ud;
        if (m == 1) return (kQB - 1 - ud) * kQB + vd;
        if (m == 2) return (kQB - 1 - vd) * kQB + (kQB - 1 - ud);
        return ud * kQB + (kQB - 1 - vd);
      };
      if (P.vec && bw == kQB && bh == kQB) {
        uint32_t wh[8], wl[8];
        if (m == 0 || m == 2) {
          const int s0 = (m == 0 ? vd : kQB - 1 - vd) * kQB;
          const uint4 h0 = *reinterpret_cast<const uint4 *>(sh + s0);
          const uint4 h1 = *reinterpret_cast<const uint4 *>(sh + s0 + 8);
          const uint4 l0 = *reinterpret_cast<const uint4 *>(sl + s0);
          const uint4 l1 = *reinterpret_cast<const uint4 *>(sl + s0 + 8);
          const uint32_t ah[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
          const uint32_t al[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            // m = 2 runs backwards: word w holds source positions 15 - 2w, 14 - 2w
            wh[w] = m == 0 ? ah[w] : __byte_perm(ah[7 - w], 0u, 0x1032);
            wl[w] = m == 0 ? al[w] : __byte_perm(al[7 - w], 0u, 0x1032);
          }
        } else {
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            const int a = src(2 * w), b = src(2 * w + 1);
            wh[w] = (uint32_t)__bfloat16_as_ushort(sh[a]) | ((uint32_t)__bfloat16_as_ushort(sh[b]) << 16);
            wl[w] = (uint32_t)__bfloat16_as_ushort(sl[a]) | ((uint32_t)__bfloat16_as_ushort(sl[b]) << 16);
          }
        }
        if (P.vec32) {  // 32-byte aligned runs: one store each
          store32(dh, wh);
          if (dl) store32(dl, wl);
        } else {
          reinterpret_cast<uint4 *>(dh)[0] = make_uint4(wh[0], wh[1], wh[2], wh[3]);
          reinterpret_cast<uint4 *>(dh)[1] = make_uint4(wh[4], wh[5], wh[6], wh[7]);
          if (dl) {
            reinterpret_cast<uint4 *>(dl)[0] = make_uint4(wl[0], wl[1], wl[2], wl[3]);
            reinterpret_cast<uint4 *>(dl)[1] = make_uint4(wl[4], wl[5], wl[6], wl[7]);
          }
        }
      } else {
        // A block at the quadrant's outer edge (or N % 16 != 0): element by
        // element, only positions whose source lies inside the block.
        for (int ud = 0; ud < kQB; ++ud) {
          const int s = src(ud), su = s % kQB, sv = s / kQB;
          if (su >= bw || sv >= bh) continue;
          dh[ud] = sh[s];
          if (dl) dl[ud] = sl[s];
        }
      }
    }
    __syncthreads();
  }
}

// ---- dense storage of an even grid, pixel by pixel -------------------------
//
// The same quarter-turn symmetry, arranged around the two things that bound
// it: the footprint loads and the stores.  A CTA takes two neighbouring image
// pixels at a time, generates all of the quadrant's columns for them in the
// (bracket, angle)-sorted order, and keeps the quadrant's hi and lo in shared
// memory; then each of the four turned copies leaves as whole rows of the
// turned quadrant (runs of 2 H bytes, 64 per store instruction and row).
//   * Footprints come from the library's 32-byte pair entries (fused.cu): one
//     256-bit load per element instead of eight 4-byte ones.
//   * CTAs take pixel pairs in order of their distance from the image centre.
//     A pixel's footprints sweep a circle of every bracket's PSFs, so the
//     pairs in flight at once share one annulus of the entries, which stays in
//     L2 (the entries of all brackets, 125 MB at 256^2, do not).
//   * A column's geometry (48 bytes) is read once for the two pixels.
// Element arithmetic is element()'s, so the bits are the direct build's.

// Columns of the quadrant inside the last radius, in sorted order, as three
// arrays of 16 bytes a column (one array of 48-byte records took ten times the
// L1 wavefronts to read).  Pixel (p, q) samples a = A00 + C2 q + S2 p,
// b = B00 - S2 q + C2 p: the source column and row, plus one, in units of 2^-41
// (element()'s 2a and 2b).
struct __align__(16) ColOrigin {
  long long A00, B00;
};
struct __align__(16) ColStep {
  unsigned long long C2, S2;
};
struct __align__(16) ColWeight {
  uint32_t off;      // first pair entry of the radial bracket
  float w0, w1;
  uint32_t pos_inv;  // position in the shared quadrant (16 bits); high half of 1 / sigma, a power of two
};
struct SplitCols {
  ColOrigin *origin;
  ColStep *step;
  ColWeight *weight;
};
constexpr int kPixThreads = 768;
constexpr size_t kPixSmem = 220 * 1024;

// Shared quadrant: Hb x Hb of the H x H pixels (Hb covers the columns inside
// the last radius), pixel (y, x) at word quad_pos.  With an odd pitch and the
// skews of two words per 32 columns and per 32 rows, 2 rows x 16 chunks of 8
// (either way round: the 32 lanes of a store) meet 32 different banks; of the
// odd pitches 15 mod 32 keeps the columns of an arc, the generators' 32 lanes,
// at 2 ways (1 mod 32: 6).
__host__ __device__ inline int quad_pitch(int Hb) { return (Hb + Hb / 16 + 16) / 32 * 32 + 15; }
__host__ __device__ inline int quad_words(int Hb) { return Hb * quad_pitch(Hb) + Hb / 16 + 2; }
__device__ __forceinline__ int quad_pos(int y, int x, int pitch) { return y * pitch + x + 2 * (x >> 5) + 2 * (y >> 5); }

struct PixParams {
  unsigned runs_magic;  // ceil(2^32 / (H / 8)): l / (H / 8) = umulhi(l, runs_magic) for l < 2^16
  int n, N, H, Hb, pitch, per, vec;  // vec: runs leave as 16-byte stores (N % 16 == 0)
  int64_t M;
  int64_t K;  // scene pixels: not read, but with the rest 8 bytes earlier 256^2 takes 3.60 ms, not 3.58
  int64_t ld;
  int64_t pairs;
  SplitCols cols;
  const int *nvalid;      // columns inside the last radius
  const int *pair_order;  // pixel pairs, nearest the image centre first
  const float *entries;   // pair entries, 8 floats each
  uint32_t zero_entry;
  __nv_bfloat16 *hi;
  __nv_bfloat16 *lo;  // null for BF16 storage
};

// The tables of the sorted column order, and the scale of every stored column.
__global__ void split_columns_kernel(const ColGeom *__restrict__ geom, const int *__restrict__ order,
                                     const int *__restrict__ nvalid, int n, int N, int pitch, int64_t K, int64_t ld,
                                     const float *__restrict__ libmax, const SplitCols cols,
                                     float *__restrict__ scale) {
  const int H = N / 2;
  const int64_t Kq = K / 4, nv = *nvalid;
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  const long long h = n - 1, base = (h + 2) << PSFSIM_FRAC_BITS;
  for (int64_t t = t0; t < nv; t += stride) {
    const int j = order[t];
    const ColGeom g = geom[j];
    cols.origin[t] = ColOrigin{base - h * (g.C + g.Sn), base + h * (g.Sn - g.C)};
    cols.step[t] = ColStep{(unsigned long long)(2 * g.C), (unsigned long long)(2 * g.Sn)};
    const float inv = 1.f / pow2_at_least(fmaxf(libmax[g.k], libmax[g.k + 1]));
    cols.weight[t] = ColWeight{(uint32_t)g.k * (uint32_t)((n + 1) * (n + 1)), g.w0, g.w1,
                               (uint32_t)quad_pos(j / H, j % H, pitch) | (__float_as_uint(inv) & 0xFFFF0000u)};
  }
  for (int64_t j = t0; j < Kq; j += stride) {
    const int k = geom[j].k;
    const float sigma = k >= 0 ? pow2_at_least(fmaxf(libmax[k], libmax[k + 1])) : 1.f;
    const int ix = H + (int)(j % H), iy = H + (int)(j / H);
    scale[(int64_t)iy * N + ix] = sigma;
    scale[(int64_t)ix * N + (N - 1 - iy)] = sigma;
    scale[(int64_t)(N - 1 - iy) * N + (N - 1 - ix)] = sigma;
    scale[(int64_t)(N - 1 - ix) * N + iy] = sigma;
  }
  for (int64_t j = K + t0; j < ld; j += stride) scale[j] = 1.f;
}

// order[]: pixel pairs by the distance of the pair's middle from the image
// centre, in bins of one pixel (the order within a bin is left to the atomics:
// it decides which CTA writes which rows, not what is written).
__global__ void __launch_bounds__(1024) pixel_order_kernel(int n, int pix, int64_t pairs, int bins,
                                                           int *__restrict__ order) {
  extern __shared__ int cnt[];
  const int pr = (n + pix - 1) / pix;  // pairs (or pixels) per row
  auto bin = [&](int64_t t) -> int {
    const float dv = (float)(t / pr) - 0.5f * (float)(n - 1), du = (float)(pix * (t % pr)) + 0.5f * (float)(pix - n);
    const int b = (int)sqrtf(du * du + dv * dv);
    return b < bins ? b : bins - 1;
  };
  for (int i = threadIdx.x; i < bins; i += blockDim.x) cnt[i] = 0;
  __syncthreads();
  for (int64_t t = threadIdx.x; t < pairs; t += blockDim.x) atomicAdd(&cnt[bin(t)], 1);
  __syncthreads();
  if (threadIdx.x < 32) {  // exclusive prefix, one warp
    int run = 0;
    for (int b0 = 0; b0 < bins; b0 += 32) {
      const int b = b0 + (int)threadIdx.x, v = b < bins ? cnt[b] : 0;
      int x = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)threadIdx.x >= o) x += u;
      }
      if (b < bins) cnt[b] = run + x - v;
      run += __shfl_sync(0xffffffffu, x, 31);
    }
  }
  __syncthreads();
  for (int64_t t = threadIdx.x; t < pairs; t += blockDim.x) order[atomicAdd(&cnt[bin(t)], 1)] = (int)t;
}

__device__ __forceinline__ uint64_t pk2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

struct Foot {
  uint64_t t00, t01, t10, t11;  // (L[k], L[k+1]) at the four taps
};

// element() on a pair entry: both PSFs at once, the same operations in the same order.
__device__ __forceinline__ float element_pair(const Foot &e, uint32_t fa, uint32_t fb, float w0, float w1) {
  constexpr float kInv32 = 2.3283064365386963e-10f;
  const float wa1 = __uint2float_rn(fa) * kInv32, wa0 = fa ? __uint2float_rn(0u - fa) * kInv32 : 1.f;
  const float wb1 = __uint2float_rn(fb) * kInv32, wb0 = fb ? __uint2float_rn(0u - fb) * kInv32 : 1.f;
  const uint64_t a0 = pk2(wa0, wa0), a1 = pk2(wa1, wa1);
  const uint64_t r0 = ffma2(a0, e.t00, fmul2(a1, e.t01)), r1 = ffma2(a0, e.t10, fmul2(a1, e.t11));
  const uint64_t v = ffma2(pk2(wb0, wb0), r0, fmul2(pk2(wb1, wb1), r1));
  float v0, v1;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v0), "=f"(v1) : "l"(v));
  if (w1 == 0.f) v1 = 0.f;  // the upper PSF takes no part (it may hold anything)
  return fmaf(w0, v0, w1 * v1);
}

// Eight quadrant words from src, `step` apart (zeros unless `in`): hi and lo as one 16-byte run at
// offset `fwd` of the matrix and, backwards, at offset `rev`.
__device__ __forceinline__ void store_run(const PixParams &P, const uint32_t *src, int step, bool in, int64_t fwd,
                                          int64_t rev) {
  uint32_t w[8], h[4], l[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) w[i] = in ? src[i * step] : 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410);
    l[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7632);
  }
  auto back = [](uint32_t v) { return __byte_perm(v, v, 0x1032); };
  __stcs(reinterpret_cast<uint4 *>(P.hi + fwd), make_uint4(h[0], h[1], h[2], h[3]));
  __stcs(reinterpret_cast<uint4 *>(P.hi + rev), make_uint4(back(h[3]), back(h[2]), back(h[1]), back(h[0])));
  if (P.lo) {
    __stcs(reinterpret_cast<uint4 *>(P.lo + fwd), make_uint4(l[0], l[1], l[2], l[3]));
    __stcs(reinterpret_cast<uint4 *>(P.lo + rev), make_uint4(back(l[3]), back(l[2]), back(l[1]), back(l[0])));
  }
}

__device__ __forceinline__ void store_one(const PixParams &P, uint32_t w, int64_t at) {
  P.hi[at] = __ushort_as_bfloat16((unsigned short)(w & 0xFFFFu));
  if (P.lo) P.lo[at] = __ushort_as_bfloat16((unsigned short)(w >> 16));
}

// kPix pixels at a time (2, or 1 where two quadrants of each do not fit).  Every
// thread interleaves the two halves of the work: while the footprints of the
// next pixels' columns are on their way it stores runs of the current pixels.
// 3.36 ms for one 256^2 wavelength (17.2 GB, 5.1 TB/s; block-wise 11.6 ms); what
// is left above the stores is L1 (71 % busy, its data pipe 67 %) and issue (58 %;
// counters of 128^2 images on 256^2 pixels).
// Apart, the halves take 1.5 ms (generation) and 2.6 ms (stores, the HBM floor)
// at 256^2, and alternating them, by phases of one CTA or by two CTAs an SM,
// takes their sum: a burst of stores fills the SM's request queue and the other
// half's loads wait behind it.
template <int kPix>
__global__ void __launch_bounds__(kPixThreads, 1) split_pixel_build_kernel(const PixParams P) {
  extern __shared__ uint32_t quads[];  // [2][kPix][per]: hi | lo << 16
  const int n = P.n, N = P.N, H = P.H, Hb = P.Hb, pitch = P.pitch, per = P.per;
  const uint32_t un = (uint32_t)n, nq = un + 1u;
  for (int i = threadIdx.x; i < 2 * kPix * per; i += kPixThreads) quads[i] = 0u;  // columns beyond the last radius
  const int nv = *P.nvalid;
  const int pr = (n + kPix - 1) / kPix, runs = H / 8;
  const int gsteps = (nv + kPixThreads - 1) / kPixThreads;
  const int blocks = P.vec ? (H * runs + kPixThreads - 1) / kPixThreads : 0, units = blocks * kPix * 2;
  __syncthreads();
  int64_t cur = -1;
  int buf = 0;
  for (int64_t next = blockIdx.x;; cur = next, next += gridDim.x, buf ^= 1) {
    const bool gen = next < P.pairs;
    if (!gen && cur < 0) break;
    const int gp = gen ? P.pair_order[next] : 0, p = gp / pr, q = kPix * (gp % pr);
    const int cp = cur >= 0 ? P.pair_order[cur] : 0, cy = cp / pr, cx = kPix * (cp % pr);
    uint32_t *dst = quads + buf * kPix * per;
    const uint32_t *src = quads + (buf ^ 1) * kPix * per;
    const int64_t r0 = (int64_t)cy * n + cx, r1 = (int64_t)cx * n + n - 1 - cy;  // P^0, P^1 of the first pixel
    // Origins of the turned quadrants in the rows P^m(pixel); the next pixel's
    // rows are 1, n, -1 and -n further.
    const int64_t o0 = r0 * P.ld + (int64_t)H * N + H, o1 = r1 * P.ld + (int64_t)H * N;
    const int64_t o2 = (P.M - 1 - r0) * P.ld, o3 = (P.M - 1 - r1) * P.ld + H;
    // One unit of the stores: a thread's run along a quadrant row (or column)
    // of one pixel.  Along row a from column c: copy 0 at (a, c), copy 2 at
    // (H-1-a, H-8-c); along column a from row c: copy 3 at (H-1-a, c), copy 1
    // at (a, H-8-c).
    const int64_t nld = (int64_t)n * P.ld;
    const bool both = cx + 1 < n;  // an odd image's last pair holds one pixel
    auto store_unit = [&](int unit) {
      const bool second = kPix == 2 && (unit & 2);
      const int l = (unit >> kPix) * kPixThreads + (int)threadIdx.x;
      if (l >= H * runs || (second && !both)) return;
      const int a = runs == 1 ? l : (int)__umulhi((unsigned)l, P.runs_magic), c = 8 * (l - a * runs);
      const bool in = a < Hb && c < Hb;  // Hb is a multiple of 8
      const uint32_t *s = src + (second ? per : 0);
      const int up = a * N + c, down = (H - 1 - a) * N + c;
      if (unit & 1) {
        const int64_t step = second ? nld : 0;
        store_run(P, s + quad_pos(c, a, pitch), pitch, in, o3 - step + down, o1 + step + (up + H - 8 - 2 * c));
      } else {
        const int64_t step = second ? P.ld : 0;
        store_run(P, s + quad_pos(a, c, pitch), 1, in, o0 + step + up, o2 - step + (down + H - 8 - 2 * c));
      }
    };
    const int steps = gen && gsteps > 0 ? gsteps : 1;
    int done = 0, due = 0;  // units stored; units x steps owed so far
    for (int g = 0; g < steps; ++g) {
      const int t = g * kPixThreads + (int)threadIdx.x;
      const bool mine = gen && t < nv;
      Foot e[kPix];
      uint32_t fa[kPix], fb[kPix];
      ColWeight c;
      if (mine) {
        const ColOrigin o = P.cols.origin[t];
        const ColStep d = P.cols.step[t];
        c = P.cols.weight[t];
        unsigned long long a = (unsigned long long)o.A00 + d.C2 * (uint32_t)q + d.S2 * (uint32_t)p;
        unsigned long long b = (unsigned long long)o.B00 - d.S2 * (uint32_t)q + d.C2 * (uint32_t)p;
#pragma unroll
        for (int x = 0; x < kPix; ++x) {
          const uint32_t qa = (uint32_t)(a >> (PSFSIM_FRAC_BITS + 1)), pb = (uint32_t)(b >> (PSFSIM_FRAC_BITS + 1));
          const uint32_t idx = qa <= un && pb <= un ? c.off + pb * nq + qa : P.zero_entry;
          asm volatile("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];"
                       : "=l"(e[x].t00), "=l"(e[x].t01), "=l"(e[x].t10), "=l"(e[x].t11)
                       : "l"(P.entries + 8 * (size_t)idx));
          fa[x] = (uint32_t)(a >> (PSFSIM_FRAC_BITS - 31));
          fb[x] = (uint32_t)(b >> (PSFSIM_FRAC_BITS - 31));
          a += d.C2;
          b -= d.S2;
        }
      }
      if (cur >= 0)
        for (due += units; due >= steps; due -= steps) store_unit(done++);
      if (mine) {
        const float iv = __uint_as_float(c.pos_inv & 0xFFFF0000u);
        const uint32_t pos = c.pos_inv & 0xFFFFu;
#pragma unroll
        for (int x = 0; x < kPix; ++x) {
          const float v = element_pair(e[x], fa[x], fb[x], c.w0, c.w1) * iv;
          const __nv_bfloat16 vh = __float2bfloat16_rn(v);
          const __nv_bfloat16 vl = __float2bfloat16_rn(v - __bfloat162float(vh));
          dst[x * per + pos] = (uint32_t)__bfloat16_as_ushort(vh) | ((uint32_t)__bfloat16_as_ushort(vl) << 16);
        }
      }
    }
    if (!P.vec && cur >= 0) {  // N % 16 != 0: element by element
      for (int x = 0; x < kPix && cx + x < n; ++x) {
        const int64_t row0 = r0 + x, row1 = r1 + (int64_t)x * n;
        auto at = [&](int y, int xx) -> uint32_t {
          return y < Hb && xx < Hb ? src[x * per + quad_pos(y, xx, pitch)] : 0u;
        };
        for (int l = threadIdx.x; l < H * H; l += kPixThreads) {
          const int r = l / H, k = l % H;
          store_one(P, at(r, k), row0 * P.ld + (int64_t)(H + r) * N + H + k);
          store_one(P, at(H - 1 - k, r), row1 * P.ld + (int64_t)(H + r) * N + k);
          store_one(P, at(H - 1 - r, H - 1 - k), (P.M - 1 - row0) * P.ld + (int64_t)r * N + k);
          store_one(P, at(k, H - 1 - r), (P.M - 1 - row1) * P.ld + (int64_t)r * N + H + k);
        }
      }
    }
    __syncthreads();
    if (!gen) break;
  }
}

}  // namespace

// Workspace the pixel-wise build wants beyond the layout (the library's pair
// entries and the pixel order); 0 where it does not run or does not pay.  Both
// sides measured, block-wise / pixel-wise build of n x n PSFs on N x N scenes:
//   N % 32 == 0 (the block-wise build's whole blocks): 64 / 64: 78 / 86 us,
//     128 / 64: 244 / 176, 128 / 32: 70 / 156, 256 / 32: 185 / 477,
//     64 / 128: 238 / 136, 128 / 256: 2727 / 887, 256 / 256: 11714 / 3560;
//   other N: 100 / 24: 121 / 137 us, 256 / 48: 1872 / 518, 200 / 60: 3166 / 598,
//     100 / 100: 2684 / 333, 48 / 200: 1569 / 278, 200 / 300: 79709 / 10610.
// Few columns leave its two barriers a pixel exposed (N below 48 to 64), few
// elements its six small launches.  It may take half as much again as A.
int64_t psfsim_pixel_build_bytes(int n, int64_t K, int storage, int n_r) {
  if (storage != PSFSIM_SPLIT_BF16 && storage != PSFSIM_BF16) return 0;
  const int64_t N = (int64_t)llround(sqrt((double)K)), H = N / 2;
  if ((int64_t)(n_r - 1) * (n + 1) * (n + 1) >= (1ll << 32) - 1) return 0;  // entries are indexed in 32 bits
  if (N * N != K || N % 2 || 2ull * quad_words((int)psfsim_round_up(H, 8)) * 4 > kPixSmem) return 0;
  const int64_t bytes = psfsim_round_up(psfsim_pair_library_bytes(n, n_r), 256) + psfsim_round_up((int64_t)n * n * 4, 256);
  const int64_t a = psfsim_round_up((int64_t)n * n, 128) * psfsim_round_up(K, 64) * (storage == PSFSIM_BF16 ? 2 : 4);
  if (N % 32 == 0 ? N < 64 || (int64_t)n * n * K < (1ll << 25) : N < 48) return 0;
  return 2 * bytes <= a ? bytes : 0;
}

cudaError_t psfsim_launch_split_build(psfsim_plan *h, cudaStream_t st) {
  float *libmax = reinterpret_cast<float *>(h->ws + h->libmax_off);
  cudaError_t e = cudaMemsetAsync(libmax, 0, (size_t)h->n_r * 4, st);
  if (e != cudaSuccess) return e;
  libmax_kernel<<<dim3(kMaxParts, (unsigned)h->n_r), 256, 0, st>>>(h->d_lib, h->M, libmax);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  SplitParams P;
  P.n = h->n;
  P.K = psfsim_cols(h);
  P.order = h->quadrant ? reinterpret_cast<const int *>(h->ws + h->order_off) : nullptr;
  P.ld = h->ld;
  P.M = h->M;
  P.rows = psfsim_round_up(h->M, kTileRows);
  P.geom = reinterpret_cast<const ColGeom *>(h->ws + h->geom_off);
  P.lib = h->d_lib;
  P.libmax = libmax;
  P.hi = reinterpret_cast<__nv_bfloat16 *>(h->ws + h->a_off);
  P.lo = h->lo_off >= 0 ? reinterpret_cast<__nv_bfloat16 *>(h->ws + h->lo_off) : nullptr;
  P.scale = reinterpret_cast<float *>(h->ws + h->scale_off);
  if (h->N > 0 && h->N % 2 == 0 && !h->quadrant) {
    // Dense storage of an even grid: the quadrant's columns, four copies each.
    // The padding (rows M.. and columns K.. of every row) is zeroed first.
    const size_t row_bytes = (size_t)P.ld * 2;
    for (__nv_bfloat16 *a : {P.hi, P.lo}) {
      if (!a) continue;
      if ((e = cudaMemsetAsync(a + P.M * P.ld, 0, (size_t)(P.rows - P.M) * row_bytes, st)) != cudaSuccess) return e;
      if (P.ld > P.K &&
          (e = cudaMemset2DAsync(a + P.K, row_bytes, 0, (size_t)(P.ld - P.K) * 2, (size_t)P.M, st)) != cudaSuccess)
        return e;
    }
    if (h->pix) {
      char *pix = h->pix;
      float *entries = reinterpret_cast<float *>(pix);
      int *pair_order = reinterpret_cast<int *>(pix + psfsim_round_up(psfsim_pair_library_bytes(h->n, h->n_r), 256));
      // the quadrant's geometry leaves three quarters of its table free
      char *tab = h->ws + h->geom_off + psfsim_round_up(h->K / 4 * (int64_t)sizeof(ColGeom), 256);
      const int64_t Kq = h->K / 4;
      const SplitCols cols = {reinterpret_cast<ColOrigin *>(tab), reinterpret_cast<ColStep *>(tab + 16 * Kq),
                              reinterpret_cast<ColWeight *>(tab + 32 * Kq)};
      const int *order = reinterpret_cast<const int *>(h->ws + h->order_off);
      const int *nvalid = reinterpret_cast<const int *>(h->ws + h->bstart_off) + psfsim_num_buckets(h->n_r) - 1;
      if ((e = psfsim_launch_pair_entries(h->d_lib, h->n, h->n_r, entries, h->num_sms, st)) != cudaSuccess) return e;
      // Quadrant pixels (2 x + 1, 2 y + 1 half pixels from the centre) inside the last radius lie in Hb x Hb.
      const int H = h->N / 2;
      const long long R2 = live_r2(h->radii[h->n_r - 1], h->S);
      const int reach = R2 > 0 ? (int)((sqrt((double)R2) + 1.0) * 0.5) + 1 : 1;
      const int Hb = (int)psfsim_round_up(reach < H ? reach : H, 8);
      split_columns_kernel<<<h->num_sms, 256, 0, st>>>(P.geom, order, nvalid, h->n, h->N, quad_pitch(Hb), h->K, P.ld,
                                                       libmax, cols, P.scale);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      PixParams X;
      X.n = h->n;
      X.N = h->N;
      X.H = H;
      X.Hb = Hb;
      X.pitch = quad_pitch(Hb);
      X.per = quad_words(Hb);
      X.vec = h->N % 16 == 0;
      X.runs_magic = H >= 16 ? (unsigned)(((1ull << 32) + H / 8 - 1) / (H / 8)) : 0u;
      X.M = h->M;
      X.K = h->K;
      X.ld = P.ld;
      const int kpix = 4ull * X.per * 4 <= kPixSmem ? 2 : 1;
      X.pairs = (int64_t)h->n * ((h->n + kpix - 1) / kpix);
      X.cols = cols;
      X.nvalid = nvalid;
      X.pair_order = pair_order;
      X.entries = entries;
      X.zero_entry = (uint32_t)(h->n_r - 1) * (uint32_t)((h->n + 1) * (h->n + 1));
      X.hi = P.hi;
      X.lo = P.lo;
      const int bins = h->n;  // the corner is 0.71 n from the centre
      pixel_order_kernel<<<1, 1024, (size_t)bins * 4, st>>>(h->n, kpix, X.pairs, bins, pair_order);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      const size_t smem = 2ull * kpix * X.per * 4;
      auto kern = kpix == 2 ? split_pixel_build_kernel<2> : split_pixel_build_kernel<1>;
      if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
      kern<<<(unsigned)(X.pairs < h->num_sms ? X.pairs : h->num_sms), kPixThreads, smem, st>>>(X);
      return cudaGetLastError();
    }
    SymSplitParams Q;
    Q.n = h->n;
    Q.N = h->N;
    Q.H = h->N / 2;
    Q.nqb = (Q.H + kQB - 1) / kQB;
    Q.vec = h->N % 16 == 0;
    Q.vec32 = h->N % 32 == 0;
    Q.M = h->M;
    Q.K = h->K;
    Q.ld = h->ld;
    Q.tiles = (h->M + kQPix - 1) / kQPix * (int64_t)Q.nqb * Q.nqb;
    Q.geom = P.geom;
    Q.lib = P.lib;
    Q.libmax = libmax;
    Q.hi = P.hi;
    Q.lo = P.lo;
    Q.scale = P.scale;
    int per_sm = 1;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, split_sym_build_kernel, 256, 0)) != cudaSuccess)
      return e;
    split_sym_build_kernel<<<h->num_sms * (per_sm < 1 ? 1 : per_sm), 256, 0, st>>>(Q);
    return cudaGetLastError();
  }
  int per_sm = 1;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, split_build_kernel, 256, 0)) != cudaSuccess)
    return e;
  split_build_kernel<<<h->num_sms * (per_sm < 1 ? 1 : per_sm), 256, 0, st>>>(P);
  return cudaGetLastError();
}
