// Library build (Sec. 2): per-column geometry, bracket sort, and the kernels
// that write every column of A = [I_1 ... I_K] (Eq. 4-5).
#include <cudaTypedefs.h>

#include <climits>
#include <cstring>

#include "psfsim_internal.cuh"
#include "ptx_util.cuh"

namespace {

constexpr double kFix = 1099511627776.0;  // 2^PSFSIM_FRAC_BITS
static_assert(PSFSIM_FRAC_BITS == 40, "kFix");

struct GeomParams {
  int n_r, N, interp, quadrant;
  int64_t K;
  double S;
  const double *pts;
  double radii[PSFSIM_MAX_RADII];
};

// a1-a2: field offset (Eq. 2-3), polar angle as x/r, y/r, radial bracket + weight.
__global__ void geom_kernel(const __grid_constant__ GeomParams P, ColGeom *geom) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= P.K) return;
  double x, y;
  if (P.pts) {
    x = P.pts[2 * j];
    y = P.pts[2 * j + 1];
  } else if (P.quadrant) {  // x > 0, y > 0 quadrant of an even N x N grid
    const int H = P.N / 2;
    const int iy = H + (int)(j / H), ix = H + (int)(j % H);
    const double half = 0.5 * (double)(P.N - 1);
    x = __dmul_rn((double)ix - half, P.S);
    y = __dmul_rn((double)iy - half, P.S);
  } else {
    const int iy = (int)(j / P.N), ix = (int)(j % P.N);
    const double half = 0.5 * (double)(P.N - 1);
    x = __dmul_rn((double)ix - half, P.S);
    y = __dmul_rn((double)iy - half, P.S);
  }
  const double r = __dsqrt_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)));
  double c = 1.0, s = 0.0;
  if (r > 0.0) {
    c = __ddiv_rn(x, r);
    s = __ddiv_rn(y, r);
  }
  ColGeom g;
  {
    const float th = atan2f((float)y, (float)x);  // ordering only
    int bin = (int)((th + 3.14159265f) * (PSFSIM_THETA_BINS / 6.2831853f));
    g.bin = bin < 0 ? 0 : (bin >= PSFSIM_THETA_BINS ? PSFSIM_THETA_BINS - 1 : bin);
  }
  g.C = __double2ll_rn(c * kFix);
  g.Sn = __double2ll_rn(s * kFix);
  if (!(r <= P.radii[P.n_r - 1])) {
    g.k = -1;
    g.w0 = 0.f;
    g.w1 = 0.f;
  } else {
    int lo = 0, hi = P.n_r - 2;  // largest k in [0, n_r-2] with radii[k] <= r
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (P.radii[mid] <= r) lo = mid; else hi = mid - 1;
    }
    double w = __ddiv_rn(__dsub_rn(r, P.radii[lo]), __dsub_rn(P.radii[lo + 1], P.radii[lo]));
    if (w < 0.0) w = 0.0;
    if (P.interp == PSFSIM_NEAREST) w = (w > 0.5) ? 1.0 : 0.0;
    g.k = lo;
    g.w0 = (float)(1.0 - w);
    g.w1 = (float)w;
  }
  geom[j] = g;
}

__device__ __forceinline__ int column_bucket(const ColGeom &g, int n_r) {
  return g.k < 0 ? psfsim_num_buckets(n_r) - 1 : g.k * PSFSIM_THETA_BINS + g.bin;
}

// Stable counting sort of the columns by (radial bracket, angle bin), zero
// columns last, so that a CTA can stage one bracket pair for many columns and
// neighbouring columns read nearby library pixels.  One CTA; warp w of W takes
// the w-th contiguous chunk of the columns, with its own row of bucket
// counters in shared memory (W x buckets ints): the chunks are counted, every
// bucket's cursor for chunk w starts after the bucket's earlier buckets and
// the bucket's entries of chunks < w, and each warp scatters its chunk in
// index order with match_any ranks.  The order is deterministic: by bucket,
// ties by column index.
__global__ void __launch_bounds__(1024) bracket_sort_kernel(const ColGeom *geom, int64_t K, int n_r, int W,
                                                            int *order, int *bstart) {
  extern __shared__ int cnt[];  // [W][nb]
  const int nb = psfsim_num_buckets(n_r);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < W * nb; i += blockDim.x) cnt[i] = 0;
  __syncthreads();
  const int64_t c0 = K * warp / W, c1 = K * (warp + 1) / W;
  if (warp < W)
    for (int64_t j = c0 + lane; j < c1; j += 32) atomicAdd(&cnt[warp * nb + column_bucket(geom[j], n_r)], 1);
  __syncthreads();
  // Per bucket: its total, then the cursors of the chunks within it.
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    int t = 0;
    for (int w = 0; w < W; ++w) {
      const int c = cnt[w * nb + b];
      cnt[w * nb + b] = t;
      t += c;
    }
    bstart[b] = t;  // total for now
  }
  __syncthreads();
  // Bucket starts: exclusive prefix of the totals, in bucket order (one warp).
  if (warp == 0) {
    int run = 0;
    for (int b0 = 0; b0 < nb; b0 += 32) {
      const int b = b0 + lane;
      const int v = b < nb ? bstart[b] : 0;
      int x = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (b < nb) bstart[b] = run + x - v;
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) bstart[nb] = run;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < W * nb; i += blockDim.x) cnt[i] += bstart[i % nb];
  __syncthreads();
  if (warp < W) {
    int *cur = cnt + warp * nb;
    const unsigned lt = (1u << lane) - 1u;
    for (int64_t base = c0; base < c1; base += 32) {
      const int64_t j = base + lane;
      const int key = j < c1 ? column_bucket(geom[j], n_r) : -1;
      const unsigned peers = __match_any_sync(0xffffffffu, key);
      const int leader = __ffs(peers) - 1;
      int pos0 = 0;
      if (lane == leader && key >= 0) pos0 = cur[key];
      pos0 = __shfl_sync(0xffffffffu, pos0, leader);
      if (key >= 0) order[pos0 + __popc(peers & lt)] = (int)j;
      __syncwarp();
      if (lane == leader && key >= 0) cur[key] = pos0 + __popc(peers);
      __syncwarp();
    }
  }
}

// Within each radial bracket, orders the columns by polar angle (the sine in
// fixed point, increasing over the x > 0, y > 0 quadrant; ties by column
// index, so the order is deterministic).  One CTA per bracket sorts its
// segment of the bracket-sorted list in shared memory (bitonic); a segment
// longer than kAngleSortMax keeps its (bracket, angle bin) order.  Any
// column order gives the same product; this one puts columns of nearly the
// same angle next to each other, so neighbouring columns read nearly the
// same library pixels for a given image pixel.
constexpr int kAngleSortMax = 4096;
__global__ void __launch_bounds__(1024) angle_sort_kernel(const ColGeom *geom, int n_r, int *order,
                                                          const int *bstart) {
  __shared__ long long key[kAngleSortMax];
  __shared__ int val[kAngleSortMax];
  const int k = blockIdx.x;
  const int begin = bstart[k * PSFSIM_THETA_BINS], end = bstart[(k + 1) * PSFSIM_THETA_BINS];
  const int m = end - begin;
  if (m < 2 || m > kAngleSortMax) return;
  int pow2 = 1;
  while (pow2 < m) pow2 <<= 1;
  for (int i = threadIdx.x; i < pow2; i += blockDim.x) {
    if (i < m) {
      const int j = order[begin + i];
      key[i] = geom[j].Sn;
      val[i] = j;
    } else {
      key[i] = LLONG_MAX;
      val[i] = INT_MAX;
    }
  }
  __syncthreads();
  for (int size = 2; size <= pow2; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < pow2; i += blockDim.x) {
        const int partner = i ^ stride;
        if (partner > i) {
          const bool up = (i & size) == 0;
          const bool gt = key[i] > key[partner] || (key[i] == key[partner] && val[i] > val[partner]);
          if (gt == up) {
            const long long tk = key[i];
            key[i] = key[partner];
            key[partner] = tk;
            const int tv = val[i];
            val[i] = val[partner];
            val[partner] = tv;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < m; i += blockDim.x) order[begin + i] = val[i];
}

struct BuildParams {
  int n, n_r, Wp, compact;  // compact: column c of the sorted list is stored at position c
  int N;                    // scene side of a grid build (0: field points)
  int64_t K, ld;
  const ColGeom *geom;
  const int *order;
  const int *bstart;
  const float *lib;
  float *A;
  int *status;
};

// Radial lerp of one library pixel (a3).  A PSF of weight zero above takes no
// part (it may hold anything).
__device__ __forceinline__ float lerp_pixel(float w0, float w1, float l0, float l1) {
  const float t = __fmul_rn(w0, l0);
  return w1 != 0.f ? fmaf(w1, l1, t) : t;
}

// Bilinear sample (a4) of a lerped 2 x 2 footprint at the 32-bit fractions fa
// and fb of its column and row.  Each weight is formed from its own exact
// integer, so a tiny one is accurate relative to itself too (2^32 - f as
// (2^32 - 1 - f) + 1: the sum is exact below 2^24 and under half an ulp above).
// Lerping before sampling halves the taps.  Every FP32 build samples with these
// operations, so all store the same bits.
__device__ __forceinline__ float bilinear(float t00, float t01, float t10, float t11, unsigned fa, unsigned fb) {
  constexpr float kInv32 = 2.3283064365386963e-10f;  // 2^-32
  const float wa1 = __uint2float_rn(fa) * kInv32, wa0 = (__uint2float_rn(~fa) + 1.f) * kInv32;
  const float wb1 = __uint2float_rn(fb) * kInv32, wb0 = (__uint2float_rn(~fb) + 1.f) * kInv32;
  const float r0 = fmaf(wa0, t00, __fmul_rn(wa1, t01));
  const float r1 = fmaf(wa0, t10, __fmul_rn(wa1, t11));
  return fmaf(wb0, r0, __fmul_rn(wb1, r1));
}

// One element from the two library PSFs: a2/b2 hold 2a and 2b in fixed point
// with PSFSIM_FRAC_BITS fraction bits; tap(row, col, l0, l1) fetches both PSFs'
// pixel (zeros outside).  The taps are all requested before any is used.
template <typename TapFn>
__device__ __forceinline__ float rotated_value(long long a2, long long b2, int n, float w0, float w1, TapFn tap) {
  constexpr int kShift = PSFSIM_FRAC_BITS + 1;
  const int q0 = (int)(a2 >> kShift);
  const int p0 = (int)(b2 >> kShift);
  if (q0 < -1 || q0 > n - 1 || p0 < -1 || p0 > n - 1) return 0.f;
  float l0[4], l1[4];
  tap(p0, q0, l0[0], l1[0]);
  tap(p0, q0 + 1, l0[1], l1[1]);
  tap(p0 + 1, q0, l0[2], l1[2]);
  tap(p0 + 1, q0 + 1, l0[3], l1[3]);
  return bilinear(lerp_pixel(w0, w1, l0[0], l1[0]), lerp_pixel(w0, w1, l0[1], l1[1]), lerp_pixel(w0, w1, l0[2], l1[2]),
                  lerp_pixel(w0, w1, l0[3], l1[3]), (unsigned)((unsigned long long)a2 >> (kShift - 32)),
                  (unsigned)((unsigned long long)b2 >> (kShift - 32)));
}

// Writes column j of A (FP32, column-major) with one warp.
template <bool kSmem, bool kVec4>
__device__ __forceinline__ void build_column(const BuildParams &P, int j, int64_t dest, const float *s0,
                                             const float *s1, int lane) {
  const ColGeom g = P.geom[j];
  float *col = P.A + dest * P.ld;
  const int n = P.n;
  const int64_t M = (int64_t)n * n;
  if (g.k < 0) {
    for (int64_t i = lane; i < P.ld; i += 32) col[i] = 0.f;
    return;
  }
  const float *L0 = P.lib + (int64_t)g.k * M;
  const float *L1 = L0 + M;
  const int Wp = P.Wp;
  auto tap = [&](int r, int c, float &l0, float &l1) {
    if (kSmem) {
      const int i = (r + 1) * Wp + (c + 4);
      l0 = s0[i];
      l1 = s1[i];
    } else {
      l0 = l1 = 0.f;
      if (r >= 0 && r < n && c >= 0 && c < n) {
        l0 = __ldg(L0 + r * n + c);
        l1 = __ldg(L1 + r * n + c);
      }
    }
  };
  const long long h = n - 1;
  const long long base = h << PSFSIM_FRAC_BITS;
  if (kVec4) {
    const int n4 = n >> 2;
    int q4 = lane, p = 0;
    while (q4 >= n4) { q4 -= n4; ++p; }
    const int total = (int)(M >> 2);
    for (int f = lane; f < total; f += 32) {
      const int q = q4 << 2;
      long long a2 = base + g.C * (2 * q - h) + g.Sn * (2 * p - h);
      long long b2 = base - g.Sn * (2 * q - h) + g.C * (2 * p - h);
      float4 v;
      v.x = rotated_value(a2, b2, n, g.w0, g.w1, tap);
      a2 += 2 * g.C; b2 -= 2 * g.Sn;
      v.y = rotated_value(a2, b2, n, g.w0, g.w1, tap);
      a2 += 2 * g.C; b2 -= 2 * g.Sn;
      v.z = rotated_value(a2, b2, n, g.w0, g.w1, tap);
      a2 += 2 * g.C; b2 -= 2 * g.Sn;
      v.w = rotated_value(a2, b2, n, g.w0, g.w1, tap);
      __stcs(reinterpret_cast<float4 *>(col + (int64_t)p * n + q), v);
      q4 += 32;
      while (q4 >= n4) { q4 -= n4; ++p; }
    }
  } else {
    for (int64_t i = lane; i < M; i += 32) {
      const int p = (int)(i / n), q = (int)(i % n);
      const long long a2 = base + g.C * (2 * q - h) + g.Sn * (2 * p - h);
      const long long b2 = base - g.Sn * (2 * q - h) + g.C * (2 * p - h);
      col[i] = rotated_value(a2, b2, n, g.w0, g.w1, tap);
    }
  }
  for (int64_t i = M + lane; i < P.ld; i += 32) col[i] = 0.f;
}

// Walks this CTA's contiguous range of the bracket-sorted column list group
// by group (one radial bracket, every angle bin; or the zero columns).  With
// kSmem, a group's bracket pair L[k], L[k+1] (zero-padded by one pixel) is
// staged in shared memory at s0 by one TMA tensor load whenever the bracket
// changes; then work(pos, gend) runs for the group's list positions.  The
// whole CTA calls it (it synchronizes); mbar must be initialised.  A staging
// copy that times out sets PSFSIM_ERR_TIMEOUT and ends the walk.
template <bool kSmem, class GroupWork>
__device__ __forceinline__ void for_each_bracket_group(const CUtensorMap *map, const BuildParams &P, float *s0,
                                                       uint64_t *mbar, GroupWork work) {
  const int64_t begin = P.K * blockIdx.x / gridDim.x;
  const int64_t end = P.K * (blockIdx.x + 1) / gridDim.x;
  const uint32_t tx_bytes = 2u * (uint32_t)((P.n + 2) * P.Wp) * 4u;
  int cur_k = -2;
  uint32_t phase = 0;
  bool failed = false;
  for (int64_t pos = begin; pos < end;) {
    const int j0 = P.order[pos];
    const int k = P.geom[j0].k;
    const int group_end = k < 0 ? psfsim_num_buckets(P.n_r) : (k + 1) * PSFSIM_THETA_BINS;
    const int64_t gend = min(end, (int64_t)P.bstart[group_end]);
    if (kSmem && k >= 0 && k != cur_k) {
      __syncthreads();  // every warp is done with the previous pair
      if (threadIdx.x == 0) {
        ptx::mbar_arrive_expect_tx(mbar, tx_bytes);
        ptx::tma_load_3d(s0, map, -4, -1, k, mbar);
      }
      if (!ptx::mbar_wait_bounded(mbar, phase)) failed = true;
      cur_k = k;
      if (__syncthreads_or(failed)) {
        // The copy may still be landing in shared memory: give it one more
        // bounded wait before the CTA exits.
        if (threadIdx.x == 0) {
          ptx::mbar_wait_bounded(mbar, phase);
          atomicExch(P.status, PSFSIM_ERR_TIMEOUT);
        }
        return;
      }
      phase ^= 1u;
    }
    work(pos, gend);
    pos = gend;
  }
}

// Each CTA owns a contiguous range of the bracket-sorted column list; its warps
// build whole columns, one warp per column.
template <bool kSmem, bool kVec4>
__global__ void __launch_bounds__(512) build_fp32_kernel(const __grid_constant__ CUtensorMap map,
                                                         const BuildParams P) {
  extern __shared__ __align__(128) float smem[];
  __shared__ __align__(8) uint64_t mbar;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  float *s0 = smem;
  float *s1 = smem + (P.n + 2) * P.Wp;
  if (kSmem && threadIdx.x == 0) {
    ptx::mbar_init(&mbar, 1);
    ptx::fence_mbar_init();
  }
  __syncthreads();
  for_each_bracket_group<kSmem>(&map, P, s0, &mbar, [&](int64_t pos, int64_t gend) {
    for (int64_t c = pos + warp; c < gend; c += nwarps) {
      const int j = P.order[c];
      build_column<kSmem, kVec4>(P, j, P.compact ? c : (int64_t)j, s0, s1, lane);
    }
  });
}

// Dense FP32 storage of an even N x N grid through the exact quarter-turn
// symmetry: R(ix, iy) = (N-1-iy, ix) on the scene and P(p, q) = (q, n-1-p) on
// the image leave the fixed-point source coordinates unchanged, so column R(j)
// holds at pixel P(i) the bits column j holds at i.  A warp builds one 32 x 32
// pixel block of a column of the x > 0, y > 0 quadrant at a time (in shared
// memory) and writes it to its four turned places, A[P^m(block), R^m(j)]:
// every copy is 32 rows of 32 contiguous floats.
constexpr int kSymBlk = 32, kSymPitch = 33;  // block side; shared pitch (transposed reads without conflicts)

// A column of the x > 0, y > 0 quadrant and its three turned copies.
struct TurnedColumns {
  float *at[4];
};
__device__ __forceinline__ TurnedColumns turned_columns(const BuildParams &P, int jq) {
  const int N = P.N, H = N / 2;
  const int iy = H + jq / H, ix = H + jq % H;  // quadrant entry jq
  return TurnedColumns{{P.A + ((int64_t)iy * N + ix) * P.ld, P.A + ((int64_t)ix * N + (N - 1 - iy)) * P.ld,
                        P.A + ((int64_t)(N - 1 - iy) * N + (N - 1 - ix)) * P.ld,
                        P.A + ((int64_t)(N - 1 - ix) * N + iy) * P.ld}};
}

// One 32 x 32 pixel block at (p0, q0) of a quadrant column, to its four turned
// places.  value(a2, b2) samples; lane: pixel column q0 + lane, down the rows in
// exact steps.  Copies 0 and 2 leave as the rows are made, 32 contiguous floats
// each (copy 2 backwards); the block goes through shared memory for copies 1 and
// 3, whose rows are its columns.
template <class ValueFn, class RowFn>
__device__ __forceinline__ void build_block_sym(int n, const ColGeom &g, const TurnedColumns &A, int p0, int q0,
                                                float *blk, int lane, ValueFn value, RowFn each_row) {
  __syncwarp();  // the previous block's copies have read the buffer
  const long long h = n - 1;
  const long long base = h << PSFSIM_FRAC_BITS;
  const int q = q0 + lane;
  long long a2 = base + g.C * (2 * q - h) + g.Sn * (2 * p0 - h);
  long long b2 = base - g.Sn * (2 * q - h) + g.C * (2 * p0 - h);
  float *r0 = A.at[0] + (int64_t)p0 * n + q, *r2 = A.at[2] + (int64_t)(n - 1 - p0) * n + (n - 1 - q);
#pragma unroll 4
  for (int a = 0; a < kSymBlk; ++a, r0 += n, r2 -= n) {
    each_row(a);
    const float v = value(a2, b2);
    blk[a * kSymPitch + lane] = v;
    __stcs(r0, v);
    __stcs(r2, v);
    a2 += 2 * g.Sn;
    b2 += 2 * g.C;
  }
  __syncwarp();
  // Copy 1: row q0 + r, columns n-32-p0 .. (source column r, rows reversed);
  // copy 3: row n-1-q0-r, columns p0 .. (source column r).
  float *r1 = A.at[1] + (int64_t)q0 * n + (n - kSymBlk - p0) + lane, *r3 = A.at[3] + (int64_t)(n - 1 - q0) * n + p0 + lane;
#pragma unroll 4
  for (int r = 0; r < kSymBlk; ++r, r1 += n, r3 -= n) {
    __stcs(r1, blk[(kSymBlk - 1 - lane) * kSymPitch + r]);
    __stcs(r3, blk[lane * kSymPitch + r]);
  }
}

// Dense FP32 storage of an even grid, n % 32 == 0: the CTAs deal the sorted
// quadrant columns round-robin (neighbours in the list, so the same PSFs, are in
// work at once, and the columns beyond the last radius spread evenly); the warps
// of a CTA take the 32 x 32 blocks of its column.
// kLerped: the column's lerped PSF sits in shared memory, zero-bordered by one
// pixel, and while a column is sampled its CTA lerps the next one into the other
// of two buffers, loads eight rows ahead of their use.  Four taps an element
// instead of eight, at a row pitch where a rotated line of 32 taps meets few bank
// conflicts, and half the passes through shared memory for the copies: 1156 ->
// 960 us for the paper's 16384 x 65536 A (4.5 TB/s written; no pipe is the bound
// alone: issue 55 %, L1 data pipe 58 %, with 16 warps an SM in shared memory's
// reach).  32 warps of 16-row blocks, whose turned rows are 64 bytes: 1040 us.
template <bool kLerped>
__global__ void __launch_bounds__(512, 1) build_fp32_sym_kernel(const BuildParams P) {
  extern __shared__ __align__(128) float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const int n = P.n, Wp = P.Wp, plane = kLerped ? (n + 2) * Wp : 0;
  const int64_t M = (int64_t)n * n;
  float *blk = smem + 2 * plane + warp * (kSymBlk * kSymPitch);
  const int nbq = n / kSymBlk, nblocks = nbq * nbq;
  if (kLerped)
    for (int i = threadIdx.x; i < 2 * plane; i += blockDim.x) smem[i] = 0.f;  // the borders stay zero
  // The thread's share of a column, two quads of pixels at a time: quads
  // threadIdx.x + blockDim.x i of the plane.
  constexpr int kBatch = 2;
  const int quads = (int)(M >> 2), rowq = n >> 2;
  const int per = (quads + (int)blockDim.x * kBatch - 1) / ((int)blockDim.x * kBatch);  // batches a thread
  float4 l0[kBatch], l1[kBatch];
  auto fetch = [&](const ColGeom &g, int batch) {
    const float4 *L0 = reinterpret_cast<const float4 *>(P.lib + (int64_t)g.k * M) + threadIdx.x;
    const float4 *L1 = reinterpret_cast<const float4 *>(P.lib + (int64_t)(g.k + 1) * M) + threadIdx.x;
#pragma unroll
    for (int e = 0; e < kBatch; ++e) {
      const int i = (batch * kBatch + e) * (int)blockDim.x;
      if (i + (int)threadIdx.x < quads) {
        l0[e] = __ldg(L0 + i);
        l1[e] = __ldg(L1 + i);
      }
    }
  };
  auto put = [&](const ColGeom &g, int batch, float *dst) {
#pragma unroll
    for (int e = 0; e < kBatch; ++e) {
      const int i = (batch * kBatch + e) * (int)blockDim.x + (int)threadIdx.x;
      if (i < quads) {
        const int r = i / rowq;
        *reinterpret_cast<float4 *>(dst + (r + 1) * Wp + 4 * (i - r * rowq) + 4) =
            make_float4(lerp_pixel(g.w0, g.w1, l0[e].x, l1[e].x), lerp_pixel(g.w0, g.w1, l0[e].y, l1[e].y),
                        lerp_pixel(g.w0, g.w1, l0[e].z, l1[e].z), lerp_pixel(g.w0, g.w1, l0[e].w, l1[e].w));
      }
    }
  };
  ColGeom g;
  int jq = 0;
  int64_t pos = blockIdx.x;
  if (pos < P.K) {
    jq = P.order[pos];
    g = P.geom[jq];
  }
  if (kLerped) {
    __syncthreads();
    if (pos < P.K && g.k >= 0)
      for (int b = 0; b < per; ++b) {
        fetch(g, b);
        put(g, b, smem);
      }
    __syncthreads();
  }
  for (int buf = 0; pos < P.K; pos += gridDim.x, buf ^= 1) {
    const bool more = pos + gridDim.x < P.K;
    int jn = 0;
    ColGeom gn;
    gn.k = -1;
    if (more) {
      jn = P.order[pos + gridDim.x];
      gn = P.geom[jn];
    }
    const float *cur = smem + buf * plane;
    float *dst = smem + (buf ^ 1) * plane;
    const bool lerp = kLerped && gn.k >= 0;
    int fetched = 0, done = 0;  // batches of the next column loaded, and lerped
    const TurnedColumns A = turned_columns(P, jq);
    for (int b = warp; b < nblocks; b += nwarps) {
      const int p0 = (b / nbq) * kSymBlk, q0 = (b % nbq) * kSymBlk;
      if (g.k < 0) {  // beyond the last radius: zeros
        build_block_sym(n, g, A, p0, q0, blk, lane, [](long long, long long) { return 0.f; }, [](int) {});
      } else if (kLerped) {
        build_block_sym(
            n, g, A, p0, q0, blk, lane,
            [&](long long a2, long long b2) {
              // Pixel (p, q) sits at (p + 1, q + 4); a footprint wholly outside reads
              // the zeros right of the first row's border.
              constexpr int kShift = PSFSIM_FRAC_BITS + 1;
              const unsigned qa = (unsigned)((int)(a2 >> kShift) + 1), pb = (unsigned)((int)(b2 >> kShift) + 1);
              const bool in = qa <= (unsigned)n && pb <= (unsigned)n;
              const float *t = cur + (in ? pb * (unsigned)Wp + qa + 3u : (unsigned)n + 4u);
              return bilinear(t[0], t[1], t[Wp], t[Wp + 1], (unsigned)((unsigned long long)a2 >> (kShift - 32)),
                              (unsigned)((unsigned long long)b2 >> (kShift - 32)));
            },
            [&](int a) {
              if (lerp && (a & 7) == 0) {
                if (done < fetched) put(gn, done++, dst);
                if (fetched < per) fetch(gn, fetched++);
              }
            });
      } else {
        const float *L0 = P.lib + (int64_t)g.k * M, *L1 = L0 + M;
        build_block_sym(
            n, g, A, p0, q0, blk, lane,
            [&](long long a2, long long b2) {
              return rotated_value(a2, b2, n, g.w0, g.w1, [&](int r, int c, float &l0, float &l1) {
                l0 = l1 = 0.f;
                if (r >= 0 && r < n && c >= 0 && c < n) {
                  l0 = __ldg(L0 + r * n + c);
                  l1 = __ldg(L1 + r * n + c);
                }
              });
            },
            [](int) {});
      }
    }
    if (kLerped) {
      if (lerp) {
        if (done < fetched) put(gn, done++, dst);
        for (; fetched < per; ++fetched) {
          fetch(gn, fetched);
          put(gn, done++, dst);
        }
      }
      __syncthreads();
    }
    jq = jn;
    g = gn;
  }
}

// Row pitch of a lerped plane: a multiple of 4 (quads of pixels are stored at
// once), at least n + 8 (the border, and zeros beyond it).  Of those up to 28
// more, 20 and then 28 mod 32 meet a rotated line of 32 taps with the fewest bank
// conflicts over the angles (2.3 ways; 0 mod 32: 8), where two planes and the
// block buffers then fit.
constexpr size_t kSymSmem = 226 * 1024;
inline size_t sym_smem(int n, int pitch, int warps) {
  return (2ull * (n + 2) * pitch + (size_t)warps * kSymBlk * kSymPitch) * 4;
}
inline int sym_pitch(int n, int warps) {
  for (int residue : {20, 28}) {
    const int p = (n + 8 - residue + 31) / 32 * 32 + residue;
    if (sym_smem(n, p, warps) <= kSymSmem) return p;
  }
  return n + 8;
}

}  // namespace

WsLayout psfsim_layout(int n, int64_t K, int storage, int n_r) {
  WsLayout L{};
  const int64_t M = (int64_t)n * n;
  int64_t off = 0;
  auto take = [&](int64_t bytes) {
    const int64_t at = off;
    off = psfsim_round_up(off + bytes, 256);
    return at;
  };
  L.lo_off = L.scale_off = -1;
  if (storage == PSFSIM_FP32 || storage == PSFSIM_FP32_SYM) {
    L.ld = psfsim_round_up(M, 32);
    // FP32_SYM stores at most the x > 0, y > 0 quadrant's columns.
    L.a_off = take(L.ld * (storage == PSFSIM_FP32_SYM ? (K + 3) / 4 : K) * 4);
  } else if (storage == PSFSIM_SPLIT_BF16 || storage == PSFSIM_BF16 || storage == PSFSIM_SPLIT_BF16_SYM) {
    // SPLIT_BF16_SYM stores at most the x > 0, y > 0 quadrant's columns.
    L.ld = psfsim_round_up(storage == PSFSIM_SPLIT_BF16_SYM ? (K + 3) / 4 : K, 64);
    const int64_t rows = psfsim_round_up(M, 128);
    L.a_off = take(rows * L.ld * 2);
    if (storage != PSFSIM_BF16) L.lo_off = take(rows * L.ld * 2);
    L.scale_off = take(L.ld * 4);
  } else {  // FUSED: nothing but the tables
    L.ld = 0;
    L.a_off = -1;
  }
  L.geom_off = take(K * (int64_t)sizeof(ColGeom));
  L.order_off = take(K * 4);
  L.bstart_off = take((int64_t)(psfsim_num_buckets(PSFSIM_MAX_RADII) + 1) * 4);
  L.pts_off = take(K * 16);
  L.status_off = take(16);
  L.libmax_off = take(PSFSIM_MAX_RADII * 4);
  // FUSED keeps the library as pair entries (both PSFs of a radial bracket,
  // each pixel's 2 x 2 bilinear footprint tap by tap, 32 bytes)
  L.plib_off = storage == PSFSIM_FUSED ? take(psfsim_pair_library_bytes(n, n_r)) : -1;
  // ... and the generators' column table.
  L.cols_off = storage == PSFSIM_FUSED ? take(psfsim_fused_columns_bytes(K)) : -1;
  L.mtorder_off = storage == PSFSIM_FUSED ? take(psfsim_fused_mtile_order_bytes(n)) : -1;
  L.total = L.total_pix = off;
  L.pix_off = -1;
  if (const int64_t extra = psfsim_pixel_build_bytes(n, K, storage, n_r)) {
    L.pix_off = take(extra);
    L.total_pix = off;
  }
  return L;
}

static cudaError_t launch_tables_and_build(psfsim_plan *h, cudaStream_t st);

static bool encode_library_map(psfsim_plan *h, int Wp) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
      return false;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  const int n = h->n;
  cuuint64_t dims[3] = {(cuuint64_t)n, (cuuint64_t)n, (cuuint64_t)h->n_r};
  cuuint64_t strides[2] = {(cuuint64_t)n * 4, (cuuint64_t)n * n * 4};
  cuuint32_t box[3] = {(cuuint32_t)Wp, (cuuint32_t)(n + 2), 2};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode(&h->lib_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void *)h->d_lib, dims, strides, box,
                      estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

cudaError_t psfsim_launch_build(psfsim_plan *h, cudaStream_t st) {
  const cudaError_t e = launch_tables_and_build(h, st);
  if (e != cudaSuccess || h->storage == PSFSIM_FUSED) return e;
  if (const cudaError_t e2 = psfsim_launch_live_table(h, st)) return e2;  // the column order is free from here on
  // The retrieval's forward kernels read A and the column list before they wait
  // for the kernel ahead of them (programmatic launch), so that kernel must not
  // be one that writes them: end with an operation that waits for those (split
  // storages have no such reader).
  if (h->storage != PSFSIM_FP32 && h->storage != PSFSIM_FP32_SYM) return cudaSuccess;
  return cudaMemsetAsync(h->ws + h->status_off + 8, 0, 8, st);
}

static cudaError_t launch_tables_and_build(psfsim_plan *h, cudaStream_t st) {
  // Dense storage of an even grid is built from the x > 0, y > 0 quadrant's
  // columns, four quarter-turned copies each, so the geometry tables cover
  // the quadrant only (entry (iy - N/2) (N/2) + ix - N/2).  The split
  // builds without pair entries take no column order.
  const bool dense_split = h->storage == PSFSIM_SPLIT_BF16 || h->storage == PSFSIM_BF16;
  const bool sym = !h->quadrant && h->N > 0 && h->N % 2 == 0 &&
                   (dense_split || (h->storage == PSFSIM_FP32 && h->n % kSymBlk == 0));
  const int64_t Kg = sym ? h->K / 4 : h->Kg;
  GeomParams G;
  std::memset(&G, 0, sizeof(G));
  G.n_r = h->n_r;
  G.N = h->N;
  G.interp = h->interp;
  G.K = Kg;
  G.S = h->S;
  G.pts = h->N ? nullptr : reinterpret_cast<const double *>(h->ws + h->pts_off);
  G.quadrant = h->quadrant || sym ? 1 : 0;
  for (int i = 0; i < h->n_r; ++i) G.radii[i] = h->radii[i];
  ColGeom *geom = reinterpret_cast<ColGeom *>(h->ws + h->geom_off);
  int *order = reinterpret_cast<int *>(h->ws + h->order_off);
  int *bstart = reinterpret_cast<int *>(h->ws + h->bstart_off);
  int *status = reinterpret_cast<int *>(h->ws + h->status_off);
  cudaError_t e = cudaMemsetAsync(status, 0, 16, st);
  if (e != cudaSuccess) return e;
  geom_kernel<<<(unsigned)((Kg + 255) / 256), 256, 0, st>>>(G, geom);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (!dense_split || (sym && h->pix)) {
    // chunks of at least 256 columns, and as many as fit in shared memory
    const int nb = psfsim_num_buckets(h->n_r);
    int W = (int)((Kg + 255) / 256);
    const int fit = (int)((200 * 1024) / ((size_t)nb * sizeof(int)));
    W = W < 1 ? 1 : (W > 32 ? 32 : W);
    W = W > fit ? fit : W;
    const size_t smem = (size_t)W * nb * sizeof(int);
    if ((e = cudaFuncSetAttribute(bracket_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
        cudaSuccess)
      return e;
    bracket_sort_kernel<<<1, 1024, smem, st>>>(geom, Kg, h->n_r, W, order, bstart);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (dense_split) {
      angle_sort_kernel<<<h->n_r - 1, 1024, 0, st>>>(geom, h->n_r, order, bstart);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  if (h->quadrant) {
    // The host needs the number of columns inside the last radius to size launches.
    int kv = 0;
    if ((e = cudaMemcpyAsync(&kv, bstart + psfsim_num_buckets(h->n_r) - 1, sizeof(int), cudaMemcpyDeviceToHost,
                             st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
      return e;
    h->K_valid = kv;
    if (h->storage == PSFSIM_FUSED) {
      angle_sort_kernel<<<h->n_r - 1, 1024, 0, st>>>(geom, h->n_r, order, bstart);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      return psfsim_launch_pair_library(h, st);
    }
    // Compact split-BF16 rows hold just the valid columns (the layout reserved
    // the whole quadrant, an upper bound, before the count was known).
    if (h->storage == PSFSIM_SPLIT_BF16_SYM) h->ld = psfsim_round_up(kv > 0 ? kv : 1, 64);
  }
  psfsim_live_count(h);
  if (h->storage == PSFSIM_SPLIT_BF16 || h->storage == PSFSIM_BF16 || h->storage == PSFSIM_SPLIT_BF16_SYM)
    return psfsim_launch_split_build(h, st);
  if (h->storage != PSFSIM_FP32 && h->storage != PSFSIM_FP32_SYM) return cudaErrorNotSupported;
  const bool compact = h->storage == PSFSIM_FP32_SYM;

  const int n = h->n;
  const int Wp = (int)psfsim_round_up(n, 4) + 8;
  const size_t smem = 2ull * (size_t)(n + 2) * Wp * 4;
  const bool vec4 = (n % 4) == 0;
  const bool use_smem = vec4 && smem <= 200 * 1024 && Wp <= 256 && encode_library_map(h, Wp);
  BuildParams P;
  P.n = n;
  P.n_r = h->n_r;
  P.Wp = Wp;
  P.compact = compact ? 1 : 0;
  P.N = h->N;
  P.K = compact ? h->K_valid : h->K;
  P.ld = h->ld;
  P.geom = geom;
  P.order = order;
  P.bstart = bstart;
  P.lib = h->d_lib;
  P.A = reinterpret_cast<float *>(h->ws + h->a_off);
  P.status = status;
  CUtensorMap dummy;
  std::memset(&dummy, 0, sizeof(dummy));
  int threads = 512, per_sm = 1;
  if (sym) {
    // Even grid: the quadrant's columns (the sorted list holds just those),
    // four turned copies each.
    P.K = Kg;
    const int nblocks = (n / kSymBlk) * (n / kSymBlk), warps = nblocks < 16 ? nblocks : 16;
    P.Wp = sym_pitch(n, warps);
    const bool lerped = sym_smem(n, P.Wp, warps) <= kSymSmem;
    const size_t total = lerped ? sym_smem(n, P.Wp, warps) : (size_t)warps * kSymBlk * kSymPitch * 4;
    auto kern = lerped ? build_fp32_sym_kernel<true> : build_fp32_sym_kernel<false>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)total)) != cudaSuccess)
      return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * warps, total)) != cudaSuccess) return e;
    per_sm = per_sm < 1 ? 1 : per_sm;
    const int64_t grid = (int64_t)h->num_sms * per_sm;
    kern<<<(unsigned)(grid < Kg ? grid : Kg), 32 * warps, total, st>>>(P);
    return cudaGetLastError();
  }
  if (use_smem) {
    threads = smem > 100 * 1024 ? 512 : 256;
    auto kern = build_fp32_kernel<true, true>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
      return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem)) != cudaSuccess)
      return e;
    per_sm = per_sm < 1 ? 1 : per_sm;
    kern<<<h->num_sms * per_sm, threads, smem, st>>>(h->lib_map, P);
  } else {
    threads = 256;
    per_sm = 8;
    if (vec4)
      build_fp32_kernel<false, true><<<h->num_sms * per_sm, threads, 0, st>>>(dummy, P);
    else
      build_fp32_kernel<false, false><<<h->num_sms * per_sm, threads, 0, st>>>(dummy, P);
  }
  return cudaGetLastError();
}
