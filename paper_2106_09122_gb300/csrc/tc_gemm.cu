// Batched S = A Z (Eq. 6) on the 5th-generation tensor cores for split-BF16
// (and BF16) A.
//
// Y[b, i] = sum_j sigma_j (hi_ij + lo_ij) x_bj.  The scene batch is scaled by
// sigma_j and split exactly into three bf16 parts x' = x1 + x2 + x3 (24 bits),
// stacked as the rows of one MMA B operand, so each k-step issues two MMAs:
//   D[:, 0:3Bp] += hi * [x1 x2 x3]^T     D[:, Bp:3Bp] += lo * [x1 x2]^T
// and the epilogue sums the three column blocks: (hi + lo)(x1 + x2) + hi x3,
// i.e. only the lo * x3 term (< 2^-24 relative) is dropped; what remains is
// the 2^-17 relative storage error of hi + lo and the FP32 accumulation.  lo x1
// is as small as hi x2, and lo x2 as hi x3: added one block on, they are not cut
// at the last bit of the large hi x1 (the accumulation is not rounded to nearest).
// Errors against 64 bits, blocks 0 and 1 / 1 and 2: ten mixed plans 1.12e-6 /
// 1.07e-6, 16 scenes of 256^2 5.7e-7 / 5.3e-7, 8 residuals of 128^2 2.542e-6 /
// 2.537e-6 (the plain FP32 sums of before the tensor cores: 2.537e-6); same times.
// BF16 storage has no lo: one MMA per k-step over two x parts,
// D[:, 0:2Bp] += hi * [x1 x2]^T, so the result carries the 2^-8 relative
// storage error of hi and the dropped hi * x3 term (< 2^-16 relative).
//
// The adjoint A^T g of the same storages (but of one residual where nearly all columns
// are read: split_adjoint.cu) is the same kernel with A's tiles
// transposed: an M-tile is 128 columns (two 64-column k-tiles of the forward,
// live ones only), the contraction runs over the image rows 64 at a time, A's
// tiles arrive as two M-major boxes of 64 columns x 64 rows, and the residuals
// take x's place, always in three parts.  adj_finish_kernel adds the k-splits
// and scales the columns.
//
// Dense plans on a scene grid are mostly zero columns (beyond the last library
// radius): only the 64-column k-tiles that hold a live column are loaded
// (live.cu; TMA starts them at multiples of 32 columns).
//
// Persistent warp-specialised kernel, one CTA per SM:
//   warp 0  TMA producer (2D tiled loads, 128-byte swizzle) into a smem ring
//   warp 1  MMA issuer (tcgen05.mma, accumulators in TMEM, double-buffered)
//   warps 2-5 epilogue (tcgen05.ld -> FP32 sums -> partial images)
// Work unit = (128-row m-tile, k-range); k is split KS ways for balance and
// the KS partial images are summed in a fixed order (deterministic).
// Every mbarrier wait is bounded; a timeout sets PSFSIM_ERR_TIMEOUT.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <cstring>

#include "live.cuh"
#include "psfsim_internal.cuh"
#include "ptx_util.cuh"
#include "reduce.cuh"

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kMaxStages = 8;
constexpr int kThreads = 192;
// TMEM per CTA: two accumulators of up to 256 columns (one CTA per SM), or,
// when every accumulator fits in 128 columns (BF16 storage, 64 scenes or
// fewer), two of 128 so that two CTAs, two load/MMA pipelines, share an SM.
constexpr uint32_t kTmemColsWide = 512, kAccStrideWide = 256;
constexpr uint32_t kTmemColsNarrow = 256, kAccStrideNarrow = 128;
constexpr uint32_t kTileBytes = BM * BK * 2;
constexpr int kMaxBp = 80;       // 3 * Bp <= 256 (MMA N and TMA box limits), Bp % 16 == 0
constexpr int kMaxJobs = 16;
constexpr int kDefaultChunk = 4; // k-tiles (of 64) per TMEM accumulation, split-BF16 storage
// One job of split storage: fewer splits sum longer runs (choose_ks), and draining
// more often pays that back without costing time: 16 scenes of 128^2 take 142 us at
// 4, 2 and 1 k-tiles, and their product errs 4.2e-7, 2.5e-7 and 1.7e-7 (against the
// stored A in 64 bits).  Accumulators of more than 128 columns are drained slower
// than they fill: 64 scenes take 156 us at 4 and 3, 159 at 2, 176 at 1.
constexpr int kSingleChunk = 1, kSingleChunkWide = 3;
constexpr int kDefaultChunkHiMulti = 2;  // BF16 storage (hi alone), several jobs in one launch
// Adjoint of split storage: residuals change sign, so its sums cancel and the
// drift weighs more: 8 residuals of 128^2 err 2.537e-6 against 64 bits with plain
// FP32 sums, 2.552 at 4 k-tiles, 2.537 at one; 124 us a call either way (8 of 256^2
// 1.50 and 1.51 ms).
constexpr int kAdjointChunk = 1;
constexpr int kAdjointRun = 160;  // and the most k-tiles a unit adds up, with one job or several
constexpr int kMaxMmas = 64;     // accumulating MMAs between drains (bounds the FP32 drift)

// One product S_j = A_j Z_j of a (possibly multi-job) launch.
struct TcJob {
  int Bp, KS, m_tiles, k_tiles;
  int tiles, ld;       // adjoint: 64-column tiles of A (ktab's), and A's row pitch
  int has_lo;          // split-BF16 (hi + lo) or BF16 (hi alone)
  int xparts;          // bf16 parts of x in the B operand: 3 (split-BF16) or 2 (BF16)
  int unit_begin;      // first work unit of this job
  int cap;             // scenes in the job's buffers (<= Bp)
  const int *ktab;     // first column of every k-tile (NULL: k-tile t starts at column 64 t)
  const int *count;    // device int: scenes present (NULL: all cap)
  float *out;          // partial images [KS][cap][out_ld]; with one split, the images themselves
  int64_t out_ld, out_rows;  // out_ld = out_rows = rows, or M for the images themselves
};

// Kernel parameter block: tensor maps (hi, lo, x) and geometry of every job.
struct TcMulti {
  CUtensorMap map[kMaxJobs][3];
  TcJob job[kMaxJobs];
  int njobs, units, stages, chunk;
  uint32_t stage_bytes;
  uint32_t x_off;  // byte offset of the x tile in a stage: after hi and lo, or after hi alone
  int adjoint;     // A transposed: M-tiles of columns, k-tiles of 64 image rows
  int interleave;  // jobs share one A and one unit count: unit u is job u % njobs, unit u / njobs
  uint32_t tmem_cols, acc_stride;
  int *status;
  uint64_t wait_ns;  // limit of every bounded wait
  int64_t stall_it;  // test hook: the producer never issues this load (-1: none)
};

// One job's scene split (xsplit_kernel).
struct XJob {
  const float *x;
  const int *count;    // scenes present (NULL: all B)
  const int *ktab;     // k-tile table, dead groups after it (live.cu), or NULL
  const int *order;    // compact storage: quadrant pixel of every column (else NULL)
  int turn;            // adjoint of compact storage: image side n, x holds whole images (else 0)
  const float *scale;  // per column (adjoint: NULL)
  __nv_bfloat16 *xs;   // [3][Bp][width]
  int64_t K, width, dead_groups;
  int B, Bp, N, first; // compact storage: slot b is rotated scene first + b, i.e. scene / 4 turned % 4 times
};
struct XMulti {
  XJob job[kMaxJobs];
};

// xs[part][b][t] of job blockIdx.y: the three bf16 parts of scene b at the t-th
// column that the k-tiles cover, times the column's scale (width = 64 k-tiles
// columns).  The columns in no k-tile are zero in A; a non-finite scene value
// there still makes the whole image NaN (0 x inf), as it does when they are
// multiplied out: position t adds 0 x for its share of them.  Compact storage
// reads the four rotated pixels of a column straight from the scene.  One
// launch serves every job (ten jobs: 12 us, against 33 us and the gaps of ten).
__global__ void __launch_bounds__(256) xsplit_kernel(const __grid_constant__ XMulti P) {
  const XJob &J = P.job[blockIdx.y];
  const int64_t width = J.width, total = (int64_t)J.Bp * width;
  const int nb = J.count ? min(*J.count, J.B) : J.B;
  const int *dead = J.ktab + width / BK;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(t / width);
    const int64_t c = t % width;
    float v = 0.f;
    if (b < nb) {
      if (J.turn) {
        if (c < J.K) {
          int p = (int)(c / J.turn), q = (int)(c % J.turn);
          const int r = J.first + b;
          for (int k = 0; k < (r & 3); ++k) {  // P(p, q) = (q, n-1-p)
            const int np = q;
            q = J.turn - 1 - p;
            p = np;
          }
          v = J.x[(int64_t)(r >> 2) * J.K + (int64_t)p * J.turn + q];
        }
      } else if (J.order) {
        if (c < J.K) {
          const int H = J.N / 2, j0 = J.order[c], r = J.first + b;
          int ix = H + j0 % H, iy = H + j0 / H;
          for (int k = 0; k < (r & 3); ++k) {  // R(ix, iy) = (N-1-iy, ix)
            const int nx = J.N - 1 - iy;
            iy = ix;
            ix = nx;
          }
          v = J.x[(int64_t)(r >> 2) * J.N * J.N + (int64_t)iy * J.N + ix] * J.scale[c];
        }
      } else {
        const float *xb = J.x + (int64_t)b * J.K;
        const int64_t j = J.ktab ? J.ktab[c / BK] + c % BK : c;
        if (j < J.K) v = J.scale ? xb[j] * J.scale[j] : xb[j];
#pragma unroll 4
        for (int64_t e = c; e < J.dead_groups * kLiveGroup; e += width) {
          const int64_t jd = (int64_t)dead[e / kLiveGroup] * kLiveGroup + e % kLiveGroup;
          v += 0.f * xb[min(jd, J.K - 1)];
        }
      }
    }
    const __nv_bfloat16 x1 = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(x1);
    const __nv_bfloat16 x2 = __float2bfloat16_rn(r1);
    const float r2 = r1 - __bfloat162float(x2);
    J.xs[t] = x1;
    J.xs[total + t] = x2;
    J.xs[2 * total + t] = __float2bfloat16_rn(r2);
  }
}

// One job's sum over its k-splits (tc_reduce_kernel).
struct RJob {
  const float *part;  // [KS][cap][rows]
  float *y;           // [cap][M]
  const int *count;
  int64_t rows, M;
  int KS, cap;
};
struct RMulti {
  RJob job[kMaxJobs];
};

// y[b, i] = sum_ks part[ks, b, i] of job blockIdx.z (reduce.cuh).  One launch serves every job.
template <bool kSerial>
__global__ void __launch_bounds__(256) tc_reduce_kernel(const __grid_constant__ RMulti P) {
  const RJob &J = P.job[blockIdx.z];
  const int b = blockIdx.y;
  if (b >= J.cap || (J.count && b >= *J.count)) return;
  reduce_partials<kSerial>(J.part + (int64_t)b * J.rows, (int64_t)J.cap * J.rows, J.KS, J.rows, J.M,
                           J.y + (int64_t)b * J.M);
}

// The adjoint's result from its partial sums, part[KS][cap][rows] per block of
// kMaxBp residuals: thread t of residual b adds the k-splits of compact column
// t, scales it and stores it at its column (dense), or at the turned pixel of
// scene b / 4 (compact storage).  Threads beyond the compact columns serve the
// columns in no tile: zero.  A residual value that is not finite gives NaN in
// its split parts; such a column is summed again from the stored elements, as
// the plain product would, so that infinities come out as they always did.  So is
// a sum below M 2^-108, which a column has where it meets only values below 2^-108
// (M rows of elements up to 1): the lesser bf16 parts of still smaller ones are
// subnormal and have lost bits (residuals of 2^-112 err 1.7e-6, of 2^-120 2.5e-5).
struct AdjFinish {
  const float *part[kMaxJobs];
  int cap[kMaxJobs];
  int KS, n, N;
  long long R2;        // dense grid: live pixels are within it (live.cuh); else -1
  int64_t rows, width, dead_groups, K, Kv, M, ld;  // width: compact columns
  const int *ktab, *order;
  const float *scale;
  const __nv_bfloat16 *hi, *lo;
  const float *g;
  float *gx;
};

__device__ __noinline__ float plain_adjoint(const AdjFinish &P, int b, int64_t j) {
  const float *g = P.g + (int64_t)(P.order ? b >> 2 : b) * P.M;
  float acc = 0.f;
#pragma unroll 4
  for (int64_t i = 0; i < P.M; ++i) {
    int64_t k = i;
    if (P.order) {
      int p = (int)(i / P.n), q = (int)(i % P.n);
      for (int m = 0; m < (b & 3); ++m) {
        const int np = q;
        q = P.n - 1 - p;
        p = np;
      }
      k = (int64_t)p * P.n + q;
    }
    const float a = __bfloat162float(P.hi[i * P.ld + j]) + (P.lo ? __bfloat162float(P.lo[i * P.ld + j]) : 0.f);
    acc = fmaf(a, g[k], acc);
  }
  return acc;
}

__global__ void __launch_bounds__(256) adj_finish_kernel(const __grid_constant__ AdjFinish P) {
  const int b = blockIdx.y, blk = b / kMaxBp, slot = b % kMaxBp;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const float *part = P.part[blk] + (int64_t)slot * P.rows;
  const int64_t step = (int64_t)P.cap[blk] * P.rows;
  auto sum = [&](int64_t at) {
    float s = 0.f;
#pragma unroll 4
    for (int ks = 0; ks < P.KS; ++ks) s += part[ks * step + at];
    return s;
  };
  const int64_t j = t >= P.width ? P.Kv : P.ktab ? P.ktab[t / BK] + t % BK : t;
  const bool column = j < P.Kv;
  float s = column ? sum(t) : 0.f;
  // A sum of zero that is not a dead column's (the k-tiles hold some): zero it is
  // where the residual has a larger value, which the CTA looks for.
  bool again = s != s || (column && s != 0.f && fabsf(s) < (float)P.M * 0x1p-108f);
  bool zero = column && s == 0.f;
  if (zero && P.R2 >= 0) {
    const long long X = 2 * (j % P.N) - (P.N - 1), Y = 2 * (j / P.N) - (P.N - 1);
    zero = X * X + Y * Y <= P.R2;
  }
  if (__syncthreads_or(zero)) {
    const float *g = P.g + (int64_t)(P.order ? b >> 2 : b) * P.M;
    bool some = false, large = false;
    for (int64_t i0 = 0; !large && i0 < P.M; i0 += 4 * 256) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t i = i0 + 256 * u + threadIdx.x;
        const float v = i < P.M ? fabsf(g[i]) : 0.f;
        some = some || v != 0.f;
        large = large || v >= 0x1p-108f;
      }
      large = __syncthreads_or(large);
    }
    if (!large && __syncthreads_or(some)) again = again || zero;
  }
  if (column) {
    if (again) s = plain_adjoint(P, b, j);
    s *= P.scale[j];
    if (P.order) {
      const int H = P.N / 2, j0 = P.order[j];
      int ix = H + j0 % H, iy = H + j0 / H;
      for (int k = 0; k < (b & 3); ++k) {  // R(ix, iy) = (N-1-iy, ix)
        const int nx = P.N - 1 - iy;
        iy = ix;
        ix = nx;
      }
      P.gx[(int64_t)(b >> 2) * P.K + (int64_t)iy * P.N + ix] = s;
    } else {
      P.gx[(int64_t)b * P.K + j] = s;
    }
  } else if (t >= P.width && t - P.width < P.dead_groups * kLiveGroup) {
    const int64_t e = t - P.width, jd = (int64_t)P.ktab[P.width / BK + e / kLiveGroup] * kLiveGroup + e % kLiveGroup;
    if (jd >= P.Kv) return;
    const float s0 = sum(0);
    P.gx[(int64_t)b * P.K + jd] = s0 != s0 ? plain_adjoint(P, b, jd) * P.scale[jd] : 0.f;
  }
}

__device__ __forceinline__ void set_abort(volatile int *abort_flag, int *status) {
  *abort_flag = 1;
  atomicExch(status, PSFSIM_ERR_TIMEOUT);
}

__device__ __forceinline__ int find_job(const TcMulti &P, int u) {
  int j = 0;
  while (j + 1 < P.njobs && u >= P.job[j + 1].unit_begin) ++j;
  return j;
}

// Work unit u -> (job, unit within the job).  Interleaved jobs (several scene
// blocks against one A) put the same (m-tile, k-range) of every job on
// neighbouring units, so CTAs running together read the same A tiles and L2
// serves all but the first read.
__device__ __forceinline__ void unit_of(const TcMulti &P, int u, int &jb, int &lu) {
  if (P.interleave) {
    jb = u % P.njobs;
    lu = u / P.njobs;
  } else {
    jb = find_job(P, u);
    lu = u - P.job[jb].unit_begin;
  }
}

__device__ __forceinline__ int k_begin(const TcJob &J, int ks) { return (int)((int64_t)J.k_tiles * ks / J.KS); }

__global__ void __launch_bounds__(kThreads, 2) tc_gemm_kernel(const __grid_constant__ TcMulti P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], tfull_bar[2], tempty_bar[2];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t lim = P.wait_ns;
  if (threadIdx.x == 0) {
    for (int s = 0; s < P.stages; ++s) {
      ptx::mbar_init(&full_bar[s], 1);
      ptx::mbar_init(&empty_bar[s], 1);
    }
    ptx::mbar_init(&drain_bar, 1);
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull_bar[a], 1);
      ptx::mbar_init(&tempty_bar[a], 4);
    }
    abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(&tmem_base_sh, P.tmem_cols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tbase = tmem_base_sh;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    uint32_t it = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok && !abort_flag; u += gridDim.x) {
      int jb, lu;
      unit_of(P, u, jb, lu);
      const TcJob &J = P.job[jb];
      const int ks = lu / J.m_tiles, mt = lu % J.m_tiles;
      const uint32_t tx = (J.has_lo ? 2 : 1) * kTileBytes + (uint32_t)(J.xparts * J.Bp) * BK * 2;
      const int k0 = k_begin(J, ks), k1 = k_begin(J, ks + 1);
      int next = J.ktab && !P.adjoint ? __ldg(J.ktab + k0) : 0;  // read one k-tile ahead of its use
      int ca = 0, cb = 0;  // adjoint: the M-tile's two runs of 64 columns (the last may be absent: past A's edge)
      if (P.adjoint) {
        ca = J.ktab ? __ldg(J.ktab + 2 * mt) : 2 * mt * BK;
        cb = 2 * mt + 1 >= J.tiles ? J.ld : J.ktab ? __ldg(J.ktab + 2 * mt + 1) : (2 * mt + 1) * BK;
      }
      for (int kt = k0; kt < k1; ++kt, ++it) {
        const int col = J.ktab ? next : kt * BK;
        if (J.ktab && !P.adjoint && kt + 1 < k1) next = __ldg(J.ktab + kt + 1);
        const int s = (int)(it % P.stages);
        if (!ptx::mbar_wait_bounded(&empty_bar[s], ((it / P.stages) & 1) ^ 1, lim)) {
          set_abort(&abort_flag, P.status);
          ok = false;
          break;
        }
        if ((int64_t)it == P.stall_it) continue;  // test hook: this stage is never filled
        uint8_t *st = smem + (size_t)s * P.stage_bytes;
        ptx::mbar_arrive_expect_tx(&full_bar[s], tx);
        if (P.adjoint) {
          for (int part = 0; part < (J.has_lo ? 2 : 1); ++part) {
            ptx::tma_load_2d(st + part * kTileBytes, &P.map[jb][part], ca, kt * BK, &full_bar[s]);
            ptx::tma_load_2d(st + part * kTileBytes + kTileBytes / 2, &P.map[jb][part], cb, kt * BK, &full_bar[s]);
          }
        } else {
          ptx::tma_load_2d(st, &P.map[jb][0], col, mt * BM, &full_bar[s]);
          if (J.has_lo) ptx::tma_load_2d(st + kTileBytes, &P.map[jb][1], col, mt * BM, &full_bar[s]);
        }
        ptx::tma_load_2d(st + P.x_off, &P.map[jb][2], kt * BK, 0, &full_bar[s]);
      }
    }
    // Drain: the last `stages` loads issued may not have been consumed (after
    // a timeout the MMA issuer stops early); wait for each to land so that no
    // copy into this CTA's shared memory is in flight when the CTA exits.
    // Nothing re-armed these stages afterwards, so their phases are final.
    for (uint32_t i = it > (uint32_t)P.stages ? it - (uint32_t)P.stages : 0u; i < it; ++i)
      if ((int64_t)i != P.stall_it && !ptx::mbar_wait_bounded(&full_bar[i % P.stages], (i / P.stages) & 1, lim))
        set_abort(&abort_flag, P.status);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    uint32_t it = 0, c = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok && !abort_flag; u += gridDim.x) {
      int jb, lu;
      unit_of(P, u, jb, lu);
      const TcJob &J = P.job[jb];
      const int ks = lu / J.m_tiles;
      const int k0 = k_begin(J, ks), k1 = k_begin(J, ks + 1);
      const uint32_t major = P.adjoint ? 1u << 15 : 0u;  // A is M-major
      const uint32_t idesc3 = ptx::idesc_bf16_f32(BM, J.xparts * J.Bp) | major;
      const uint32_t idesc2 = ptx::idesc_bf16_f32(BM, 2 * J.Bp) | major;
      const bool has_lo = J.has_lo != 0;
      for (int kc = k0; kc < k1 && ok; kc += P.chunk, ++c) {
        const int kc1 = min(kc + P.chunk, k1);
        const uint32_t acc = c & 1;
        if (!ptx::mbar_wait_bounded(&tempty_bar[acc], ((c >> 1) & 1) ^ 1, lim)) {
          set_abort(&abort_flag, P.status);
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        const uint32_t d_tmem = tbase + acc * P.acc_stride;
        const uint32_t d_lo = d_tmem + (uint32_t)J.Bp;  // lo's products: one block on
        for (int kt = kc; kt < kc1; ++kt, ++it) {
          const int s = (int)(it % P.stages);
          if (!ptx::mbar_wait_bounded(&full_bar[s], (it / P.stages) & 1, lim)) {
            set_abort(&abort_flag, P.status);
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          const uint8_t *st = smem + (size_t)s * P.stage_bytes;
          const uint64_t dh = P.adjoint ? ptx::smem_desc_mn_sw128(st, kTileBytes / 2, 1024) : ptx::smem_desc_sw128(st);
          const uint64_t dl = P.adjoint ? ptx::smem_desc_mn_sw128(st + kTileBytes, kTileBytes / 2, 1024)
                                        : ptx::smem_desc_sw128(st + kTileBytes);
          const uint64_t dx = ptx::smem_desc_sw128(st + P.x_off);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t adv = (uint64_t)(kk * 32) >> 4;  // 16 bf16 = 32 bytes along K
            const uint64_t adva = P.adjoint ? (uint64_t)(kk * 2048) >> 4 : adv;  // M-major: two groups of 8 rows
            ptx::mma_bf16(d_tmem, dh + adva, dx + adv, idesc3, (kt > kc || kk > 0) ? 1u : 0u);
            if (has_lo) ptx::mma_bf16(d_lo, dl + adva, dx + adv, idesc2, 1u);
          }
          ptx::mma_commit(&empty_bar[s]);
        }
        if (ok) ptx::mma_commit(&tfull_bar[acc]);
      }
    }
    // Drain: wait until every MMA this thread issued has completed, so that
    // none still reads shared memory or writes TMEM when the CTA releases them.
    ptx::mma_commit(&drain_bar);
    if (!ptx::mbar_wait_bounded(&drain_bar, 0, lim)) set_abort(&abort_flag, P.status);
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    // The tensor core's FP32 accumulation is not rounded to nearest, so its
    // error grows with the number of accumulating MMAs.  Each accumulator
    // therefore holds at most P.chunk k-tiles; the epilogue drains it into
    // FP32 register sums and hands it back (double-buffered).
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    uint32_t c = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
      int jb, lu;
      unit_of(P, u, jb, lu);
      const TcJob &J = P.job[jb];
      const int ks = lu / J.m_tiles, mt = lu % J.m_tiles;
      const int k0 = k_begin(J, ks), k1 = k_begin(J, ks + 1);
      const int Bp = J.Bp;
      const bool third = J.xparts == 3;
      float sum[kMaxBp];
#pragma unroll
      for (int t = 0; t < kMaxBp; ++t) sum[t] = 0.f;
      for (int kc = k0; kc < k1; kc += P.chunk, ++c) {
        // Lane 0 alone takes the bounded wait and the abort decision, so the
        // warp stays converged for the .sync.aligned TMEM loads below.
        const uint32_t acc = c & 1;
        int good = 0;
        if (lane == 0) {
          good = !abort_flag && ptx::mbar_wait_bounded(&tfull_bar[acc], (c >> 1) & 1, lim);
          if (!good) set_abort(&abort_flag, P.status);
        }
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) {
          ok = false;
          break;
        }
        // Already complete (lane 0 saw it): this gives every lane its acquire.
        if (!ptx::mbar_wait_bounded(&tfull_bar[acc], (c >> 1) & 1, lim)) set_abort(&abort_flag, P.status);
        ptx::tc_fence_after();
        const uint32_t tacc = tbase + ((uint32_t)(quarter * 32) << 16) + acc * P.acc_stride;
#pragma unroll
        for (int q = 0; q < kMaxBp / 16; ++q) {
          if (q * 16 < Bp) {
            float v0[16], v1[16], v2[16];
            ptx::tmem_ld16(tacc + q * 16, v0);
            ptx::tmem_ld16(tacc + Bp + q * 16, v1);
            if (third) ptx::tmem_ld16(tacc + 2 * Bp + q * 16, v2);
            ptx::tmem_ld_wait();
            if (third) {
#pragma unroll
              for (int t = 0; t < 16; ++t) sum[q * 16 + t] += (v0[t] + v1[t]) + v2[t];
            } else {
#pragma unroll
              for (int t = 0; t < 16; ++t) sum[q * 16 + t] += v0[t] + v1[t];
            }
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&tempty_bar[acc]);
      }
      if (!ok) break;
      const int nb = J.count ? min(*J.count, J.cap) : J.cap;
      const int64_t i = (int64_t)mt * BM + row;
      float *out = J.out + (int64_t)ks * J.cap * J.out_ld + i;
      if (i < J.out_rows) {
#pragma unroll
        for (int t = 0; t < kMaxBp; ++t)
          if (t < nb) out[(int64_t)t * J.out_ld] = sum[t];
      }
    }
  }
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tbase, P.tmem_cols);
  }
}

// ---- many scenes of one plan -------------------------------------------------
//
// With scenes along the MMA's N, a step reads A's 128-row tiles and every x part
// from shared memory for each of its two MMAs: about 200 bytes a clock against
// the 128 it delivers, which held 256 rotated scenes of 256^2 to half the tensor
// rate (998 us).  Beyond 80 scenes (wide_form) the roles are swapped: 128 scenes are
// the MMA's M, 256 image pixels its N, and all five products
//     x1 hi + x2 hi + x3 hi + x1 lo + x2 lo      (BF16: x1 hi + x2 hi)
// accumulate into one accumulator of 256 columns, two of which alternate, so
// each MMA is a full 128 x 256 x 16 (96 bytes of operands a clock).  Every
// k-tile is drained into FP32 sums by itself (20 accumulating MMAs: less drift
// than the narrow form's 32), by eight epilogue warps of 128 pixels each.
// Two stages of x (three parts of 128 scenes, 48 KB) and A (hi and lo of 256
// pixels, 64 KB).  Blocks of 128 scenes interleave, so A comes from L2.
constexpr int kWideScenes = 128, kWidePix = 256;
constexpr int kWideThreads = 320;
constexpr uint32_t kWideX = kWideScenes * BK * 2, kWideA = kWidePix * BK * 2;
constexpr int kWideStages = 2;

struct TcWide {
  CUtensorMap hi, lo, x;
  int njobs, KS, n_tiles, k_tiles, units, has_lo, scenes;
  int x_rows;  // rows of one x part (128 njobs)
  const int *ktab;
  float *out;  // [KS][scenes][out_ld]
  int64_t out_ld, out_rows;
  int *status;
  uint64_t wait_ns;
  int64_t stall_it;  // test hook: the producer never issues this load (-1: none)
};

__global__ void __launch_bounds__(kWideThreads, 1) tc_wide_kernel(const __grid_constant__ TcWide P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full_bar[kWideStages], empty_bar[kWideStages], tfull_bar[2], tempty_bar[2];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t lim = P.wait_ns;
  const int xparts = P.has_lo ? 3 : 2;
  const uint32_t a_off = 3 * kWideX, stage_bytes = a_off + 2 * kWideA;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kWideStages; ++s) {
      ptx::mbar_init(&full_bar[s], 1);
      ptx::mbar_init(&empty_bar[s], 1);
    }
    ptx::mbar_init(&drain_bar, 1);
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull_bar[a], 1);
      ptx::mbar_init(&tempty_bar[a], 8);
    }
    abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(&tmem_base_sh, 512);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tbase = tmem_base_sh;
  auto k_at = [&](int ks) { return (int)((int64_t)P.k_tiles * ks / P.KS); };

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    uint32_t it = 0;
    bool ok = true;
    const uint32_t tx = xparts * kWideX + (P.has_lo ? 2 : 1) * kWideA;
    for (int u = blockIdx.x; u < P.units && ok && !abort_flag; u += gridDim.x) {
      const int jb = u % P.njobs, nt = u / P.njobs % P.n_tiles, ks = u / P.njobs / P.n_tiles;
      const int k0 = k_at(ks), k1 = k_at(ks + 1);
      int next = P.ktab ? __ldg(P.ktab + k0) : 0;
      for (int kt = k0; kt < k1; ++kt, ++it) {
        const int col = P.ktab ? next : kt * BK;
        if (P.ktab && kt + 1 < k1) next = __ldg(P.ktab + kt + 1);
        const int s = (int)(it % kWideStages);
        if (!ptx::mbar_wait_bounded(&empty_bar[s], ((it / kWideStages) & 1) ^ 1, lim)) {
          set_abort(&abort_flag, P.status);
          ok = false;
          break;
        }
        if ((int64_t)it == P.stall_it) continue;  // test hook: this stage is never filled
        uint8_t *st = smem + (size_t)s * stage_bytes;
        ptx::mbar_arrive_expect_tx(&full_bar[s], tx);
        ptx::tma_load_2d(st + a_off, &P.hi, col, nt * kWidePix, &full_bar[s]);
        if (P.has_lo) ptx::tma_load_2d(st + a_off + kWideA, &P.lo, col, nt * kWidePix, &full_bar[s]);
        for (int part = 0; part < xparts; ++part)
          ptx::tma_load_2d(st + part * kWideX, &P.x, kt * BK, part * P.x_rows + jb * kWideScenes, &full_bar[s]);
      }
    }
    // Drain: the last loads issued may not have been consumed (as in tc_gemm_kernel).
    for (uint32_t i = it > (uint32_t)kWideStages ? it - (uint32_t)kWideStages : 0u; i < it; ++i)
      if ((int64_t)i != P.stall_it && !ptx::mbar_wait_bounded(&full_bar[i % kWideStages], (i / kWideStages) & 1, lim))
        set_abort(&abort_flag, P.status);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    uint32_t it = 0;
    bool ok = true;
    const uint32_t idesc = ptx::idesc_bf16_f32(kWideScenes, kWidePix);
    for (int u = blockIdx.x; u < P.units && ok && !abort_flag; u += gridDim.x) {
      const int ks = u / P.njobs / P.n_tiles;
      for (int kt = k_at(ks); kt < k_at(ks + 1); ++kt, ++it) {
        const uint32_t acc = it & 1;
        const int s = (int)(it % kWideStages);
        if (!ptx::mbar_wait_bounded(&tempty_bar[acc], ((it >> 1) & 1) ^ 1, lim) ||
            !ptx::mbar_wait_bounded(&full_bar[s], (it / kWideStages) & 1, lim)) {
          set_abort(&abort_flag, P.status);
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        const uint8_t *st = smem + (size_t)s * stage_bytes;
        const uint64_t x1 = ptx::smem_desc_sw128(st), x2 = ptx::smem_desc_sw128(st + kWideX),
                       x3 = ptx::smem_desc_sw128(st + 2 * kWideX);
        const uint64_t dh = ptx::smem_desc_sw128(st + a_off), dl = ptx::smem_desc_sw128(st + a_off + kWideA);
        const uint32_t d = tbase + acc * 256;
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) {
          const uint64_t adv = (uint64_t)(kk * 32) >> 4;
          ptx::mma_bf16(d, x1 + adv, dh + adv, idesc, kk > 0 ? 1u : 0u);
          ptx::mma_bf16(d, x2 + adv, dh + adv, idesc, 1u);
          if (P.has_lo) {
            ptx::mma_bf16(d, x3 + adv, dh + adv, idesc, 1u);
            ptx::mma_bf16(d, x1 + adv, dl + adv, idesc, 1u);
            ptx::mma_bf16(d, x2 + adv, dl + adv, idesc, 1u);
          }
        }
        ptx::mma_commit(&empty_bar[s]);
        ptx::mma_commit(&tfull_bar[acc]);
      }
    }
    ptx::mma_commit(&drain_bar);
    if (!ptx::mbar_wait_bounded(&drain_bar, 0, lim)) set_abort(&abort_flag, P.status);
  } else if (warp >= 2) {
    // ---------------- epilogue: scene 32 (warp % 4) + lane, pixels 128 half .. +127 ----------------
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    uint32_t it = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
      const int jb = u % P.njobs, nt = u / P.njobs % P.n_tiles, ks = u / P.njobs / P.n_tiles;
      float sum[128];
#pragma unroll
      for (int t = 0; t < 128; ++t) sum[t] = 0.f;
      for (int kt = k_at(ks); kt < k_at(ks + 1); ++kt, ++it) {
        const uint32_t acc = it & 1;
        int good = 0;
        if (lane == 0) {
          good = !abort_flag && ptx::mbar_wait_bounded(&tfull_bar[acc], (it >> 1) & 1, lim);
          if (!good) set_abort(&abort_flag, P.status);
        }
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) {
          ok = false;
          break;
        }
        // Already complete (lane 0 saw it): this gives every lane its acquire.
        if (!ptx::mbar_wait_bounded(&tfull_bar[acc], (it >> 1) & 1, lim)) set_abort(&abort_flag, P.status);
        ptx::tc_fence_after();
        const uint32_t t0 = tbase + ((uint32_t)(quarter * 32) << 16) + acc * 256 + half * 128;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float v[16];
          ptx::tmem_ld16(t0 + q * 16, v);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int t = 0; t < 16; ++t) sum[q * 16 + t] += v[t];
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&tempty_bar[acc]);
      }
      if (!ok) break;
      const int scene = jb * kWideScenes + quarter * 32 + lane;
      const int64_t px = (int64_t)nt * kWidePix + half * 128;
      if (scene < P.scenes && px < P.out_rows) {
        float *out = P.out + ((int64_t)ks * P.scenes + scene) * P.out_ld + px;
#pragma unroll
        for (int t = 0; t < 128; t += 8)
          if (px + t < P.out_rows)
            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out + t), "f"(sum[t]),
                         "f"(sum[t + 1]), "f"(sum[t + 2]), "f"(sum[t + 3]), "f"(sum[t + 4]), "f"(sum[t + 5]),
                         "f"(sum[t + 6]), "f"(sum[t + 7])
                         : "memory");
      }
    }
  }
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tbase, 512);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  return encode;
}

bool encode_bf16_2d(CUtensorMap *map, const void *base, uint64_t inner, uint64_t outer, uint32_t box_inner,
                    uint32_t box_outer, CUtensorMapL2promotion promotion = CU_TENSOR_MAP_L2_PROMOTION_L2_256B) {
  auto encode = get_encoder();
  if (!encode) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, promotion,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


struct JobSpec {
  const psfsim_plan *h;
  const float *x;
  float *y;
  int cap;
  const int *count;
  int first;  // compact storage: x holds whole scenes, and slot b is rotated scene first + b (-1: plain)
};

struct JobPlan {
  int Bp, KS, m_tiles, k_tiles;
  int64_t rows;
  size_t xs_off, part_off;
};

// Split over k of a single job: the cheapest by the launch's clocks.  CTAs walk the
// units in rounds of `slots`; a k-tile of a round takes what its TMA pipeline needs
// alone (1750 clocks, 1300 without lo), its share of memory at 4000 bytes a clock,
// or its SM's shared memory under the MMAs, whichever is longest.  A unit's start
// and store cost 1800; partial images 2700 for their launch and their bytes
// written and read again.  The constants are a fit to 96 products (64^2..256^2
// pixels and grids, 1..64 scenes, both directions, both storages) at 15 splits
// each: 1.4 % above the best split on average, 12 % at worst.  The smallest split
// that fills the SMs evenly was 9.3 % above on average: 23 scenes of a 100^2 BF16
// plan on 85^2 pixels ran 1817 units in 43 us, 237 in 37; 64 of a 256^2 one on
// 64^2 pixels took 121 us in three splits, 78 in one.  At most `most` k-tiles a
// unit: the drained sums add up one after another in FP32, and the adjoint of
// 256^2 split storage errs 2 % more with its 1024 in one chain than in runs of
// 146 (kAdjointRun; 8 residuals 1.51 ms, 1.45 in one).
int choose_ks(const JobPlan &p, int cap, int x_rows, bool lo, bool direct1, int most, int slots,
              int num_sms) {
  const double a_bytes = lo ? 2.0 * kTileBytes : kTileBytes, x_bytes = x_rows * BK * 2.0;
  const double alone = lo ? 1750.0 : 1300.0, mma = (lo ? 2.0 : 1.0) * (kTileBytes + x_bytes) / 48.0;
  auto tile = [&](int64_t active) {
    const double mem = (double)active * (a_bytes + x_bytes) / 4000.0;
    const double sm = (double)((active + num_sms - 1) / num_sms) * mma;
    return fmax(alone, fmax(mem, sm));
  };
  const int fewest = (p.k_tiles + most - 1) / most < 64 ? (p.k_tiles + most - 1) / most : 64;
  int best = fewest;
  double least = 1e300;
  for (int ks = fewest; ks <= 64 && ks <= p.k_tiles; ++ks) {
    const int64_t units = (int64_t)p.m_tiles * ks, full = units / slots, rest = units % slots;
    const double kt = (p.k_tiles + ks - 1) / ks;
    double cost = (double)full * (kt * tile(slots) + 1800.0);
    if (rest) cost += kt * tile(rest) + 1800.0;
    if (ks > 1 || !direct1) cost += 2700.0 + (double)ks * cap * (double)p.rows * 4.0 / 3000.0;
    if (cost < least * 0.9999) {
      least = cost;
      best = ks;
    }
  }
  return best;
}

struct MultiPlan {
  JobPlan jp[kMaxJobs];
  int njobs, units, stages, chunk, ctas_per_sm;
  uint32_t stage_bytes, x_off, tmem_cols, acc_stride;
  size_t smem, scratch;
};

// Tile/launch shape of a multi-job product.  `tune` fields of 0 take defaults:
// chunk = kDefaultChunk k-tiles per TMEM accumulation; without lo, the most
// that fit for one job and kDefaultChunkHiMulti for several (the fastest
// measured on one 128^2 job and on eight 256^2 jobs); split factors chosen so
// that the whole launch has about units_per_sm work units per SM (or, for a
// single job without tuning, by choose_ks); as many smem stages as fit.
MultiPlan plan_multi(const JobSpec *jobs, int nj, const psfsim_tuning_t *tune, bool adjoint = false) {
  MultiPlan mp;
  std::memset(&mp, 0, sizeof(mp));
  mp.njobs = nj;
  const int num_sms = jobs[0].h->num_sms;
  const int ups = tune && tune->units_per_sm > 0 ? tune->units_per_sm : 0;
  // A stage holds hi, lo (when any job has one) and the x tile; without lo
  // the stage is smaller, so more stages (bytes in flight) fit.
  bool any_lo = false;
  int x_rows = 0;  // largest B operand: x parts x Bp
  int64_t total = 0;
  for (int j = 0; j < nj; ++j) {
    const psfsim_plan *h = jobs[j].h;
    JobPlan &p = mp.jp[j];
    p.Bp = (int)psfsim_round_up(jobs[j].cap, 16);
    p.rows = adjoint ? psfsim_round_up(h->k_tiles, 2) * BK : psfsim_round_up(h->M, BM);
    p.m_tiles = (int)(p.rows / BM);
    p.k_tiles = adjoint ? (int)(psfsim_round_up(h->M, BM) / BK) : h->k_tiles;
    total += (int64_t)p.m_tiles * p.k_tiles;
    const bool lo = h->lo_off >= 0;
    any_lo = any_lo || lo;
    const int r = (lo || adjoint ? 3 : 2) * p.Bp;
    x_rows = r > x_rows ? r : x_rows;
  }
  // Accumulators of at most 128 columns: two CTAs per SM, each with half the
  // shared memory and half the tensor memory.
  const bool narrow = x_rows <= (int)kAccStrideNarrow;
  mp.ctas_per_sm = narrow ? 2 : 1;
  const int64_t target_units = (int64_t)(ups ? ups : 4) * num_sms;
  const int64_t per_unit = (total + target_units - 1) / target_units;
  int units = 0;
  size_t off = 0;
  for (int j = 0; j < nj; ++j) {
    JobPlan &p = mp.jp[j];
    if (nj == 1 && !ups) {
      p.KS = choose_ks(p, jobs[j].cap, x_rows, any_lo, jobs[j].first < 0 && !adjoint,
                       adjoint && any_lo ? kAdjointRun : p.k_tiles, num_sms * mp.ctas_per_sm, num_sms);
    } else {
      int ks = (int)((p.k_tiles + per_unit - 1) / (per_unit > 0 ? per_unit : 1));
      const int fewest = adjoint && any_lo ? (p.k_tiles + kAdjointRun - 1) / kAdjointRun : 1;
      ks = ks < fewest ? fewest : ks;
      ks = ks > 64 ? 64 : ks;
      p.KS = ks > p.k_tiles ? p.k_tiles : ks;
    }
    units += p.m_tiles * p.KS;
    const psfsim_plan *h = jobs[j].h;
    p.xs_off = off;
    off += (size_t)psfsim_round_up(3ll * p.Bp * p.k_tiles * BK * 2, 256);
    p.part_off = off;
    off += (size_t)psfsim_round_up((int64_t)p.KS * jobs[j].cap * p.rows * 4, 256);
  }
  mp.units = units;
  mp.scratch = off;
  mp.x_off = (any_lo ? 2 : 1) * kTileBytes;
  mp.stage_bytes = (uint32_t)psfsim_round_up(mp.x_off + (int64_t)x_rows * BK * 2, 1024);
  mp.tmem_cols = narrow ? kTmemColsNarrow : kTmemColsWide;
  mp.acc_stride = narrow ? kAccStrideNarrow : kAccStrideWide;
  int fit = (int)(((narrow ? 108 : 220) * 1024) / mp.stage_bytes);
  fit = fit > kMaxStages ? kMaxStages : fit;
  mp.stages = tune && tune->stages >= 2 && tune->stages < fit ? tune->stages : fit;
  // A k-tile is 4 MMAs per accumulator (8 with lo), so at most 16 (8) k-tiles
  // accumulate between drains.
  const int max_chunk = kMaxMmas / ((any_lo ? 2 : 1) * (BK / 16));
  mp.chunk = tune && tune->chunk > 0 ? (tune->chunk > max_chunk ? max_chunk : tune->chunk)
                                     : (adjoint && any_lo ? kAdjointChunk
                                        : any_lo && !adjoint && nj == 1 ? (narrow ? kSingleChunk : kSingleChunkWide)
                                        : any_lo || adjoint ? kDefaultChunk
                                        : (nj > 1 ? kDefaultChunkHiMulti : max_chunk));
  mp.smem = (size_t)mp.stages * mp.stage_bytes + 1024;
  return mp;
}

// Test hook of a launch: a short wait limit, one load the producer never
// issues, and a single CTA (see psfsim_debug_forward_stall).
struct StallHook {
  uint64_t wait_ns;
  int64_t stall_it;
  bool one_cta;
};
constexpr StallHook kNoStall = {2000000000ull, -1, false};

cudaError_t launch_multi(const JobSpec *jobs, int nj, const MultiPlan &mp, void *scratch, cudaStream_t st,
                         const StallHook &hook = kNoStall, bool adjoint = false) {
  char *base = static_cast<char *>(scratch);
  cudaError_t e;
  TcMulti P;  // kernel parameter blocks, copied at launch
  XMulti XP;
  RMulti RP;
  std::memset(&P, 0, sizeof(P));
  std::memset(&XP, 0, sizeof(XP));
  std::memset(&RP, 0, sizeof(RP));
  int64_t x_blocks = 1, red_M = 0, red_rows = 0;
  int nred = 0, red_cap = 0, red_KS = 1;
  for (int j = 0; j < nj; ++j) {
    const psfsim_plan *h = jobs[j].h;
    const JobPlan &p = mp.jp[j];
    __nv_bfloat16 *xs = reinterpret_cast<__nv_bfloat16 *>(base + p.xs_off);
    const float *scale = reinterpret_cast<const float *>(h->ws + h->scale_off);
    XJob &X = XP.job[j];
    X.x = jobs[j].x;
    X.count = jobs[j].count;
    X.ktab = h->live ? reinterpret_cast<const int *>(h->ws + h->order_off) : nullptr;
    X.order = jobs[j].first >= 0 && !adjoint ? reinterpret_cast<const int *>(h->ws + h->order_off) : nullptr;
    X.turn = jobs[j].first >= 0 && adjoint ? h->n : 0;
    X.scale = adjoint ? nullptr : scale;
    X.xs = xs;
    X.K = adjoint ? h->M : psfsim_cols(h);
    X.width = (int64_t)p.k_tiles * BK;
    X.dead_groups = adjoint ? 0 : h->dead_groups;
    X.B = jobs[j].cap;
    X.Bp = p.Bp;
    X.N = h->N;
    X.first = jobs[j].first;
    const int64_t blocks = ((int64_t)p.Bp * X.width + 255) / 256;
    x_blocks = blocks > x_blocks ? blocks : x_blocks;
    const bool has_lo = h->lo_off >= 0;
    const uint64_t a_rows = (uint64_t)psfsim_round_up(h->M, BM);
    const uint32_t box_rows = adjoint ? BK : BM;
    const int xparts = has_lo || adjoint ? 3 : 2;
    // What an L2 miss on A fetches.  256 bytes suit rows read from end to end
    // (all of a 128^2 plan's columns: 185 us, 210 at 64 bytes) and still runs of
    // three tiles a scene row (256^2, 12 of 16 lambda/D: 1752 against 1837); where
    // a row holds a tile or two, half of it is thrown away (50 scenes on ten
    // plans: 765 us, 703 at 64 bytes).  The adjoint reads a run's tiles side by
    // side, and takes 64 bytes wherever columns are skipped (256^2: 1869 / 1460).
    const auto promotion = h->live && (adjoint || h->short_runs) ? CU_TENSOR_MAP_L2_PROMOTION_L2_64B
                                                                 : CU_TENSOR_MAP_L2_PROMOTION_L2_256B;
    if (!encode_bf16_2d(&P.map[j][0], h->ws + h->a_off, (uint64_t)h->ld, a_rows, BK, box_rows, promotion) ||
        (has_lo &&
         !encode_bf16_2d(&P.map[j][1], h->ws + h->lo_off, (uint64_t)h->ld, a_rows, BK, box_rows, promotion)) ||
        !encode_bf16_2d(&P.map[j][2], xs, (uint64_t)p.k_tiles * BK, (uint64_t)(3 * p.Bp), BK,
                        (uint32_t)(xparts * p.Bp)))
      return cudaErrorInvalidValue;
    TcJob &J = P.job[j];
    J.has_lo = has_lo ? 1 : 0;
    J.xparts = xparts;
    J.tiles = h->k_tiles;
    J.ld = (int)h->ld;
    J.Bp = p.Bp;
    J.KS = p.KS;
    J.m_tiles = p.m_tiles;
    J.k_tiles = p.k_tiles;
    J.unit_begin = j == 0 ? 0 : P.job[j - 1].unit_begin + P.job[j - 1].m_tiles * P.job[j - 1].KS;
    J.cap = jobs[j].cap;
    J.ktab = X.ktab;
    if (adjoint) X.ktab = nullptr;
    J.count = jobs[j].count;
    // One split: the accumulated sums are the images (compact storage still
    // has its four rotations to add).
    const bool direct = p.KS == 1 && jobs[j].first < 0 && !adjoint;
    J.out = direct ? jobs[j].y : reinterpret_cast<float *>(base + p.part_off);
    J.out_ld = J.out_rows = direct ? h->M : p.rows;
    if (!direct && !adjoint) {
      RJob &R = RP.job[nred++];
      R.part = J.out;
      R.y = jobs[j].y;
      R.count = jobs[j].count;
      R.rows = p.rows;
      R.M = h->M;
      R.KS = p.KS;
      R.cap = jobs[j].cap;
      red_M = h->M > red_M ? h->M : red_M;
      red_KS = p.KS > red_KS ? p.KS : red_KS;
      red_rows += (int64_t)R.cap * h->M;
      red_cap = R.cap > red_cap ? R.cap : red_cap;
    }
  }
  const int64_t x_cap = (int64_t)jobs[0].h->num_sms * 8;
  xsplit_kernel<<<dim3((unsigned)(x_blocks < x_cap ? x_blocks : x_cap), (unsigned)nj), 256, 0, st>>>(XP);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  P.njobs = nj;
  P.units = mp.units;
  bool same = nj > 1;
  for (int j = 1; j < nj; ++j)
    same = same && jobs[j].h == jobs[0].h &&
           mp.jp[j].m_tiles * mp.jp[j].KS == mp.jp[0].m_tiles * mp.jp[0].KS;
  P.interleave = same ? 1 : 0;
  P.adjoint = adjoint ? 1 : 0;
  P.tmem_cols = mp.tmem_cols;
  P.acc_stride = mp.acc_stride;
  P.stages = mp.stages;
  P.chunk = mp.chunk;
  P.stage_bytes = mp.stage_bytes;
  P.x_off = mp.x_off;
  P.status = reinterpret_cast<int *>(jobs[0].h->ws + jobs[0].h->status_off);
  P.wait_ns = hook.wait_ns;
  P.stall_it = hook.stall_it;
  if ((e = cudaFuncSetAttribute(tc_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mp.smem)) !=
      cudaSuccess)
    return e;
  const int num_sms = jobs[0].h->num_sms;
  const int slots = hook.one_cta ? 1 : num_sms * mp.ctas_per_sm;
  tc_gemm_kernel<<<mp.units < slots ? mp.units : slots, kThreads, mp.smem, st>>>(P);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (jobs[0].first >= 0 || adjoint) return cudaSuccess;  // the caller adds the rotations (SymSum), or finishes
  if (nred > 0) {
    const bool serial = reduce_serial(red_KS, red_rows);
    const dim3 grid((unsigned)reduce_ctas(serial, red_M), (unsigned)red_cap, (unsigned)nred);
    if (serial)
      tc_reduce_kernel<true><<<grid, 256, 0, st>>>(RP);
    else
      tc_reduce_kernel<false><<<grid, 256, 0, st>>>(RP);
  }
  return cudaGetLastError();
}

}  // namespace

namespace {

// A batch of B scenes (compact storage: rotated scenes) against one plan as jobs
// of at most kMaxBp scenes (at most kMaxJobs of them), run by one interleaved
// persistent launch.  The launch fills in x and y.
int tc_jobs(const psfsim_plan *h, int B, JobSpec *js) {
  int nj = 0;
  for (int b0 = 0; b0 < B && nj < kMaxJobs; b0 += kMaxBp, ++nj) {
    const int c = (B - b0) < kMaxBp ? (B - b0) : kMaxBp;
    js[nj] = JobSpec{h, nullptr, nullptr, c, nullptr, h->quadrant ? b0 : -1};
  }
  return nj;
}

constexpr int kMaxLaunchScenes = kMaxJobs * kMaxBp;

// Whether `scenes` scenes (or rotated scenes) of a plan take the wide form.  One
// job of up to 80 never does: the narrow form reads A at HBM rate there.  Beyond,
// compact and BF16 storage always (us a call, narrow / wide: compact 128^2, 132
// rotated scenes 91 / 71, 256: 129 / 76; BF16 128^2, 130 scenes 290 / 187); dense
// split storage, whose A weighs twice, where its shared-memory traffic per
// 128-pixel tile and k-tile is less, 1375 clocks per 128 scenes against 512 a job
// and 8 a scene (128^2, 90 scenes: 268 narrow, 178 wide; 160: 275 and 292).
bool wide_form(const psfsim_plan *h, int scenes) {
  if (scenes <= kMaxBp) return false;
  if (h->quadrant || h->lo_off < 0) return true;
  const int narrow = 512 * ((scenes + kMaxBp - 1) / kMaxBp) + 8 * scenes;
  return 1375 * ((scenes + kWideScenes - 1) / kWideScenes) < narrow;
}

struct WidePlan {
  int njobs, KS, n_tiles, k_tiles;
  int64_t rows;
  size_t part_off, scratch;
};

WidePlan plan_wide(const psfsim_plan *h, int scenes) {
  WidePlan w;
  w.njobs = (scenes + kWideScenes - 1) / kWideScenes;
  w.rows = psfsim_round_up(h->M, BM);
  w.n_tiles = (int)((w.rows + kWidePix - 1) / kWidePix);
  w.k_tiles = h->k_tiles;
  // Splits by their cost in clocks: the rounds of units, a unit's k-tiles at 2750
  // and its partial image's 128 KB at 6000, and the partial images read again at
  // HBM rate.  (Filling the last round alone cost a 256^2 image of a 64^2 scene
  // more in partial images than in products: 148 us for 32 scenes, 75 now.)
  w.KS = 1;
  double best = 1e300;
  for (int ks = 1; ks <= 16 && ks <= w.k_tiles; ++ks) {
    const int64_t units = (int64_t)w.n_tiles * w.njobs * ks, rounds = (units + h->num_sms - 1) / h->num_sms;
    const double cost = (double)rounds * (2750.0 * ((w.k_tiles + ks - 1) / ks) + 6000.0) +
                        (double)ks * (double)scenes * (double)w.rows * 4.0 / 3400.0;
    if (cost < best) {
      best = cost;
      w.KS = ks;
    }
  }
  w.part_off = (size_t)psfsim_round_up(3ll * kWideScenes * w.njobs * w.k_tiles * BK * 2, 256);
  w.scratch = w.part_off + (size_t)w.KS * scenes * w.rows * 4;
  return w;
}

// Partial images part[KS][scenes][rows] in the scratch; compact storage: x holds
// whole scenes and the batch is their rotations.
cudaError_t launch_wide(const psfsim_plan *h, const float *x, int scenes, const WidePlan &w, void *scratch,
                        cudaStream_t st, const StallHook &hook = kNoStall) {
  __nv_bfloat16 *xs = static_cast<__nv_bfloat16 *>(scratch);
  const int *tab = reinterpret_cast<const int *>(h->ws + h->order_off);
  XMulti XP;
  TcWide P;
  std::memset(&XP, 0, sizeof(XP));
  std::memset(&P, 0, sizeof(P));
  XJob &X = XP.job[0];
  X.x = x;
  X.ktab = h->live ? tab : nullptr;
  X.order = h->quadrant ? tab : nullptr;
  X.scale = reinterpret_cast<const float *>(h->ws + h->scale_off);
  X.xs = xs;
  X.K = psfsim_cols(h);
  X.width = (int64_t)w.k_tiles * BK;
  X.dead_groups = h->dead_groups;
  X.B = scenes;
  X.Bp = kWideScenes * w.njobs;
  X.N = h->N;
  const int64_t blocks = ((int64_t)X.Bp * X.width + 255) / 256, cap = (int64_t)h->num_sms * 16;
  xsplit_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, st>>>(XP);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  P.has_lo = h->lo_off >= 0 ? 1 : 0;
  if (!encode_bf16_2d(&P.hi, h->ws + h->a_off, (uint64_t)h->ld, (uint64_t)w.rows, BK, kWidePix) ||
      (P.has_lo && !encode_bf16_2d(&P.lo, h->ws + h->lo_off, (uint64_t)h->ld, (uint64_t)w.rows, BK, kWidePix)) ||
      !encode_bf16_2d(&P.x, xs, (uint64_t)X.width, (uint64_t)(3 * X.Bp), BK, kWideScenes))
    return cudaErrorInvalidValue;
  P.njobs = w.njobs;
  P.KS = w.KS;
  P.n_tiles = w.n_tiles;
  P.k_tiles = w.k_tiles;
  P.units = w.njobs * w.n_tiles * w.KS;
  P.scenes = scenes;
  P.x_rows = X.Bp;
  P.ktab = X.ktab;
  P.out = reinterpret_cast<float *>(static_cast<char *>(scratch) + w.part_off);
  P.out_ld = P.out_rows = w.rows;
  P.status = reinterpret_cast<int *>(h->ws + h->status_off);
  P.wait_ns = hook.wait_ns;
  P.stall_it = hook.stall_it;
  const size_t smem = kWideStages * (3 * kWideX + 2 * kWideA) + 1024;
  if ((e = cudaFuncSetAttribute(tc_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return e;
  const int slots = hook.one_cta ? 1 : h->num_sms;
  tc_wide_kernel<<<P.units < slots ? P.units : slots, kWideThreads, smem, st>>>(P);
  return cudaGetLastError();
}

}  // namespace

namespace {

// One launch of a product of `count` scenes or, adjoint, residuals (compact storage:
// turned ones).  What sizes the scratch and what runs are this same plan.
struct Launch {
  bool wide;  // forward: scenes as the product's rows
  bool one;   // adjoint: one residual on CUDA cores
  int nj;
  JobSpec js[kMaxJobs];
  MultiPlan multi;
  WidePlan w;
  size_t scratch;
};

Launch plan_launch(const psfsim_plan *h, int count, bool adjoint) {
  Launch L;
  L.wide = !adjoint && wide_form(h, count);
  L.one = adjoint && count == 1 && psfsim_adjoint_one_better(h);
  L.nj = 0;
  if (L.one) {
    L.scratch = psfsim_adjoint_one_scratch(h);
  } else if (L.wide) {
    L.w = plan_wide(h, count);
    L.scratch = L.w.scratch;
  } else {
    L.nj = tc_jobs(h, count, L.js);
    L.multi = plan_multi(L.js, L.nj, nullptr, adjoint);
    L.scratch = L.multi.scratch;
  }
  return L;
}

// A batch beyond kMaxLaunchScenes runs as several launches, the last of which
// may be smaller and of the other form: the scenes of launch i.
int launch_count(int B, int i) {
  const int64_t left = B - (int64_t)i * kMaxLaunchScenes;
  return left < 0 ? 0 : (int)(left < kMaxLaunchScenes ? left : kMaxLaunchScenes);
}

// What the caller is told: enough for every batch up to B, so that a buffer for a
// large batch serves a smaller one, whose split of k may be finer and take more
// (and the remainder launch of a batch beyond kMaxLaunchScenes).
size_t tc_scratch(const psfsim_plan *h, int B, bool adjoint) {
  const int step = h->quadrant ? 4 : 1, top = launch_count(B, 0);
  size_t most = 0;
  for (int c = step; c <= top; c += step) {
    // Narrow launches of equally many jobs split alike: the last of them takes the most.
    if (c > kMaxBp && c % kMaxBp && c < top && (adjoint || !(wide_form(h, c) || wide_form(h, c + step)))) continue;
    const size_t need = plan_launch(h, c, adjoint).scratch;
    most = need > most ? need : most;
  }
  return most;
}

}  // namespace

size_t psfsim_forward_tc_scratch(const psfsim_plan *h, int B) { return tc_scratch(h, B, false); }

// What a call of B itself takes: its first launch's, or its last's (those between
// are as the first).
size_t psfsim_tc_taken(const psfsim_plan *h, int B, bool adjoint) {
  const size_t first = plan_launch(h, launch_count(B, 0), adjoint).scratch;
  if (B <= kMaxLaunchScenes) return first;
  const size_t last = plan_launch(h, launch_count(B, (B - 1) / kMaxLaunchScenes), adjoint).scratch;
  return last > first ? last : first;
}

int psfsim_tc_run(const psfsim_plan *h, int B, bool adjoint) {
  int most = 0;
  for (int i = 0, c; (c = launch_count(B, i)) > 0; ++i) {
    const Launch L = plan_launch(h, c, adjoint);
    if (L.one) continue;
    const int k = L.wide ? L.w.k_tiles : L.multi.jp[0].k_tiles, ks = L.wide ? L.w.KS : L.multi.jp[0].KS;
    const int run = (k + ks - 1) / ks;
    most = run > most ? run : most;
  }
  return most;
}

// A call of several launches is refused whole: the first launch refuses by itself.
static bool fits(const psfsim_plan *h, int total, bool adjoint, size_t scratch_bytes) {
  return total <= kMaxLaunchScenes || psfsim_tc_taken(h, total, adjoint) <= scratch_bytes;
}

static cudaError_t launch_forward(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                  size_t scratch_bytes, cudaStream_t st, const StallHook &hook) {
  if (!fits(h, B, false, scratch_bytes)) return kScratchTooSmall;
  for (int i = 0, c; (c = launch_count(B, i)) > 0; ++i) {
    Launch L = plan_launch(h, c, false);
    if (L.scratch > scratch_bytes) return kScratchTooSmall;
    const float *xb = x + (int64_t)i * kMaxLaunchScenes * h->K;
    float *yb = y + (int64_t)i * kMaxLaunchScenes * h->M;
    cudaError_t e;
    if (L.wide) {
      if ((e = launch_wide(h, xb, c, L.w, scratch, st, hook)) != cudaSuccess) return e;
      e = psfsim_launch_reduce_partials(reinterpret_cast<const float *>(static_cast<char *>(scratch) + L.w.part_off),
                                        L.w.KS, c, L.w.rows, h->M, yb, st);
    } else {
      for (int j = 0; j < L.nj; ++j) {
        L.js[j].x = xb + (int64_t)j * kMaxBp * h->K;
        L.js[j].y = yb + (int64_t)j * kMaxBp * h->M;
      }
      e = launch_multi(L.js, L.nj, L.multi, scratch, st, hook);
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t psfsim_launch_forward_tc(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                     size_t scratch_bytes, cudaStream_t st) {
  return launch_forward(h, x, B, y, scratch, scratch_bytes, st, kNoStall);
}

// Compact split storage: the four rotations of up to kMaxLaunchScenes / 4
// scenes are the launch's jobs, gathered from the scenes by xsplit_kernel; the
// partial images of all rotations are added through the inverse turns at the
// end.
cudaError_t psfsim_launch_forward_tc_sym(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                         size_t scratch_bytes, cudaStream_t st) {
  constexpr int kScenes = kMaxLaunchScenes / 4;
  static_assert(kMaxBp % 4 == 0, "a scene's rotations share a job");
  if (!fits(h, 4 * B, false, scratch_bytes)) return kScratchTooSmall;
  for (int i = 0, c; (c = launch_count(4 * B, i)) > 0; ++i) {
    Launch L = plan_launch(h, c, false);
    if (L.scratch > scratch_bytes) return kScratchTooSmall;
    if (h->K_valid == 0) return cudaMemsetAsync(y, 0, (size_t)B * h->M * 4, st);
    const float *xb = x + (int64_t)i * kScenes * h->K;
    SymSum S;
    std::memset(&S, 0, sizeof(S));
    S.n = h->n;
    cudaError_t e;
    if (L.wide) {
      e = launch_wide(h, xb, c, L.w, scratch, st);
      S.part[0] = reinterpret_cast<const float *>(static_cast<char *>(scratch) + L.w.part_off);
      S.cap[0] = S.per = c;
      S.KS[0] = L.w.KS;
      S.rows = L.w.rows;
    } else {
      for (int j = 0; j < L.nj; ++j) L.js[j].x = xb;
      e = launch_multi(L.js, L.nj, L.multi, scratch, st);
      S.per = kMaxBp;
      S.rows = L.multi.jp[0].rows;
      for (int j = 0; j < L.nj; ++j) {
        S.part[j] = reinterpret_cast<const float *>(static_cast<char *>(scratch) + L.multi.jp[j].part_off);
        S.cap[j] = L.js[j].cap;
        S.KS[j] = L.multi.jp[j].KS;
      }
    }
    if (e != cudaSuccess) return e;
    if ((e = psfsim_launch_sym_sum(S, c / 4, y + (int64_t)i * kScenes * h->M, st)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Compact storage: the four turns of the residuals are the batch.
size_t psfsim_adjoint_tc_scratch(const psfsim_plan *h, int B) { return tc_scratch(h, B, true); }

cudaError_t psfsim_launch_adjoint_tc(const psfsim_plan *h, const float *g, int B, float *gx, void *scratch,
                                     size_t scratch_bytes, cudaStream_t st) {
  const int turns = h->quadrant ? 4 : 1;
  if (!fits(h, turns * B, true, scratch_bytes)) return kScratchTooSmall;
  for (int i = 0, c; (c = launch_count(turns * B, i)) > 0; ++i) {
    Launch L = plan_launch(h, c, true);
    if (L.scratch > scratch_bytes) return kScratchTooSmall;
    if (h->quadrant && i == 0) {  // scene pixels without a column
      const cudaError_t e = cudaMemsetAsync(gx, 0, (size_t)B * h->K * 4, st);
      if (e != cudaSuccess || h->K_valid == 0) return e;
    }
    const MultiPlan &mp = L.multi;
    const int64_t b0 = (int64_t)i * (kMaxLaunchScenes / turns);
    const float *gb = g + b0 * h->M;
    if (L.one) {
      const cudaError_t e = psfsim_launch_adjoint_one(h, gb, gx + b0 * h->K, scratch, st);
      if (e != cudaSuccess) return e;
      continue;
    }
    for (int j = 0; j < L.nj; ++j) L.js[j].x = h->quadrant ? gb : gb + (int64_t)j * kMaxBp * h->M;
    cudaError_t e = launch_multi(L.js, L.nj, mp, scratch, st, kNoStall, true);
    if (e != cudaSuccess) return e;
    AdjFinish F;
    std::memset(&F, 0, sizeof(F));
    for (int j = 0; j < L.nj; ++j) {
      F.part[j] = reinterpret_cast<const float *>(static_cast<char *>(scratch) + mp.jp[j].part_off);
      F.cap[j] = L.js[j].cap;
    }
    const int *tab = reinterpret_cast<const int *>(h->ws + h->order_off);
    F.KS = mp.jp[0].KS;
    F.n = h->n;
    F.N = h->N;
    F.R2 = h->N > 0 && !h->quadrant ? live_r2(h->radii[h->n_r - 1], h->S) : -1;
    F.rows = mp.jp[0].rows;
    F.width = (int64_t)h->k_tiles * BK;
    F.dead_groups = h->dead_groups;
    F.K = h->K;
    F.Kv = psfsim_cols(h);
    F.M = h->M;
    F.ld = h->ld;
    F.ktab = h->live ? tab : nullptr;
    F.order = h->quadrant ? tab : nullptr;
    F.scale = reinterpret_cast<const float *>(h->ws + h->scale_off);
    F.hi = reinterpret_cast<const __nv_bfloat16 *>(h->ws + h->a_off);
    F.lo = h->lo_off >= 0 ? reinterpret_cast<const __nv_bfloat16 *>(h->ws + h->lo_off) : nullptr;
    F.g = gb;
    F.gx = gx + b0 * h->K;
    const int64_t threads = F.width + F.dead_groups * kLiveGroup;
    adj_finish_kernel<<<dim3((unsigned)((threads + 255) / 256), (unsigned)c), 256, 0, st>>>(F);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int psfsim_multi_validate(const psfsim_job_t *jobs, int njobs) {
  if (!jobs || njobs < 1 || njobs > kMaxJobs) return PSFSIM_ERR_ARG;
  for (int j = 0; j < njobs; ++j) {
    const psfsim_plan *h = jobs[j].plan;
    if (!h || !jobs[j].d_x || !jobs[j].d_y || jobs[j].capacity < 1 || jobs[j].capacity > kMaxBp)
      return PSFSIM_ERR_ARG;
    if (h->storage != PSFSIM_SPLIT_BF16 && h->storage != PSFSIM_BF16) return PSFSIM_ERR_UNSUPPORTED;
    if (h->device != jobs[0].plan->device) return PSFSIM_ERR_ARG;
  }
  return PSFSIM_OK;
}

static MultiPlan plan_jobs(const psfsim_job_t *jobs, int njobs, const psfsim_tuning_t *tune, JobSpec *js) {
  for (int j = 0; j < njobs; ++j) js[j] = JobSpec{jobs[j].plan, jobs[j].d_x, jobs[j].d_y, jobs[j].capacity, jobs[j].d_count, -1};
  return plan_multi(js, njobs, tune);
}

// Enough for smaller capacities too: one job's split of k depends on its capacity.
size_t psfsim_forward_multi_scratch(const psfsim_job_t *jobs, int njobs, const psfsim_tuning_t *tune) {
  JobSpec js[kMaxJobs];
  if (njobs > 1) return plan_jobs(jobs, njobs, tune, js).scratch;
  psfsim_job_t one = jobs[0];
  size_t most = 0;
  for (one.capacity = 1; one.capacity <= jobs[0].capacity; ++one.capacity) {
    const size_t need = plan_jobs(&one, 1, tune, js).scratch;
    most = need > most ? need : most;
  }
  return most;
}

cudaError_t psfsim_launch_forward_multi(const psfsim_job_t *jobs, int njobs, const psfsim_tuning_t *tune,
                                        void *scratch, size_t scratch_bytes, cudaStream_t st) {
  JobSpec js[kMaxJobs];
  const MultiPlan mp = plan_jobs(jobs, njobs, tune, js);
  if (mp.scratch > scratch_bytes) return kScratchTooSmall;
  return launch_multi(js, njobs, mp, scratch, st);
}

bool psfsim_forward_tc_one_launch(const psfsim_plan *h, int B) {
  return B <= kMaxBp || (B <= kMaxLaunchScenes && wide_form(h, B));
}

cudaError_t psfsim_launch_forward_tc_stall(const psfsim_plan *h, const float *x, int B, float *y, void *scratch,
                                           size_t scratch_bytes, uint64_t wait_ns, int64_t stall_it, cudaStream_t st) {
  const StallHook hook = {wait_ns, stall_it, true};
  return launch_forward(h, x, B, y, scratch, scratch_bytes, st, hook);
}
