// Tables of the live columns of a dense plan on a scene grid (live.cuh), in
// the column-order part of the workspace, which nothing reads after the build:
//   split storage   ktab[k_tiles]: first column (a multiple of 32) of every
//                   64-column k-tile that holds a live column, then
//                   dead[dead_groups]: the 32-column groups in no k-tile.
// What that is worth depends on the grid: the wave of 50 scenes on ten split
// plans (64..256 pixels a side, 12 lambda/D of PSFs in fields of 19 to 128)
// streams 26 % of its k-tiles, 2680 -> 852 us (651 with tc_gemm.cu's other steps);
// tiles start at multiples of 32 columns rather than 64 so that a narrow row needs
// one tile where it used to touch two, and 32 columns are the 64 bytes that HBM
// moves at least.
//   FP32 storage    the live columns, ascending, then the others, ascending.
// The host counts the same tables by the same integer arithmetic, to size
// launches without reading anything back.
#include "live.cuh"
#include "psfsim_internal.cuh"

namespace {

// Exclusive block scans over 1024 threads (max and sum), with the block total.
__device__ __forceinline__ int scan_max(int v, int *sh, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v = max(v, u);
  }
  if (lane == 31) sh[warp] = v;
  __syncthreads();
  int pre = -1;
  total = -1;
  for (int w = 0; w < 32; ++w) {
    if (w < warp) pre = max(pre, sh[w]);
    total = max(total, sh[w]);
  }
  __syncthreads();
  return max(v, pre);  // inclusive
}

__device__ __forceinline__ int scan_sum(int v, int *sh, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += u;
  }
  if (lane == 31) sh[warp] = x;
  __syncthreads();
  int pre = 0;
  total = 0;
  for (int w = 0; w < 32; ++w) {
    if (w < warp) pre += sh[w];
    total += sh[w];
  }
  __syncthreads();
  return pre + x - v;  // exclusive
}

__device__ __forceinline__ bool group_live(int N, int64_t K, long long R2, int64_t g, int64_t groups) {
  if (g >= groups) return false;
  if (g == 0 && R2 < (N & 1 ? 0 : 2)) return true;  // no live pixel at all: keep one tile
  const int64_t j0 = g * kLiveGroup, j1 = min(j0 + kLiveGroup, K);
  for (int iy = (int)(j0 / N); (int64_t)iy * N < j1; ++iy) {  // the one or two (narrow scenes: more) rows it spans
    int a, b;
    live_row(N, R2, iy, a, b);
    if (a < b && (int64_t)iy * N + a < j1 && (int64_t)iy * N + b > j0) return true;
  }
  return false;
}

// One CTA walks the groups, 1024 at a time.  Within a run of live groups every
// second one starts a k-tile; the group after a run of odd length falls inside
// the run's last tile.
__global__ void __launch_bounds__(1024) ktile_table_kernel(int N, int64_t K, long long R2, int *ktab, int k_tiles,
                                                           int *dead, int64_t dead_groups) {
  __shared__ int sh[32];
  __shared__ bool flag[1024];
  bool carry = false;  // the last group of the block before is live
  const int64_t groups = (K + kLiveGroup - 1) / kLiveGroup;
  int run_carry = -1, tile_carry = 0, dead_carry = 0;
  for (int64_t base = 0; base < groups; base += blockDim.x) {
    const int64_t g = base + threadIdx.x;
    const bool live = group_live(N, K, R2, g, groups);
    flag[threadIdx.x] = live;
    __syncthreads();
    const bool before = threadIdx.x ? flag[threadIdx.x - 1] : carry;
    carry = flag[blockDim.x - 1];
    int total;
    const int start = max(run_carry, scan_max(live && !before ? (int)g : -1, sh, total));  // of g's, or the last, run
    run_carry = max(run_carry, total);
    const bool tile = live && (((int)g - start) & 1) == 0;
    const bool covered = live || (before && (((int)g - 1 - start) & 1) == 0);
    const int t = tile_carry + scan_sum(tile ? 1 : 0, sh, total);
    if (tile && t < k_tiles) ktab[t] = (int)(g * kLiveGroup);
    tile_carry += total;
    const int d = dead_carry + scan_sum(g < groups && !covered ? 1 : 0, sh, total);
    if (g < groups && !covered && d < dead_groups) dead[d] = (int)g;
    dead_carry += total;
  }
}

// FP32 storage: list[0 .. L) the live columns, list[L .. K) the others.  A CTA
// takes kListRows scene rows; the rows before them are counted by all threads.
constexpr int kListRows = 8;
__global__ void __launch_bounds__(256) column_list_kernel(int N, long long R2, int64_t live_cols, int *list) {
  __shared__ int before[8];
  const int y0 = blockIdx.x * kListRows;
  int a, b, n = 0;
  for (int iy = threadIdx.x; iy < y0; iy += blockDim.x) {
    live_row(N, R2, iy, a, b);
    n += b - a;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if ((threadIdx.x & 31) == 0) before[threadIdx.x >> 5] = n;
  __syncthreads();
  int64_t at = 0;
  for (int w = 0; w < 8; ++w) at += before[w];
  for (int iy = y0; iy < y0 + kListRows && iy < N; ++iy) {
    live_row(N, R2, iy, a, b);
    const int64_t row = (int64_t)iy * N;
    int *dead = list + live_cols + (row - at);  // the row's others follow the others of the rows before
    for (int ix = threadIdx.x; ix < N; ix += blockDim.x) {
      if (ix >= a && ix < b)
        list[at + ix - a] = (int)(row + ix);
      else
        dead[ix < a ? ix : ix - (b - a)] = (int)(row + ix);
    }
    at += b - a;
  }
}

}  // namespace

void psfsim_live_count(psfsim_plan *h) {
  const bool split = h->storage == PSFSIM_SPLIT_BF16 || h->storage == PSFSIM_BF16;
  h->live = false;
  h->k_tiles = (int)(h->ld / 64);
  h->dead_groups = 0;
  h->live_cols = psfsim_cols(h);
  if (h->N < 1 || h->quadrant) return;
  const long long R2 = live_r2(h->radii[h->n_r - 1], h->S);
  if (!split) {
    int64_t cols = 0;
    for (int iy = 0; iy < h->N; ++iy) {
      int a, b;
      live_row(h->N, R2, iy, a, b);
      cols += b - a;
    }
    h->live = cols < h->K;
    h->live_cols = cols;
    return;
  }
  const int64_t groups = (h->K + kLiveGroup - 1) / kLiveGroup;
  int64_t runs = 0, tiles = 0, covered = 0, run0 = -1, run1 = -1;  // current run of live groups [run0, run1)
  auto close = [&] {
    if (run0 < 0) return;
    const int64_t t = (run1 - run0 + 1) / 2, end = run0 + 2 * t;
    tiles += t;
    ++runs;
    covered += (end < groups ? end : groups) - run0;
  };
  for (int iy = 0; iy < h->N; ++iy) {
    int a, b;
    live_row(h->N, R2, iy, a, b);
    if (a == b) continue;
    const int64_t g0 = ((int64_t)iy * h->N + a) / kLiveGroup, g1 = ((int64_t)iy * h->N + b - 1) / kLiveGroup + 1;
    if (run0 >= 0 && g0 <= run1) {
      run1 = g1;
      continue;
    }
    close();
    run0 = g0;
    run1 = g1;
  }
  if (run0 < 0) {
    run0 = 0;
    run1 = 1;
  }
  close();
  if (covered >= groups) return;  // nothing to skip
  h->live = true;
  h->k_tiles = (int)tiles;
  h->short_runs = 2 * tiles <= 5 * runs;
  h->dead_groups = groups - covered;
}

cudaError_t psfsim_launch_live_table(psfsim_plan *h, cudaStream_t st) {
  if (!h->live) return cudaSuccess;
  int *tab = reinterpret_cast<int *>(h->ws + h->order_off);
  if (h->storage == PSFSIM_FP32) {
    column_list_kernel<<<(unsigned)((h->N + kListRows - 1) / kListRows), 256, 0, st>>>(
        h->N, live_r2(h->radii[h->n_r - 1], h->S), h->live_cols, tab);
    return cudaGetLastError();
  }
  ktile_table_kernel<<<1, 1024, 0, st>>>(h->N, h->K, live_r2(h->radii[h->n_r - 1], h->S), tab, h->k_tiles,
                                         tab + h->k_tiles, h->dead_groups);
  return cudaGetLastError();
}
