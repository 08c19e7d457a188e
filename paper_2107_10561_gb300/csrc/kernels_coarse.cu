// Direct coarse solve of Algorithm 1 (d_1 = J_1^{-1} r_1, or J_1^{-T} r_1 in the adjoint V-cycle) through
// the twisted block factors of J_1 in x-slab order (kernels_factor.cu), for coarse levels too large for
// the dense explicit inverse to pay (3D: 18,000 DoFs, 2.6 GB as a dense inverse).
//
// In slab order J_1 is block tridiagonal. Its slabs are eliminated from both ends towards the twist
// slab t; with Sinv_b the inverse Schur complements, the solve of J_1 x = r is
//   z_b = Sinv_b r_b                                         (all slabs at once)
//   y_b = z_b - Lo_b y_{b-1},  b = 1 .. t-1   together with  y_b = z_b - Up_b y_{b+1},  b = nx-2 .. t+1
//   x_t = z_t - Lo_t y_{t-1} - Up_t y_{t+1}
//   x_b = y_b - Bk_b x_{b+1},  b = t-1 .. 0   together with  x_b = y_b - Bk_b x_{b-1},  b = t+1 .. nx-1
// (Lo_b = Sinv_b A_{b,b-1}, Up_b = Sinv_b A_{b,b+1}, Bk_b the back-substitution block). J_1^T has its
// own blocks of the same shapes (kinds 4..7), so both directions run the same kernel. The dependent steps
// (about nx, each working on the two slabs at the ends of the chains) run inside one cooperative kernel
// with a grid-wide barrier between steps; before a step's barrier every thread requests into L2 a share of
// the blocks the next step reads.
//
// The products run on the tensor cores in FP64 accuracy (digits.h): the blocks are kept as base-256 digits
// (eight bytes per value, a power of two per row and 96 columns), in fragment order, 16 x 16 values in 2 KB;
// the vector is cut into digits where it is used, scaled per 96 entries.
//   - One vector: a CTA takes 16 rows, its warps 96 columns each; M = 16 rows, N = 8 the digits of the
//     vector, so all 64 digit pairs of a product are formed; the warps' sums are added in a fixed order.
//   - 32 interleaved columns: a CTA takes 64 rows and 96 columns of a block, a warp 16 rows x 16 of the
//     vectors, the 36 digit pairs above 2^-62; the sums of the column groups are added in a fixed order
//     behind a second barrier.
// Measured on the 18,000-DoF 3D coarse level (16 slabs): 213 us per solve, against 290 us with FP64 dot
// products and 560 us for the explicit inverse; 32 columns 0.90 ms against 6.0 ms. What bounds it is the
// chain of about 18 steps of 10 us: a barrier, the values' way from L2, the vector's digits, the sums'
// joining. Looking the blocks up once and joining in integers took 222 to 213 us; requesting the next
// step's blocks before instead of after a step's products: 218 us.
#include <cooperative_groups.h>

#include "digits.h"
#include "internal.h"

namespace cg = cooperative_groups;

namespace stm {
namespace {

constexpr int kChunk = 96, kChunkK = kChunk / 16;  // columns that share a power of two

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

struct SlabView {
  int nx, t;
  long long n;
  const long long* off;   // [nx + 1] first permuted row of every slab
  const long long* wpos;  // [8][nx] block offsets in words, in tiles of 16 x 16 (-1: absent)
  const long long* epos;  // [8][nx] offsets in exps
  const int* perm;        // [n] permuted position of every row of J_1
  long long block, dR;    // unknowns of a time node, the first pressure among them
  double scale;           // the factors are those of J_1 with pressure rows and columns scaled
  const uint4* words;
  const int* exps;        // per block [row tiles x 16][column groups]
};

enum { K_INV = 0, K_LO = 1, K_UP = 2, K_BACK = 3 };

// One product of a step: rows of slab b, y_b (-)= M x_c (M: nb x nc).
struct Task {
  const uint4* w = nullptr;
  const int* e = nullptr;
  long long r0 = 0, c0 = 0;
  int nb = 0, nc = 0, tiles = 0, chunks = 0;
};

__device__ __forceinline__ double scaled(const SlabView& S, long long row, double v) {
  return row % S.block >= S.dR ? v * S.scale : v;
}
__host__ __device__ __forceinline__ int groups_of(long long n, int g) { return (int)((n + g - 1) / g); }

__device__ __forceinline__ Task make_task(const SlabView& S, int kind, int b, int c) {
  Task k;
  k.w = S.words + S.wpos[kind * S.nx + b] * 128;
  k.e = S.exps + S.epos[kind * S.nx + b];
  k.r0 = S.off[b];
  k.nb = (int)(S.off[b + 1] - k.r0);
  k.c0 = S.off[c];
  k.nc = (int)(S.off[c + 1] - k.c0);
  k.tiles = groups_of(k.nb, 16);
  k.chunks = groups_of(k.nc, kChunk);
  return k;
}

// Every thread of the grid requests a share of the 128-byte lines of the task's block into L2.
__device__ __forceinline__ void task_prefetch(const Task& T, long long gt, long long nt) {
  if (!T.w) return;
  const char* p = reinterpret_cast<const char*>(T.w);
  const long long bytes = (long long)T.tiles * T.chunks * kChunkK * 2048;
  for (long long o = gt * 128; o < bytes; o += nt * 128) prefetch_l2(p + o);
}

// Chain tasks of step s (1-based) of the forward elimination, of the twist slab and of the back substitution.
__device__ __forceinline__ void chain_tasks(const SlabView& S, int base, int s, Task& A, Task& B) {
  const int t = S.t, nx = S.nx;
  A = s <= t - 1 ? make_task(S, base + K_LO, s, s - 1) : Task();
  B = nx - 1 - s >= t + 1 ? make_task(S, base + K_UP, nx - 1 - s, nx - s) : Task();
}
__device__ __forceinline__ void twist_tasks(const SlabView& S, int base, Task& A, Task& B) {
  const int t = S.t, nx = S.nx;
  A = t >= 1 ? make_task(S, base + K_LO, t, t - 1) : Task();
  B = t + 1 < nx ? make_task(S, base + K_UP, t, t + 1) : Task();
}
__device__ __forceinline__ void back_tasks(const SlabView& S, int base, int s, Task& A, Task& B) {
  const int t = S.t, nx = S.nx;
  A = t - s >= 0 ? make_task(S, base + K_BACK, t - s, t - s + 1) : Task();
  B = t + s <= nx - 1 ? make_task(S, base + K_BACK, t + s, t + s - 1) : Task();
}
// The two tasks of up to kSteps steps, looked up once by one thread: a step then starts without three
// dependent loads.
constexpr int kSteps = 32;
// Step p of a solve: 1 .. nchain the chains, then the twist, then the back substitution
__device__ __forceinline__ void step_tasks(const SlabView& S, int base, int p, int nchain, Task& A, Task& B) {
  if (p <= nchain) chain_tasks(S, base, p, A, B);
  else if (p == nchain + 1) twist_tasks(S, base, A, B);
  else back_tasks(S, base, p - nchain - 1, A, B);
}

// Fills the table with the tasks of steps p0 .. p0 + kSteps - 1; every thread of the CTA calls.
__device__ __forceinline__ void fill_tasks(const SlabView& S, int base, int p0, int last, int nchain, Task (*tab)[2]) {
  __syncthreads();
  for (int i = threadIdx.x; i < kSteps; i += blockDim.x)
    if (p0 + i <= last) step_tasks(S, base, p0 + i, nchain, tab[i][0], tab[i][1]);
  __syncthreads();
}

constexpr int kWarps1 = 12;

// Rows 16 tile .. 16 tile + 15 of M x (x: slab part of a vector), summed over the CTA's warps; threads 0 .. 15
// return one row's sum.
__device__ __forceinline__ double tile_dot(const Task& T, int tile, const double* x, __half (*xs)[kChunk * 8],
                                           double (*red)[16]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = lane >> 2, q = lane & 3;
  double tot0 = 0.0, tot1 = 0.0;
  for (int c = warp; c < T.chunks; c += kWarps1) {
    const uint4* w = T.w + ((long long)tile * T.chunks + c) * (kChunkK * 128) + lane;
    uint4 a[kChunkK][4];  // all of the warp's values are on their way while x is cut
#pragma unroll
    for (int kk = 0; kk < kChunkK; ++kk)
#pragma unroll
      for (int k = 0; k < 4; ++k) a[kk][k] = __ldg(w + kk * 128 + 32 * k);
    const int er0 = T.e[(long long)(16 * tile + n) * T.chunks + c], er8 = T.e[(long long)(16 * tile + n + 8) * T.chunks + c];
    // this group of x: one power of two, digits as [pair][digit] of two FP16
    double v[kChunk / 32];
    int e = kExpZero;
#pragma unroll
    for (int j = 0; j < kChunk / 32; ++j) {
      const int k = c * kChunk + 32 * j + lane;
      v[j] = k < T.nc ? x[k] : 0.0;
      e = max(e, exp_above(v[j]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kChunk / 32; ++j) {
      const unsigned long long p = digits_of(e > 1024 ? 0.0 : v[j], e);
      const int k = 32 * j + lane;
#pragma unroll
      for (int d = 0; d < kDig; ++d) xs[warp][((k >> 1) * 8 + d) * 2 + (k & 1)] = digit_half(p, d);
    }
    __syncwarp();
    // a byte in the low half of an FP16 number is that integer times 2^-24; the bytes carry the bias 128,
    // which the sums of x's digits (A = ones) take off again
    float acc[kDig + 1][4];
#pragma unroll
    for (int d = 0; d <= kDig; ++d)
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[d][m] = 0.f;
    const uint32_t* xw = reinterpret_cast<const uint32_t*>(xs[warp]);
#pragma unroll
    for (int kk = 0; kk < kChunkK; ++kk) {
      const uint32_t b0 = xw[(8 * kk + q) * 8 + n], b1 = xw[(8 * kk + 4 + q) * 8 + n];
      const uint32_t ww[4][4] = {{a[kk][0].x, a[kk][0].y, a[kk][0].z, a[kk][0].w}, {a[kk][1].x, a[kk][1].y, a[kk][1].z, a[kk][1].w},
                                 {a[kk][2].x, a[kk][2].y, a[kk][2].z, a[kk][2].w}, {a[kk][3].x, a[kk][3].y, a[kk][3].z, a[kk][3].w}};
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        mma_f16(acc[d], ww[0][d] & 0x00FF00FFu, ww[1][d] & 0x00FF00FFu, ww[2][d] & 0x00FF00FFu, ww[3][d] & 0x00FF00FFu, b0, b1);
        mma_f16(acc[d + 4], __byte_perm(ww[0][d], 0u, 0x4341), __byte_perm(ww[1][d], 0u, 0x4341),
                __byte_perm(ww[2][d], 0u, 0x4341), __byte_perm(ww[3][d], 0u, 0x4341), b0, b1);
      }
      mma_f16(acc[kDig], 0x00010001u, 0x00010001u, 0x00010001u, 0x00010001u, b0, b1);
    }
    // acc[d][m]: row n (m < 2) or n + 8, digit 2 q + (m & 1) of x; 255 x 128 x 96 terms stay below 2^24
    const int x0 = __float2int_rn(acc[kDig][0] * 16777216.f) * 128, x1 = __float2int_rn(acc[kDig][1] * 16777216.f) * 128;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      long long hi = 0, lo = 0;
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const int u0 = __float2int_rn(acc[d][2 * h] * 16777216.f) - x0, u1 = __float2int_rn(acc[d][2 * h + 1] * 16777216.f) - x1;
        const int v0 = __float2int_rn(acc[d + 4][2 * h] * 16777216.f) - x0, v1 = __float2int_rn(acc[d + 4][2 * h + 1] * 16777216.f) - x1;
        hi += ((long long)u0 * 256 + u1) * (1 << (24 - 8 * d));
        lo += ((long long)v0 * 256 + v1) * (1 << (24 - 8 * d));
      }
      const int er = h ? er8 : er0;
      double s = 0.0;
      if (e > 1024 || er > 1024) s = __hiloint2double(0x7FF80000, 0);  // a vector or block that is not finite
      else if (e != kExpZero && er != kExpZero) s = join_pow2(hi, lo, er + e - 124 + 48 - 16 * q);
      (h ? tot1 : tot0) += s;
    }
  }
  tot0 += __shfl_xor_sync(0xffffffffu, tot0, 1);
  tot1 += __shfl_xor_sync(0xffffffffu, tot1, 1);
  tot0 += __shfl_xor_sync(0xffffffffu, tot0, 2);
  tot1 += __shfl_xor_sync(0xffffffffu, tot1, 2);
  __syncthreads();  // the sums of the tile before are read
  if (q == 0) {
    red[warp][n] = tot0;
    red[warp][n + 8] = tot1;
  }
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 16) {
    double r[kWarps1];
#pragma unroll
    for (int k = 0; k < kWarps1; ++k) r[k] = red[k][threadIdx.x];
#pragma unroll
    for (int o = kWarps1 / 2; o >= 3; o /= 2)
#pragma unroll
      for (int k = 0; k < o; ++k) r[k] += r[k + o];
    s = (r[0] + r[1]) + r[2];
  }
  return s;
}

__global__ void __launch_bounds__(32 * kWarps1) k_coarse_slab(SlabView S, const double* __restrict__ r,
                                                              double* __restrict__ d, double* u, double* v,
                                                              int transpose) {
  cg::grid_group grid = cg::this_grid();
  __shared__ __half xs[kWarps1][kChunk * 8];
  __shared__ double red[kWarps1][16];
  __shared__ Task tab[kSteps][2];
  const long long gt = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nt = (long long)gridDim.x * blockDim.x;
  const int nx = S.nx, t = S.t;
  const int base = transpose ? 4 : 0;
  const int nchain = max(max(t - 1, nx - 2 - t), 0), nback = max(t, nx - 1 - t);
  // gather into slab order
  for (long long e = gt; e < S.n; e += nt) u[S.perm[e]] = scaled(S, e, r[e]);
  grid.sync();
  // z_b = Sinv_b r_b for every slab
  int first = 0;
  for (int b = 0; b < nx; ++b) {
    const Task T = make_task(S, base + K_INV, b, b);
    int tile = (int)blockIdx.x - first % (int)gridDim.x;  // tiles of all slabs are dealt out in turn
    if (tile < 0) tile += gridDim.x;
    for (; tile < T.tiles; tile += gridDim.x) {
      const double s = tile_dot(T, tile, u + T.c0, xs, red);
      const int row = 16 * tile + threadIdx.x;
      if (threadIdx.x < 16 && row < T.nb) v[T.r0 + row] = s;
    }
    first += T.tiles;
  }
  const int last = nchain + 1 + nback;
  for (int p = 1; p <= last; ++p) {
    if ((p - 1) % kSteps == 0) {
      fill_tasks(S, base, p, last, nchain, tab);
      task_prefetch(tab[0][0], gt, nt);
      task_prefetch(tab[0][1], gt, nt);
    }
    const Task &A = tab[(p - 1) % kSteps][0], &B = tab[(p - 1) % kSteps][1];
    grid.sync();
    const bool twist = p == nchain + 1;
    const int tiles = twist ? max(A.tiles, B.tiles) : A.tiles + B.tiles;
    for (int i = blockIdx.x; i < tiles; i += gridDim.x) {
      const bool second = !twist && i >= A.tiles;
      const Task& T = second ? B : A;
      const int tile = second ? i - A.tiles : i;
      double s = 0.0;
      if (T.w) s = tile_dot(T, tile, v + T.c0, xs, red);
      if (twist && B.w) s += tile_dot(B, tile, v + B.c0, xs, red);
      const Task& Y = T.w ? T : B;
      const int row = 16 * tile + threadIdx.x;
      if (threadIdx.x < 16 && row < Y.nb) v[Y.r0 + row] -= s;
    }
    if (p < last && p % kSteps) {
      task_prefetch(tab[p % kSteps][0], gt, nt);
      task_prefetch(tab[p % kSteps][1], gt, nt);
    }
  }
  grid.sync();
  // back to the row order of J_1
  for (long long e = gt; e < S.n; e += nt) d[e] = scaled(S, e, v[S.perm[e]]);
}

// --- 32 interleaved columns ---------------------------------------------------------------------------
constexpr int NR = 32;

// Partial sums of rows 64 g .. 64 g + 63 of M X over column group c, into part[row][32].
__device__ __forceinline__ void block_part(const Task& T, int g, int c, const double* X, double* part, uint4 (*xs)[NR],
                                           int (*ex)[NR]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = lane >> 2, q = lane & 3;
  constexpr int RPW = kChunk / 8;  // rows of X per warp
  const int tile = 4 * g + (warp & 3), cb = (warp >> 2) * 16;
  // all of the warp's values are on their way while X is cut
  const uint4* w = T.w + ((long long)min(tile, T.tiles - 1) * T.chunks + c) * (kChunkK * 128) + lane;
  uint4 a[kChunkK][4];
#pragma unroll
  for (int kk = 0; kk < kChunkK; ++kk)
#pragma unroll
    for (int k = 0; k < 4; ++k) a[kk][k] = __ldg(w + kk * 128 + 32 * k);
  double v[RPW];
  int e = kExpZero;
#pragma unroll
  for (int j = 0; j < RPW; ++j) {
    const int k = c * kChunk + warp * RPW + j;
    v[j] = k < T.nc ? X[(long long)k * NR + lane] : 0.0;
    e = max(e, exp_above(v[j]));
  }
  __syncthreads();  // the operands of the unit before are read
  ex[warp][lane] = e;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k) e = max(e, ex[k][lane]);
  // pair p of column col sits at (col + 2 p) mod 32: eight lanes of a read then meet eight banks
#pragma unroll
  for (int j = 0; j < RPW; j += 2) {
    const int p = (warp * RPW + j) >> 1;
    xs[p][(lane + 2 * p) & 31] = words_of(digits_of(e > 1024 ? 0.0 : v[j], e), digits_of(e > 1024 ? 0.0 : v[j + 1], e));
  }
  __syncthreads();
  if (tile < T.tiles) {
    float acc[kDig][8];
#pragma unroll
    for (int d = 0; d < kDig; ++d)
#pragma unroll
      for (int m = 0; m < 8; ++m) acc[d][m] = 0.f;
#pragma unroll
    for (int kk = 0; kk < kChunkK; ++kk) {
      const uint32_t ww[4][4] = {{a[kk][0].x, a[kk][0].y, a[kk][0].z, a[kk][0].w}, {a[kk][1].x, a[kk][1].y, a[kk][1].z, a[kk][1].w},
                                 {a[kk][2].x, a[kk][2].y, a[kk][2].z, a[kk][2].w}, {a[kk][3].x, a[kk][3].y, a[kk][3].z, a[kk][3].w}};
      const int p0 = 8 * kk + q, p1 = p0 + 4;
      uint32_t b[2][kDig][2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int col = cb + 8 * h + n;
        const uint4 x0 = xs[p0][(col + 2 * p0) & 31], x1 = xs[p1][(col + 2 * p1) & 31];
        const uint32_t y0[4] = {x0.x, x0.y, x0.z, x0.w}, y1[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
        for (int d = 0; d < kDig; ++d) {
          b[h][d][0] = digit_pair(y0[d & 3], d >= 4);
          b[h][d][1] = digit_pair(y1[d & 3], d >= 4);
        }
      }
#pragma unroll
      for (int d = 0; d < kDig; ++d) {
        uint32_t f[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) f[k] = digit_pair(ww[k][d & 3], d >= 4);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int o = 0; d + o < kDig; ++o) mma_f16(acc[d + o] + 4 * h, f[0], f[1], f[2], f[3], b[h][o][0], b[h][o][1]);
      }
    }
    // 8 pairs x 96 terms x 2^14 < 2^24
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int row = 16 * tile + n + ((m & 2) ? 8 : 0), col = cb + (m >> 2) * 8 + 2 * q + (m & 1);
      long long hi = 0, lo = 0;
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        hi += (long long)__float2int_rn(acc[d][m]) * (1 << (24 - 8 * d));
        lo += (long long)__float2int_rn(acc[d + 4][m]) * (1 << (24 - 8 * d));
      }
      const int er = T.e[(long long)row * T.chunks + c], ec = __shfl_sync(0xffffffffu, e, col);
      double s = 0.0;
      if (er > 1024 || ec > 1024) s = __hiloint2double(0x7FF80000, 0);
      else if (er != kExpZero && ec != kExpZero)
        s = join_pow2(hi, lo, er + ec - 124 + 56);
      part[(long long)row * NR + col] = s;
    }
  }
}

constexpr int kBatch = 8;  // slabs whose inverses are applied between two barriers

// part: [column groups][rows][32] per task: the two tasks of a step, or kBatch slabs' inverses, at a time
__global__ void __launch_bounds__(256, 1) k_coarse_slab_multi(SlabView S, const double* __restrict__ R,
                                                              double* __restrict__ Dm, double* u, double* v,
                                                              double* part, long long stride) {
  cg::grid_group grid = cg::this_grid();
  __shared__ uint4 xs[kChunk / 2][NR];
  __shared__ int ex[8][NR];
  const long long gt = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nt = (long long)gridDim.x * blockDim.x;
  const int nx = S.nx, t = S.t;
  const int nchain = max(max(t - 1, nx - 2 - t), 0), nback = max(t, nx - 1 - t);
  for (long long e = gt; e < S.n * NR; e += nt) {
    const long long i = e / NR;
    u[(long long)S.perm[i] * NR + (e - i * NR)] = scaled(S, i, R[e]);
  }
  grid.sync();
  auto units = [](const Task& T) { return groups_of(T.tiles, 4) * T.chunks; };
  auto product = [&](const Task& T, int k, const double* X, double* out) {
    const int c = k % T.chunks;
    block_part(T, k / T.chunks, c, X + T.c0 * NR, out + (long long)c * T.tiles * 16 * NR, xs, ex);
  };
  auto sum = [&](const Task& T, const double* in, long long e) {
    double s = 0.0;
    for (int c = 0; c < T.chunks; ++c) s += in[(long long)c * T.tiles * 16 * NR + e];
    return s;
  };
  for (int b0 = 0; b0 < nx; b0 += kBatch) {
    int first = 0;  // units of all slabs of the batch are dealt out in turn
    for (int b = b0; b < min(nx, b0 + kBatch); ++b) {
      const Task T = make_task(S, K_INV, b, b);
      const int m = units(T);
      int k = (int)blockIdx.x - first % (int)gridDim.x;
      if (k < 0) k += gridDim.x;
      for (; k < m; k += gridDim.x) product(T, k, u, part + (b - b0) * stride);
      first += m;
    }
    grid.sync();
    for (int b = b0; b < min(nx, b0 + kBatch); ++b) {
      const Task T = make_task(S, K_INV, b, b);
      for (long long e = gt; e < (long long)T.nb * NR; e += nt) v[T.r0 * NR + e] = sum(T, part + (b - b0) * stride, e);
    }
    grid.sync();
  }
  for (int p = 1; p <= nchain + 1 + nback; ++p) {
    Task A, B;
    step_tasks(S, 0, p, nchain, A, B);
    const bool joined = p == nchain + 1;  // both tasks end in the twist slab
    const int ma = units(A), mb = units(B);
    for (int k = blockIdx.x; k < ma + mb; k += gridDim.x)
      if (k < ma) product(A, k, v, part);
      else product(B, k - ma, v, part + stride);
    if (p < nchain + 1 + nback) {
      Task nA, nB;
      step_tasks(S, 0, p + 1, nchain, nA, nB);
      task_prefetch(nA, gt, nt);
      task_prefetch(nB, gt, nt);
    }
    grid.sync();
    const long long na = (long long)A.nb * NR, nb = (long long)B.nb * NR;
    for (long long e = gt; e < (joined ? max(na, nb) : na + nb); e += nt) {
      const long long f = joined ? e : e - na;
      double s = 0.0;
      if (e < na) s += sum(A, part, e);
      if (f >= 0 && f < nb) s += sum(B, part + stride, f);
      v[e < na ? A.r0 * NR + e : B.r0 * NR + f] -= s;
    }
    grid.sync();
  }
  for (long long e = gt; e < S.n * NR; e += nt) {
    const long long i = e / NR;
    Dm[e] = scaled(S, i, v[(long long)S.perm[i] * NR + (e - i * NR)]);
  }
}

// Words and exponents of one block (rows x cols, row-major): one warp per row and group of 96 columns.
__global__ void __launch_bounds__(256) k_block_words(const double* __restrict__ M, int rows, int cols,
                                                     uint4* __restrict__ words, int* __restrict__ exps) {
  const int lane = threadIdx.x & 31;
  const int tiles = groups_of(rows, 16), chunks = groups_of(cols, kChunk);
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < (long long)tiles * 16 * chunks; i += nwarps) {
    const int row = (int)(i / chunks), c = (int)(i - (long long)row * chunks);
    const double* a = M + (long long)row * cols + (long long)c * kChunk;
    const int len = row < rows ? min(kChunk, cols - c * kChunk) : 0;
    // lane l < 16 x 3: pairs l, l + 32 of the 48
    double v[2][2];
    int e = kExpZero;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int j = 2 * (lane + 32 * h) + k;
        v[h][k] = j < len ? a[j] : 0.0;
        e = max(e, exp_above(v[h][k]));
      }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) exps[i] = e;
    uint4* w = words + ((long long)(row >> 4) * chunks + c) * (kChunkK * 128) + ((row >> 3) & 1) * 32 + (row & 7) * 4;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int p = lane + 32 * h;
      if (p < kChunk / 2)
        w[(p >> 3) * 128 + ((p >> 2) & 1) * 64 + (p & 3)] =
            words_of(digits_of(e > 1024 ? 0.0 : v[h][0], e), digits_of(e > 1024 ? 0.0 : v[h][1], e));
    }
  }
}

SlabView view_of(const Hierarchy& H) {
  SlabView S;
  S.nx = H.cs_nx;
  S.t = H.cs_t;
  S.n = H.N0;
  S.off = H.cs_off;
  S.wpos = H.cs_wpos;
  S.epos = H.cs_wpos + 8LL * H.cs_nx;
  S.perm = H.cs_perm;
  S.block = H.L[0].block;
  S.dR = (long long)H.L[0].dim * H.L[0].R;
  S.scale = H.cs_scale;
  S.words = (const uint4*)H.cs_words;
  S.exps = H.cs_exps;
  return S;
}

template <typename F, typename... Args>
stm_status launch_cooperative(F kernel, int threads, int per_sm, cudaStream_t s, Args... args) {
  int occ = 0;
  STM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, 0));
  if (occ < 1) {
    set_error("coarse slab solve: kernel does not fit on an SM");
    return STM_ERR_CUDA;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(std::min(occ, per_sm) * sm_count()));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  STM_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
  note_launch();
  return STM_OK;
}

}  // namespace

// The digits of the slab factors in cs_store (after each factorisation). rows: of every slab; cpos: [8][nx]
// block offsets in cs_store (-1: absent).
stm_status coarse_slab_words(Hierarchy& H, const std::vector<long long>& off, const std::vector<long long>& cpos,
                             cudaStream_t s) {
  const int nx = H.cs_nx, t = H.cs_t;
  auto rows = [&](int b) { return (int)(off[b + 1] - off[b]); };
  auto cols = [&](int kind, int b) {
    switch (kind & 3) {
      case K_INV: return rows(b);
      case K_LO: return rows(b - 1);
      case K_UP: return rows(b + 1);
      default: return b < t ? rows(b + 1) : rows(b - 1);
    }
  };
  std::vector<long long> pos(16 * (size_t)nx, -1);
  long long tiles = 0, ne = 0;
  for (int kind = 0; kind < 8; ++kind)
    for (int b = 0; b < nx; ++b)
      if (cpos[kind * nx + b] >= 0) {
        const long long rt = groups_of(rows(b), 16), ch = groups_of(cols(kind, b), kChunk);
        pos[kind * nx + b] = tiles;
        pos[(8 + kind) * nx + b] = ne;
        tiles += rt * ch * kChunkK;
        ne += rt * 16 * ch;
      }
  if ((!H.cs_words && cudaMalloc(&H.cs_words, 2048 * (size_t)tiles)) ||
      (!H.cs_exps && cudaMalloc((void**)&H.cs_exps, sizeof(int) * (size_t)ne)) ||
      (!H.cs_wpos && cudaMalloc((void**)&H.cs_wpos, sizeof(long long) * 16 * nx))) {
    cudaGetLastError();
    set_error("coarse factorisation: out of device memory");
    return STM_ERR_OOM;
  }
  for (int kind = 0; kind < 8; ++kind)
    for (int b = 0; b < nx; ++b)
      if (cpos[kind * nx + b] >= 0) {
        const long long warps = (long long)groups_of(rows(b), 16) * 16 * groups_of(cols(kind, b), kChunk);
        k_block_words<<<(int)std::min<long long>((warps + 7) / 8, sm_count() * 8LL), 256, 0, s>>>(
            H.cs_store + cpos[kind * nx + b], rows(b), cols(kind, b),
            (uint4*)H.cs_words + pos[kind * nx + b] * 128, H.cs_exps + pos[(8 + kind) * nx + b]);
        note_launch();
      }
  STM_CUDA(cudaGetLastError());
  // pos is pageable: the copy returns only when it has been read
  STM_CUDA(cudaMemcpyAsync(H.cs_wpos, pos.data(), sizeof(long long) * pos.size(), cudaMemcpyHostToDevice, s));
  return STM_OK;
}

stm_status coarse_slab_apply(Hierarchy& H, const double* r, double* d, int transpose, cudaStream_t s) {
  return launch_cooperative(k_coarse_slab, 32 * kWarps1, 2, s, view_of(H), r, d, H.cs_u, H.cs_v, transpose);
}

stm_status coarse_slab_apply_multi(Hierarchy& H, const double* R, double* D, cudaStream_t s) {
  const long long stride = (long long)groups_of(H.cs_maxnb, kChunk) * groups_of(H.cs_maxnb, 16) * 16 * NR;
  if (!H.cs_mu || !H.cs_mv) {
    cudaFree(H.cs_mu);
    H.cs_mu = nullptr;
    STM_TRY(device_alloc(H, &H.cs_mu, sizeof(double) * 32 * (size_t)H.N0));
    STM_TRY(device_alloc(H, &H.cs_mv, sizeof(double) * 32 * (size_t)H.N0));
  }
  if (!H.cs_part) STM_TRY(device_alloc(H, &H.cs_part, sizeof(double) * std::max(2, std::min(kBatch, H.cs_nx)) * (size_t)stride));
  return launch_cooperative(k_coarse_slab_multi, 256, 1, s, view_of(H), R, D, H.cs_mu, H.cs_mv, H.cs_part, stride);
}

}  // namespace stm
