// 32-column product with the slab Jacobian J_g or its transpose whose velocity rows run on the tensor cores:
// Y = J X or Y = B - J X in FP64 accuracy.
//
// 32 columns make 32 FMAs per value of J, and at 2 FP64 FMAs per clock and SM those take 40 times as long
// as the bytes take from HBM. Here the values of J and the entries of X are 63-bit integers (one power of
// two per row of J, and one per node and column of X) cut into eight balanced base-256 digits, whose
// products add up exactly in the FP32 accumulators of FP16 tensor instructions (digits.h). The 36 digit
// pairs (s, t) with s + t <= 7 are accumulated per weight and joined in 64-bit integers every 128
// positions; the rounding is that of the digits left out and of one conversion per result.
//   - One warp per node and 16 columns. M = 16 of an MMA holds the columns, N = 8 the K d <= 6 rows of the
//     node, K = 16 consecutive positions: the entries (time, component) of each neighbour node in pairs,
//     then the pressures of the node's cells once per time node (a row multiplies those of its own time
//     node, the others are zero).
//   - Both operands are stored as the fragments want them: a lane's two neighbouring positions as four words
//     [u_i, u_{i+4}, v_i, v_{i+4}] of biased bytes; a byte permute and an FP16 subtraction give a register
//     of an operand. X is brought into this form by a pass of its own, per node and column scaled to a
//     common base (a multiple of eight bits); a node takes the largest base around it per column, and
//     neighbours with a smaller one are shifted by whole digits, so rows far from the largest entries of a
//     column lose nothing. Nodes and cells have bases of their own, and their sums are joined in FP64.
//   - Rows of the pressure equations (3 % of the values) stay on the FP64 pipe, interleaved.
//   - What bounds it (127,920 unknowns, 3D dG(1)): 340 warp instructions per 16 positions x 6 rows x 16 columns
//     (36 MMAs, 96 to form the digits, a shift around nodes where magnitudes cross a digit), issued at 40 %
//     with sixteen warps per SM; the tensor pipe is 31 % busy. With one step's operands loaded ahead and
//     twelve warps it is slower (0.82 against 0.71 ms per product with X's passes); FP64 FMAs took 2.52 ms.
//   - Columns whose neighbourhood holds an infinity or a NaN, and nodes whose rows do, are summed from the
//     CSR values in plain FP64.
#include "digits.h"
#include "internal.h"

namespace stm {
namespace {

constexpr int NR = 32;                   // columns of a multi-vector
constexpr int kZeroBase = -20000;        // base of entries that are all zero
constexpr int kBadBase = 20000;          // base of entries that are not all finite
constexpr int kThreads = 256, kCtas = 2;
constexpr int kDrain = 8;                // steps of 16 positions after which the FP32 sums are joined:
                                         // 8 pairs x 128 positions x 2^14 = 2^24

template <int K, int D>
struct Shape {
  static constexpr int KD = K * D;               // velocity rows of a node
  static constexpr int NP = D + 1, MAXC = 1 << D, MAXN = D == 2 ? 25 : 125, NV = D == 2 ? 9 : 27;
  static constexpr int PAIRS = (KD + 1) / 2;     // position pairs of a neighbour node
  static constexpr int CPAIRS = 2 * K;           // position pairs of a cell: four per time node
  static constexpr int LANES = 4 * KD;           // lanes that hold values of J
  static constexpr int TAB = PAIRS * MAXN + CPAIRS * MAXC + 16;
};

// base g with |v| <= 2^(8 g + 6) for |v| < 2^e
__device__ __forceinline__ int base_of(int e) { return e == kExpZero ? kZeroBase : e > 1024 ? kBadBase : (e + 1) >> 3; }

// words shifted down by sh <= most digits: one digit turns word i into word i - 1, and word 0 into the low
// halves of word 3 under a zero
__device__ __forceinline__ uint4 shift_words(uint4 w, int sh, int most) {
  for (int k = 0; k < most; ++k)
    if (k < sh) {
      const uint32_t z = __byte_perm(w.w, 0x80808080u, 0x2404);
      w.w = w.z;
      w.z = w.y;
      w.y = w.x;
      w.x = z;
    }
  return w;
}
// Words and bases of X: one warp per node or cell, lane = column.
template <int K, int D>
__global__ void __launch_bounds__(256) k_xm_words(const double* __restrict__ X, long long block, int R, int C,
                                                  uint4* __restrict__ xw, short* __restrict__ xb) {
  using S = Shape<K, D>;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < (long long)R + C; e += nwarps) {
    constexpr int MV = 2 * (S::PAIRS > S::CPAIRS ? S::PAIRS : S::CPAIRS);
    double v[MV];
    int em = kExpZero;
    const bool vel = e < R;
#pragma unroll
    for (int k = 0; k < MV; ++k) {
      v[k] = 0.0;
      if (vel && k < S::KD) v[k] = X[((k / D) * block + (long long)(k % D) * R + e) * NR + lane];
      if (!vel && k < 2 * S::CPAIRS && k % 4 < S::NP)
        v[k] = X[((k / 4) * block + (long long)D * R + (e - R) * S::NP + k % 4) * NR + lane];
      em = max(em, exp_above(v[k]));
    }
    const int g = base_of(em);
    xb[e * NR + lane] = (short)g;
    uint4* o = (vel ? xw + e * (S::PAIRS * NR) : xw + (long long)R * (S::PAIRS * NR) + (e - R) * (S::CPAIRS * NR)) + lane;
#pragma unroll
    for (int c = 0; c < MV / 2; ++c)
      if (c < (vel ? S::PAIRS : S::CPAIRS))
        o[c * NR] = words_of(digits_of(g == kBadBase ? 0.0 : v[2 * c], 8 * g + 6),
                             digits_of(g == kBadBase ? 0.0 : v[2 * c + 1], 8 * g + 6));
  }
}

// Around every node: the largest base of its neighbours and of its cells per column, and per 16 columns the
// largest shift that brings one of them to it (127: a base that is not finite). One warp per node, lane =
// column.
template <int K, int D>
__global__ void __launch_bounds__(256) k_xm_bases(const short* __restrict__ xb, const int* __restrict__ nbr_ptr,
                                                  const int* __restrict__ nbr, const int* __restrict__ ncell,
                                                  const int* __restrict__ node_cells, int R, short* __restrict__ nb,
                                                  uchar4* __restrict__ most) {
  using S = Shape<K, D>;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < R; i += nwarps) {
    const int p0 = nbr_ptr[i], nn = nbr_ptr[i + 1] - p0, nc = ncell[i];
    int m[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int cnt = h ? nc : nn;
      int hi = kZeroBase, lo = kBadBase;
      for (int j0 = 0; j0 < cnt; j0 += 8) {
        int g[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          g[j] = kZeroBase;
          if (j0 + j < cnt) {
            const long long at = h ? (long long)R + node_cells[i * S::MAXC + j0 + j] : nbr[p0 + j0 + j];
            g[j] = xb[at * NR + lane];
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          hi = max(hi, g[j]);
          if (g[j] != kZeroBase) lo = min(lo, g[j]);
        }
      }
      nb[(i * 2 + h) * NR + lane] = (short)hi;
      m[h] = hi == kBadBase ? 127 : lo < hi ? min(hi - lo, 8) : 0;
    }
    const unsigned half = 0xFFFFu << (lane & 16);
    const int a = __reduce_max_sync(half, m[0]), b = __reduce_max_sync(half, m[1]);
    const int a1 = __shfl_sync(0xffffffffu, a, 16), b1 = __shfl_sync(0xffffffffu, b, 16);
    if (lane == 0) most[i] = make_uchar4((unsigned char)a, (unsigned char)b, (unsigned char)a1, (unsigned char)b1);
  }
}

// Words of the velocity rows of J in fragment order, and each row's exponent: one warp per node.
template <int K, int D>
__global__ void __launch_bounds__(256) k_j_words(const long long* __restrict__ rowptr, const double* __restrict__ val,
                                                 const int* __restrict__ nbr_ptr, const int* __restrict__ ncell,
                                                 const int* __restrict__ dbase, uint4* __restrict__ jw,
                                                 int* __restrict__ jexp, long long block, int R) {
  using S = Shape<K, D>;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < R; i += nwarps) {
    const int nn = nbr_ptr[i + 1] - nbr_ptr[i], nc = ncell[i], npc = S::NP * nc;
    const int len = S::KD * nn + npc;
    const int r = lane >> 2, q = lane & 3;
    int e = kExpZero;
#pragma unroll
    for (int k = 0; k < S::KD; ++k) {
      const double* v = val + rowptr[(k / D) * block + (long long)(k % D) * R + i];
      int t = kExpZero;
      for (int p = lane; p < len; p += 32) t = max(t, exp_above(v[p]));
      t = __reduce_max_sync(0xffffffffu, t);
      if (k == r) e = t;
    }
    if (r < S::KD && q == 0) jexp[i * S::KD + r] = e;
    if (r >= S::KD) continue;
    const int a = r / D, l = r - a * D;
    const double* v = val + rowptr[a * block + (long long)l * R + i];
    const int steps = dbase[i + 1] - dbase[i], vsteps = (S::PAIRS * nn + 7) >> 3;
    for (int t = 0; t < steps; ++t)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int pr = 8 * t + 4 * h + q;
        unsigned long long p[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          int pos = -1;
          if (t < vsteps) {  // velocity: entry 2 c + k of neighbour j
            const int j = pr / S::PAIRS, bm = 2 * (pr - j * S::PAIRS) + k, b = bm / D, m = bm - b * D;
            if (j < nn && bm < S::KD) pos = b * D * nn + (b > a ? npc : 0) + m * nn + j;
          } else {  // pressure qq of cell ci at time at
            const int pp = pr - 8 * vsteps, ci = pp / S::CPAIRS, at = (pp - ci * S::CPAIRS) / 2, qq = 2 * (pp & 1) + k;
            if (ci < nc && at == a && qq < S::NP) pos = (a + 1) * D * nn + ci * S::NP + qq;
          }
          p[k] = digits_of(pos >= 0 && e <= 1024 ? v[pos] : 0.0, e);
        }
        jw[((long long)dbase[i] + t) * (2 * S::LANES) + h * S::LANES + lane] = words_of(p[0], p[1]);
      }
  }
}

struct SpmmArgs {
  const uint4 *jw[2];       // J, J^T
  const int* jexp[2];
  const double* val[2];     // CSR values
  const long long* rowptr;
  const int* col;
  const int *dbase, *nbr_ptr, *nbr, *ncell, *node_cells, *cell_nodes, *jobs;
  const uint4* xw;
  const short *xb, *nb;
  const uchar4* most;
  long long block;
  int R, C;
  const double *X, *B;
  double* Y;
  int mode, split;
  uint32_t* T16;
  unsigned* work;
  unsigned ntot;             // node halves and cells
  unsigned long long pstep;  // cells per unit, times 2^32
};

__device__ __forceinline__ void put(const SpmmArgs& s, long long o, double v) {
  const double y = s.mode == 1 ? s.B[o] - v : v;
  s.Y[o] = y;
  if (s.T16) {
    uint32_t h, l;
    bf16_split_rn(y, h, l);
    s.T16[o] = (l << 16) | h;
  }
}

// Work units from a device counter: one node and 16 columns (nodes with most neighbours first; the two halves
// of a node follow one another, so the second finds J in a cache), or the pressure rows of one cell.
template <int K, int D>
__global__ void __launch_bounds__(kThreads, kCtas) k_spmm_digits(const __grid_constant__ SpmmArgs s) {
  using S = Shape<K, D>;
  __shared__ uint32_t tab[kThreads / 32][S::TAB];                       // first word of every pair of X
  const int lane = threadIdx.x & 31, n = lane >> 2, q = lane & 3;
  uint32_t* tb = tab[threadIdx.x >> 5];
  auto cells_before = [&](unsigned u) { return (unsigned)(((unsigned long long)u * s.pstep) >> 32); };
  unsigned u = 0;
  if (lane == 0) u = atomicAdd(s.work, 1u);
  u = __shfl_sync(0xffffffffu, u, 0);
  while (u < s.ntot) {
    unsigned unext = 0;
    if (lane == 0) unext = atomicAdd(s.work, 1u);
    const unsigned cb = cells_before(u);
    if (cells_before(u + 1) == cb) {
      const int c0 = ((u - cb) & 1) * 16;
      const int i = s.jobs[s.R - 1 - (int)((u - cb) >> 1)];
      const int tr = c0 >= s.split;
      const int p0 = s.nbr_ptr[i], nn = s.nbr_ptr[i + 1] - p0, nc = s.ncell[i];
      const int db = s.dbase[i], steps = s.dbase[i + 1] - db;
      const int vsteps = (S::PAIRS * nn + 7) >> 3;
      const int er = n < S::KD ? s.jexp[tr][(long long)i * S::KD + n] : kExpZero;
      __syncwarp();  // the tables of the node before are free
      // neighbour nodes and cells one per lane: their pairs of X
#pragma unroll
      for (int k = 0; k < (S::MAXN + 31) / 32; ++k)
        if (32 * k + lane < nn) {
          const uint32_t v = s.nbr[p0 + 32 * k + lane];
#pragma unroll
          for (int c = 0; c < S::PAIRS; ++c) tb[S::PAIRS * (32 * k + lane) + c] = v * S::PAIRS + c;
        }
      if (lane < nc) {
        const uint32_t v = s.node_cells[(long long)i * S::MAXC + lane];
#pragma unroll
        for (int c = 0; c < S::CPAIRS; ++c)
          tb[8 * vsteps + S::CPAIRS * lane + c] = (uint32_t)s.R * S::PAIRS + v * S::CPAIRS + c;
      }
      // the rest of a segment's last step meets zeros of J
      if (lane < 8) {
        if (S::PAIRS * nn + lane < 8 * vsteps) tb[S::PAIRS * nn + lane] = 0u;
        tb[8 * vsteps + S::CPAIRS * nc + lane] = 0u;
      }
      // bases of this lane's columns n and n + 8 (nodes, cells), and the largest shifts
      const short* nb = s.nb + (long long)i * (2 * NR) + c0 + n;
      const int g00 = nb[0], g08 = nb[8], g10 = nb[NR], g18 = nb[NR + 8];
      const uchar4 mm = s.most[i];
      const int most0 = c0 ? mm.z : mm.x, most1 = c0 ? mm.w : mm.y;
      const bool rows_bad = __any_sync(0xffffffffu, er > 1024);
      unsigned bad = 0;  // columns (of the 16) that are summed in plain FP64
      if (rows_bad || most0 == 127 || most1 == 127) {
        const unsigned b0 = __ballot_sync(0xffffffffu, q == 0 && (rows_bad || g00 == kBadBase || g10 == kBadBase));
        const unsigned b8 = __ballot_sync(0xffffffffu, q == 0 && (rows_bad || g08 == kBadBase || g18 == kBadBase));
#pragma unroll
        for (int c = 0; c < 8; ++c) bad |= ((b0 >> (4 * c)) & 1u) << c | ((b8 >> (4 * c)) & 1u) << (c + 8);
      }
      __syncwarp();
      const int row = n < S::KD ? n : S::KD - 1;  // lanes past the last row follow it; their sums are not used
      const uint4* jw = s.jw[tr] + (size_t)db * (2 * S::LANES) + row * 4 + q;
      const uint4* xw = s.xw + c0 + n;
      float acc[8][4];
#pragma unroll
      for (int l = 0; l < 8; ++l)
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[l][m] = 0.f;
      long long hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
      double sum[4] = {0.0, 0.0, 0.0, 0.0};
      const uint32_t* tq = tb + q;
      int left = kDrain;
      for (int t = 0; t < steps; ++t) {
        const uint4* a0 = xw + (size_t)tq[8 * t] * NR;
        const uint4* a1 = xw + (size_t)tq[8 * t + 4] * NR;
        // (column n, n + 8) x (positions 2 q, 2 q + 1 | 2 q + 8, 2 q + 9)
        uint4 x[4] = {__ldg(a0), __ldg(a0 + 8), __ldg(a1), __ldg(a1 + 8)};
        const uint4 j0 = __ldg(jw + t * (2 * S::LANES)), j1 = __ldg(jw + t * (2 * S::LANES) + S::LANES);
        const bool cell = t >= vsteps;
        const int most = min(cell ? most1 : most0, 8);
        if (most) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {  // the pair's node or cell (its first pair for the rest of a last step)
            const uint32_t w = tb[8 * t + 4 * h + q];
            const uint32_t e = w < (uint32_t)s.R * S::PAIRS ? w / S::PAIRS : s.R + (w - (uint32_t)s.R * S::PAIRS) / S::CPAIRS;
            const short* xb = s.xb + (long long)e * NR + c0 + n;
            x[2 * h] = shift_words(x[2 * h], (cell ? g10 : g00) - xb[0], most);
            x[2 * h + 1] = shift_words(x[2 * h + 1], (cell ? g18 : g08) - xb[8], most);
          }
        }
        uint32_t b[8][2];
        {
          const uint32_t w0[4] = {j0.x, j0.y, j0.z, j0.w}, w1[4] = {j1.x, j1.y, j1.z, j1.w};
#pragma unroll
          for (int d = 0; d < 8; ++d) {
            b[d][0] = digit_pair(w0[d & 3], d >= 4);
            b[d][1] = digit_pair(w1[d & 3], d >= 4);
          }
        }
        const uint32_t xx[4][4] = {{x[0].x, x[0].y, x[0].z, x[0].w}, {x[1].x, x[1].y, x[1].z, x[1].w},
                                   {x[2].x, x[2].y, x[2].z, x[2].w}, {x[3].x, x[3].y, x[3].z, x[3].w}};
#pragma unroll
        for (int d = 0; d < 8; ++d) {
          uint32_t a[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) a[k] = digit_pair(xx[k][d & 3], d >= 4);
#pragma unroll
          for (int e = 0; d + e < 8; ++e) mma_f16(acc[d + e], a[0], a[1], a[2], a[3], b[e][0], b[e][1]);
        }
        const bool end = t == vsteps - 1 || t == steps - 1;
        if (--left == 0 || end) {
          left = kDrain;
#pragma unroll
          for (int m = 0; m < 4; ++m) {
#pragma unroll
            for (int d = 0; d < 4; ++d) {  // one wide multiply-add each
              hi[m] += (long long)__float2int_rn(acc[d][m]) * (1 << (24 - 8 * d));
              lo[m] += (long long)__float2int_rn(acc[d + 4][m]) * (1 << (24 - 8 * d));
              acc[d][m] = 0.f;
              acc[d + 4][m] = 0.f;
            }
          }
        }
        // acc[m]: column n (m < 2) or n + 8, row 2 q + (m & 1); a segment is hi 2^(er + 8 base - 30) + lo 2^(er + 8 base - 62)
        if (end) {
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int r = 2 * q + (m & 1);
            const int e = __shfl_sync(0xffffffffu, er, (4 * r) & 31);
            const int g = m < 2 ? (cell ? g10 : g00) : (cell ? g18 : g08);
            if (e != kExpZero && g != kZeroBase)
              sum[m] += scale_pow2(fma((double)hi[m], 4294967296.0, (double)lo[m]), e - 62 + 8 * g);
            hi[m] = lo[m] = 0;
          }
        }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int r = 2 * q + (m & 1), c = n + (m < 2 ? 0 : 8);
        if (r < S::KD && !((bad >> c) & 1u)) put(s, ((r / D) * s.block + (long long)(r % D) * s.R + i) * NR + c0 + c, sum[m]);
      }
      if (bad) {
        if (lane < 16 && ((bad >> lane) & 1u))
          for (int r = 0; r < S::KD; ++r) {
            const long long y = (r / D) * s.block + (long long)(r % D) * s.R + i;
            double t = 0.0;
            for (long long e = s.rowptr[y]; e < s.rowptr[y + 1]; ++e)
              t = fma(s.val[tr][e], s.X[(long long)s.col[e] * NR + c0 + lane], t);
            put(s, y * NR + c0 + lane, t);
          }
        __syncwarp();
      }
    } else {
      // pressure rows of cell cb: lane = column, each value broadcast
      const long long c = cb;
      const double* val = s.val[lane >= s.split];
      long long rp[K * S::NP];
      double acc[K * S::NP];
#pragma unroll
      for (int a = 0; a < K; ++a)
#pragma unroll
        for (int p = 0; p < S::NP; ++p) {
          rp[a * S::NP + p] = s.rowptr[a * s.block + (long long)D * s.R + c * S::NP + p];
          acc[a * S::NP + p] = 0.0;
        }
      const int mine = lane < S::NV ? s.cell_nodes[c * S::NV + lane] : 0;
#pragma unroll 1
      for (int m = 0; m < D; ++m)
#pragma unroll 3
        for (int jj = 0; jj < S::NV; ++jj) {
          const long long node = __shfl_sync(0xffffffffu, mine, jj);
#pragma unroll
          for (int a = 0; a < K; ++a) {
            const double xa = s.X[(a * s.block + (long long)m * s.R + node) * NR + lane];
#pragma unroll
            for (int p = 0; p < S::NP; ++p) acc[a * S::NP + p] += __ldg(val + rp[a * S::NP + p] + m * S::NV + jj) * xa;
          }
        }
#pragma unroll
      for (int a = 0; a < K; ++a)
#pragma unroll
        for (int p = 0; p < S::NP; ++p)
          put(s, (a * s.block + (long long)D * s.R + c * S::NP + p) * NR + lane, acc[a * S::NP + p]);
    }
    u = __shfl_sync(0xffffffffu, unext, 0);
  }
  // the last CTA to finish resets the counter: every warp has drawn a unit past the end by then
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(s.work + 1, 1u) == gridDim.x - 1) {
      s.work[0] = 0u;
      s.work[1] = 0u;
      __threadfence();
    }
  }
}

template <int K, int D>
stm_status words(const Level& L, const double* val, uint4* jw, int* jexp, cudaStream_t s) {
  const int blocks = (int)std::min<long long>(((long long)L.R * 32 + 255) / 256, sm_count() * 8LL);
  k_j_words<K, D><<<blocks, 256, 0, s>>>(L.rowptr, val, L.nbr_ptr, L.ncell, L.dbase, jw, jexp, L.block, L.R);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

template <int K, int D>
stm_status launch(const Level& L, SpmmArgs& a, cudaStream_t s) {
  static int occ = 0;  // resident CTAs per SM
  if (!occ) {
    STM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_spmm_digits<K, D>, kThreads, 0));
    if (occ < 1) occ = 1;
  }
  const int xblocks = (int)std::min<long long>(((long long)L.R + L.C + 7) / 8, sm_count() * 16LL);
  k_xm_words<K, D><<<xblocks, 256, 0, s>>>(a.X, L.block, L.R, L.C, (uint4*)L.xw, L.xb);
  note_launch();
  k_xm_bases<K, D><<<xblocks, 256, 0, s>>>(L.xb, L.nbr_ptr, L.nbr, L.ncell, L.node_cells, L.R, L.xnb, (uchar4*)L.xmost);
  note_launch();
  a.ntot = 2u * (unsigned)L.R + (unsigned)L.C;
  a.pstep = (((unsigned long long)L.C << 32) + a.ntot - 1) / a.ntot;
  const int blocks = (int)std::max<long long>(1, std::min<long long>((long long)occ * sm_count(), (a.ntot + kThreads / 32 - 1) / (kThreads / 32)));
  k_spmm_digits<K, D><<<blocks, kThreads, 0, s>>>(a);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

}  // namespace

bool spmm_digits_supported(const Level& L) { return L.K * L.dim <= 6; }

// J's words (and J^T's when transpose is set) for the present values; work space on first use
stm_status ensure_spmm_digits(Level& L, int transpose, cudaStream_t s) {
  const int KD = L.K * L.dim, pairs = (KD + 1) / 2, cpairs = 2 * L.K;
  if (!L.dbase) {
    std::vector<int> nbr_ptr(L.R + 1), ncell(L.R), dbase(L.R + 1, 0);
    STM_CUDA(cudaMemcpy(nbr_ptr.data(), L.nbr_ptr, sizeof(int) * (L.R + 1), cudaMemcpyDeviceToHost));
    STM_CUDA(cudaMemcpy(ncell.data(), L.ncell, sizeof(int) * L.R, cudaMemcpyDeviceToHost));
    for (int i = 0; i < L.R; ++i)
      dbase[i + 1] = dbase[i] + (pairs * (nbr_ptr[i + 1] - nbr_ptr[i]) + 7) / 8 + (cpairs * ncell[i] + 7) / 8;
    STM_CUDA(cudaMalloc((void**)&L.dbase, sizeof(int) * (L.R + 1)));
    STM_CUDA(cudaMemcpy(L.dbase, dbase.data(), sizeof(int) * (L.R + 1), cudaMemcpyHostToDevice));
    L.dsteps = dbase[L.R];
  }
  if (!L.xw) STM_CUDA(cudaMalloc(&L.xw, sizeof(uint4) * NR * ((size_t)L.R * pairs + (size_t)L.C * cpairs)));
  if (!L.xb) STM_CUDA(cudaMalloc((void**)&L.xb, sizeof(short) * NR * ((size_t)L.R + L.C)));
  if (!L.xnb) STM_CUDA(cudaMalloc((void**)&L.xnb, sizeof(short) * 2 * NR * (size_t)L.R));
  if (!L.xmost) STM_CUDA(cudaMalloc(&L.xmost, sizeof(uchar4) * (size_t)L.R));
  for (int t = 0; t <= (transpose ? 1 : 0); ++t) {
    if (!L.jw[t]) STM_CUDA(cudaMalloc(&L.jw[t], sizeof(uint4) * 8 * KD * (size_t)L.dsteps));
    if (!L.jwexp[t]) STM_CUDA(cudaMalloc((void**)&L.jwexp[t], sizeof(int) * KD * (size_t)L.R));
    if (L.jw_current[t]) continue;
    const double* val = t ? L.valT : L.val;
    switch (L.dim * 10 + L.K) {
      case 21: STM_TRY((words<1, 2>(L, val, (uint4*)L.jw[t], L.jwexp[t], s))); break;
      case 22: STM_TRY((words<2, 2>(L, val, (uint4*)L.jw[t], L.jwexp[t], s))); break;
      case 23: STM_TRY((words<3, 2>(L, val, (uint4*)L.jw[t], L.jwexp[t], s))); break;
      case 31: STM_TRY((words<1, 3>(L, val, (uint4*)L.jw[t], L.jwexp[t], s))); break;
      default: STM_TRY((words<2, 3>(L, val, (uint4*)L.jw[t], L.jwexp[t], s))); break;
    }
    L.jw_current[t] = true;
  }
  return STM_OK;
}

stm_status spmm_digits(Level& L, const double* X, const double* B, double* Y, int mode, cudaStream_t s, int split,
                       uint32_t* T16) {
  STM_TRY(ensure_spmm_digits(L, split < NR, s));
  SpmmArgs a{};
  for (int t = 0; t < 2; ++t) {
    a.jw[t] = (const uint4*)L.jw[t];
    a.jexp[t] = L.jwexp[t];
  }
  a.val[0] = L.val;
  a.val[1] = L.valT;
  a.rowptr = L.rowptr;
  a.col = L.colidx;
  a.dbase = L.dbase;
  a.nbr_ptr = L.nbr_ptr;
  a.nbr = L.nbr;
  a.ncell = L.ncell;
  a.node_cells = L.node_cells;
  a.cell_nodes = L.cell_nodes;
  a.jobs = L.job_nodes;
  a.xw = (const uint4*)L.xw;
  a.xb = L.xb;
  a.nb = L.xnb;
  a.most = (const uchar4*)L.xmost;
  a.block = L.block;
  a.R = L.R;
  a.C = L.C;
  a.X = X;
  a.B = B;
  a.Y = Y;
  a.mode = mode;
  a.split = split;
  a.T16 = T16;
  a.work = L.spmv_work;
  switch (L.dim * 10 + L.K) {
    case 21: return launch<1, 2>(L, a, s);
    case 22: return launch<2, 2>(L, a, s);
    case 23: return launch<3, 2>(L, a, s);
    case 31: return launch<1, 3>(L, a, s);
    default: return launch<2, 3>(L, a, s);
  }
}

}  // namespace stm
