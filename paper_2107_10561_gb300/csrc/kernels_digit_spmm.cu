// 32-column product with the slab Jacobian J_g or its transpose whose velocity columns run on the tensor cores:
// Y = J X or Y = B - J X, every entry as accurate as an FP64 sum of its row is held to be.
//
// 32 columns make 32 FMAs per value of J, and at 2 FP64 FMAs per clock and SM those take 40 times as long
// as the bytes take from HBM. Here the values of J and the entries of X are 63-bit integers cut into eight balanced
// base-256 digits, whose products add up exactly in the FP32 accumulators of FP16 tensor instructions (digits.h). The
// 36 digit pairs (s, t) with s + t <= 7 are accumulated per weight and joined in 64-bit integers.
//   - One warp per node and 16 columns. M = 16 of an MMA holds the columns, N = 8 the K d <= 6 rows of the
//     node, K = 16 neighbour nodes. The velocity components (of all time nodes) are gone through one after the other,
//     each with scales of its own: a power of two per row of J, and one per node and column of X (a multiple of eight
//     bits). A node takes the largest base around it per component and column, and neighbours with a smaller one are
//     shifted by whole digits. A component's sum is added to the row's in FP64.
//     Whole product with X's passes, 3D dG(1), 129,094 unknowns: 1.27 ms inside FGMRES, in FP64 2.57 ms; 2D dG(2), 137,094:
//     598 against 656 us. A step of 16 neighbours takes about 360 warp instructions (37 MMAs, 96 to form the digits).
//   - What the digits leave out is 2^-61 of a component's product of scales, usually far less than 2^-53 of |J||X|. The
//     components' sums, a product of the leading digits' magnitudes (one MMA in 37) and the pressures' terms bound
//     |J||X| from below; where they stay 2^-kSpare below the largest product of scales the row is summed again in FP64,
//     by the whole warp: of V-cycles' results one entry in 13, most in rows at walls, where J is large and X small
//     (0.2 ms of the 1.27; entry by entry 0.45). With one scale for all components of a node and the pressures in
//     the same rows the error was 1e-14 of |J||X| at components 1e-2 apart and 1e-10 at 1e-6.
//   - Both operands are stored as the fragments want them: four words [u_i, u_{i+4}, v_i, v_{i+4}] of biased bytes per
//     pair of neighbours u, v of J, the halves [u_i, u_{i+4}] of X; byte permutes and an FP16 subtraction give a register
//     of an operand.
//   - Pressure columns (4 % of the values) and the rows of the pressure equations (3 %) stay on the FP64 pipe.
//   - Entries whose neighbourhood or row holds an infinity or a NaN are summed in FP64.
#include "digits.h"
#include "internal.h"

namespace stm {
namespace {

constexpr int NR = 32;                   // columns of a multi-vector
constexpr int kZeroBase = -20000;        // base of entries that are all zero
constexpr int kBadBase = 20000;          // base of entries that are not all finite
constexpr int kThreads = 256, kCtas = 2;
constexpr int kSpare = 12;               // bits by which an entry's magnitudes may lie below its scale

template <int K, int D>
struct Shape {
  static constexpr int KD = K * D;               // velocity rows of a node, components of X
  static constexpr int NP = D + 1, MAXC = 1 << D, MAXN = D == 2 ? 25 : 125, NV = D == 2 ? 9 : 27;
  static constexpr int LANES = 4 * KD;           // lanes that hold values of J
  // 16 neighbours a step: 8 pairs of digits x 128 positions x 2^14 = 2^24, FP32 sums of a component are exact
  static_assert(MAXN <= 128, "drain");
};

// base g with |v| <= 2^(8 g + 6) for |v| < 2^e
__device__ __forceinline__ int base_of(int e) { return e == kExpZero ? kZeroBase : e > 1024 ? kBadBase : (e + 1) >> 3; }

// The halves of a value's words: bytes [u0 u4 u1 u5], [u2 u6 u3 u7]
__device__ __forceinline__ uint2 halves_of(unsigned long long u) {
  const uint32_t h = (uint32_t)(u >> 32), l = (uint32_t)u;
  return make_uint2(__byte_perm(h, l, 0x6273), __byte_perm(h, l, 0x4051));
}
// The same shifted down by sh <= most digits
__device__ __forceinline__ uint2 shift_halves(uint2 w, int sh, int most) {
  for (int k = 0; k < most; ++k)
    if (k < sh) w = make_uint2((__byte_perm(w.x, w.y, 0x1060) & 0xFFFFFF00u) | 0x80u, __byte_perm(w.x, w.y, 0x5432));
  return w;
}
__device__ __forceinline__ uint4 join_halves(uint2 u, uint2 v) {
  return make_uint4(__byte_perm(u.x, v.x, 0x5410), __byte_perm(u.x, v.x, 0x7632), __byte_perm(u.y, v.y, 0x5410),
                    __byte_perm(u.y, v.y, 0x7632));
}

// Halves and bases of X: one warp per node, lane = column.
template <int K, int D>
__global__ void __launch_bounds__(256) k_xm_words(const double* __restrict__ X, long long block, int R,
                                                  uint2* __restrict__ xw, short* __restrict__ xb) {
  using S = Shape<K, D>;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < R; i += nwarps) {
    double v[S::KD];
#pragma unroll
    for (int k = 0; k < S::KD; ++k) v[k] = X[((k / D) * block + (long long)(k % D) * R + i) * NR + lane];
#pragma unroll
    for (int k = 0; k < S::KD; ++k) {
      const int g = base_of(exp_above(v[k]));
      xb[(i * S::KD + k) * NR + lane] = (short)g;
      xw[(i * S::KD + k) * NR + lane] = halves_of(digits_of(g == kBadBase ? 0.0 : v[k], 8 * g + 6));
    }
  }
}

// Largest and smallest base (of entries that are not zero) in each cell, per component and column: one warp per cell
// and component, lane = column.
template <int K, int D>
__global__ void __launch_bounds__(256) k_xm_cells(const short* __restrict__ xb, const int* __restrict__ cell_nodes, int C,
                                                  short2* __restrict__ cb) {
  using S = Shape<K, D>;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < (long long)C * S::KD; e += nwarps) {
    const int c = (int)(e / S::KD), k = (int)(e - (long long)c * S::KD);
    const int mine = lane < S::NV ? cell_nodes[(long long)c * S::NV + lane] : 0;
    int hi = kZeroBase, lo = kBadBase;
#pragma unroll 9
    for (int j = 0; j < S::NV; ++j) {
      const long long node = __shfl_sync(0xffffffffu, mine, j);
      const int g = xb[(node * S::KD + k) * NR + lane];
      hi = max(hi, g);
      if (g != kZeroBase) lo = min(lo, g);
    }
    cb[e * NR + lane] = make_short2((short)hi, (short)lo);
  }
}

// Around every node: the largest base per component and column, and per 16 columns the largest shift that brings a
// neighbour to it (127: a base that is not finite). One warp per node, lane = column.
template <int K, int D>
__global__ void __launch_bounds__(256) k_xm_bases(const short2* __restrict__ cb, const int* __restrict__ ncell,
                                                  const int* __restrict__ node_cells, int R, short* __restrict__ nb,
                                                  unsigned char* __restrict__ most) {
  using S = Shape<K, D>;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < R; i += nwarps) {
    const int nc = ncell[i];
    int hi[S::KD], lo[S::KD];
#pragma unroll
    for (int k = 0; k < S::KD; ++k) hi[k] = kZeroBase, lo[k] = kBadBase;
    for (int j = 0; j < nc; ++j) {
      const long long c = node_cells[i * S::MAXC + j];
#pragma unroll
      for (int k = 0; k < S::KD; ++k) {
        const short2 g = cb[(c * S::KD + k) * NR + lane];
        hi[k] = max(hi[k], (int)g.x);
        lo[k] = min(lo[k], (int)g.y);
      }
    }
#pragma unroll
    for (int k = 0; k < S::KD; ++k) {
      nb[(i * S::KD + k) * NR + lane] = (short)hi[k];
      const int m = hi[k] == kBadBase ? 127 : lo[k] < hi[k] ? min(hi[k] - lo[k], 8) : 0;
      const int a = __reduce_max_sync(0xFFFFu << (lane & 16), m);
      if ((lane & 15) == 0) most[(i * 2 + (lane >> 4)) * 8 + k] = (unsigned char)a;
    }
  }
}

// Words of the velocity columns of J's velocity rows in fragment order, and each row's exponent per component: one
// warp per node.
template <int K, int D>
__global__ void __launch_bounds__(256) k_j_words(const long long* __restrict__ rowptr, const double* __restrict__ val,
                                                 const int* __restrict__ nbr_ptr, const int* __restrict__ ncell,
                                                 const int* __restrict__ dbase, uint4* __restrict__ jw,
                                                 int* __restrict__ jexp, long long block, int R) {
  using S = Shape<K, D>;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < R; i += nwarps) {
    const int nn = nbr_ptr[i + 1] - nbr_ptr[i], npc = S::NP * ncell[i], steps = (nn + 15) >> 4;
    const int r = lane >> 2, q = lane & 3;
    for (int k = 0; k < S::KD; ++k) {
      const int b = k / D, m = k - b * D;
      int e = kExpZero;
#pragma unroll
      for (int y = 0; y < S::KD; ++y) {
        const int a = y / D;
        const double* v = val + rowptr[a * block + (long long)(y - a * D) * R + i] + (b * D + m) * nn + (b > a ? npc : 0);
        int t = kExpZero;
        for (int p = lane; p < nn; p += 32) t = max(t, exp_above(v[p]));
        t = __reduce_max_sync(0xffffffffu, t);
        if (y == r) e = t;
      }
      if (r < S::KD && q == 0) jexp[(i * S::KD + k) * S::KD + r] = e;
      if (r >= S::KD) continue;
      const int a = r / D;
      const double* v = val + rowptr[a * block + (long long)(r - a * D) * R + i] + (b * D + m) * nn + (b > a ? npc : 0);
      for (int t = 0; t < steps; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = 16 * t + 8 * h + 2 * q;
          const unsigned long long p0 = digits_of(j < nn && e <= 1024 ? v[j] : 0.0, e);
          const unsigned long long p1 = digits_of(j + 1 < nn && e <= 1024 ? v[j + 1] : 0.0, e);
          jw[((long long)dbase[i] + k * steps + t) * (2 * S::LANES) + h * S::LANES + lane] = words_of(p0, p1);
        }
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
  const uint2* xw;
  const short *xb, *nb;
  const unsigned char* most;
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
  __shared__ __align__(8) uint32_t tab[kThreads / 32][128];  // the neighbours
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
      const int p0 = s.nbr_ptr[i], nn = s.nbr_ptr[i + 1] - p0, nc = s.ncell[i], steps = (nn + 15) >> 4;
      __syncwarp();  // the table of the node before is free
#pragma unroll
      for (int k = 0; k < (S::MAXN + 31) / 32; ++k)  // the rest of the last step meets zeros of J
        if (32 * k + lane < 16 * steps) tb[32 * k + lane] = 32 * k + lane < nn ? (uint32_t)s.nbr[p0 + 32 * k + lane] : 0u;
      __syncwarp();
      // rows 2 q, 2 q + 1 (m & 1) x columns n, n + 8 (m >> 1) of the unit
      const int row = n < S::KD ? n : S::KD - 1;  // lanes past the last row follow it; their sums are not used
      const uint4* jw = s.jw[tr] + (size_t)s.dbase[i] * (2 * S::LANES) + row * 4 + q;
      const int* je = s.jexp[tr] + (long long)i * (S::KD * S::KD);
      const double* val = s.val[tr];
      double sum[4] = {0.0, 0.0, 0.0, 0.0};
      int top[4], lead[4];  // the largest product of scales; |J||X| is at least 2^(lead - 1)
      bool again = false;   // an infinity or a NaN
#pragma unroll
      for (int m = 0; m < 4; ++m) top[m] = lead[m] = kExpZero;
#pragma unroll 1
      for (int k = 0; k < S::KD; ++k) {
        const short* nb = s.nb + ((long long)i * S::KD + k) * NR + c0 + n;
        const int g0 = nb[0], g8 = nb[8], er = je[k * S::KD + row];
        const int shifts = s.most[((long long)i * 2 + (c0 >> 4)) * 8 + k], most = min(shifts, 8);
        again = again || shifts == 127 || er > 1024;
        const uint2* xw = s.xw + k * NR + c0 + n;
        const short* xb = s.xb + k * NR + c0 + n;
        float acc[8][4], mag[4] = {0.f, 0.f, 0.f, 0.f};  // and the sum of magnitudes over the leading digits
#pragma unroll
        for (int l = 0; l < 8; ++l)
#pragma unroll
          for (int m = 0; m < 4; ++m) acc[l][m] = 0.f;
#pragma unroll 1
        for (int t = 0; t < steps; ++t) {
          const uint2 i0 = *reinterpret_cast<const uint2*>(tb + 16 * t + 2 * q);
          const uint2 i1 = *reinterpret_cast<const uint2*>(tb + 16 * t + 8 + 2 * q);
          const uint32_t at[4] = {i0.x * (S::KD * NR), i0.y * (S::KD * NR), i1.x * (S::KD * NR), i1.y * (S::KD * NR)};
          uint2 x[4][2];  // neighbours 2 q, 2 q + 1, 2 q + 8, 2 q + 9 of the step x columns n, n + 8
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            x[p][0] = __ldg(xw + at[p]);
            x[p][1] = __ldg(xw + at[p] + 8);
          }
          const uint4 j0 = __ldg(jw + t * (2 * S::LANES)), j1 = __ldg(jw + t * (2 * S::LANES) + S::LANES);
          if (most) {
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              x[p][0] = shift_halves(x[p][0], g0 - xb[at[p]], most);
              x[p][1] = shift_halves(x[p][1], g8 - xb[at[p] + 8], most);
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
          uint32_t xx[4][4];
#pragma unroll
          for (int p = 0; p < 4; ++p) {  // (column n, n + 8) x (neighbours 2 q, 2 q + 1 | 2 q + 8, 2 q + 9)
            const uint4 w = join_halves(x[2 * (p >> 1)][p & 1], x[2 * (p >> 1) + 1][p & 1]);
            xx[p][0] = w.x, xx[p][1] = w.y, xx[p][2] = w.z, xx[p][3] = w.w;
          }
#pragma unroll
          for (int d = 0; d < 8; ++d) {
            uint32_t a[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) a[p] = digit_pair(xx[p][d & 3], d >= 4);
#pragma unroll
            for (int e = 0; d + e < 8; ++e) mma_f16(acc[d + e], a[0], a[1], a[2], a[3], b[e][0], b[e][1]);
            if (d == 0) {
              constexpr uint32_t abs2 = 0x7FFF7FFFu;
              mma_f16(mag, a[0] & abs2, a[1] & abs2, a[2] & abs2, a[3] & abs2, b[0][0] & abs2, b[0][1] & abs2);
            }
          }
        }
        jw += steps * (2 * S::LANES);
        // acc[m]: column n (m < 2) or n + 8, row 2 q + (m & 1); the component's sum is (hi 2^32 + lo) 2^(er + 8 base - 62)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          long long hi = 0, lo = 0;
#pragma unroll
          for (int d = 0; d < 4; ++d) {  // one wide multiply-add each
            hi += (long long)__float2int_rn(acc[d][m]) * (1 << (24 - 8 * d));
            lo += (long long)__float2int_rn(acc[d + 4][m]) * (1 << (24 - 8 * d));
          }
          const int e = __shfl_sync(0xffffffffu, er, (4 * (2 * q + (m & 1))) & 31), g = m < 2 ? g0 : g8;
          if (e != kExpZero && g != kZeroBase) {
            const double v = join_pow2(hi, lo, e - 62 + 8 * g);
            sum[m] += v;
            top[m] = max(top[m], e + 8 * g + 6);
            lead[m] = max(lead[m], exp_above(v));
            // a leading digit of 1 stands for 2^-7 of its scale at least
            if (mag[m] > 0.f) lead[m] = max(lead[m], e + 8 * g + 6 - 13 + (int)(__float_as_uint(mag[m]) >> 23) - 127);
          }
        }
      }
      // pressure columns: a row meets those of its own time node
      const int cell = lane < nc ? s.node_cells[(long long)i * S::MAXC + lane] : 0;
      const double* vr[2];
      long long xr[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = min(2 * q + h, S::KD - 1), a = r / D;
        vr[h] = val + s.rowptr[a * s.block + (long long)(r - a * D) * s.R + i] + (a + 1) * D * nn;
        xr[h] = (a * s.block + (long long)D * s.R) * NR + c0 + n;
      }
#pragma unroll 1
      for (int c = 0; c < nc; ++c) {
        const long long at = (long long)__shfl_sync(0xffffffffu, cell, c) * (S::NP * NR);
#pragma unroll
        for (int p = 0; p < S::NP; ++p)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const double v = __ldg(vr[h] + c * S::NP + p), x0 = __ldg(s.X + xr[h] + at + p * NR), x8 = __ldg(s.X + xr[h] + at + p * NR + 8);
            sum[h] = fma(v, x0, sum[h]);
            sum[2 + h] = fma(v, x8, sum[2 + h]);
            const int e = exp_above(v), e0 = exp_above(x0), e8 = exp_above(x8);
            if (e != kExpZero && e0 != kExpZero) lead[h] = max(lead[h], e + e0 - 1);
            if (e != kExpZero && e8 != kExpZero) lead[2 + h] = max(lead[2 + h], e + e8 - 1);
          }
      }
      again = __any_sync(0xffffffffu, again);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 2 * q + h;
        bool fail = false;
#pragma unroll
        for (int m = h; m < 4; m += 2) fail = fail || (top[m] != kExpZero && lead[m] - 1 < top[m] - kSpare);
        const unsigned f = __ballot_sync(0xffffffffu, r < S::KD && (again || fail));
        // rows with such an entry in FP64 from the CSR values, the 16 columns together: four lanes take a sector of X each
        if (f)
#pragma unroll 1
          for (int w = 0; w < 4; ++w) {
            if (!(f & (0x11111111u << w))) continue;
            const int y = 2 * w + h;
            const long long at = (y / D) * s.block + (long long)(y % D) * s.R + i, end = s.rowptr[at + 1];
            const double* xc = s.X + c0 + 4 * (lane >> 3);
            double t[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
            for (long long e = s.rowptr[at] + (lane & 7); e < end; e += 8) {
              const double v = val[e];
              const double2* xe = reinterpret_cast<const double2*>(xc + (long long)s.col[e] * NR);
              const double2 x0 = xe[0], x1 = xe[1];
              t[0] = fma(v, x0.x, t[0]);
              t[1] = fma(v, x0.y, t[1]);
              t[2] = fma(v, x1.x, t[2]);
              t[3] = fma(v, x1.y, t[3]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
              for (int off = 4; off >= 1; off >>= 1) t[j] += __shfl_xor_sync(0xffffffffu, t[j], off);
#pragma unroll
            for (int g = 0; g < 2; ++g)
#pragma unroll
              for (int j = 0; j < 4; ++j) {  // column n + 8 g is entry n mod 4 of lanes 8 (n / 4) + 16 g
                const double v = __shfl_sync(0xffffffffu, t[j], 8 * (n >> 2) + 16 * g);
                if (q == w && (n & 3) == j) sum[h + 2 * g] = v;
              }
          }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int r = 2 * q + (m & 1), c = n + (m < 2 ? 0 : 8);
        if (r < S::KD) put(s, ((r / D) * s.block + (long long)(r % D) * s.R + i) * NR + c0 + c, sum[m]);
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
  const int xblocks = (int)std::min<long long>(((long long)L.R + 7) / 8, sm_count() * 16LL);
  const int cblocks = (int)std::min<long long>(((long long)L.C * K * D + 7) / 8, sm_count() * 16LL);
  k_xm_words<K, D><<<xblocks, 256, 0, s>>>(a.X, L.block, L.R, (uint2*)L.xw, L.xb);
  note_launch();
  k_xm_cells<K, D><<<cblocks, 256, 0, s>>>(L.xb, L.cell_nodes, L.C, (short2*)L.xcb);
  note_launch();
  k_xm_bases<K, D><<<xblocks, 256, 0, s>>>((const short2*)L.xcb, L.ncell, L.node_cells, L.R, L.xnb, (unsigned char*)L.xmost);
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

// Nodes of fewer than six rows are faster in FP64, or no slower (2D dG(1), 91,396 unknowns: 323 us per product against
// 361, dG(0), 45,698: 106 against 221; 3D dG(0), 64,547: 708 against 725).
bool spmm_digits_supported(const Level& L) { return L.K * L.dim == 6; }

void free_spmm_digits(Level& L) {
  void* ptrs[] = {L.xw, L.xb, L.xcb, L.xnb, L.xmost, L.jw[0], L.jw[1], L.jwexp[0], L.jwexp[1]};
  for (void* q : ptrs) cudaFree(q);
  L.xw = L.xcb = L.xmost = L.jw[0] = L.jw[1] = nullptr;
  L.xb = L.xnb = nullptr;
  L.jwexp[0] = L.jwexp[1] = nullptr;
  L.jw_current[0] = L.jw_current[1] = false;
}

// J's words (and J^T's when transpose is set) for the present values; work space on first use. STM_ERR_OOM where it
// does not fit, and nothing is kept then.
stm_status ensure_spmm_digits(Level& L, int transpose, cudaStream_t s) {
  const int KD = L.K * L.dim;
  if (!L.dbase) {
    std::vector<int> nbr_ptr(L.R + 1), dbase(L.R + 1, 0);
    STM_CUDA(cudaMemcpy(nbr_ptr.data(), L.nbr_ptr, sizeof(int) * (L.R + 1), cudaMemcpyDeviceToHost));
    for (int i = 0; i < L.R; ++i)
      dbase[i + 1] = dbase[i] + KD * ((nbr_ptr[i + 1] - nbr_ptr[i] + 15) / 16);
    STM_CUDA(cudaMalloc((void**)&L.dbase, sizeof(int) * (L.R + 1)));
    STM_CUDA(cudaMemcpy(L.dbase, dbase.data(), sizeof(int) * (L.R + 1), cudaMemcpyHostToDevice));
    L.dsteps = dbase[L.R];
  }
  struct { void** p; size_t bytes; } want[] = {
      {&L.xw, sizeof(uint2) * NR * KD * (size_t)L.R}, {(void**)&L.xb, sizeof(short) * NR * KD * (size_t)L.R},
      {&L.xcb, sizeof(short2) * NR * KD * (size_t)L.C}, {(void**)&L.xnb, sizeof(short) * NR * KD * (size_t)L.R},
      {&L.xmost, 16 * (size_t)L.R}, {&L.jw[0], sizeof(uint4) * 8 * KD * (size_t)L.dsteps},
      {(void**)&L.jwexp[0], sizeof(int) * KD * KD * (size_t)L.R}, {&L.jw[1], sizeof(uint4) * 8 * KD * (size_t)L.dsteps},
      {(void**)&L.jwexp[1], sizeof(int) * KD * KD * (size_t)L.R}};
  for (int i = 0; i < (transpose ? 9 : 7); ++i)
    if (!*want[i].p && cudaMalloc(want[i].p, want[i].bytes) != cudaSuccess) {
      cudaGetLastError();
      *want[i].p = nullptr;
      STM_CUDA(cudaStreamSynchronize(s));  // products that still read them
      free_spmm_digits(L);
      return STM_ERR_OOM;
    }
  for (int t = 0; t <= (transpose ? 1 : 0); ++t) {
    if (L.jw_current[t]) continue;
    const double* val = t ? L.valT : L.val;
    switch (L.dim * 10 + L.K) {
      case 23: STM_TRY((words<3, 2>(L, val, (uint4*)L.jw[t], L.jwexp[t], s))); break;
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
  a.xw = (const uint2*)L.xw;
  a.xb = L.xb;
  a.nb = L.xnb;
  a.most = (const unsigned char*)L.xmost;
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
    case 23: return launch<3, 2>(L, a, s);
    default: return launch<2, 3>(L, a, s);
  }
}

}  // namespace stm
