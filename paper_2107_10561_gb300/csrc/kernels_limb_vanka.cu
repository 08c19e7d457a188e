// Cell solves y_T = J_T^{-1} t_T over FP64 inverses, on the INT32 pipe, every row as accurate as an FP64 sum of it is held
// to be.
//
// Every entry of an inverse is read once and needs one multiply-add; in FP64 that is the limit (2D dG(2), 16,384 cells,
// 528 MB: 150 us against 78 us for the bytes at the measured copy rate). The inverses are therefore kept a second time as
// two-limb integers (limbs.h), three integer multiply-adds each: 105 us; 2D dG(1) 97 -> 65 us, 3D dG(0) 280 -> 219.
//   - A sum of integers has one scale. An inverse has an exponent per row and class of columns (a velocity component or
//     the pressures of one time node), t one per class; a class's columns are summed at the product of the two and the
//     sum is shifted to the largest such product of the row. What is cut off is 2^-57 of that product. The classes'
//     sums bound |J_T^{-1}||t| from below: a row where they stay 2^-kSpare below the largest product is summed again
//     in FP64. kSpare = 8 keeps what one term may lose (2^-56.4) below m 2^-53 |J_T^{-1}||t|, the bound of an FP64 chain of
//     m >= 42 terms. Right-hand sides and residuals have no such row in 2D, one in 100 cells in 3D dG(1) and one in 20
//     to 50 in 3D dG(0). With one scale per row and one offset for the pressures (91 us) the error was 3 to 400 times
//     that of FP64 (normally distributed t, tau 1e-2 to 1e-5).
//   - A warp per cell, whole lines per load; lanes own row pairs and t's limbs are broadcast from shared memory, so
//     a column costs a load, a shared load and six multiply-adds per lane. Exponents and the first columns are on their
//     way while t is cut.
//   - Few cells stay with the FP64 kernel, which takes several warps per cell (limb_cells_pay; 3D dG(1), 1,536 cells,
//     whole sweep: 185 against 168 us; with several warps here 360 cells took 46 us against 31), and so does the transpose (2D dG(2): 204 us against 145; the scales of its products differ from row to row of
//     the inverse and class of columns). So do cells of fewer than 32 rows (2D dG(0): 21) and levels without
//     room for the second copy, which is made on the first solve and given back when memory runs short.
//   - Cells with an infinity or a NaN, in the inverse or in t, are summed in FP64 from the FP64 inverses.
#include "digits.h"
#include "internal.h"
#include "limbs.h"

namespace stm {
namespace {

constexpr int kNone = -20000;  // exponent where every entry is zero (16 bits)
constexpr int kPlain = 20000;  // exponent of a row's class that holds an infinity or a NaN
constexpr int kCtas = 2;       // per SM, of eight warps
constexpr int kSpare = 8;      // bits by which a row's sum of magnitudes may lie below its scale

// The columns of a cell by class: per time node the D velocity components, then the pressures.
template <int K, int D>
struct Cell {
  static constexpr int NV = D == 2 ? 9 : 27, NP = D + 1, NT = D * NV + NP, PT = D + 1;  // PT classes per time node
  static constexpr int n = K * NT, nk = K * PT;
  // batches of three columns, within a class each: the last one of a time node is short in 3D
  static constexpr int BT = (D * NV + NP + 2) / 3, batches = K * BT;
  static __device__ __forceinline__ int column(int b) { return b / BT * NT + b % BT * 3; }
  static __device__ __forceinline__ int width(int b) { return min(3, NT - b % BT * 3); }
  static __device__ __forceinline__ bool last(int b) { return b % BT == BT - 1 || (b % BT < D * NV / 3 && b % BT % (NV / 3) == NV / 3 - 1); }
  static __device__ __forceinline__ int cls(int j) {
    const int a = j / NT, r = j - a * NT;
    return a * PT + min(r / NV, D);
  }
  static __device__ __forceinline__ int begin(int k) { return k / PT * NT + k % PT * NV; }
};

__device__ __forceinline__ int exponent_of(double v) {
  const int e = exp_above(v);
  return e == kExpZero ? kNone : e > 1024 ? kPlain : e;
}

// Limbs of a cell's inverse in the layout of the inverse; lexp: [C][classes][ld], the exponents. One CTA per cell.
template <int K, int D>
__global__ void __launch_bounds__(256) k_inverse_limbs(const double* __restrict__ inv, int ld, int2* __restrict__ out,
                                                       short* __restrict__ lexp) {
  using S = Cell<K, D>;
  constexpr int n = S::n, nk = S::nk;
  __shared__ short ex[nk][256];
  const int c = blockIdx.x, i = threadIdx.x;
  const double* M = inv + (size_t)c * n * ld;
  if (i < ld) {
    for (int k = 0; k < nk; ++k) {
      int e = kNone;
      const int end = k + 1 < nk ? S::begin(k + 1) : n;
      if (i < n)
        for (int j = S::begin(k); j < end; ++j) e = max(e, exponent_of(M[(size_t)j * ld + i]));
      ex[k][i] = (short)e;
      lexp[((size_t)c * nk + k) * ld + i] = (short)e;
    }
  }
  __syncthreads();
  for (int e = i; e < n * ld; e += 256) {
    const int j = e / ld, r = e - j * ld, x = ex[S::cls(j)][r];
    out[(size_t)c * n * ld + e] = x == kNone || x == kPlain ? make_int2(0, 0) : limbs_of(M[e], x);
  }
}

__device__ __forceinline__ double join(long long h, long long m) { return fma((double)h, (double)(1ll << kLimbBits), (double)m); }
// The exponent of a sum of limb products at the scale 2^top
__device__ __forceinline__ int scale_exp(int top) { return top - (2 * kLimbTotal - kLimbBits); }

// (H, M) += (h, m) >> sh, 0 <= sh; returns the part of it in units of H
__device__ __forceinline__ long long merge(long long h, long long m, int sh, long long& H, long long& M) {
  constexpr unsigned mask = (1u << kLimbBits) - 1;
  h += m >> kLimbBits;
  unsigned lo = (unsigned)m & mask;
  for (; sh >= kLimbBits; sh -= kLimbBits) {  // classes that hardly matter
    lo = (unsigned)h & mask;
    h >>= kLimbBits;
  }
  M += (((unsigned)h << (kLimbBits - sh)) & mask) | (lo >> sh);
  h >>= sh;
  H += h;
  return h;
}

// One row in plain FP64
__device__ __forceinline__ double plain_row(const double* M, const int* ic, const double* t, int n, int stride) {
  double y = 0.0;
#pragma unroll 8
  for (int j = 0; j < n; ++j) y = fma(M[(size_t)j * stride], t[ic[j]], y);
  return y;
}

// A warp per cell, eight cells per CTA. Lane l of a warp owns the row pairs l, l + 32, .. (NR of them); batches of three
// columns are loaded PD - 1 ahead, t's limbs stand in the warp's own shared memory. The next cell's t is gathered while
// the present one is streamed.
template <int K, int D>
__global__ void __launch_bounds__(256, kCtas) k_limb_cells(const int4* __restrict__ lim, const short* __restrict__ lexp,
                                                       const double* __restrict__ inv, const int* __restrict__ idx,
                                                       const double* __restrict__ t, double* __restrict__ Y,
                                                       const int* __restrict__ cell_list, int ncells, int ld,
                                                       double* __restrict__ d_scatter, double omega) {
  using S = Cell<K, D>;
  constexpr int n = S::n, nk = S::nk, NR = (n + 63) / 64, NT = 2 * NR, PD = NR == 1 ? 4 : NR == 2 ? 2 : 1;
  // a class's sums stay below 2^63: 27 columns of 2^56 in h and 2^58 in m
  static_assert(S::NV <= 31, "m overflows");
  __shared__ double2 tsh[8][32 * NR];
  __shared__ int te[8][nk];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, LDV = ld / 2;
  int2* tl = reinterpret_cast<int2*>(tsh[warp]);
  int cls[NT];
#pragma unroll
  for (int k = 0; k < NT; ++k) cls[k] = S::cls(min(lane + 32 * k, n - 1));
  auto cell_of = [&](int ci) { return ci < ncells ? (cell_list ? cell_list[ci] : ci) : -1; };
  double tv[NT];
  int at[NT];
  auto lookup = [&](int c) {
#pragma unroll
    for (int k = 0; k < NT; ++k) at[k] = c >= 0 && lane + 32 * k < n ? idx[(long long)c * n + lane + 32 * k] : -1;
  };
  auto gather = [&]() {
#pragma unroll
    for (int k = 0; k < NT; ++k) tv[k] = at[k] >= 0 ? t[at[k]] : 0.0;
  };
  unsigned off[NR];  // lanes beyond the rows repeat the last pair
#pragma unroll
  for (int r = 0; r < NR; ++r) off[r] = (unsigned)min(lane + 32 * r, LDV - 1);
  const int step = gridDim.x * 8;
  int ci = blockIdx.x * 8 + warp, c = cell_of(ci);
  lookup(c);
  gather();
  for (; c >= 0; ci += step) {
    const int4* A = lim + (size_t)c * n * LDV;
    int4 raw[PD][3][NR];
    auto load = [&](int b, int4 (*to)[NR]) {
      const int w = b < S::batches ? S::width(b) : 0;
      const int4* col = A + (unsigned)(S::column(b) * LDV);
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (u < w)
#pragma unroll
          for (int r = 0; r < NR; ++r) to[u][r] = __ldcs(col + u * LDV + off[r]);
    };
#pragma unroll
    for (int p = 0; p < PD - 1; ++p) load(p, raw[p]);
    // t's exponents by class, the scale of the lane's rows
    const short2* ex = reinterpret_cast<const short2*>(lexp + (size_t)c * nk * ld);
    short2 x[nk][NR];
#pragma unroll
    for (int k = 0; k < nk; ++k)
#pragma unroll
      for (int r = 0; r < NR; ++r) x[k][r] = __ldg(ex + k * LDV + off[r]);
    int e[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) e[k] = exponent_of(tv[k]);
    int top[NR][2];
    bool plain = false;
#pragma unroll
    for (int r = 0; r < NR; ++r) top[r][0] = top[r][1] = 2 * kNone;
#pragma unroll
    for (int k = 0; k < nk; ++k) {
      int v = kNone;
#pragma unroll
      for (int q = 0; q < NT; ++q)
        if (cls[q] == k) v = max(v, e[q]);
      v = __reduce_max_sync(0xffffffffu, v);
      if (lane == 0) te[warp][k] = v;
      plain = plain || v == kPlain;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        plain = plain || x[k][r].x == kPlain || x[k][r].y == kPlain;
        top[r][0] = max(top[r][0], x[k][r].x + v);
        top[r][1] = max(top[r][1], x[k][r].y + v);
      }
    }
    plain = __any_sync(0xffffffffu, plain);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NT; ++k) tl[lane + 32 * k] = plain || e[k] == kNone ? make_int2(0, 0) : limbs_of(tv[k], te[warp][cls[k]]);
    __syncwarp();
    const int cn = cell_of(ci + step);
    lookup(cn);
    long long H[NR][2], M[NR][2], h[NR][2], m[NR][2];
    unsigned sum[NR][2];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int v = 0; v < 2; ++v) H[r][v] = M[r][v] = h[r][v] = m[r][v] = 0, sum[r][v] = 0;
    if (!plain) {
#pragma unroll 1
      for (int bb = 0; bb < S::batches; bb += PD)
#pragma unroll
        for (int p = 0; p < PD; ++p) {
          const int b = bb + p;
          if (b >= S::batches) break;
          load(b + PD - 1, raw[(p + PD - 1) % PD]);
          const int w = S::width(b), j = S::column(b);
#pragma unroll
          for (int u = 0; u < 3; ++u)
            if (u < w) {
              const int2 y = tl[j + u];
#pragma unroll
              for (int r = 0; r < NR; ++r) {
                limb_fma(make_int2(raw[p][u][r].x, raw[p][u][r].y), y, h[r][0], m[r][0]);
                limb_fma(make_int2(raw[p][u][r].z, raw[p][u][r].w), y, h[r][1], m[r][1]);
              }
            }
          if (S::last(b)) {
            const int k = S::cls(j), tk = te[warp][k];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              const short2 z = __ldg(ex + k * LDV + off[r]);
#pragma unroll
              for (int v = 0; v < 2; ++v) {
                // one bit lower than the scale, so that 254 columns fit
                const long long q = merge(h[r][v], m[r][v], min(top[r][v] + 1 - (v ? z.y : z.x) - tk, 4 * kLimbBits), H[r][v], M[r][v]);
                sum[r][v] += (unsigned)abs((int)(q >> 32));
                h[r][v] = m[r][v] = 0;
              }
            }
          }
        }
    }
    gather();
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int i = 2 * (lane + 32 * r) + v;
        if (i >= n) continue;
        double y = scale_pow2(join(H[r][v], M[r][v]), scale_exp(top[r][v] + 1));
        if (top[r][v] < kNone / 2) y = 0.0;  // the row or all entries that it meets are zero
        else if (plain || sum[r][v] < (1u << (23 - kSpare)))
          y = plain_row(inv + (size_t)c * n * ld + i, idx + (long long)c * n, t, n, ld);
        if (d_scatter) d_scatter[idx[(long long)c * n + i]] += omega * y;
        else Y[(long long)c * n + i] = y;
      }
    c = cn;
  }
}

template <int K, int D>
stm_status launch_cells(const Level& L, const double* t, const int* cells, int nc, double* scatter, double omega,
                        cudaStream_t s) {
  const int ld = inv_layout(Cell<K, D>::n, STM_F64).ld;
  // as few CTAs as give the same number of rounds, so that none idles through a last partial one
  const int most = kCtas * sm_count(), ctas = (nc + 7) / 8, rounds = (ctas + most - 1) / most;
  k_limb_cells<K, D><<<(ctas + rounds - 1) / rounds, 256, 0, s>>>((const int4*)L.lim, L.lexp, (const double*)L.inv, L.idx,
                                                                  t, L.Y, cells, nc, ld, scatter, omega);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

}  // namespace

// In V-cycles, whose residuals send some rows to the FP64 sums, against the FP64 kernel. 2D, from four fifths of the
// resident warps on (1,945 cells): dG(1), 4,096 cells 29 -> 24 us, 16,384 98 -> 66; dG(2), 2,560 34 -> 32, 4,096 43 -> 35,
// 16,384 150 -> 107. 3D, from one and a half rounds of them on (3,648 cells): dG(0), 2,048 cells 41 -> 48 us, 3,072 70 -> 74,
// 4,608 90 -> 76, 16,384 281 -> 214; dG(1), 2,048 116 -> 130, 3,072 168 -> 204, 4,608 243 -> 234, 16,384 854 -> 680.
bool limb_cells_pay(int dim, int nc) {
  const int warps = 8 * kCtas * sm_count();
  return dim == 2 ? 5 * nc > 4 * warps : 2 * nc > 3 * warps;
}

// The elements whose cells have 32 rows and more and whose inverse is formed at all: 42 and 63 rows in 2D, 85 and 170 in 3D
#define STM_CELLS(L, call)                          \
  switch ((L).dim * 10 + (L).K) {                   \
    case 22: { constexpr int K = 2, D = 2; call; break; } \
    case 23: { constexpr int K = 3, D = 2; call; break; } \
    case 31: { constexpr int K = 1, D = 3; call; break; } \
    case 32: { constexpr int K = 2, D = 3; call; break; } \
    default: break;                                 \
  }

void free_inverse_limbs(Level& L) {
  cudaFree(L.lim);
  cudaFree(L.lexp);
  L.lim = nullptr;
  L.lexp = nullptr;
  L.lim_current = false;
}

// A second copy of the inverses, on the first cell solve after a factorisation. Where it would not leave room for the
// Krylov basis, J^T and something for others the FP64 kernels serve.
stm_status ensure_inverse_limbs(Hierarchy& H, int g, cudaStream_t s) {
  Level& L = H.L[g];
  if (H.p.inv_precision != STM_F64 || L.lim_current || L.lim_off || !L.inv) return STM_OK;
  const int ld = inv_layout(L.n, STM_F64).ld, nk = L.K * (L.dim + 1);
  // the coloured smoother solves on the cells of one colour at a time
  const int nc = H.p.smoother == STM_VANKA_COLOURED ? L.C >> L.dim : L.C;
  if (ld % 2 || L.n < 32 || L.n > 192 || !limb_cells_pay(L.dim, nc)) return STM_OK;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  STM_CUDA(cudaStreamIsCapturing(s, &capture));
  if (capture != cudaStreamCaptureStatusNone) return STM_OK;
  if (!L.lim) {
    const size_t limbs = sizeof(int2) * (size_t)L.C * L.n * ld, exps = sizeof(short) * (size_t)L.C * nk * ld;
    size_t room = 0, all = 0, later = (size_t)2 << 30;
    if (!H.V) later += sizeof(double) * 62 * (size_t)H.L.back().N;
    for (const Level& l : H.L)
      if (!l.valT) later += sizeof(double) * (size_t)(l.nnz + l.nval_cap + l.pval_len);
    STM_CUDA(cudaMemGetInfo(&room, &all));
    if (room < limbs + exps + later || cudaMalloc((void**)&L.lim, limbs) != cudaSuccess ||
        cudaMalloc((void**)&L.lexp, exps) != cudaSuccess) {
      cudaGetLastError();
      free_inverse_limbs(L);
      L.lim_off = true;
      return STM_OK;
    }
  }
  STM_CELLS(L, (k_inverse_limbs<K, D><<<L.C, 256, 0, s>>>((const double*)L.inv, ld, L.lim, L.lexp)));
  note_launch();
  STM_CUDA(cudaGetLastError());
  L.lim_current = true;
  return STM_OK;
}

stm_status vanka_limbs(const Level& L, const double* t, const int* cells, int nc, double* scatter, double omega,
                       cudaStream_t s) {
  STM_CELLS(L, return (launch_cells<K, D>(L, t, cells, nc, scatter, omega, s)));
  set_error("cell solves over limbs: unsupported (dim, k)");
  return STM_ERR_INVALID_ARG;
}

}  // namespace stm
