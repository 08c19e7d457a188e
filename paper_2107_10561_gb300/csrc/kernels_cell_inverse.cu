// Cell inverses J_T^{-1} (Sec. 4.3): after each Jacobian update the inverse of every cell's local Jacobian, the
// rows and columns of the ASSEMBLED global matrix on the cell's DoFs (Sec. 4.4), stored column-major per cell
// in FP64, FP32 or BF16.
//
// Pressure rows and columns are inverted near the size of the velocity ones (pressure_scale): without it the residual
// |A B - I| of an inverse against |A||B| grew with falling time steps (3D dG(0): 6e-15 at tau = 1e-2, 2e-10 at 1e-8;
// with it 1e-15 and 4e-15).
// One CTA per cell: blocked Gauss-Jordan elimination with partial pivoting (largest |pivot| in the column,
// lowest row on ties), 16 pivots per panel. A panel runs in shared memory on the FP64 pipe and ends as a block
// transform M; after the panel's row exchanges every other column c becomes (c with the panel's rows
// cleared) + M c_panel. That product runs on the tensor cores over base-256 digits (digits.h: the rows of M
// and the columns of c_panel scaled by powers of two, the 43 digit pairs above 2^-70: with the 36 above 2^-62
// the residual of 85-row cells was 6e-15 against 1e-15 by FP64 FMAs), so the FP64 pipe (2 FMAs per clock and SM) carries 16 n^2 / 2 + n^2 / 16 x n operations instead of n^3. The matrix sits in
// shared memory where it fits beside the operands, else in a scratch block that L2 holds for the most part.
// Measured, 2,016 cells of 170 x 170: 25.0 -> 9.6 ms; 21,420 cells of 63 x 63: 14.7 -> 9.3 ms (a Gauss-
// Jordan with n^3 FP64 FMAs in shared memory before). What bounds it now are chains of dependent instructions
// at 16 warps per SM (issue slots 46 % used, FP64 pipe 42 %): 2.5 million warp instructions per 170 x 170 cell,
// half of them in the update (43 MMAs, 32 to form digits and about 200 to join the sums and add them, per 16 x 8
// entries).
#include "digits.h"
#include "internal.h"

namespace stm {
namespace {

constexpr int kPanel = 16;
constexpr int kPitch = kPanel + 1;

template <typename S> __device__ __forceinline__ S to_store(double v);
template <> __device__ __forceinline__ double to_store<double>(double v) { return v; }
template <> __device__ __forceinline__ float to_store<float>(double v) { return (float)v; }
template <> __device__ __forceinline__ __nv_bfloat16 to_store<__nv_bfloat16>(double v) {
  return __ushort_as_bfloat16((unsigned short)bf16_bits_rn(v));  // one rounding, straight from FP64
}

// Position in the CSR values of J_g of the entry (local row al, local col be) of cell c.
__device__ __forceinline__ long long entry_pos(int c, int al, int be, const int* __restrict__ idx,
                                               const int* __restrict__ cell_nodes,
                                               const unsigned char* __restrict__ rank,
                                               const unsigned char* __restrict__ cellrank,
                                               const int* __restrict__ nn, const int* __restrict__ ncell,
                                               const long long* __restrict__ rowptr, int d, int nv,
                                               int np, int nt, int n) {
  const int a = al / nt, ra = al - a * nt;
  const int b = be / nt, rb = be - b * nt;
  const long long row = idx[(long long)c * n + al];
  const int dnv = d * nv;
  if (ra < dnv) {
    const int i = ra % nv;
    const int node = cell_nodes[(long long)c * nv + i];
    const int nni = nn[node];
    if (rb < dnv) {
      const int m = rb / nv, j = rb - m * nv;
      return rowptr[row] + (long long)b * d * nni + (b > a ? np * ncell[node] : 0) + (long long)m * nni +
             rank[((long long)c * nv + i) * nv + j];
    }
    if (b != a) return -1;
    const int q = rb - dnv;
    return rowptr[row] + (long long)a * d * nni + (long long)d * nni + (long long)cellrank[(long long)c * nv + i] * np + q;
  }
  if (rb >= dnv || b != a) return -1;
  return rowptr[row] + rb;  // pressure row: columns (a, m, j) in order m * nv + j
}

struct CellArgs {
  const int *idx, *cell_nodes, *nn, *ncell;
  const unsigned char *rank, *cellrank;
  const long long* rowptr;
  const double* val;
  int C, d, nv, np, nt, n, ld;
  double scale;     // of the pressure rows and columns while the matrix is inverted
  double* scratch;  // [CTAs][n * n], or null: the matrix is kept in shared memory
  int* flag;
  long long* bad;
};

// Shared memory: panel, operands, their exponents, candidates, row bookkeeping, the matrix
struct CellSmem {
  int tiles, cols, pitch;  // 16-row tiles, 8-column tiles, pitch of the column operand
  size_t words_m, words_r, exps, keys, rows, matrix, total;
};
__host__ __device__ inline CellSmem cell_smem(int n, bool matrix) {
  CellSmem s;
  s.tiles = (n + 15) / 16;
  s.cols = (n + 7) / 8;
  s.pitch = 8 * s.cols + 2;  // eight lanes of a read meet eight groups of banks
  // the column operand takes the place of the panel, which is done when it is formed
  size_t o = sizeof(double) * (size_t)n * kPitch;
  o = (o + 15) / 16 * 16;
  s.words_r = 0;
  if (o < sizeof(uint4) * 8 * (size_t)s.pitch) o = sizeof(uint4) * 8 * (size_t)s.pitch;
  s.words_m = o;
  o += sizeof(uint4) * 128 * (size_t)s.tiles;
  s.exps = o;
  o += sizeof(int) * (16 * (size_t)s.tiles + 8 * (size_t)s.cols);
  s.keys = o = (o + 15) / 16 * 16;
  o += 8 * (sizeof(long long) + sizeof(int)) + 2 * kPanel * sizeof(double);
  s.rows = o = (o + 15) / 16 * 16;
  o += sizeof(int) * (2 * (size_t)n + 3 * kPanel);
  s.matrix = o = (o + 15) / 16 * 16;
  if (matrix) o += sizeof(double) * (size_t)n * n;
  s.total = o;
  return s;
}

template <typename S, int kThreads>
__global__ void __launch_bounds__(kThreads, 512 / kThreads) k_cell_inverse(const __grid_constant__ CellArgs g, S* __restrict__ inv) {
  constexpr int kWarps = kThreads / 32;
  extern __shared__ __align__(16) unsigned char sm[];
  const int n = g.n, dnv = g.d * g.nv;
  const CellSmem L = cell_smem(n, g.scratch == nullptr);
  double* P = reinterpret_cast<double*>(sm);                 // [n][17]: the panel
  uint4* wm = reinterpret_cast<uint4*>(sm + L.words_m);      // [tiles][4][32]: M as row operand
  uint4* wr = reinterpret_cast<uint4*>(sm + L.words_r);      // [8 pairs][pitch]: the panel's rows as column operand
  int* em = reinterpret_cast<int*>(sm + L.exps);             // [16 tiles]
  int* ec = em + 16 * L.tiles;                               // [8 cols]
  double* ubuf = reinterpret_cast<double*>(sm + L.keys);     // [16] scaled pivot row
  double* kbuf = ubuf + kPanel;                              // [16] row to be exchanged
  long long* wkey = reinterpret_cast<long long*>(kbuf + kPanel);
  int* widx = reinterpret_cast<int*>(wkey + 8);
  int* at = reinterpret_cast<int*>(sm + L.rows);             // [n] row that now sits at r; at the end columns
  int* piv = at + n;                                         // [n]
  int *top = piv + n, *dst = top + kPanel, *src = dst + kPanel;
  double* A = g.scratch ? g.scratch + (size_t)blockIdx.x * n * n : reinterpret_cast<double*>(sm + L.matrix);  // column-major
  __shared__ int s_bad, s_piv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int half = lane >> 4, j16 = lane & 15;  // panel: two rows per warp instruction
  const int nq = lane >> 2, q = lane & 3;       // MMA fragments

  for (int c = blockIdx.x; c < g.C; c += gridDim.x) {
    __syncthreads();
    if (tid == 0) s_bad = 0;
    for (int e0 = tid; e0 < n * n; e0 += 4 * kThreads) {  // four look-ups in flight
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int e = e0 + k * kThreads, be = e / n, al = e - be * n;
        v[k] = 0.0;
        if (e < n * n) {
          const long long pos = entry_pos(c, al, be, g.idx, g.cell_nodes, g.rank, g.cellrank, g.nn, g.ncell, g.rowptr,
                                          g.d, g.nv, g.np, g.nt, n);
          if (pos >= 0) v[k] = __ldg(g.val + pos);
          if (al % g.nt >= dnv) v[k] *= g.scale;
          if (be % g.nt >= dnv) v[k] *= g.scale;
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (e0 + k * kThreads < n * n) A[e0 + k * kThreads] = v[k];
    }
    for (int p0 = 0; p0 < n; p0 += kPanel) {
      const int w = min(kPanel, n - p0);
      __syncthreads();
      // the panel; candidates of its first column
      for (int e = tid; e < n * kPanel; e += kThreads) {
        const int j = e / n, i = e - j * n;
        P[i * kPitch + j] = j < w ? A[(size_t)(p0 + j) * n + i] : 0.0;
      }
      for (int i = tid; i < n; i += kThreads) at[i] = i;
      __syncthreads();
      long long bk = -1;
      int bi = n;
      for (int i = p0 + tid; i < n; i += kThreads) {
        const long long k = abs_key(P[i * kPitch]);
        if (k > bk) { bk = k; bi = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
      }
      if (lane == 0) {
        wkey[warp] = bk;
        widx[warp] = bi;
      }
      __syncthreads();
      bool singular = false;  // the same for all threads: read between two barriers that enclose no write
      for (int k = 0; k < w; ++k) {
        const int gk = p0 + k;
        if (warp == 0) {
          bk = wkey[lane & (kWarps - 1)];
          bi = widx[lane & (kWarps - 1)];
#pragma unroll
          for (int o = kWarps / 2; o > 0; o >>= 1) {
            const long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
          }
          if (bk <= 0 || bk >= 0x7FF0000000000000ll) {
            if (lane == 0) s_bad = 1;
          } else {
            const double pr = P[bi * kPitch + j16], inv1 = 1.0 / P[bi * kPitch + k];
            if (lane < kPanel) {
              kbuf[lane] = P[gk * kPitch + lane];
              ubuf[lane] = lane == k ? inv1 : pr * inv1;
            }
            if (lane == 0) {
              s_piv = bi;
              piv[gk] = bi;
              const int a = at[gk];
              at[gk] = at[bi];
              at[bi] = a;
              src[k] = bi;  // the panel's exchanges in order
            }
          }
        }
        __syncthreads();
        singular = s_bad != 0;
        if (singular) break;
        const int p = s_piv;
        const double u = ubuf[j16];
        bk = -1;
        bi = n;
        constexpr int RB = 4;  // row pairs whose loads are in flight together
        for (int i0 = 2 * warp; i0 < n; i0 += 2 * kWarps * RB) {
          double f[RB], v[RB];
#pragma unroll
          for (int b = 0; b < RB; ++b) {
            const int i = i0 + 2 * kWarps * b + half;
            const double* row = i < n && i != p ? P + i * kPitch : kbuf;
            f[b] = -row[k];
            v[b] = j16 == k ? 0.0 : row[j16];
          }
          __syncwarp();  // every lane has read the multipliers before column k is overwritten
#pragma unroll
          for (int b = 0; b < RB; ++b) {
            const int i = i0 + 2 * kWarps * b + half;
            const double nv = i == gk ? u : fma(f[b], u, v[b]);
            if (i < n) {
              P[i * kPitch + j16] = nv;
              if (j16 == k + 1 && i > gk && abs_key(nv) > bk) {
                bk = abs_key(nv);
                bi = i;
              }
            }
          }
        }
        {  // the two halves hold alternate rows
          const long long ok = __shfl_xor_sync(0xffffffffu, bk, 16);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, 16);
          if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
          if (lane == ((k + 1) & 15)) {
            wkey[warp] = bk;
            widx[warp] = bi;
          }
        }
        __syncthreads();
      }
      // not s_bad: threads that are through the pivots may already set it for a row of M that is not finite
      if (singular) break;
      // M back into the matrix and as a row operand: a warp per 16-row tile, lane = (row, position pairs)
      for (int e = tid; e < n * w; e += kThreads) {
        const int j = e / n, i = e - j * n;
        A[(size_t)(p0 + j) * n + i] = P[i * kPitch + j];
      }
      for (int r = warp * 4 + (lane >> 3); r < 16 * L.tiles; r += kWarps * 4) {  // eight lanes per row
        const int pp = lane & 7;
        const double a = r < n ? P[r * kPitch + 2 * pp] : 0.0, b = r < n ? P[r * kPitch + 2 * pp + 1] : 0.0;
        int e = max(exp_above(a), exp_above(b));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
        const bool ok = e <= 1024;
        if (!ok) s_bad = 1;
        if (pp == 0) em[r] = e;
        wm[((r >> 4) * 4 + ((r >> 3) & 1) + 2 * (pp >> 2)) * 32 + (r & 7) * 4 + (pp & 3)] =
            words_of(digits_of(ok ? a : 0.0, e), digits_of(ok ? b : 0.0, e));
      }
      if (tid < kPanel) {
        const int k = tid;
        const int p = k < w ? src[k] : 0;
        top[k] = k < w ? at[p0 + k] : 0;
        dst[k] = k < w && p >= p0 + w ? p : -1;  // rows of the panel itself are covered by top
      }
      __syncthreads();
      // row exchanges of every other column, and the panel's rows as a column operand: half a warp per column
      const int to = dst[j16], from = to >= 0 ? at[to] : 0, head = top[j16];
      constexpr int EB = 4;  // columns whose loads are in flight together
      for (int j0 = 2 * warp; j0 < 8 * L.cols; j0 += 2 * kWarps * EB) {
        double v[EB], t[EB];
#pragma unroll
        for (int b = 0; b < EB; ++b) {
          const int j = j0 + 2 * kWarps * b + half;
          const bool live = j < n && (j < p0 || j >= p0 + w);
          const double* col = A + (size_t)(live ? j : 0) * n;
          v[b] = live && j16 < w ? col[head] : 0.0;
          t[b] = live && to >= 0 ? col[from] : 0.0;
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < EB; ++b) {
          const int j = j0 + 2 * kWarps * b + half;
          if (j < n && (j < p0 || j >= p0 + w) && to >= 0) A[(size_t)j * n + to] = t[b];
          int e = exp_above(v[b]);
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
          const bool ok = e <= 1024;
          if (!ok) s_bad = 1;
          const unsigned long long pk = digits_of(ok ? v[b] : 0.0, e);
          const unsigned long long nx = __shfl_down_sync(0xffffffffu, pk, 1);
          if (j < 8 * L.cols) {
            if (!(j16 & 1)) wr[(j16 >> 1) * L.pitch + j] = words_of(pk, nx);
            if (j16 == 0) ec[j] = e;
          }
        }
      }
      __syncthreads();
      if (s_bad) break;
      // C = (C with the panel's rows cleared) + M R on every other column: a warp takes a 16-row tile and half
      // of the 8-column tiles
      const int nh = (L.cols + 1) / 2;
      for (int un = warp; un < 2 * L.tiles; un += kWarps) {
        const int mt = un >> 1, t0 = (un & 1) * nh, t1 = (un & 1) ? L.cols : nh;
        uint32_t a[kDig][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint4 x = wm[(mt * 4 + k) * 32 + lane];
          const uint32_t xx[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int d = 0; d < kDig; ++d) a[d][k] = digit_pair(xx[d & 3], d >= 4);
        }
        const int r0 = 16 * mt + nq, e0 = em[r0], e8 = em[r0 + 8];
        // the next tile's column operand and entries are loaded while this one is multiplied
        uint4 nx0, nx1;
        double nc[4];
        auto load = [&](int ct) {
          nx0 = wr[q * L.pitch + 8 * ct + nq];
          nx1 = wr[(q + 4) * L.pitch + 8 * ct + nq];
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int r = r0 + (m < 2 ? 0 : 8), j = 8 * ct + 2 * q + (m & 1);
            nc[m] = r < n && j < n && (r < p0 || r >= p0 + w) ? A[(size_t)j * n + r] : 0.0;
          }
        };
        load(t0);
#pragma unroll 1
        for (int ct = t0; ct < t1; ++ct) {
          const uint32_t y0[4] = {nx0.x, nx0.y, nx0.z, nx0.w}, y1[4] = {nx1.x, nx1.y, nx1.z, nx1.w};
          double cv[4] = {nc[0], nc[1], nc[2], nc[3]};
          if (ct + 1 < t1) load(ct + 1);
          float acc[kDig + 1][4];
#pragma unroll
          for (int d = 0; d <= kDig; ++d)
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[d][m] = kSumZero;
#pragma unroll
          for (int o = 0; o < kDig; ++o) {
            const uint32_t b0 = digit_pair(y0[o & 3], o >= 4), b1 = digit_pair(y1[o & 3], o >= 4);
#pragma unroll
            for (int d = 0; d < kDig && d + o <= kDig; ++d) mma_f16(acc[d + o], a[d][0], a[d][1], a[d][2], a[d][3], b0, b1);
          }
          const int ec0 = ec[8 * ct + 2 * q], ec1 = ec[8 * ct + 2 * q + 1];
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int r = r0 + (m < 2 ? 0 : 8), j = 8 * ct + 2 * q + (m & 1);
            // sums of at most 8 pairs x 16 terms x 2^14
            long long hi, lo;
            join_sums(acc, m, hi, lo);
            lo += (__float_as_int(acc[kDig][m]) - 0x4B400000 + 128) >> 8;  // the next digit's pairs, rounded
            const int er = m < 2 ? e0 : e8, ecj = (m & 1) ? ec1 : ec0;
            if (er != kExpZero && ecj != kExpZero) cv[m] += join_pow2(hi, lo, er + ecj - 124 + 56);
            if (r < n && j < n && (j < p0 || j >= p0 + w)) A[(size_t)j * n + r] = cv[m];
          }
        }
      }
    }
    __syncthreads();
    if (s_bad) {
      if (tid == 0 && atomicCAS(g.flag, 0, 1) == 0) *g.bad = c;
      continue;
    }
    // the row interchanges come off as column interchanges, last first
    for (int i = tid; i < n; i += kThreads) at[i] = i;
    __syncthreads();
    if (tid == 0)
      for (int k = n - 1; k >= 0; --k) {
        const int p = piv[k], a = at[k];
        at[k] = at[p];
        at[p] = a;
      }
    __syncthreads();
    S* out = inv + (size_t)c * n * g.ld;
    for (int e0 = tid; e0 < n * g.ld; e0 += 4 * kThreads) {
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int e = e0 + k * kThreads, j = e / g.ld, i = e - j * g.ld;  // column-major store: element (i, j) at j * ld + i
        v[k] = e < n * g.ld && i < n ? A[(size_t)at[j] * n + i] : 0.0;
        if (i % g.nt >= dnv) v[k] *= g.scale;
        if (j % g.nt >= dnv) v[k] *= g.scale;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (e0 + k * kThreads < n * g.ld) out[e0 + k * kThreads] = to_store<S>(v[k]);
    }
  }
}

size_t storage_bytes(int prec) { return prec == STM_F64 ? 8 : prec == STM_F32 ? 4 : 2; }

template <typename S, int T>
stm_status launch(const CellArgs& a, void* inv, int blocks, size_t smem, cudaStream_t s) {
  STM_CUDA(cudaFuncSetAttribute(k_cell_inverse<S, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_cell_inverse<S, T><<<blocks, T, smem, s>>>(a, (S*)inv);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}
template <int T>
stm_status launch(const Hierarchy& H, const CellArgs& a, void* inv, int blocks, size_t smem, cudaStream_t s) {
  if (H.p.inv_precision == STM_F64) return launch<double, T>(a, inv, blocks, smem, s);
  if (H.p.inv_precision == STM_F32) return launch<float, T>(a, inv, blocks, smem, s);
  return launch<__nv_bfloat16, T>(a, inv, blocks, smem, s);
}

}  // namespace

stm_status factor_level(Hierarchy& H, int g, cudaStream_t s) {
  Level& L = H.L[g];
  const int n = L.n;
  const InvLayout lay = inv_layout(n, H.p.inv_precision);
  if (!L.inv) STM_TRY(device_alloc(H, &L.inv, storage_bytes(H.p.inv_precision) * (size_t)n * lay.ld * L.C));
  int dev = 0, maxsm = 0;
  STM_CUDA(cudaGetDevice(&dev));
  STM_CUDA(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  if (sizeof(double) * (size_t)n * n + sizeof(short) * n + 80 > (size_t)maxsm) {
    set_error("factor_cells: cell matrix does not fit in shared memory");
    return STM_ERR_INVALID_ARG;
  }
  CellArgs a{L.idx, L.cell_nodes, L.nn, L.ncell, L.rank, L.cellrank, L.rowptr, L.val, L.C, L.dim, L.nv, L.np, L.nt,
             n, lay.ld, pressure_scale(H, L), nullptr, H.dflag, H.dbad};
  // small blocks: four CTAs of four warps per SM, so that one's panel steps fill another's barriers; the
  // matrix in shared memory where that many fit, else in scratch
  const int per_sm = n <= 96 ? 4 : 2;
  const bool in_smem = per_sm * (cell_smem(n, true).total + 1024) <= (size_t)maxsm;
  const int blocks = std::min(L.C, per_sm * sm_count());
  if (!in_smem && H.cell_scratch_len < (long long)blocks * n * n) {
    if (H.cell_scratch) cudaFree(H.cell_scratch);
    H.cell_scratch = nullptr;
    H.cell_scratch_len = 0;
    STM_TRY(device_alloc(H, &H.cell_scratch, sizeof(double) * (size_t)blocks * n * n));
    H.cell_scratch_len = (long long)blocks * n * n;
  }
  const size_t smem = cell_smem(n, in_smem).total;
  a.scratch = in_smem ? nullptr : H.cell_scratch;
  if (per_sm == 4) STM_TRY(launch<128>(H, a, L.inv, blocks, smem, s));
  else STM_TRY(launch<256>(H, a, L.inv, blocks, smem, s));
  L.lim_current = L.lim_off = false;
  return STM_OK;
}

}  // namespace stm
