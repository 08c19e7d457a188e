// Dense FP64 blocks of the coarse factorisation on the tensor cores: matrix products and inverses.
//
// FP64 arithmetic on this device issues 2 FMAs per clock and SM (1.25 TFLOP/s), while FP16 tensor
// instructions with FP32 accumulators run near 600 TFLOP/s from mma.sync. A product C = A B is
// therefore formed from digits: every row of A and every column of B is scaled by its own power of two
// to 63-bit integers and cut into eight balanced base-256 digits (-128 .. 127, exact in FP16). Digit
// products are at most 2^14, so up to 2^10 of them add up exactly in an FP32 accumulator; the 36 digit
// pairs (s, t) with s + t <= 7 are accumulated per weight s + t, and the eight sums are joined in 64-bit
// integers every 128 terms. The only errors are the digits left out, below 2^-60 of (row maximum x
// column maximum) per term, and one rounding of the result to FP64, against one rounding per term of an
// FMA chain. Measured on 1125 x 1125 x 1125: 0.34 ms (36 x 2.85 GFLOP of digit products; 2.1 waves of
// tiles) and 0.035 ms for cutting both operands, against 3.3 ms for a tiled FP64 kernel; error 6e-17
// |A||B| against 1.3e-15 of an FMA chain.
#include <cfloat>

#include "digits.h"
#include "internal.h"

namespace stm {
namespace {

constexpr int kTileM = 64, kTileN = 48, kTileK = 32;
constexpr int kStages = 3;
constexpr int kGemmThreads = 384;  // 4 x 3 warps, one 16 x 16 tile each
constexpr int kRowB = 112;         // bytes of one k-row of B in shared memory (96 used): conflict-free
constexpr int kStageA = kDig * kTileM * kTileK * 2;  // 32 KB
constexpr int kStageB = kDig * kTileK * kRowB;       // 28 KB
constexpr int kPanel = 32;   // pivots per panel of the blocked inverse
constexpr int kSmallInv = 192;  // up to this size one panel is the whole matrix
constexpr int kCluster = 16;
constexpr int kPanelRows = 512;    // panel rows per CTA at most: 32 columns fill 130 KB

struct SliceTask {
  const double* src;   // rows x cols, row-major
  long long ld;
  int rows, cols;
  __half* out;         // [8][...][pitch]
  long long plane;     // elements per digit plane
  int pitch;           // row operand: padded columns (K); column operand: padded columns (N)
  int kpad;            // column operand: padded rows (K)
  int* exps;           // [rows] or [cols]
};
struct SliceTasks {
  SliceTask t[6];
};

// Row operand: one warp per row, scaled by the row's largest entry; columns up to `pitch` are zero.
__global__ void __launch_bounds__(256) k_slice_rows(const __grid_constant__ SliceTasks ts, int* flag) {
  const SliceTask& t = ts.t[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row >= t.rows) return;
  const double* a = t.src + row * t.ld;
  int e = kExpZero;
  for (int j = lane; j < t.cols; j += 32) e = max(e, exp_above(a[j]));
  for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  const bool bad = e > 1024;
  if (lane == 0) {
    t.exps[row] = e;
    if (bad) atomicExch(flag, 1);
  }
  __half* o = t.out + row * t.pitch;
  for (int j = 2 * lane; j < t.pitch; j += 64) {
    const unsigned long long p0 = digits_of(j < t.cols && !bad ? a[j] : 0.0, e);
    const unsigned long long p1 = digits_of(j + 1 < t.cols && !bad ? a[j + 1] : 0.0, e);
#pragma unroll
    for (int d = 0; d < kDig; ++d)
      *reinterpret_cast<__half2*>(o + d * t.plane + j) = __halves2half2(digit_half(p0, d), digit_half(p1, d));
  }
}

// Column operand, two passes so that both fill the chip: the largest exponent of every column (one CTA per
// 64 columns and 64 rows, two adjacent columns per lane, joined by atomicMax over kExpZero), then the
// digits; rows from `rows` to `kpad` are zero.
__global__ void __launch_bounds__(256) k_col_exps(const __grid_constant__ SliceTasks ts) {
  const SliceTask& t = ts.t[blockIdx.z];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = blockIdx.x * 64 + 2 * lane, rb = blockIdx.y * 64;
  if (blockIdx.x * 64 >= t.cols || rb >= t.rows) return;
  __shared__ int red[8][64];
  const bool l0 = c0 < t.cols, l1 = c0 + 1 < t.cols;
  int e0 = kExpZero, e1 = kExpZero;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int r = rb + warp + 8 * q;
    if (r >= t.rows) break;
    const double* a = t.src + (long long)r * t.ld + c0;
    if (l0) e0 = max(e0, exp_above(a[0]));
    if (l1) e1 = max(e1, exp_above(a[1]));
  }
  red[warp][2 * lane] = e0;
  red[warp][2 * lane + 1] = e1;
  __syncthreads();
  if (threadIdx.x < 64 && blockIdx.x * 64 + threadIdx.x < t.cols) {
    int e = kExpZero;
#pragma unroll
    for (int q = 0; q < 8; ++q) e = max(e, red[q][threadIdx.x]);
    if (e != kExpZero) atomicMax(t.exps + blockIdx.x * 64 + threadIdx.x, e);
  }
}
__global__ void __launch_bounds__(256) k_slice_cols(const __grid_constant__ SliceTasks ts, int* flag) {
  const SliceTask& t = ts.t[blockIdx.z];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = blockIdx.x * 64 + 2 * lane;
  if (c0 >= t.pitch) return;
  const bool l0 = c0 < t.cols, l1 = c0 + 1 < t.cols;
  const int e0 = l0 ? t.exps[c0] : kExpZero, e1 = l1 ? t.exps[c0 + 1] : kExpZero;
  const bool b0 = e0 > 1024, b1 = e1 > 1024;
  if (b0 || b1) atomicExch(flag, 1);
#pragma unroll 2
  for (int q = 0; q < 4; ++q) {
    const int r = blockIdx.y * 32 + warp + 8 * q;
    if (r >= t.kpad) break;
    const double* a = t.src + (long long)r * t.ld + c0;
    const bool in = r < t.rows;
    const unsigned long long p0 = digits_of(in && l0 && !b0 ? a[0] : 0.0, e0);
    const unsigned long long p1 = digits_of(in && l1 && !b1 ? a[1] : 0.0, e1);
    __half* o = t.out + (long long)r * t.pitch + c0;
#pragma unroll
    for (int d = 0; d < kDig; ++d)
      *reinterpret_cast<__half2*>(o + d * t.plane) = __halves2half2(digit_half(p0, d), digit_half(p1, d));
  }
}

struct GemmTask {
  const __half *A, *B;      // digits [8][m rows][kp] and [8][kp][np]
  long long pa, pb;         // elements per plane
  const int *ea, *eb;       // exponents per row of A, per column of B
  int m, n, kp, np;
  double alpha;             // +-1
  const double* C0;         // added (row-major, ldc0) unless null
  long long ldc0;
  double* C;                // row-major, ldc; trans: C[j * ldc + i]
  long long ldc;
  int trans;
  int skip0, skip1;         // columns in [skip0, skip1) are not written
};
struct GemmTasks {
  GemmTask t[4];
  int tiles[5];  // first tile of each task
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void ldsm4(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// C = [C0] + alpha A B from digits. 64 x 48 tile per CTA, 12 warps of 16 x 16; per 16 terms a warp loads
// its eight A and eight B digit fragments once and issues 72 MMAs, so the tensor pipe is the limit (a
// 64 x 64 tile with sixteen warps has no room for the eight weights' accumulators). Operand tiles of
// 32 terms come through a three-stage cp.async ring.
__global__ void __launch_bounds__(kGemmThreads) k_digit_gemm(const __grid_constant__ GemmTasks ts) {
  extern __shared__ __align__(128) unsigned char sm[];
  int ti = 0;
  while (ti < 3 && (int)blockIdx.x >= ts.tiles[ti + 1]) ++ti;
  const GemmTask& t = ts.t[ti];
  const int tile = blockIdx.x - ts.tiles[ti];
  const int tn = (t.n + kTileN - 1) / kTileN;
  const int m0 = (tile / tn) * kTileM, n0 = (tile % tn) * kTileN;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = (warp & 3) * 16, wn = (warp >> 2) * 16;
  const uint32_t sbase = smem_addr(sm);
  const int nk = t.kp / kTileK;

  auto load = [&](int st, int kc) {
    const uint32_t sa = sbase + st * (kStageA + kStageB), sb = sa + kStageA;
    // A: 8 planes x 64 rows x 4 chunks of 16 bytes; chunk c of row r at c ^ ((r >> 1) & 3)
    for (int e = threadIdx.x; e < kDig * kTileM * 4; e += kGemmThreads) {
      const int c = e & 3, r = (e >> 2) & (kTileM - 1), p = e >> 8;
      const int row = min(m0 + r, t.m - 1);
      cp16(sa + ((p * kTileM + r) * 4 + (c ^ ((r >> 1) & 3))) * 16,
           t.A + p * t.pa + (long long)row * t.kp + kc * kTileK + c * 8);
    }
    // B: 8 planes x 32 k-rows x 6 chunks
    for (int e = threadIdx.x; e < kDig * kTileK * 6; e += kGemmThreads) {
      const int c = e % 6, r = (e / 6) & (kTileK - 1), p = e / (6 * kTileK);
      cp16(sb + (p * kTileK + r) * kRowB + c * 16,
           t.B + p * t.pb + (long long)(kc * kTileK + r) * t.np + n0 + c * 8);
    }
  };

  float acc[kDig][8];
  long long hi[8], lo[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) hi[i] = lo[i] = 0;
#pragma unroll
  for (int d = 0; d < kDig; ++d)
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[d][i] = 0.f;

#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (s < nk) load(s, s);
    asm volatile("cp.async.commit_group;");
  }
  for (int kc = 0; kc < nk; ++kc) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2));
    __syncthreads();
    if (kc + kStages - 1 < nk) load((kc + kStages - 1) % kStages, kc + kStages - 1);
    asm volatile("cp.async.commit_group;");
    const uint32_t sa = sbase + (kc % kStages) * (kStageA + kStageB), sb = sa + kStageA;
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      uint32_t a[kDig][4];
      const int ar = wm + ((lane >> 3) & 1) * 8 + (lane & 7), ac = kk * 2 + (lane >> 4);
      const int br = kk * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), bc = wn / 8 + (lane >> 4);
#pragma unroll
      for (int d = 0; d < kDig; ++d)
        ldsm4(a[d], sa + ((d * kTileM + ar) * 4 + (ac ^ ((ar >> 1) & 3))) * 16);
#pragma unroll
      for (int tt = 0; tt < kDig; ++tt) {
        uint32_t b[4];
        ldsm4t(b, sb + (tt * kTileK + br) * kRowB + bc * 16);
#pragma unroll
        for (int s = 0; s + tt < kDig; ++s) {
          mma_f16(acc[s + tt], a[s][0], a[s][1], a[s][2], a[s][3], b[0], b[1]);
          mma_f16(acc[s + tt] + 4, a[s][0], a[s][1], a[s][2], a[s][3], b[2], b[3]);
        }
      }
    }
    // 128 terms x 8 pairs x 2^14 = 2^24: the FP32 sums are still exact; join them
    if ((kc & 3) == 3 || kc == nk - 1) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        long long h = 0, l = 0;
#pragma unroll
        for (int d = 0; d < 4; ++d) {
          h = h * 256 + __float2int_rn(acc[d][i]);
          l = l * 256 + __float2int_rn(acc[d + 4][i]);
          acc[d][i] = 0.f;
          acc[d + 4][i] = 0.f;
        }
        hi[i] += h;
        lo[i] += l;
      }
    }
  }
  asm volatile("cp.async.wait_group 0;");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = m0 + wm + (lane >> 2) + ((i & 2) ? 8 : 0);
    const int c = n0 + wn + (i >> 2) * 8 + (lane & 3) * 2 + (i & 1);
    if (r >= t.m || c >= t.n || (c >= t.skip0 && c < t.skip1)) continue;
    const int ea = t.ea[r], eb = t.eb[c];  // value: hi 2^(ea + eb - 36) + lo 2^(ea + eb - 68)
    double v = 0.0;
    if (ea != kExpZero && eb != kExpZero) v = t.alpha * scale_pow2(fma((double)hi[i], 4294967296.0, (double)lo[i]), ea + eb - 68);
    if (t.C0) v += t.C0[(long long)r * t.ldc0 + c];
    if (t.trans) t.C[(long long)c * t.ldc + r] = v;
    else t.C[(long long)r * t.ldc + c] = v;
  }
}

// ---------------------------------------------------------------------------------------------
// Inverse of an n x n block: blocked Gauss-Jordan with partial pivoting
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void remote_store(uint32_t addr, uint32_t rank, double v) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t addr, uint32_t rank, int v) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(ra), "r"(v) : "memory");
}

// Row pitch of the panel in shared memory (odd, so that a column is read without bank conflicts) and the
// shared memory of one CTA: its rows, two mailboxes (every CTA's candidate row, the row to be exchanged, the
// candidates' keys, rows and reciprocals) and the warps' candidates.
__host__ __device__ inline int panel_pitch(int w) { return w | 1; }
__host__ __device__ inline size_t panel_smem(int rpc, int w) {
  return sizeof(double) * ((size_t)rpc * panel_pitch(w) + 2 * (size_t)(kCluster + 1) * w) +
         2 * kCluster * (sizeof(long long) + sizeof(double) + sizeof(int)) + 8 * (sizeof(long long) + sizeof(int));
}
// |v| as an integer key that orders like |v|; NaN orders below everything
__device__ __forceinline__ long long abs_key(double v) {
  const long long k = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll;
  return k > 0x7FF0000000000000ll ? -1 : k;
}
// 1 / a: the hardware's approximation and two Newton steps, four dependent FP64 operations
__device__ __forceinline__ double reciprocal(double a) {
  const int ex = (__double2hiint(a) >> 20) & 0x7FF;
  if (ex < 64 || ex > 1982) return 1.0 / a;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  r = fma(r, fma(-a, r, 1.0), r);
  return fma(r, fma(-a, r, 1.0), r);
}

// In-place Gauss-Jordan on columns [k0, k0 + w) of the n x n matrix A, rows kept in the shared memory of
// one 16-CTA cluster. Pivot k is the largest entry of column k0 + k among rows >= k0 + k (lowest row on
// ties). Each CTA pushes its best row and that row's reciprocal pivot into every CTA's mailbox before the
// one cluster barrier of the pivot, so the winner is known and at hand everywhere after it. The panel ends
// as the block transform M: any other column c becomes (c with the panel's rows cleared) + M c_panel after
// the row exchanges. What bounds it: an FP64 instruction occupies its pipe for 64 clocks, so per pivot the
// update (one FMA per row and 32 columns), the reciprocal and the barrier follow one another; keys are
// compared as integers, and the next pivot's candidates are taken while the rows are updated. With digits
// set, M is also written as a row operand of the digit product (w <= 32 only). Measured: 5.1 ms for the
// inverse of a 1125 x 1125 block (36 panels of 32), 0.27 ms at 99 x 99 (one panel), against 34 ms with one
// pivot per four launches and 1.23 ms for a Gauss-Jordan in one CTA's shared memory.
template <int Q>  // 32-column blocks: w <= 32 Q
__global__ void __launch_bounds__(256) k_gj_panel(double* __restrict__ A, int n, int k0, int w, int* __restrict__ piv,
                                                  int* flag, __half* __restrict__ dig, long long plane,
                                                  int* __restrict__ exps) {
  extern __shared__ __align__(16) double sd[];
  const int rank = (int)cluster_rank();
  const int rpc = (n + kCluster - 1) / kCluster, ws = panel_pitch(w);
  const int r0 = min(rank * rpc, n), r1 = min(r0 + rpc, n), nr = r1 - r0;
  double* P = sd;                          // [rpc][ws]
  double* mail = P + (size_t)rpc * ws;     // [2][17][w]: candidate rows, then row k0 + k
  long long* ckey = reinterpret_cast<long long*>(mail + 2 * (size_t)(kCluster + 1) * w);  // [2][16]
  double* cinv = reinterpret_cast<double*>(ckey + 2 * kCluster);                           // [2][16]
  long long* wkey = reinterpret_cast<long long*>(cinv + 2 * kCluster);                     // [8]
  int* cidx = reinterpret_cast<int*>(wkey + 8);                                            // [2][16]
  int* widx = cidx + 2 * kCluster;                                                         // [8]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // candidate of this warp's rows for column k0 (later columns: while the rows are updated)
  long long bk = -1;
  int bi = n;
  for (int i = warp; i < nr; i += 8)
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = 32 * q + lane;
      if (j < w) {
        const double v = A[(long long)(r0 + i) * n + k0 + j];
        P[(size_t)i * ws + j] = v;
        if (q == 0 && lane == 0 && r0 + i >= k0 && abs_key(v) > bk) {
          bk = abs_key(v);
          bi = r0 + i;
        }
      }
    }
  if (lane == 0) {
    wkey[warp] = bk;
    widx[warp] = bi;
  }
  cluster_sync();
  for (int k = 0; k < w; ++k) {
    const int gk = k0 + k, buf = k & 1;
    double* box = mail + (size_t)buf * (kCluster + 1) * w;
    // this CTA's candidate: every warp takes the best of the eight (lowest row on ties)
    bk = wkey[lane & 7];
    bi = widx[lane & 7];
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
      const long long ok = __shfl_xor_sync(0xffffffffu, bk, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
    }
    const bool mine = gk >= r0 && gk < r1;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = 32 * q + lane;
      const double cand = bk >= 0 && j < w ? P[(size_t)(bi - r0) * ws + j] : 0.0;
      const double old = mine && j < w ? P[(size_t)(gk - r0) * ws + j] : 0.0;
      if (j < w)
#pragma unroll
        for (int d = 0; d < kCluster; d += 8) {
          if (bk >= 0) remote_store(smem_addr(box + (size_t)rank * w + j), d + warp, cand);
          if (mine) remote_store(smem_addr(box + (size_t)kCluster * w + j), d + warp, old);
        }
    }
    if (warp == 7) {
      const double inv = bk >= 0 ? reciprocal(P[(size_t)(bi - r0) * ws + k]) : 0.0;
      if (lane < kCluster) {
        remote_store(smem_addr(ckey + buf * kCluster + rank), lane, __longlong_as_double(bk));
        remote_store(smem_addr(cinv + buf * kCluster + rank), lane, inv);
        remote_store(smem_addr(cidx + buf * kCluster + rank), lane, bi);
      }
    }
    cluster_sync();
    bk = ckey[buf * kCluster + (lane & 15)];
    bi = cidx[buf * kCluster + (lane & 15)];
    int who = lane & 15;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
      const long long ok = __shfl_xor_sync(0xffffffffu, bk, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      const int ow = __shfl_xor_sync(0xffffffffu, who, off);
      if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; who = ow; }
    }
    const int p = bi;
    if (bk <= 0 || bk >= 0x7FF0000000000000ll) {  // the same decision in every CTA of the cluster
      if (rank == 0 && tid == 0) {
        atomicExch(flag, 1);
        for (int q = k; q < w; ++q) piv[k0 + q] = k0 + q;
      }
      break;
    }
    if (rank == 0 && tid == 0) piv[gk] = p;
    const double* prow = box + (size_t)who * w;
    const double* krow = box + (size_t)kCluster * w;
    const double pinv = cinv[buf * kCluster + who];
    // one warp per row, lanes over the columns: row p takes the old row k0 + k, row k0 + k the scaled
    // pivot row, every other row loses its multiple of it; column k becomes the transform's column
    // (0 - f pinv), so one FMA serves all columns
    double u[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = 32 * q + lane;
      u[q] = j == k ? pinv : j < w ? prow[j] * pinv : 0.0;
    }
    bk = -1;
    bi = n;
    for (int i = warp; i < nr; i += 8) {
      const int gi = r0 + i;
      double* row = P + (size_t)i * ws;
      const double* c = gi == p ? krow : row;
      const double f = -c[k];
      double v[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int j = 32 * q + lane;
        v[q] = j == k || j >= w ? 0.0 : c[j];
      }
      __syncwarp();  // every lane has read the multiplier before column k is overwritten
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int j = 32 * q + lane;
        const double nv = gi == gk ? u[q] : fma(f, u[q], v[q]);
        if (j < w) row[j] = nv;
        if (j == k + 1 && gi > gk && abs_key(nv) > bk) {  // strict: the lowest row wins ties
          bk = abs_key(nv);
          bi = gi;
        }
      }
    }
    if (((k + 1) & 31) == lane) {
      wkey[warp] = bk;
      widx[warp] = bi;
    }
    __syncthreads();
  }
  for (int i = warp; i < nr; i += 8)
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = 32 * q + lane;
      if (j < w) A[(long long)(r0 + i) * n + k0 + j] = P[(size_t)i * ws + j];
    }
  if (Q == 1 && dig) {
    for (int i = warp; i < nr; i += 8) {
      const double v = lane < w ? P[(size_t)i * ws + lane] : 0.0;
      int e = exp_above(v);
      for (int off = 16; off > 0; off >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
      const bool bad = e > 1024;
      if (bad && lane == 0) atomicExch(flag, 1);
      const unsigned long long pk = digits_of(bad ? 0.0 : v, e);
#pragma unroll
      for (int d = 0; d < kDig; ++d) dig[d * plane + (long long)(r0 + i) * kPanel + lane] = digit_half(pk, d);
      if (lane == 0) exps[r0 + i] = e;
    }
  }
  cluster_sync();  // no CTA leaves while another may still write into its mailbox
}

// The row exchanges of one panel on every other column, the panel's rows as a column operand of the digit
// product (scaled per column), and zeros in their place. One thread per column; the exchanges are first
// composed into source rows, so that all loads of a column are independent.
__global__ void __launch_bounds__(128) k_gj_rows(double* __restrict__ A, int n, int k0, int w, const int* __restrict__ piv,
                                                 int* flag, __half* __restrict__ dig, long long plane, int pitch,
                                                 int* __restrict__ exps) {
  extern __shared__ int at[];  // at[r]: row that now sits at r
  for (int r = threadIdx.x; r < n; r += 128) at[r] = r;
  __shared__ int dst[kPanel], src[kPanel], top[kPanel];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0; k < w; ++k) {
      const int p = piv[k0 + k], a = at[k0 + k];
      at[k0 + k] = at[p];
      at[p] = a;
    }
  __syncthreads();
  if (threadIdx.x < kPanel) {
    const int k = threadIdx.x;
    const int p = k < w ? piv[k0 + k] : k0;
    top[k] = k < w ? at[k0 + k] : k0;
    const bool out = k < w && p >= k0 + w;  // rows of the panel itself are covered by top
    dst[k] = out ? p : -1;
    src[k] = out ? at[p] : k0;
  }
  __syncthreads();
  const int j = blockIdx.x * 128 + threadIdx.x;
  if (j >= pitch) return;
  const bool live = j < n && (j < k0 || j >= k0 + w);
  double v[kPanel], t[kPanel];
#pragma unroll
  for (int k = 0; k < kPanel; ++k) {
    v[k] = live && k < w ? A[(long long)top[k] * n + j] : 0.0;
    t[k] = live && dst[k] >= 0 ? A[(long long)src[k] * n + j] : 0.0;
  }
  int e = kExpZero;
#pragma unroll
  for (int k = 0; k < kPanel; ++k) e = max(e, exp_above(v[k]));
  const bool bad = e > 1024;
  if (bad) atomicExch(flag, 1);
#pragma unroll
  for (int k = 0; k < kPanel; ++k) {
    if (live && k < w) A[(long long)(k0 + k) * n + j] = 0.0;
    if (live && dst[k] >= 0) A[(long long)dst[k] * n + j] = t[k];
  }
#pragma unroll
  for (int k = 0; k < kPanel; ++k) {
    const unsigned long long pk = digits_of(bad ? 0.0 : v[k], e);
#pragma unroll
    for (int d = 0; d < kDig; ++d) dig[d * plane + (long long)k * pitch + j] = digit_half(pk, d);
  }
  if (j < n) exps[j] = e;
}

// Undo the row exchanges as column exchanges, last first: out[:, j] = A[:, from[j]].
__global__ void k_gj_compose(const int* __restrict__ piv, int n, int* __restrict__ from) {
  extern __shared__ unsigned short sc[];
  unsigned short *at = sc, *pv = sc + n;
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    at[r] = (unsigned short)r;
    pv[r] = (unsigned short)piv[r];
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = n - 1; k >= 0; --k) {
      const unsigned short p = pv[k], a = at[k];
      at[k] = at[p];
      at[p] = a;
    }
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += blockDim.x) from[r] = at[r];
}
__global__ void k_gj_columns(const double* __restrict__ A, int n, const int* __restrict__ from, double* __restrict__ out) {
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int j = threadIdx.x; j < n; j += blockDim.x) out[(long long)i * n + j] = A[(long long)i * n + from[j]];
}

int up(int v, int m) { return (v + m - 1) / m * m; }

constexpr int kMaxCluster = kCluster * kPanelRows;  // rows of the largest block inverted by clusters

template <int Q>
stm_status launch_panel(double* A, int n, int k0, int w, int* piv, int* flag, __half* dig, long long plane, int* exps,
                        cudaStream_t s) {
  const size_t smem = panel_smem((n + kCluster - 1) / kCluster, w);
  STM_CUDA(cudaFuncSetAttribute(k_gj_panel<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  STM_CUDA(cudaFuncSetAttribute(k_gj_panel<Q>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kCluster);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kCluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  STM_CUDA(cudaLaunchKernelEx(&cfg, k_gj_panel<Q>, A, n, k0, w, piv, flag, dig, plane, exps));
  note_launch();
  return STM_OK;
}

template <typename T>
bool grow(T*& p, long long& have, long long want) {
  if (have >= want) return true;
  if (p) cudaFree(p);
  p = nullptr;
  have = 0;
  if (cudaMalloc((void**)&p, sizeof(T) * (size_t)want) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  have = want;
  return true;
}

}  // namespace

long long dense_max_inverse() { return kMaxCluster; }

stm_status dense_reserve(DenseWork& w, int slot, long long rows, long long cols) {
  const long long halves = (long long)kDig * (up((int)rows, kTileK) + kTileK) * (up((int)cols, kTileN) + kTileN);
  __half* d = reinterpret_cast<__half*>(w.dig[slot]);
  const bool ok = grow(d, w.halves[slot], halves) && grow(w.exps[slot], w.nexp[slot], std::max(rows, cols));
  w.dig[slot] = d;
  if (!ok) {
    set_error("coarse factorisation: out of device memory");
    return STM_ERR_OOM;
  }
  return STM_OK;
}

stm_status dense_reserve_inverse(DenseWork& w, long long n) {
  STM_TRY(dense_reserve(w, 0, n, kPanel));
  STM_TRY(dense_reserve(w, 1, kPanel, n));
  if (!grow(w.tmp, w.ntmp, n * n) || !grow(w.piv, w.npiv, n) || !grow(w.from, w.nfrom, n)) {
    set_error("coarse factorisation: out of device memory");
    return STM_ERR_OOM;
  }
  return STM_OK;
}

void dense_free(DenseWork& w) {
  for (int i = 0; i < DenseWork::kSlots; ++i) {
    cudaFree(w.dig[i]);
    cudaFree(w.exps[i]);
  }
  cudaFree(w.tmp);
  cudaFree(w.piv);
  cudaFree(w.from);
  w = DenseWork{};
}

stm_status dense_slice(DenseWork& w, const DenseSlice* sl, int count, int* flag, cudaStream_t s) {
  SliceTasks tr{}, tc{};
  int nr = 0, nc = 0, gr = 0, gc = 0, gk = 0;
  for (int i = 0; i < count; ++i) {
    const DenseSlice& d = sl[i];
    if (d.rows <= 0 || d.cols <= 0) continue;
    SliceTask t{};
    t.src = d.src;
    t.ld = d.ld;
    t.rows = d.rows;
    t.cols = d.cols;
    t.out = reinterpret_cast<__half*>(w.dig[d.slot]);
    t.exps = w.exps[d.slot];
    if (d.column) {
      t.pitch = up(d.cols, kTileN);
      t.kpad = up(d.rows, kTileK);
      t.plane = (long long)t.kpad * t.pitch;
      tc.t[nc++] = t;
      gc = std::max(gc, (t.pitch + 63) / 64);
      gk = std::max(gk, t.kpad);
    } else {
      t.pitch = up(d.cols, kTileK);
      t.plane = (long long)d.rows * t.pitch;
      tr.t[nr++] = t;
      gr = std::max(gr, (d.rows + 7) / 8);
    }
  }
  if (nr) {
    k_slice_rows<<<dim3(gr, nr), 256, 0, s>>>(tr, flag);
    note_launch();
  }
  if (nc) {
    for (int i = 0; i < nc; ++i) STM_CUDA(cudaMemsetAsync(tc.t[i].exps, kExpZero & 0xFF, sizeof(int) * tc.t[i].cols, s));
    k_col_exps<<<dim3(gc, (gk + 63) / 64, nc), 256, 0, s>>>(tc);
    note_launch();
    k_slice_cols<<<dim3(gc, gk / 32, nc), 256, 0, s>>>(tc, flag);
    note_launch();
  }
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

stm_status dense_products(const DenseWork& w, const DenseProduct* pr, int count, cudaStream_t s) {
  GemmTasks g{};
  int used = 0, tiles = 0;
  for (int i = 0; i < count; ++i) {
    const DenseProduct& p = pr[i];
    if (p.m <= 0 || p.n <= 0) continue;
    GemmTask t{};
    t.A = reinterpret_cast<const __half*>(w.dig[p.a]);
    t.B = reinterpret_cast<const __half*>(w.dig[p.b]);
    t.ea = w.exps[p.a];
    t.eb = w.exps[p.b];
    t.m = p.m;
    t.n = p.n;
    t.kp = up(p.k, kTileK);
    t.np = up(p.n, kTileN);
    t.pa = (long long)p.m * t.kp;
    t.pb = (long long)t.kp * t.np;
    t.alpha = p.alpha;
    t.C0 = p.C0;
    t.ldc0 = p.ldc0;
    t.C = p.C;
    t.ldc = p.ldc;
    t.trans = p.trans;
    t.skip0 = p.skip0;
    t.skip1 = p.skip1;
    g.t[used] = t;
    g.tiles[used++] = tiles;
    tiles += ((p.m + kTileM - 1) / kTileM) * ((p.n + kTileN - 1) / kTileN);
  }
  if (!used) return STM_OK;
  for (int i = used; i < 5; ++i) g.tiles[i] = tiles;
  const int smem = kStages * (kStageA + kStageB);
  STM_CUDA(cudaFuncSetAttribute(k_digit_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  k_digit_gemm<<<tiles, kGemmThreads, smem, s>>>(g);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

stm_status dense_inverse(DenseWork& w, double* A, int n, double* out, int* flag, cudaStream_t s) {
  if (n <= kSmallInv) {
    if (n <= 32) STM_TRY(launch_panel<1>(A, n, 0, n, w.piv, flag, nullptr, 0, nullptr, s));
    else if (n <= 96) STM_TRY(launch_panel<3>(A, n, 0, n, w.piv, flag, nullptr, 0, nullptr, s));
    else STM_TRY(launch_panel<kSmallInv / 32>(A, n, 0, n, w.piv, flag, nullptr, 0, nullptr, s));
  } else {
    __half *dm = reinterpret_cast<__half*>(w.dig[0]), *dr = reinterpret_cast<__half*>(w.dig[1]);
    const int pitch = up(n, kTileN);
    for (int k0 = 0; k0 < n; k0 += kPanel) {
      const int pw = std::min(kPanel, n - k0);
      STM_TRY(launch_panel<1>(A, n, k0, pw, w.piv, flag, dm, (long long)n * kPanel, w.exps[0], s));
      k_gj_rows<<<(pitch + 127) / 128, 128, sizeof(int) * n, s>>>(A, n, k0, pw, w.piv, flag, dr,
                                                                  (long long)kPanel * pitch, pitch, w.exps[1]);
      note_launch();
      STM_CUDA(cudaGetLastError());
      DenseProduct p;
      p.a = 0;
      p.b = 1;
      p.m = p.n = n;
      p.k = kPanel;
      p.C0 = p.C = A;
      p.ldc0 = p.ldc = n;
      p.skip0 = k0;
      p.skip1 = k0 + pw;
      STM_TRY(dense_products(w, &p, 1, s));
    }
  }
  k_gj_compose<<<1, 1024, 2 * sizeof(unsigned short) * n, s>>>(w.piv, n, w.from);
  note_launch();
  k_gj_columns<<<std::min(n, sm_count() * 8), 256, 0, s>>>(A, n, w.from, out);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

}  // namespace stm
