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
#include <climits>

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
constexpr int kSmallInv = 128;  // up to this size one panel is the whole matrix (144 rows: 0.37 ms against 0.30 blocked)
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
    if (r >= t.m || c >= t.n) continue;
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
// Asynchronous 16-byte store into the shared memory of another CTA of the cluster, counted by its barrier.
__device__ __forceinline__ void remote_store(uint32_t addr, uint32_t bar, uint32_t rank, double v0, double v1) {
  uint32_t ra, rb;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(bar), "r"(rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(ra),
               "l"(__double_as_longlong(v0)), "l"(__double_as_longlong(v1)), "r"(rb)
               : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Waits for the barrier's phase for one second at most; false if it did not come.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  uint32_t done = 0;
  unsigned long long t0 = 0;
  for (int i = 0;; ++i) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    if (done) return true;
    if ((i & 255) == 255) {
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      else if (t - t0 > 1000000000ull) return false;
    }
  }
}
// Lane (of `lanes`) with the largest key, the smallest row among equal keys; every lane of the warp calls.
__device__ __forceinline__ int best_lane(long long key, int row, int lanes) {
  const int lane = threadIdx.x & 31;
  const int hi = lane < lanes ? (int)(key >> 32) : INT_MIN;  // keys are >= -1
  const int mh = __reduce_max_sync(0xffffffffu, hi);
  unsigned m = __ballot_sync(0xffffffffu, hi == mh);
  if (m & (m - 1)) {
    const unsigned lo = hi == mh ? (unsigned)key : 0u;
    const unsigned ml = __reduce_max_sync(0xffffffffu, lo);
    m = __ballot_sync(0xffffffffu, hi == mh && (unsigned)key == ml);
    if (m & (m - 1)) {
      const int r = (m >> lane) & 1u ? row : INT_MAX;
      const int mr = __reduce_min_sync(0xffffffffu, r);
      m = __ballot_sync(0xffffffffu, ((m >> lane) & 1u) && row == mr);
    }
  }
  return __ffs(m) - 1;
}

// Row pitch of the panel in shared memory (odd, so that a column is read without bank conflicts), pitch of the
// rows that are sent (even: 16-byte pieces), and the shared memory of one CTA: two mailboxes (every CTA's
// candidate row, the row to be exchanged, the candidates' keys, reciprocals and rows), its rows, the warps'
// candidates.
__host__ __device__ inline int panel_pitch(int w) { return w | 1; }
__host__ __device__ inline int mail_pitch(int w) { return (w + 1) & ~1; }
__host__ __device__ inline size_t mail_doubles(int nc, int w) { return (size_t)(nc + 1) * mail_pitch(w) + 4 * nc; }
__host__ __device__ inline size_t panel_smem(int nc, int rpc, int w) {
  return sizeof(double) * (2 * mail_doubles(nc, w) + (size_t)rpc * panel_pitch(w)) + 8 * (sizeof(long long) + sizeof(int));
}

// In-place Gauss-Jordan on columns [k0, k0 + w) of the n x n matrix A, rows kept in the shared memory of
// one 16-CTA cluster. Pivot k is the largest entry of column k0 + k among rows >= k0 + k (lowest row on
// ties). Each CTA sends its best row with that row's key and reciprocal pivot to every CTA, by asynchronous
// stores that the receivers' barriers count, so a pivot costs one flight between CTAs and no cluster-wide
// barrier: a CTA goes on when all sixteen have sent. (It cannot run more than one pivot ahead of any other,
// so two mailboxes are enough.) The panel ends as the block transform M: any other column c becomes (c with
// the panel's rows cleared) + M c_panel after the row exchanges. What bounds it: the flight, and an FP64
// instruction that occupies its pipe for 64 clocks (one FMA per row and 32 columns); keys are compared as
// integers, and the next pivot's candidates are taken while the rows are updated. With words set, M is
// also written as the row operand of the update (w <= 32 only). Measured: 1.3 us per pivot at 32 rows (with a
// cluster barrier per pivot 1.8 us), 0.16 ms for a whole 96 x 96 block; blocked inverse of 1125 rows 3.7 ms,
// against 34 ms with one pivot per four launches and 1.23 ms at 99 rows for one CTA's shared memory.
template <int Q, int NC>  // 32-column blocks: w <= 32 Q; CTAs of the cluster
__global__ void __launch_bounds__(256) k_gj_panel(double* __restrict__ A, int n, int k0, int w, int* __restrict__ piv,
                                                  int* flag, uint4* __restrict__ words, int* __restrict__ exps) {
  extern __shared__ __align__(16) double sd[];
  __shared__ __align__(8) unsigned long long bars[2];
  __shared__ int s_late;
  const int rank = (int)cluster_rank();
  const int rpc = (n + NC - 1) / NC, ws = panel_pitch(w), wp = mail_pitch(w);
  const int r0 = min(rank * rpc, n), r1 = min(r0 + rpc, n), nr = r1 - r0;
  // a mailbox: [16][wp] candidate rows, [wp] row k0 + k, [16][2] key and reciprocal, [16][2] row
  const size_t box_len = mail_doubles(NC, w);
  double* P = sd + 2 * box_len;            // [rpc][ws]
  long long* wkey = reinterpret_cast<long long*>(P + (size_t)rpc * ws);  // [8]
  int* widx = reinterpret_cast<int*>(wkey + 8);                          // [8]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t bytes = (uint32_t)(NC * (wp * 8 + 32) + wp * 8);  // received per pivot
  if (tid == 0) {
    s_late = 0;
    for (int i = 0; i < 2; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bars + i)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
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
    double* box = sd + buf * box_len;
    const uint32_t bar = smem_addr(bars + buf);
    // this CTA's candidate: every warp takes the best of the eight (lowest row on ties)
    {
      const long long key = wkey[lane & 7];
      const int row = widx[lane & 7], l = best_lane(key, row, 8);
      bk = __shfl_sync(0xffffffffu, key, l);
      bi = __shfl_sync(0xffffffffu, row, l);
    }
    if (warp == 7) {  // the reciprocal takes longest
      const double inv = bk >= 0 ? 1.0 / P[(size_t)(bi - r0) * ws + k] : 0.0;
      const uint32_t at = smem_addr(box + (size_t)(NC + 1) * wp + 2 * rank);
      if (lane < NC) remote_store(at, bar, lane, __longlong_as_double(bk), inv);
      else if (lane < 2 * NC) remote_store(at + 16 * NC, bar, lane - NC, __longlong_as_double(bi), 0.0);
      if (lane == 0) bar_expect(bar, bytes);
    } else {
      const bool mine = gk >= r0 && gk < r1;
      const int h = wp >> 1;  // 16-byte pieces of a row
      for (int e = tid; e < NC * h; e += 224) {
        const int d = Q == 1 && w == 32 ? e >> 4 : e / h, j = 2 * (e - d * h);
        double c0 = 0.0, c1 = 0.0;
        if (bk >= 0) {
          c0 = P[(size_t)(bi - r0) * ws + j];
          if (j + 1 < w) c1 = P[(size_t)(bi - r0) * ws + j + 1];
        }
        remote_store(smem_addr(box + (size_t)rank * wp + j), bar, d, c0, c1);
        if (mine) {
          const double o0 = P[(size_t)(gk - r0) * ws + j], o1 = j + 1 < w ? P[(size_t)(gk - r0) * ws + j + 1] : 0.0;
          remote_store(smem_addr(box + (size_t)NC * wp + j), bar, d, o0, o1);
        }
      }
    }
    if (!bar_wait(bar, (k >> 1) & 1)) s_late = 1;
    const double* cand = box + (size_t)(NC + 1) * wp;
    int who;
    {
      const long long key = __double_as_longlong(cand[2 * (lane & (NC - 1))]);
      const int row = (int)__double_as_longlong(cand[2 * NC + 2 * (lane & (NC - 1))]);
      who = best_lane(key, row, NC);
      bk = __shfl_sync(0xffffffffu, key, who);
      bi = __shfl_sync(0xffffffffu, row, who);
    }
    const int p = bi;
    // the same decision in every CTA of the cluster
    if (bk <= 0 || bk >= 0x7FF0000000000000ll) {
      if (rank == 0 && tid == 0) {
        atomicExch(flag, 1);
        for (int q = k; q < w; ++q) piv[k0 + q] = k0 + q;
      }
      break;
    }
    // after a wait that ran out the row may be anything: what follows indexes with it
    if (rank == 0 && tid == 0) piv[gk] = p >= gk && p < n ? p : gk;
    const double* prow = box + (size_t)who * wp;
    const double* krow = box + (size_t)NC * wp;
    const double pinv = cand[2 * who + 1];
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
    if (s_late) {  // a CTA that does not hear from the others gives up, and then they do
      if (tid == 0) atomicExch(flag, 1);
      for (int q = k + 1 + tid; rank == 0 && q < w; q += 256) piv[k0 + q] = k0 + q;
      break;
    }
  }
  for (int i = warp; i < nr; i += 8)
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = 32 * q + lane;
      if (j < w) A[(long long)(r0 + i) * n + k0 + j] = P[(size_t)i * ws + j];
    }
  if (Q == 1 && words) {  // [16-row tile][16 positions][4][32 lanes], two neighbouring positions per word set
    for (int i = warp; i < nr; i += 8) {
      const int r = r0 + i;
      const double v = lane < w ? P[(size_t)i * ws + lane] : 0.0;
      const int e = __reduce_max_sync(0xffffffffu, exp_above(v));
      const bool bad = e > 1024;
      if (bad && lane == 0) atomicExch(flag, 1);
      const unsigned long long pk = digits_of(bad ? 0.0 : v, e);
      const unsigned long long nx = __shfl_down_sync(0xffffffffu, pk, 1);
      if (!(lane & 1)) {
        const int pp = lane >> 1;
        words[((r >> 4) * 2 + (pp >> 3)) * 128 + (((r >> 3) & 1) + 2 * ((pp >> 2) & 1)) * 32 + (r & 7) * 4 + (pp & 3)] =
            words_of(pk, nx);
      }
      if (lane == 0) exps[r] = e;
    }
  }
  cluster_sync();  // no CTA leaves while another may still write into its mailbox
}

// The row exchanges of one panel on the columns [c0, c1) without the panel's own and without [x0, x1), and the
// panel's rows as the column operand of the update ([pair][column] word sets, scaled per column). One thread
// per column; the exchanges are first composed into source rows, so that all loads of a column are
// independent.
__global__ void __launch_bounds__(128) k_gj_rows(double* __restrict__ A, int n, int k0, int w, const int* __restrict__ piv,
                                                 int c0, int c1, int x0, int x1, int* flag, uint4* __restrict__ words,
                                                 int pitch, int* __restrict__ exps) {
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
  const int j = c0 + blockIdx.x * 128 + threadIdx.x;
  if (j >= c1 || (j >= k0 && j < k0 + w) || (j >= x0 && j < x1)) return;
  double v[kPanel], t[kPanel];
#pragma unroll
  for (int k = 0; k < kPanel; ++k) {
    v[k] = k < w ? A[(long long)top[k] * n + j] : 0.0;
    t[k] = dst[k] >= 0 ? A[(long long)src[k] * n + j] : 0.0;
  }
  int e = kExpZero;
#pragma unroll
  for (int k = 0; k < kPanel; ++k) e = max(e, exp_above(v[k]));
  const bool bad = e > 1024;
  if (bad) atomicExch(flag, 1);
#pragma unroll
  for (int k = 0; k < kPanel; ++k)
    if (dst[k] >= 0) A[(long long)dst[k] * n + j] = t[k];
#pragma unroll
  for (int k = 0; k < kPanel; k += 2)
    words[(long long)(k >> 1) * pitch + j] = words_of(digits_of(bad ? 0.0 : v[k], e), digits_of(bad ? 0.0 : v[k + 1], e));
  exps[j] = e;
}

constexpr int kUpCols = 48;  // columns per warp of the update

// C = (C with the panel's rows cleared) + M R on the columns [c0, c1) without the panel's own and without [x0, x1): a
// warp takes 16 rows and 48 columns with M's digits in registers; the next eight columns' operands and
// entries are loaded while the present ones are multiplied. At 1125 rows that is one wave of twelve warps
// per SM.
__global__ void __launch_bounds__(128, 3) k_gj_update(double* __restrict__ A, int n, int k0, int w,
                                                      const uint4* __restrict__ mw, const int* __restrict__ em,
                                                      const uint4* __restrict__ rw, const int* __restrict__ er, int pitch,
                                                      int c0, int c1, int x0, int x1) {
  const int lane = threadIdx.x & 31, nq = lane >> 2, q = lane & 3;
  const int groups = (c1 - c0 + kUpCols - 1) / kUpCols, tiles = (n + 15) / 16;
  const int un = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (un >= groups * tiles) return;
  const int mt = un / groups, j0 = c0 + (un - mt * groups) * kUpCols, j1 = min(j0 + kUpCols, c1);
  uint32_t a[2][kDig][4];
#pragma unroll
  for (int kk = 0; kk < 2; ++kk)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint4 x = __ldg(mw + (mt * 2 + kk) * 128 + k * 32 + lane);
      const uint32_t xx[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int d = 0; d < kDig; ++d) a[kk][d][k] = digit_pair(xx[d & 3], d >= 4);
    }
  const int r0 = 16 * mt + nq, e0 = em[min(r0, n - 1)], e8 = em[min(r0 + 8, n - 1)];
  auto live = [&](int j) { return j < j1 && (j < k0 || j >= k0 + w) && (j < x0 || j >= x1); };
  uint4 nx[4];
  double nc[4];
  auto load = [&](int jb) {
    const int jc = min(jb + nq, c1 - 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) nx[k] = __ldg(rw + (long long)(4 * k + q) * pitch + jc);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int r = r0 + (m < 2 ? 0 : 8), j = jb + 2 * q + (m & 1);
      nc[m] = r < n && live(j) && (r < k0 || r >= k0 + w) ? A[(long long)r * n + j] : 0.0;
    }
  };
  load(j0);
#pragma unroll 1
  for (int jb = j0; jb < j1; jb += 8) {
    uint4 y[4] = {nx[0], nx[1], nx[2], nx[3]};
    double cv[4] = {nc[0], nc[1], nc[2], nc[3]};
    if (jb + 8 < j1) load(jb + 8);
    float acc[kDig][4];
#pragma unroll
    for (int d = 0; d < kDig; ++d)
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[d][m] = kSumZero;
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      const uint32_t y0[4] = {y[2 * kk].x, y[2 * kk].y, y[2 * kk].z, y[2 * kk].w};
      const uint32_t y1[4] = {y[2 * kk + 1].x, y[2 * kk + 1].y, y[2 * kk + 1].z, y[2 * kk + 1].w};
#pragma unroll
      for (int o = 0; o < kDig; ++o) {
        const uint32_t b0 = digit_pair(y0[o & 3], o >= 4), b1 = digit_pair(y1[o & 3], o >= 4);
#pragma unroll
        for (int d = 0; d + o < kDig; ++d) mma_f16(acc[d + o], a[kk][d][0], a[kk][d][1], a[kk][d][2], a[kk][d][3], b0, b1);
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int r = r0 + (m < 2 ? 0 : 8), j = jb + 2 * q + (m & 1);
      if (r >= n || !live(j)) continue;
      // sums of 8 pairs x 32 terms, products at most 2^14 (2^13 where a leading digit takes part)
      long long hi, lo;
      join_sums(acc, m, hi, lo);
      const int ea = m < 2 ? e0 : e8, eb = er[j];
      if (ea != kExpZero && eb != kExpZero) cv[m] += join_pow2(hi, lo, ea + eb - 124 + 56);
      A[(long long)r * n + j] = cv[m];
    }
  }
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

template <int Q, int NC>
stm_status launch_panel(double* A, int n, int k0, int w, int* piv, int* flag, uint4* words, int* exps, cudaStream_t s) {
  const size_t smem = panel_smem(NC, (n + NC - 1) / NC, w);
  STM_CUDA(cudaFuncSetAttribute(k_gj_panel<Q, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  STM_CUDA(cudaFuncSetAttribute(k_gj_panel<Q, NC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(NC);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = NC;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  STM_CUDA(cudaLaunchKernelEx(&cfg, k_gj_panel<Q, NC>, A, n, k0, w, piv, flag, words, exps));
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
  // two buffers of M's and of the panel rows' words: 64 halves per row and column each, twice
  STM_TRY(dense_reserve(w, 0, 2 * n + 64, kPanel));
  STM_TRY(dense_reserve(w, 1, kPanel, 2 * n + 2 * kUpCols));
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
  if (w.side) cudaStreamDestroy(w.side);
  for (cudaEvent_t e : w.ev)
    if (e) cudaEventDestroy(e);
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

// Panel k + 1 needs only its own columns of update k: those come first, on s, and the other columns are updated on
// w.side while panel k + 1 runs. Operands alternate between two buffers, since update k may still read its own
// when panel k + 1 writes; the columns of panel k + 2 wait for update k. Where the caller allows no second stream
// (w.overlap) all of it runs on s: once two streams have run in a context, every launch after that costs a little
// more, for good (a 2D adjoint solve of 13 iterations: 5.43 -> 5.68 ms), and one update of all columns costs a 2D
// Newton step no more than two side by side (58.1 against 59.5 ms). The slab chains of 3D use two streams anyway
// (dG(0) step: 43.5 -> 39.1 ms with the overlap).
stm_status dense_inverse(DenseWork& w, double* A, int n, double* out, int* flag, cudaStream_t s) {
  if (n <= kSmallInv) {
    if (n <= 32) STM_TRY((launch_panel<1, 4>(A, n, 0, n, w.piv, flag, nullptr, nullptr, s)));
    else if (n <= 64) STM_TRY((launch_panel<2, 8>(A, n, 0, n, w.piv, flag, nullptr, nullptr, s)));
    else if (n <= 96) STM_TRY((launch_panel<3, kCluster>(A, n, 0, n, w.piv, flag, nullptr, nullptr, s)));
    else STM_TRY((launch_panel<kSmallInv / 32, kCluster>(A, n, 0, n, w.piv, flag, nullptr, nullptr, s)));
  } else {
    if (w.overlap) {
      if (!w.side) STM_CUDA(cudaStreamCreateWithFlags(&w.side, cudaStreamNonBlocking));
      for (cudaEvent_t& e : w.ev)
        if (!e) STM_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    }
    const int pitch = up(n, kUpCols), tiles = (n + 15) / 16;
    const long long mwords = 256LL * tiles, rwords = 16LL * pitch;
    auto update = [&](int k0, int pw, int par, int c0, int c1, int x0, int x1, cudaStream_t st) -> stm_status {
      uint4 *mw = (uint4*)w.dig[0] + par * mwords, *rw = (uint4*)w.dig[1] + par * rwords;
      int *em = w.exps[0] + par * n, *er = w.exps[1] + par * n;
      k_gj_rows<<<(c1 - c0 + 127) / 128, 128, sizeof(int) * n, st>>>(A, n, k0, pw, w.piv, c0, c1, x0, x1, flag, rw, pitch, er);
      note_launch();
      const int units = tiles * ((c1 - c0 + kUpCols - 1) / kUpCols);
      k_gj_update<<<(units + 3) / 4, 128, 0, st>>>(A, n, k0, pw, mw, em, rw, er, pitch, c0, c1, x0, x1);
      note_launch();
      STM_CUDA(cudaGetLastError());
      return STM_OK;
    };
    for (int k0 = 0, k = 0; k0 < n; k0 += kPanel, ++k) {
      const int pw = std::min(kPanel, n - k0), next = k0 + pw, nend = std::min(next + kPanel, n);
      const int par = w.overlap ? k & 1 : 0;
      STM_TRY((launch_panel<1, kCluster>(A, n, k0, pw, w.piv, flag, (uint4*)w.dig[0] + par * mwords, w.exps[0] + par * n, s)));
      if (!w.overlap) {
        STM_TRY(update(k0, pw, par, 0, n, n, n, s));
        continue;
      }
      STM_CUDA(cudaEventRecord(w.ev[0], s));
      if (k > 0) STM_CUDA(cudaStreamWaitEvent(s, w.ev[1], 0));  // update k - 1 is through
      STM_CUDA(cudaStreamWaitEvent(w.side, w.ev[0], 0));
      STM_TRY(update(k0, pw, par, 0, n, next, nend, w.side));
      STM_CUDA(cudaEventRecord(w.ev[1], w.side));
      if (next < n) STM_TRY(update(k0, pw, par, next, nend, n, n, s));
    }
    if (w.overlap) STM_CUDA(cudaStreamWaitEvent(s, w.ev[1], 0));
  }
  k_gj_compose<<<1, 1024, 2 * sizeof(unsigned short) * n, s>>>(w.piv, n, w.from);
  note_launch();
  k_gj_columns<<<std::min(n, sm_count() * 8), 256, 0, s>>>(A, n, w.from, out);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

}  // namespace stm
