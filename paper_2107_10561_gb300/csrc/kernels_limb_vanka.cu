// Cell solves y_T = J_T^{-1} t_T (or with the transpose) over FP64 inverses, on the INT32 pipe.
//
// Every entry of an inverse is read once and needs one multiply-add; in FP64 that takes 74 clocks per warp
// instruction and sub-core, while HBM delivers the next 256 bytes after 44. The inverses are therefore kept a second
// time as two-limb integers (limbs.h), each row at a scale of its own, which takes 13 clocks. On 16,128 cells of 2D
// dG(2) (528 MB) a launch takes 91 us, 76 % of the copy rate, where the FP64 kernel took 150; whole sweeps: 243 ->
// 181 us, 2D dG(1) 156 -> 104, 3D dG(0) 449 -> 375, 3D dG(1) (2,016 cells) 195 -> 159. Cutting the FP64 values into
// limbs as they are read instead took 126 us.
//   - A warp per cell, whole lines per load; lanes own row pairs and t's limbs are broadcast from shared memory, so
//     a column costs a load, a shared load and six multiply-adds per lane. Several warps per cell (each a block of
//     columns, sums joined in FP64) where cells are fewer than resident warps.
//   - t is cut below the largest entry of the cell, the pressure columns with one offset per cell against the
//     velocity columns. Against the FP64 kernel results differ by 2e-16 to 1e-15 of the largest entry.
//   - The transpose goes a thread per column (2D dG(2) 236 us as in FP64, 3D dG(0) 413 -> 384, dG(1) 217 -> 186).
//   - Cells with an infinity, a NaN or a scale near the ends of the exponent range, in the inverse or in t, are
//     summed in FP64 from the FP64 inverses, which the 32-column products and the copy to the host read anyway.
//   - Cells of fewer than 32 rows (2D dG(0): 21) stay with the FP64 kernel: 11 of 32 lanes would own rows (63 against
//     65 us per sweep, and 38 against 35 on 4,032 cells). So do levels without room for the second copy.
#include "digits.h"
#include "internal.h"
#include "limbs.h"

namespace stm {
namespace {

constexpr int kNone = -(1 << 20);  // biased exponent where every entry is zero
constexpr int kPlain = 1 << 20;    // pressure offset of a cell whose inverse holds an infinity, a NaN or tiny rows

__device__ __forceinline__ int biased(double v) {
  const int hi = __double2hiint(v) & 0x7FFFFFFF;
  return (hi | __double2loint(v)) == 0 ? kNone : hi >> 20;
}

// Limbs of a cell's inverse in the layout of the inverse, each row at the biased exponent of its largest velocity
// column, the pressure columns delta above; lexp: [C][n + 1], the rows' exponents and delta. One CTA per cell.
__global__ void __launch_bounds__(256) k_inverse_limbs(const double* __restrict__ inv, int n, int ld, int nt, int nvel,
                                                       int2* __restrict__ out, int* __restrict__ lexp) {
  __shared__ int row[256], offset, bad;
  const int c = blockIdx.x, i = threadIdx.x;
  const double* M = inv + (size_t)c * n * ld;
  if (i == 0) offset = kNone, bad = 0;
  __syncthreads();
  if (i < n) {
    int ev = kNone, ep = kNone;
    for (int k = 0, r = 0; k < n; ++k) {
      const int e = biased(M[(size_t)k * ld + i]);
      if (r < nvel) ev = max(ev, e);
      else ep = max(ep, e);
      if (++r == nt) r = 0;
    }
    const int most = max(ev, ep);
    if (most >= 2047 || (most != kNone && most < 128)) bad = 1;
    if (ev == kNone) ev = ep == kNone ? 1023 : ep;
    if (ep != kNone) atomicMax(&offset, ep - ev);
    row[i] = ev;
  }
  __syncthreads();
  const int delta = offset == kNone ? 0 : offset;
  const bool plain = bad || delta > 900 || delta < -900;
  if (i < n) lexp[(size_t)c * (n + 1) + i] = row[i];
  if (i == 0) lexp[(size_t)c * (n + 1) + n] = plain ? kPlain : delta;
  for (int e = i; e < n * ld; e += 256) {
    const int j = e / ld, r = e - j * ld;
    const bool zero = plain || r >= n;
    out[(size_t)c * n * ld + e] =
        limbs_of(zero ? 0.0 : M[e], zero ? 0 : row[r] - 1022 + (j % nt < nvel ? 0 : delta));
  }
}

// The largest exponents of t's velocities and pressures give the exponent that t is cut at, or kPlain.
__device__ __forceinline__ int common_top(int ev, int ep, int delta) {
  if (delta == kPlain) return kPlain;
  const int most = max(ev, ep);
  if (most == kNone) return 1023;
  const int top = max(ev, ep + delta);
  return most >= 2047 || min(top, top - delta) < 64 || max(top, top - delta) > 2046 ? kPlain : top;
}
__device__ __forceinline__ void carry(long long& h, long long& m) {
  h += m >> kLimbBits;
  m &= (1ll << kLimbBits) - 1;
}
__device__ __forceinline__ double join(long long h, long long m) { return fma((double)h, (double)(1ll << kLimbBits), (double)m); }
__device__ __forceinline__ int scale_exp(int row, int top) { return row + top - 2044 - (2 * kLimbTotal - kLimbBits); }

// G warps per cell (8 / G cells per CTA), each a block of columns. Lane l of a warp owns the row pairs
// l, l + 32, .. (NR of them); UB columns are in flight, t's limbs stand in the warp's own shared memory. The next cell's t is gathered while the present one is streamed.
template <int NR>
__global__ void __launch_bounds__(256, NR <= 2 ? 3 : 2) k_limb_cells(const int4* __restrict__ lim, const int* __restrict__ lexp,
                                                       const double* __restrict__ inv, const int* __restrict__ idx,
                                                       const double* __restrict__ t, double* __restrict__ Y,
                                                       const int* __restrict__ cell_list, int ncells, int n, int ld, int G,
                                                       int nt, int nvel, double* __restrict__ d_scatter, double omega) {
  constexpr int UB = NR == 1 ? 6 : NR < 4 ? 3 : 2, NT = 2 * NR;
  // h grows by less than 2^56 per column: t is cut a bit higher where a warp may see more than 127
  constexpr int kLess = NR > 1 ? 1 : 0;
  constexpr int kEvery = (21 - UB) / UB;  // batches between carries: m grows by up to 1.5 x 2^58 per column
  __shared__ double2 tsh[8][32 * NR];
  __shared__ double part[8][64 * NR];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = warp & (G - 1), LDV = ld / 2;
  const int slots = 8 / G, slot = warp / G;
  int2* tl = reinterpret_cast<int2*>(tsh[warp]);
  double* td = reinterpret_cast<double*>(tsh[warp]);
  unsigned vel = 0;
#pragma unroll
  for (int k = 0; k < NT; ++k) vel |= (unsigned)((lane + 32 * k) % nt < nvel) << k;
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
  // the warp's columns; lanes beyond the rows repeat the last pair
  const int cb = (n + G - 1) / G, j0 = min(g * cb, n), cols = min(cb, n - j0);
  unsigned off[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) off[r] = (unsigned)(j0 * LDV + min(lane + 32 * r, LDV - 1));
  const int step = gridDim.x * slots;
  int ci = blockIdx.x * slots + slot, c = cell_of(ci);
  lookup(c);
  gather();
  for (; ci - slot < ncells; ci += step) {  // the same for all warps of a CTA
    const bool has = c >= 0;
    const int* ie = lexp + (size_t)(has ? c : 0) * (n + 1);
    const int delta = ie[n];
    int ev = kNone, ep = kNone;
#pragma unroll
    for (int k = 0; k < NT; ++k) {
      const int e = biased(tv[k]);
      if (vel >> k & 1) ev = max(ev, e);
      else ep = max(ep, e);
    }
    ev = __reduce_max_sync(0xffffffffu, ev);
    ep = __reduce_max_sync(0xffffffffu, ep);
    const int top = common_top(ev, ep, delta);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NT; ++k) {
      if (top != kPlain) tl[lane + 32 * k] = limbs_below(tv[k], (vel >> k & 1 ? top : top - delta) + kLess);
      else td[lane + 32 * k] = tv[k];
    }
    __syncwarp();
    const int cn = cell_of(ci + step);
    lookup(cn);
    double a[NR][2];
#pragma unroll
    for (int r = 0; r < NR; ++r) a[r][0] = a[r][1] = 0.0;
    if (has && top != kPlain) {
      long long h[NR][2], m[NR][2];
#pragma unroll
      for (int r = 0; r < NR; ++r) h[r][0] = h[r][1] = m[r][0] = m[r][1] = 0;
      const int4* M = lim + (size_t)c * n * LDV;
      const int2* tx = tl + j0;
      auto columns = [&](int cnt) {  // cnt <= UB: constant after unrolling but for the last batch
        int4 raw[UB][NR];
#pragma unroll
        for (int u = 0; u < UB; ++u)
          if (u < cnt)
#pragma unroll
            for (int r = 0; r < NR; ++r) raw[u][r] = __ldcs(M + (off[r] + (unsigned)(u * LDV)));
#pragma unroll
        for (int u = 0; u < UB; ++u)
          if (u < cnt) {
            const int2 x = tx[u];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              limb_fma(make_int2(raw[u][r].x, raw[u][r].y), x, h[r][0], m[r][0]);
              limb_fma(make_int2(raw[u][r].z, raw[u][r].w), x, h[r][1], m[r][1]);
            }
          }
      };
      int k = 0, left = cols;
#pragma unroll 1
      for (; left >= UB; left -= UB) {
        columns(UB);
        M += UB * LDV;
        tx += UB;
        if (++k < kEvery) continue;
        k = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          carry(h[r][0], m[r][0]);
          carry(h[r][1], m[r][1]);
        }
      }
#pragma unroll 1
      for (; left > 0; --left) {
        columns(1);
        M += LDV;
        ++tx;
      }
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        a[r][0] = join(h[r][0], m[r][0]);
        a[r][1] = join(h[r][1], m[r][1]);
      }
    } else {
      if (has) {
        const double* M = inv + (size_t)c * n * ld;
        for (int j = j0; j < j0 + cols; ++j)
#pragma unroll
          for (int r = 0; r < NR; ++r)
            if (lane + 32 * r < LDV) {
              a[r][0] = fma(M[(size_t)j * ld + 2 * (lane + 32 * r)], td[j], a[r][0]);
              a[r][1] = fma(M[(size_t)j * ld + 2 * (lane + 32 * r) + 1], td[j], a[r][1]);
            }
      }
    }
    gather();
    if (G > 1) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < NR; ++r) *reinterpret_cast<double2*>(part[warp] + 2 * (lane + 32 * r)) = make_double2(a[r][0], a[r][1]);
      __syncthreads();
      // warp g of the cell finishes the row pairs g (mod G)
    }
    if (has)
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const int i = 2 * (lane + 32 * r) + v;
          if (i >= n || (lane & (G - 1)) != g) continue;
          double y = a[r][v];
          if (G > 1) {
            y = 0.0;
            for (int w = 0; w < G; ++w) y += part[slot * G + w][i];
          }
          if (top != kPlain) y = scale_pow2(y, scale_exp(ie[i], top + kLess));
          if (d_scatter) d_scatter[idx[(long long)c * n + i]] += omega * y;
          else Y[(long long)c * n + i] = y;
        }
    c = cn;
  }
}

// The transpose: a thread per column, which it streams along its rows; P cells per CTA of T threads. The rows'
// exponents go into t's.
__global__ void __launch_bounds__(256, 4) k_limb_cells_t(const int4* __restrict__ lim, const int* __restrict__ lexp,
                                                         const double* __restrict__ inv, const int* __restrict__ idx,
                                                         const double* __restrict__ t, double* __restrict__ Y,
                                                         const int* __restrict__ cell_list, int ncells, int n, int ld,
                                                         int T, int P, int nt, int nvel, double* __restrict__ d_scatter,
                                                         double omega) {
  constexpr int UB = 6;
  extern __shared__ int4 sm4[];  // [P][ld] limbs of t
  __shared__ int most[16], worst[16];
  const int slot = threadIdx.x / T, j = threadIdx.x - slot * T, LDV = ld / 2;
  int2* tl = reinterpret_cast<int2*>(sm4) + slot * ld;
  double* td = reinterpret_cast<double*>(tl);
  for (int base = blockIdx.x * P; base < ncells; base += gridDim.x * P) {
    const int ci = base + slot;
    const bool has = slot < P && ci < ncells;
    const int c = has ? (cell_list ? cell_list[ci] : ci) : 0;
    const int* ic = idx + (long long)c * n;
    const int* ie = lexp + (size_t)c * (n + 1);
    __syncthreads();
    if (threadIdx.x < 16) most[threadIdx.x] = worst[threadIdx.x] = kNone;
    __syncthreads();
    if (has)
      for (int i = j; i < ld; i += T) {
        const double v = i < n ? t[ic[i]] : 0.0;
        td[i] = v;
        const int e = biased(v);
        if (e != kNone) {
          atomicMax(&most[slot], e + ie[i]);
          atomicMax(&worst[slot], e < 64 ? 2047 : e);
        }
      }
    __syncthreads();
    const int delta = ie[n], all = has ? most[slot] : kNone;  // largest product of a row's scale and t's entry
    const bool plain = delta == kPlain || (all != kNone && (worst[slot] >= 2047 || all < 256));
    if (has && !plain)
      for (int i = j; i < ld; i += T) {
        const int top = all == kNone || i >= n ? 1023 : all - ie[i];  // below 64 only where t is zero
        tl[i] = top < 64 ? make_int2(0, 0) : limbs_below(td[i], top);
      }
    __syncthreads();
    if (has && j < n) {
      double y = 0.0;
      if (!plain) {
        const int4* col = lim + ((size_t)c * n + j) * LDV;
        long long h = 0, m = 0, hs = 0;
        for (int i0 = 0; i0 < LDV; i0 += UB) {
          int4 raw[UB];
#pragma unroll
          for (int u = 0; u < UB; ++u)
            if (i0 + u < LDV) raw[u] = __ldg(col + i0 + u);
            else raw[u] = make_int4(0, 0, 0, 0);
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            const int q = min(i0 + u, LDV - 1);
            limb_fma(make_int2(raw[u].x, raw[u].y), tl[2 * q], h, m);
            limb_fma(make_int2(raw[u].z, raw[u].w), tl[2 * q + 1], h, m);
          }
          carry(h, m);
          hs += h >> 8;  // up to 254 rows
          h &= 255;
        }
        y = fma((double)hs, 256.0, (double)h);
        y = fma(y, (double)(1ll << kLimbBits), (double)m);
        y = scale_pow2(y, scale_exp(all == kNone ? 1023 : all, (j % nt < nvel ? 0 : delta)));
      } else {
        const double* col = inv + (size_t)c * n * ld + (size_t)j * ld;
        for (int i = 0; i < n; ++i) y = fma(col[i], td[i], y);
      }
      if (d_scatter) d_scatter[ic[j]] += omega * y;
      else Y[(long long)c * n + j] = y;
    }
  }
}

template <int NR>
stm_status launch_cells(const Level& L, const double* t, const int* cells, int nc, int ld, double* scatter, double omega,
                        cudaStream_t s) {
  static int per_sm = 0;
  if (!per_sm) {
    int o = 0;
    STM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_limb_cells<NR>, 256, 0));
    per_sm = std::max(o, 1);
  }
  // a warp per cell where that keeps every resident warp busy, more where cells are few
  const long long most = 8LL * sm_count() * per_sm;
  int G = 1;
  while (G < 8 && nc * (long long)G * 2 <= most) G *= 2;
  // as few CTAs as give the same number of rounds, so that none idles through a last partial one
  const long long ctas = ((long long)nc * G + 7) / 8, rounds = (ctas + most / 8 - 1) / (most / 8);
  k_limb_cells<NR><<<(int)((ctas + rounds - 1) / rounds), 256, 0, s>>>(
      (const int4*)L.lim, L.lexp, (const double*)L.inv, L.idx, t, L.Y, cells, nc, L.n, ld, G, L.nt, L.dim * L.nv, scatter, omega);
  return STM_OK;
}

}  // namespace

stm_status inverse_limbs(Level& L, cudaStream_t s) {
  const int ld = inv_layout(L.n, STM_F64).ld;
  if (ld % 2 || L.n < 32 || L.n > 254) return STM_OK;
  if (!L.lim) {
    // a second copy of the inverses: without room for it the FP64 kernels serve
    if (cudaMalloc((void**)&L.lim, sizeof(int2) * (size_t)L.C * L.n * ld) != cudaSuccess ||
        cudaMalloc((void**)&L.lexp, sizeof(int) * (size_t)L.C * (L.n + 1)) != cudaSuccess) {
      cudaGetLastError();
      if (L.lim) cudaFree(L.lim);
      L.lim = nullptr;
      return STM_OK;
    }
  }
  k_inverse_limbs<<<L.C, 256, 0, s>>>((const double*)L.inv, L.n, ld, L.nt, L.dim * L.nv, L.lim, L.lexp);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

stm_status vanka_limbs(const Level& L, const double* t, const int* cells, int nc, int transpose, double* scatter,
                       double omega, cudaStream_t s) {
  const int n = L.n, ld = inv_layout(n, STM_F64).ld;
  if (transpose) {
    const int T = (n + 31) / 32 * 32, P = std::min(16, std::max(1, 256 / T));
    const int blocks = std::min((nc + P - 1) / P, sm_count() * 8);
    k_limb_cells_t<<<blocks, T * P, sizeof(int2) * (size_t)P * ld, s>>>((const int4*)L.lim, L.lexp, (const double*)L.inv,
                                                                       L.idx, t, L.Y, cells, nc, n, ld, T, P, L.nt,
                                                                       L.dim * L.nv, scatter, omega);
  } else if (n <= 64) {
    STM_TRY(launch_cells<1>(L, t, cells, nc, ld, scatter, omega, s));
  } else if (n <= 128) {
    STM_TRY(launch_cells<2>(L, t, cells, nc, ld, scatter, omega, s));
  } else if (n <= 192) {
    STM_TRY(launch_cells<3>(L, t, cells, nc, ld, scatter, omega, s));
  } else {
    STM_TRY(launch_cells<4>(L, t, cells, nc, ld, scatter, omega, s));
  }
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

}  // namespace stm
