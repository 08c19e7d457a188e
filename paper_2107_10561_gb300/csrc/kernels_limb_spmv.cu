// Products with the slab Jacobian J_g (or its transpose) whose velocity rows run on the INT32 pipe:
// y = J x, y = b - J x or y += J x in FP64 accuracy.
//
// The product reads every value of J once and needs one multiply-add for it. In FP64 that is the limit: at 74
// clocks per warp instruction and sub-core the finest 3D dG(1) level (962,208 unknowns, 2.6 GB of values) took
// 566 us against 382 us for the bytes at the measured copy rate. Here J's velocity rows are two-limb integers
// (limbs.h, eight bytes per value as before), three integer multiply-adds each, 13 clocks: the bytes are the limit
// again: 425 us are 6.1 TB/s of values, 6.6 TB/s of what is read (padded runs read 5 % more sectors). On smaller 3D levels: 91.7 -> 71.1 us (127,920 unknowns),
// 49.9 -> 32.4 (18,000); 3D dG(0) 175.8 -> 145 (481,104), dG(2) 651 -> 469 (735,369); 2D dG(2) 89.3 -> 78.8
// (536,448) and 35.1 -> 31.0 (135,168).
//   - Row exponents come with the values; the exponent of x is that of the largest entry around a node, found per
//     cell in a pass of its own (a node's neighbours are the nodes of its cells), so that rows far from the
//     largest entries of x lose nothing. The pressure columns of a node share one offset against the velocity
//     columns, which keeps both in one pair of accumulators.
//   - Against the sum of |J| |x| in a row the error measured 1e-16 to 4e-16 (normally distributed x), that of an
//     FP64 chain 2e-16 to 5e-16.
//   - VL lanes per node, a lane per neighbour node: its K*d positions of K*d values stand in planes of VL lanes,
//     so that all addresses but the first are constants. Positions are loaded PD ahead and entries of x K*d
//     positions ahead into registers; rings in shared memory (444 us) and bulk prefetches into L2 (438 to 477 us)
//     were slower, more warps with fewer registers too (520 us at 80 registers).
//   - Units of 32 / VL nodes or 32 pressure rows (FP64, 3 % of the values) from a device counter, the two kinds
//     interleaved; the next unit's nodes are looked up while the present one is finished.
//   - The exponent pass (5 to 8 us) ends beside the product's first loads: a programmatic dependent launch.
//   - Nodes with an infinity or a NaN in their rows or around them, or with entries of x below 2^-958 only, are
//     summed from the CSR values in plain FP64.
#include "digits.h"
#include "internal.h"
#include "limbs.h"

namespace stm {
namespace {

constexpr int kNone = -(1 << 20);    // biased exponent where every entry is zero
constexpr int kPlain = 1 << 20;      // pressure offset of a node whose rows hold an infinity or a NaN

__device__ __forceinline__ int biased(double v) {
  const int hi = __double2hiint(v) & 0x7FFFFFFF;
  return (hi | __double2loint(v)) == 0 ? kNone : hi >> 20;
}

// Largest biased exponents of x in each cell: velocities, pressures. A lane per node of the cell, whose K*d entries
// are independent loads; half a warp per cell in 2D, a warp in 3D.
template <int K, int D>
__global__ void __launch_bounds__(256) k_cell_exps(const int* __restrict__ cell_nodes, const double* __restrict__ x,
                                                   int C, long long block, int R, int2* __restrict__ cexp) {
  constexpr int NV = D == 2 ? 9 : 27, NP = D + 1, G = D == 2 ? 16 : 32;
  static_assert(K * NP <= G, "a lane per pressure");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int lane = threadIdx.x & (G - 1);
  const int c = (blockIdx.x * 256 + threadIdx.x) / G;
  int ev = kNone, ep = kNone;
  if (c < C) {
    if (lane < NV) {
      const double* xn = x + cell_nodes[(long long)c * NV + lane];
#pragma unroll
      for (int k = 0; k < K * D; ++k) ev = max(ev, biased(__ldg(xn + (k / D) * block + (long long)(k % D) * R)));
    }
    if (lane < K * NP) ep = biased(__ldg(x + (lane / NP) * block + (long long)D * R + (long long)c * NP + lane % NP));
  }
#pragma unroll
  for (int off = G / 2; off >= 1; off >>= 1) {
    ev = max(ev, __shfl_xor_sync(0xffffffffu, ev, off));
    ep = max(ep, __shfl_xor_sync(0xffffffffu, ep, off));
  }
  if (lane == 0 && c < C) cexp[c] = make_int2(ev, ep);
}

// CSR position of node-block position p in a velocity row of time node a
__device__ __forceinline__ int csr_pos(int p, int a, int npv, int npc, int dnn) {
  if (p < npv) return p + (p >= (a + 1) * dnn ? npc : 0);
  return (a + 1) * dnn + (p - npv);
}

// Limbs of the velocity rows, one warp per node: row exponents first, then the positions in runs of VL, the
// KD values of a position in KD / 2 planes of 16 bytes (KD planes of 8 for odd KD) so that the VL lanes of a
// group read whole lines.
template <int KD, int D>
__global__ void __launch_bounds__(256) k_build_limbs(const long long* __restrict__ rowptr, const double* __restrict__ val,
                                                     const int* __restrict__ nbr_ptr, const int* __restrict__ ncell,
                                                     const long long* __restrict__ lbase, int2* __restrict__ out,
                                                     int* __restrict__ nexp, long long block, int R, int VL) {
  constexpr int NP = D + 1, W = KD % 2 ? 1 : 2;
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < R; i += nwarps) {
    const int nn = nbr_ptr[i + 1] - nbr_ptr[i], npc = NP * ncell[i], npv = KD * nn, dnn = D * nn;
    const int pad = KD * ((nn + VL - 1) / VL * VL);
    const double* v[KD];
    int ev[KD], delta = kNone, top = 0;
#pragma unroll
    for (int r = 0; r < KD; ++r) {
      v[r] = val + rowptr[(r / D) * block + (long long)(r % D) * R + i];
      int e = kExpZero, ep = kExpZero;
      for (int p = lane; p < npv + npc; p += 32) {
        const int t = exp_above(v[r][csr_pos(p, r / D, npv, npc, dnn)]);
        if (p < npv) e = max(e, t);
        else ep = max(ep, t);
      }
      e = __reduce_max_sync(0xffffffffu, e);
      ep = __reduce_max_sync(0xffffffffu, ep);
      if (e == kExpZero) e = ep == kExpZero ? 0 : ep;
      if (ep != kExpZero) delta = max(delta, ep - e);
      ev[r] = e;
      top = max(top, max(e, ep));
    }
    if (delta == kNone) delta = 0;
    const bool bad = top > 1024;
    if (lane == 0) {
#pragma unroll
      for (int r = 0; r < KD; ++r) nexp[i * (KD + 1) + r] = ev[r];
      nexp[i * (KD + 1) + KD] = bad ? kPlain : delta;
    }
    for (int p = lane; p < npv + npc; p += 32) {
      const bool vel = p < npv;
      const int bm = vel ? p / nn : 0, q = vel ? p - bm * nn : p - npv;  // neighbour and its entry, or pressure
      const int c0 = q - q % VL;
      int2* o = out + lbase[i] + (vel ? c0 * KD + bm * VL : pad + c0) * KD + (q - c0) * W;
#pragma unroll
      for (int r = 0; r < KD; r += W) {
        int2 l[2];
#pragma unroll
        for (int k = 0; k < W; ++k) {
          const double t = bad ? 0.0 : v[r + k][csr_pos(p, (r + k) / D, npv, npc, dnn)];
          l[k] = limbs_of(t, ev[r + k] + (vel ? 0 : delta));
        }
        if constexpr (W == 2) *reinterpret_cast<int4*>(o + r * VL) = make_int4(l[0].x, l[0].y, l[1].x, l[1].y);
        else o[r * VL] = l[0];
      }
    }
  }
}

// The KD values of a lane's position in a run (planes of VL lanes).
template <int KD, int VL>
__device__ __forceinline__ void load_values(const char* run, int2* v) {
  if constexpr (KD % 2 == 0) {
#pragma unroll
    for (int r = 0; r < KD / 2; ++r) {
      const int4 t = __ldcs(reinterpret_cast<const int4*>(run) + r * VL);
      v[2 * r] = make_int2(t.x, t.y);
      v[2 * r + 1] = make_int2(t.z, t.w);
    }
  } else {
#pragma unroll
    for (int r = 0; r < KD; ++r) v[r] = __ldcs(reinterpret_cast<const int2*>(run) + r * VL);
  }
}

template <int VL, int NA>
__device__ __forceinline__ void reduce_scatter(double* acc, int lane) {
  int cnt = NA;
#pragma unroll
  for (int off = VL / 2; off >= 1; off >>= 1) {
    if (cnt > 1) {
      const int half = cnt / 2;
      const bool upper = (lane & off) != 0;
#pragma unroll
      for (int k = 0; k < NA / 2; ++k)
        if (k < half) {
          const double send = upper ? acc[k] : acc[k + half], keep = upper ? acc[k + half] : acc[k];
          acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, off, VL);
        }
      cnt = half;
    } else {
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off, VL);
    }
  }
}
template <int VL, int NA>
__device__ __forceinline__ int scatter_index(int lane, int& writer_mask) {
  int cnt = NA, k = 0;
  writer_mask = 0;
#pragma unroll
  for (int off = VL / 2; off >= 1; off >>= 1) {
    if (cnt > 1) {
      cnt /= 2;
      if (lane & off) k += cnt;
    } else {
      writer_mask |= off;
    }
  }
  return k;
}
__host__ __device__ constexpr int pow2ceil(int v) { return v <= 1 ? 1 : 2 * pow2ceil((v + 1) / 2); }

struct LimbArgs {
  const int2* jl;
  const int* nexp;
  const int2* cexp;
  const double* pvalT;
  const long long* lbase;
  const int *nbr_ptr, *nbr, *ncell, *node_cells, *cell_nodes, *jobs;
  const long long* rowptr;
  const int* col;
  const double* val;  // CSR values
  long long block;
  int R, C;
  const double *x, *b;
  double* y;
  int mode;
  unsigned* work;
  int njobs;
  unsigned nvu, ntot;         // units of nodes, all units
  unsigned long long pstep;   // pressure units per unit, times 2^32
};

__device__ __forceinline__ void put(const LimbArgs& s, long long row, double v) {
  if (s.mode == 0) s.y[row] = v;
  else if (s.mode == 1) s.y[row] = s.b[row] - v;
  else s.y[row] += v;
}

// 128 registers and 16 warps per SM; three rows per node (dG(0)) need half of that and gain from twice the warps
// (170 -> 145 us on 481,104 unknowns).
template <int VL, int K, int D>
__global__ void __launch_bounds__(128, K * D == 3 ? 8 : 4) k_spmv_limbs(const __grid_constant__ LimbArgs s) {
  constexpr int GPW = 32 / VL, KD = K * D, NP = D + 1, MAXC = 1 << D, NV = D == 2 ? 9 : 27, MAXN = D == 2 ? 25 : 125;
  constexpr int NAV = pow2ceil(KD), HOLD = NAV > VL ? NAV / VL : 1;
  constexpr int PD = KD % 3 ? 2 : 3;      // positions loaded ahead
  constexpr int kRun = KD * VL * 8, kChunk = KD * kRun;
  // h stays below 2^63 for 127 positions per lane; m grows by up to 1.5 x 2^58 per position and is carried over
  // to h in time
  constexpr int kRuns = (NP * MAXC + VL - 1) / VL;  // pressure runs at most
  constexpr int kMost = KD * ((MAXN + VL - 1) / VL) + kRuns;
  static_assert(kMost < 128, "h overflows");
  static_assert(VL >= MAXC, "a lane per cell");
  constexpr bool kCarry = kMost > 20;
  const int lw = threadIdx.x & 31, lane = lw & (VL - 1), gw = lw / VL;
  int wmask;
  const int kv = scatter_index<VL, NAV>(lane, wmask);
  auto pressure_before = [&](unsigned u) { return (unsigned)(((unsigned long long)u * s.pstep) >> 32); };
  unsigned u = 0, u1 = 0;
  bool first = true;
  if (lw == 0) u = atomicAdd(s.work, 1u);
  u = __shfl_sync(0xffffffffu, u, 0);
  // what a unit needs to know of its nodes is looked up while the unit before is finished
  struct Node { int i, p0, nn, npc; long long at; bool ok; };
  auto lookup = [&](unsigned w) {
    Node n{0, 0, 0, 0, 0, false};
    const unsigned p = pressure_before(w);
    const int job = (int)(s.nvu - 1 - (w - p)) * GPW + gw;
    if (w < s.ntot && pressure_before(w + 1) == p && job < s.njobs) {
      n.i = s.jobs[job];
      n.p0 = s.nbr_ptr[n.i];
      n.nn = s.nbr_ptr[n.i + 1] - n.p0;
      n.npc = NP * s.ncell[n.i];
      n.at = s.lbase[n.i];
      n.ok = true;
    }
    return n;
  };
  Node nd = lookup(u);
  while (u < s.ntot) {
    if (lw == 0) u1 = atomicAdd(s.work, 1u);
    Node nx{};
    const unsigned pu = pressure_before(u);
    if (pressure_before(u + 1) == pu) {
      const bool ok = nd.ok;
      const int i = nd.i, p0 = nd.p0, nn = nd.nn, npc = nd.npc;
      const char* blk = reinterpret_cast<const char*>(s.jl + nd.at) + lane * (KD % 2 ? 8 : 16);
      const int nch = (nn + VL - 1) / VL, nchw = __reduce_max_sync(0xffffffffu, nch);
      const int nrw = __reduce_max_sync(0xffffffffu, (npc + VL - 1) / VL);
      const char* blkp = blk + nch * kChunk;
      int2 v[PD][KD];
#pragma unroll
      for (int t = 0; t < PD; ++t)
        if (lane < nn) load_values<KD, VL>(blk + t * kRun, v[t]);
        else
#pragma unroll
          for (int r = 0; r < KD; ++r) v[t][r] = make_int2(0, 0);
      double x[KD], xp[K];
      unsigned node = 0, next = 0;
      if (lane < nn) node = (unsigned)s.nbr[p0 + lane];
      if (lane + VL < nn) next = (unsigned)s.nbr[p0 + lane + VL];
      const int cell = lane < MAXC && NP * lane < npc ? s.node_cells[(long long)i * MAXC + lane] : 0;
      const int delta = s.nexp[(long long)i * (KD + 1) + KD];
#pragma unroll
      for (int bm = 0; bm < KD; ++bm)
        x[bm] = lane < nn ? __ldg(s.x + (bm / D) * s.block + (long long)(bm % D) * s.R + node) : 0.0;
      auto pressures = [&](int r) {
        const int tq = lane + r * VL, ci = tq / NP, c = __shfl_sync(0xffffffffu, cell, ci < MAXC ? ci : 0, VL);
#pragma unroll
        for (int a = 0; a < K; ++a)
          xp[a] = tq < npc ? __ldg(s.x + a * s.block + (long long)D * s.R + (long long)c * NP + (tq - ci * NP)) : 0.0;
      };
      pressures(0);
      int bv = kNone, bp = kNone;
      if (first) {  // what came before is independent of the exponents
        asm volatile("griddepcontrol.wait;" ::: "memory");
        first = false;
      }
      if (lane < MAXC && NP * lane < npc) {
        const int2 e = __ldcg(s.cexp + cell);
        bv = e.x;
        bp = e.y;
      }
#pragma unroll
      for (int off = MAXC / 2; off >= 1; off >>= 1) {
        bv = max(bv, __shfl_xor_sync(0xffffffffu, bv, off, VL));
        bp = max(bp, __shfl_xor_sync(0xffffffffu, bp, off, VL));
      }
      if constexpr (VL > MAXC) {
        bv = __shfl_sync(0xffffffffu, bv, 0, VL);
        bp = __shfl_sync(0xffffffffu, bp, 0, VL);
      }
      int top = max(bv, bp + delta);
      if (max(bv, bp) == kNone) top = 1023;
      const bool plain = delta == kPlain || max(bv, bp) >= 2047 || min(top, top - delta) < 64 || max(top, top - delta) > 2046;
      if (plain) top = 1023;
      const int topp = plain ? 1023 : top - delta;
      long long h[KD], m[KD];
#pragma unroll
      for (int r = 0; r < KD; ++r) h[r] = m[r] = 0;
      for (int k = 0; k < nchw; ++k) {
        const bool has = lane + (k + 1) * VL < nn;
        const char* src = blk + k * kChunk;
        const unsigned node8 = 8u * next;
        if (lane + (k + 2) * VL < nn) next = (unsigned)s.nbr[p0 + lane + (k + 2) * VL];
#pragma unroll
        for (int bm = 0; bm < KD; ++bm) {
          const int2 xl = limbs_below(x[bm], top);
          const char* xb = reinterpret_cast<const char*>(s.x + (bm / D) * s.block + (long long)(bm % D) * s.R);
          x[bm] = has ? __ldg(reinterpret_cast<const double*>(xb + node8)) : 0.0;
#pragma unroll
          for (int r = 0; r < KD; ++r) limb_fma(v[bm % PD][r], xl, h[r], m[r]);
          // the position PD ahead; the last chunk's lanes beyond its end keep what they have (times x = 0)
          if (bm + PD < KD ? lane + k * VL < nn : has) load_values<KD, VL>(src + (bm + PD) * kRun, v[bm % PD]);
        }
        if constexpr (kCarry)
          if ((k & (KD <= 2 ? 7 : KD <= 4 ? 3 : 1)) == 1) {
#pragma unroll
            for (int r = 0; r < KD; ++r) {
              h[r] += m[r] >> kLimbBits;
              m[r] &= (1ll << kLimbBits) - 1;
            }
          }
      }
      u1 = __shfl_sync(0xffffffffu, u1, 0);
      nx = lookup(u1);
      for (int r = 0; r < nrw; ++r) {
        int2 w[KD];
        if (lane + r * VL < npc) load_values<KD, VL>(blkp + r * kRun, w);
        else
#pragma unroll
          for (int q = 0; q < KD; ++q) w[q] = make_int2(0, 0);
        int2 xl[K];
#pragma unroll
        for (int a = 0; a < K; ++a) xl[a] = limbs_below(xp[a], topp);
        if (r + 1 < nrw) pressures(r + 1);
#pragma unroll
        for (int a = 0; a < K; ++a)
#pragma unroll
          for (int l = 0; l < D; ++l) limb_fma(w[a * D + l], xl[a], h[a * D + l], m[a * D + l]);
      }
      double acc[NAV];
#pragma unroll
      for (int r = 0; r < NAV; ++r) acc[r] = r < KD ? fma((double)h[r], (double)(1ll << kLimbBits), (double)m[r]) : 0.0;
      reduce_scatter<VL, NAV>(acc, lane);
      if (ok && !plain && (lane & wmask) == 0) {
#pragma unroll
        for (int q = 0; q < HOLD; ++q) {
          const int r = kv + q;
          if (r < KD) {
            const int e = s.nexp[(long long)i * (KD + 1) + r] + top - 1022 - (2 * kLimbTotal - kLimbBits);
            put(s, (r / D) * s.block + (long long)(r % D) * s.R + i, scale_pow2(acc[q], e));
          }
        }
      }
      if (ok && plain)
        for (int r = lane; r < KD; r += VL) {
          const long long row = (r / D) * s.block + (long long)(r % D) * s.R + i;
          double t = 0.0;
          for (long long e = s.rowptr[row]; e < s.rowptr[row + 1]; ++e) t = fma(s.val[e], s.x[s.col[e]], t);
          put(s, row, t);
        }
      __syncwarp();
    } else {
      if (first) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        first = false;
      }
      u1 = __shfl_sync(0xffffffffu, u1, 0);
      nx = lookup(u1);
      // pressure rows pr = (a*C + c)*n_p + q: one lane per row over the warp-transposed copy
      const long long pr = (long long)pu * 32 + lw;
      if (pr < (long long)K * s.C * NP) {
        const int a = (int)(pr / ((long long)s.C * NP));
        const long long cq = pr - (long long)a * s.C * NP, c = cq / NP;
        const double* vr = s.pvalT + ((pr >> 5) * (D * NV)) * 32 + (pr & 31);
        const int* cn = s.cell_nodes + c * NV;
        const double* xa = s.x + a * s.block;
        double s3[3] = {0.0, 0.0, 0.0};  // three independent chains
#pragma unroll
        for (int m = 0; m < D; ++m)
#pragma unroll 9
          for (int jj = 0; jj < NV; ++jj)
            s3[jj % 3] = fma(__ldcs(vr + (m * NV + jj) * 32), __ldg(xa + (long long)m * s.R + __ldg(cn + jj)), s3[jj % 3]);
        put(s, a * s.block + (long long)D * s.R + cq, (s3[0] + s3[1]) + s3[2]);
      }
    }
    u = u1;
    nd = nx;
  }
  // the last CTA to finish resets the counter: every warp has fetched a unit past the end by then
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

template <int VL, int K, int D>
stm_status launch(const Level& L, LimbArgs& a, cudaStream_t s) {
  static int occ = 0;
  if (!occ) {
    int o = 0;
    STM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_spmv_limbs<VL, K, D>, 128, 0));
    occ = std::max(o, 1);
  }
  const unsigned npu = (unsigned)(((long long)K * L.C * (D + 1) + 31) / 32);
  a.nvu = (unsigned)((a.njobs + 32 / VL - 1) / (32 / VL));
  a.ntot = a.nvu + npu;
  // rounded up so that the last unit brings the count to npu
  a.pstep = (((unsigned long long)npu << 32) + a.ntot - 1) / a.ntot;
  const int blocks = (int)std::max<long long>(1, std::min<long long>((long long)occ * sm_count(), (a.ntot + 3) / 4));
  // launched while the exponents are still being found: it waits for them after its first loads
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  STM_CUDA(cudaLaunchKernelEx(&cfg, k_spmv_limbs<VL, K, D>, a));
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

template <int K, int D>
stm_status launch_vl(const Level& L, LimbArgs& a, cudaStream_t s) {
  constexpr int kCells = D == 2 ? 16 : 8;  // cells per CTA
  k_cell_exps<K, D><<<(L.C + kCells - 1) / kCells, 256, 0, s>>>(L.cell_nodes, a.x, L.C, L.block, L.R, L.cexp);
  note_launch();
  STM_CUDA(cudaGetLastError());
  if constexpr (D == 2) {
    return L.limb_lanes == 4 ? launch<4, K, D>(L, a, s) : launch<8, K, D>(L, a, s);
  } else {
    if constexpr (K < 3)  // 127 positions per lane at most
      if (L.limb_lanes == 8) return launch<8, K, D>(L, a, s);
    return L.limb_lanes == 16 ? launch<16, K, D>(L, a, s) : launch<32, K, D>(L, a, s);
  }
}

}  // namespace

stm_status build_limbs(const Level& L, const double* val, double* nval, int* nexp, cudaStream_t s) {
  const int blocks = (int)std::min<long long>(((long long)L.R * 32 + 255) / 256, sm_count() * 8LL);
  int2* o = reinterpret_cast<int2*>(nval);
#define STM_BUILD(KD, D) \
  k_build_limbs<KD, D><<<blocks, 256, 0, s>>>(L.rowptr, val, L.nbr_ptr, L.ncell, L.lbase, o, nexp, L.block, L.R, L.limb_lanes)
  switch (L.dim * 10 + L.K) {
    case 23: STM_BUILD(6, 2); break;
    case 31: STM_BUILD(3, 3); break;
    case 32: STM_BUILD(6, 3); break;
    default: STM_BUILD(9, 3); break;
  }
#undef STM_BUILD
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

// 3D levels keep limbs whatever their size (from 1,146 unknowns: 18.1 -> 12.6 us). In 2D it takes dG(2) and 12,000
// nodes: at 4,200 nodes the pass over x costs what the product gains (17.8 against 20.9 us), and with four rows or
// two per node the FP64 product is faster (dG(1), 357,632 unknowns: 47 against 50 us; dG(0), 178,816: 25 against
// 26 us) since a lane has less to multiply per entry of x that it converts. Lanes per node as in the FP64 product
// but for the 2D levels between (8: 31.0 us, 16: 37.2 us on 135,168 unknowns) and 3D dG(2) (16 at least: a lane of
// 8 would see more positions than its sums hold).
int limb_lanes(const Level& L) {
  if (L.dim == 3) return std::max(node_lanes(L), L.K == 3 ? 16 : 8);
  if (L.K < 3 || L.R < 12000) return 0;
  return node_lanes(L) == 4 ? 4 : 8;
}

stm_status spmv_limbs(const Level& L, int transpose, const double* x, const double* b, double* y, int mode,
                      cudaStream_t s, const int* jobs, int njobs) {
  LimbArgs a{};
  a.jl = reinterpret_cast<const int2*>(transpose ? L.nvalJT : L.nval);
  a.nexp = transpose ? L.nexpJT : L.nexp;
  a.cexp = L.cexp;
  a.pvalT = transpose ? L.pvalJT : L.pvalT;
  a.lbase = L.lbase;
  a.nbr_ptr = L.nbr_ptr;
  a.nbr = L.nbr;
  a.ncell = L.ncell;
  a.node_cells = L.node_cells;
  a.cell_nodes = L.cell_nodes;
  a.jobs = jobs ? jobs : L.job_nodes;
  a.njobs = jobs ? njobs : L.R;
  a.rowptr = L.rowptr;
  a.col = L.colidx;
  a.val = transpose ? L.valT : L.val;
  a.block = L.block;
  a.R = L.R;
  a.C = L.C;
  a.x = x;
  a.b = b;
  a.y = y;
  a.mode = mode;
  a.work = L.spmv_work;
  switch (L.dim * 10 + L.K) {
    case 23: return launch_vl<3, 2>(L, a, s);
    case 31: return launch_vl<1, 3>(L, a, s);
    case 32: return launch_vl<2, 3>(L, a, s);
    default: return launch_vl<3, 3>(L, a, s);
  }
}

}  // namespace stm
