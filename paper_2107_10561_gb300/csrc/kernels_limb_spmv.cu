// Products with the slab Jacobian J_g of a 3D level (or its transpose) whose velocity rows run on the INT32 pipe:
// y = J x, y = b - J x or y += J x, every row as accurate as an FP64 sum of it is held to be.
//
// The product reads every value of J once and needs one multiply-add for it. In FP64 that is the limit: the finest 3D
// dG(1) level (962,208 unknowns, 2.6 GB of values) takes 564 us against 382 us for the bytes at the measured copy rate.
// Here J's velocity rows are two-limb integers (limbs.h, eight bytes per value as before), three integer multiply-adds
// each: 459 us for normally distributed x and about 545 us for what a V-cycle returns (below). Smaller levels and other
// elements, normally distributed x, FP64 against this: 3D dG(1), 129,094 unknowns: 106 -> 85 us; 3D dG(0), 486,979:
// 188 -> 174 (V-cycles' vectors 187); 3D dG(2), 296,385: 363 -> 217.
//   - A sum of integers has one scale, FP64 terms have one each. Scales therefore go by class of unknowns (a velocity
//     component or a pressure mode of one time node): J has an exponent per component of the row, class of the column
//     and node, x one per class, the largest around a node, found per cell in a pass of its own (a node's neighbours
//     are the nodes of its cells). The sums of a component's rows stand at its largest product of scales; an entry of x
//     is cut at its own class's scale and shifted once per component of the rows, which is cheaper than shifting K*D
//     values of J (24 instructions more per position).
//   - What is cut off, about 2^-57 per term, is small against that product but not always against |J||x|: x may be large
//     where J is small. The lanes' sums and the magnitudes of the pressures' terms bound |J||x| from below; a row where
//     that stays 2^-kSpare below the largest product of scales is summed again in FP64 from the CSR values, by the lanes
//     of its node. kSpare = 7 keeps every row below the bound m 2^-53 |J||x| of an FP64 chain of m terms (8 exceeds it
//     by 8 % for x with single entries 1e12 above the others). Of normally distributed x no row in a thousand is summed
//     again, also with components or pressures 1e-8 apart. Of V-cycles' results, which peak at corners and
//     walls, so many are that a solve to 1e-10 takes 69.8 ms (71.5 ms with the FP64 product).
//   - One scale for all classes of a node, without a second sum, took 433 us and lost 2^-53 of the largest term in every
//     row: 3e-14 of |J||x| at velocity components 1e-2 apart, 2e-10 at 1e-6.
//   - VL lanes per node, a lane per neighbour node: its K*d positions of K*d values stand in planes of VL lanes,
//     so that all addresses but the first are constants. Positions are loaded PD ahead and entries of x K*d
//     positions ahead into registers. Rings in shared memory filled by bulk copies (475 us) cost more instructions than
//     they save waiting: 16 warps per SM issue at 50 % of the rate.
//   - Units of 32 / VL nodes or 32 pressure rows (FP64, 3 % of the values) from a device counter, the two kinds
//     interleaved; the next unit's nodes are looked up while the present one is finished.
//   - The exponent pass (5 to 8 us) ends beside the product's first loads: a programmatic dependent launch.
//   - Nodes with an infinity or a NaN in their rows or around them, or with a class of x below 2^-958, are summed in
//     FP64 as well.
#include "digits.h"
#include "internal.h"
#include "limbs.h"

namespace stm {
namespace {

constexpr int kNone = -20000;   // exponent where every entry is zero (16 bits)
constexpr int kPlain = 20000;   // exponent of a block of J that holds an infinity or a NaN
constexpr int kNonePair = (int)(((unsigned)kNone & 0xFFFFu) * 0x10001u);

__device__ __forceinline__ int biased(double v) {
  const int hi = __double2hiint(v) & 0x7FFFFFFF;
  return (hi | __double2loint(v)) == 0 ? kNone : hi >> 20;
}

constexpr int D = 3, NV = 27, NP = 4, MAXC = 8;  // 2D levels keep FP64 values (limb_lanes)

// Classes of unknowns: the K*D velocity components of all time nodes, then the pressure modes of each time node.
template <int K>
struct Classes {
  static constexpr int KD = K * D, count = KD + K * NP;
  static constexpr int words = K == 1 ? 4 : K == 2 ? 8 : 16;  // exponents of a cell, two to a word, padded
  // exponents of J per node: per component and class (all time nodes' velocities, the row's own pressures), per row
  static constexpr int row = KD + NP, node = D * row + KD;
};

// Largest biased exponents of x in each cell, one per class: a warp per cell, a lane per node, whose K*d entries are
// independent loads, and a lane per pressure.
template <int K>
__global__ void __launch_bounds__(256) k_cell_exps(const int* __restrict__ cell_nodes, const double* __restrict__ x,
                                                   int C, long long block, int R, short* __restrict__ cexp) {
  using S = Classes<K>;
  constexpr int NW = (S::KD + 1) / 2;
  static_assert(K * NP <= 32, "a lane per pressure");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int lane = threadIdx.x & 31, c = (blockIdx.x * 256 + threadIdx.x) >> 5;
  if (c >= C) return;
  int e[2 * NW];
#pragma unroll
  for (int k = 0; k < 2 * NW; ++k) e[k] = kNone;
  if (lane < NV) {
    const double* xn = x + cell_nodes[(long long)c * NV + lane];
#pragma unroll
    for (int k = 0; k < S::KD; ++k) e[k] = biased(__ldg(xn + (k / D) * block + (long long)(k % D) * R));
  }
  short* out = cexp + (long long)c * (2 * S::words);
  if (lane < K * NP)
    out[S::KD + lane] = (short)biased(__ldg(x + (lane / NP) * block + (long long)D * R + (long long)c * NP + lane % NP));
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    unsigned w = __byte_perm((unsigned)e[2 * k], (unsigned)e[2 * k + 1], 0x5410);
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) w = __vmaxs2(w, __shfl_xor_sync(0xffffffffu, w, off));
    if (lane == 0) {
      out[2 * k] = (short)w;
      if (2 * k + 1 < S::KD) out[2 * k + 1] = (short)(w >> 16);
    }
  }
}

// CSR position of node-block position p in a velocity row of time node a
__device__ __forceinline__ int csr_pos(int p, int a, int npv, int npc, int dnn) {
  if (p < npv) return p + (p >= (a + 1) * dnn ? npc : 0);
  return (a + 1) * dnn + (p - npv);
}

// Limbs of the velocity rows, one warp per node: exponents first, then the positions in runs of VL, the KD values of
// a position in KD / 2 planes of 16 bytes (KD planes of 8 for odd KD) so that the VL lanes of a group read whole lines.
// A value of row r (component l) and class k of columns (velocity components of all time nodes, pressure modes) is kept at
// the exponent E[l][k] + rho[r]: rho is that of the row's own component and time node, E the largest exponent above
// it among the rows of component l.
template <int K>
__global__ void __launch_bounds__(256) k_build_limbs(const long long* __restrict__ rowptr, const double* __restrict__ val,
                                                     const int* __restrict__ nbr_ptr, const int* __restrict__ ncell,
                                                     const long long* __restrict__ lbase, int2* __restrict__ out,
                                                     short* __restrict__ nexp, long long block, int R, int VL) {
  using S = Classes<K>;
  constexpr int KD = S::KD, W = KD % 2 ? 1 : 2;
  __shared__ int ex[8][KD][S::row];
  const int lane = threadIdx.x & 31;
  auto e = ex[threadIdx.x >> 5];
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < R; i += nwarps) {
    const int nn = nbr_ptr[i + 1] - nbr_ptr[i], npc = NP * ncell[i], npv = KD * nn, dnn = D * nn;
    const int pad = KD * ((nn + VL - 1) / VL * VL);
    const double* v[KD];
    bool bad = false;
#pragma unroll
    for (int r = 0; r < KD; ++r) {
      v[r] = val + rowptr[(r / D) * block + (long long)(r % D) * R + i];
      for (int k = 0; k < S::row; ++k) {
        const bool vel = k < KD;
        const int p0 = vel ? k * nn : npv + k - KD, p1 = vel ? p0 + nn : npv + npc, step = vel ? 1 : NP;
        int m = kExpZero;
        for (int p = p0 + step * lane; p < p1; p += 32 * step) m = max(m, exp_above(v[r][csr_pos(p, r / D, npv, npc, dnn)]));
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) e[r][k] = m == kExpZero ? kNone : m;
        bad = bad || m > 1024;
      }
    }
    __syncwarp();
    int rho[KD];
#pragma unroll
    for (int r = 0; r < KD; ++r) {
      rho[r] = e[r][r];
      if (rho[r] == kNone) {
        for (int k = 0; k < S::row; ++k) rho[r] = max(rho[r], e[r][k]);
        if (rho[r] == kNone) rho[r] = 0;
      }
    }
    __syncwarp();
    if (lane < S::row) {  // class = lane; e becomes the exponent that the values are kept at
#pragma unroll
      for (int l = 0; l < D; ++l) {
        int m = kNone;
#pragma unroll
        for (int a = 0; a < K; ++a)
          if (e[a * D + l][lane] != kNone) m = max(m, e[a * D + l][lane] - rho[a * D + l]);
        nexp[i * S::node + l * S::row + lane] = (short)(bad ? kPlain : m);
#pragma unroll
        for (int a = 0; a < K; ++a) e[a * D + l][lane] = m == kNone ? 0 : m + rho[a * D + l];
      }
    }
#pragma unroll
    for (int r = 0; r < KD; ++r)
      if (lane == r) nexp[i * S::node + D * S::row + r] = (short)rho[r];
    __syncwarp();
    for (int p = lane; p < npv + npc; p += 32) {
      const bool vel = p < npv;
      const int bm = vel ? p / nn : KD, q = vel ? p - bm * nn : p - npv;  // component and neighbour, or pressure
      const int k = vel ? bm : KD + q % NP;
      const int c0 = q - q % VL;
      int2* o = out + lbase[i] + (vel ? c0 * KD + bm * VL : pad + c0) * KD + (q - c0) * W;
#pragma unroll
      for (int r = 0; r < KD; r += W) {
        int2 l[2];
#pragma unroll
        for (int j = 0; j < W; ++j)
          l[j] = limbs_of(bad ? 0.0 : v[r + j][csr_pos(p, (r + j) / D, npv, npc, dnn)], e[r + j][k]);
        if constexpr (W == 2) *reinterpret_cast<int4*>(o + r * VL) = make_int4(l[0].x, l[0].y, l[1].x, l[1].y);
        else o[r * VL] = l[0];
      }
    }
    __syncwarp();
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
  const short* nexp;
  const short* cexp;
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

// 128 registers and 16 warps per SM; three rows per node (dG(0)) take 80 and 24 warps, nine (3D dG(2)) 168 and 12.
template <int VL, int K>
__global__ void __launch_bounds__(128, K == 1 ? 6 : K == 2 ? 4 : 3) k_spmv_limbs(const __grid_constant__ LimbArgs s) {
  using S = Classes<K>;
  constexpr int GPW = 32 / VL, KD = S::KD, MAXN = 125;
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
  constexpr int kSpare = 7;  // bits by which a row's sum of magnitudes may lie below its scale
  constexpr int CPL = S::words >= 8 ? S::words / 4 : 2;  // classes that each of the first eight lanes looks after
  static_assert(VL % NP == 0, "a lane meets one pressure mode");
  __shared__ int4 cut_sh[4][GPW][2 * S::words];  // per class of x the shifts for each component's rows, and where it is cut
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
      const short* jexp = s.nexp + (long long)i * S::node;
      // the first eight lanes share the classes out (k0 .. k0 + CPL - 1): J's exponents for the rows of each component
      const int k0 = lane >= MAXC ? S::count : K == 1 ? lane & 6 : CPL * lane;
      int je[CPL][D];
#pragma unroll
      for (int q = 0; q < CPL; ++q)
#pragma unroll
        for (int l = 0; l < D; ++l) {
          const int k = k0 + q;
          je[q][l] = k < S::count ? (int)__ldg(jexp + l * S::row + (k < KD ? k : KD + (k - KD) % NP)) : kNone;
        }
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
      if (first) {  // what came before is independent of the exponents
        asm volatile("griddepcontrol.wait;" ::: "memory");
        first = false;
      }
      // largest exponents of x around the node: a lane per cell, whose classes are halved from step to step
      unsigned w[S::words];
#pragma unroll
      for (int k = 0; k < S::words / 4; ++k) {
        int4 e = make_int4(kNonePair, kNonePair, kNonePair, kNonePair);
        if (lane < MAXC && NP * lane < npc) e = __ldcg(reinterpret_cast<const int4*>(s.cexp + (long long)cell * (2 * S::words)) + k);
        w[4 * k] = (unsigned)e.x, w[4 * k + 1] = (unsigned)e.y, w[4 * k + 2] = (unsigned)e.z, w[4 * k + 3] = (unsigned)e.w;
      }
#pragma unroll
      for (int off = MAXC / 2, cnt = S::words; off >= 1; off >>= 1) {
        if (cnt > 1) {
          cnt >>= 1;
          const bool upper = (lane & off) != 0;
#pragma unroll
          for (int k = 0; k < S::words / 2; ++k)
            if (k < cnt) {
              const unsigned send = upper ? w[k] : w[k + cnt], keep = upper ? w[k + cnt] : w[k];
              w[k] = __vmaxs2(keep, __shfl_xor_sync(0xffffffffu, send, off, VL));
            }
        } else {
          w[0] = __vmaxs2(w[0], __shfl_xor_sync(0xffffffffu, w[0], off, VL));
        }
      }
      int t[CPL], top[D];
      bool odd = false;
#pragma unroll
      for (int q = 0; q < CPL; ++q) {
        t[q] = k0 + q < S::count ? (int)(short)(w[q / 2] >> (16 * (q & 1))) : kNone;
        odd = odd || je[q][0] == kPlain || t[q] >= 2047 || (t[q] != kNone && t[q] < 64);
      }
      const unsigned group = (VL == 32 ? 0xffffffffu : (1u << (VL & 31)) - 1) << (VL * gw);
      const bool plain = (__ballot_sync(0xffffffffu, odd) & group) != 0;
      // The sums of a component's rows stand at the largest product of scales among the classes; the entries of the
      // other classes are shifted down to it. Classes that are zero may be cut anywhere.
#pragma unroll
      for (int l = 0; l < D; ++l) {
        top[l] = je[0][l] + t[0];
#pragma unroll
        for (int q = 1; q < CPL; ++q) top[l] = max(top[l], je[q][l] + t[q]);
#pragma unroll
        for (int off = MAXC / 2; off >= 1; off >>= 1) top[l] = max(top[l], __shfl_xor_sync(0xffffffffu, top[l], off, VL));
        if constexpr (VL > MAXC) top[l] = __shfl_sync(0xffffffffu, top[l], 0, VL);
        if (plain || top[l] < kNone / 2) top[l] = kNone;  // all products are zero
      }
#pragma unroll
      for (int q = 0; q < CPL; ++q)
        if (k0 + q < S::count) {
          int sh[3] = {63, 63, 63};
#pragma unroll
          for (int l = 0; l < D; ++l)
            if (top[l] != kNone) sh[l] = min(top[l] - je[q][l] - t[q], 63);
          cut_sh[threadIdx.x >> 5][gw][k0 + q] = make_int4(sh[0], sh[1], sh[2], plain || t[q] == kNone ? 1023 : t[q]);
        }
      __syncwarp();
      const int4* cuts = cut_sh[threadIdx.x >> 5][gw];
      // x in fixed point for the rows of each component
      auto limbs_x = [&](double v, int k, int2* xl) {
        const int4 c = cuts[k];
        const long long q = fixed_below(v, c.w);
        const int sh[3] = {c.x, c.y, c.z};
#pragma unroll
        for (int l = 0; l < D; ++l) {
          const long long u = q >> sh[l];
          xl[l] = make_int2((int)(u >> kLimbBits), (int)((unsigned)u & ((1u << kLimbBits) - 1)));
        }
      };
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
          int2 xl[D];
          limbs_x(x[bm], bm, xl);
          const char* xb = reinterpret_cast<const char*>(s.x + (bm / D) * s.block + (long long)(bm % D) * s.R);
          x[bm] = has ? __ldg(reinterpret_cast<const double*>(xb + node8)) : 0.0;
#pragma unroll
          for (int r = 0; r < KD; ++r) limb_fma(v[bm % PD][r], xl[r % D], h[r], m[r]);
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
      float sp[KD];  // sums of magnitudes over the pressures
#pragma unroll
      for (int r = 0; r < KD; ++r) sp[r] = 0.f;
      for (int r = 0; r < nrw; ++r) {
        int2 pv[KD];
        if (lane + r * VL < npc) load_values<KD, VL>(blkp + r * kRun, pv);
        else
#pragma unroll
          for (int q = 0; q < KD; ++q) pv[q] = make_int2(0, 0);
        int2 xl[K][D];
#pragma unroll
        for (int a = 0; a < K; ++a) limbs_x(xp[a], KD + a * NP + lane % NP, xl[a]);
        if (r + 1 < nrw) pressures(r + 1);
#pragma unroll
        for (int a = 0; a < K; ++a)
#pragma unroll
          for (int l = 0; l < D; ++l) {
            const int r = a * D + l;
            limb_fma(pv[r], xl[a][l], h[r], m[r]);
            sp[r] = fmaf(fabsf((float)pv[r].x), fabsf((float)xl[a][l].x), sp[r]);
          }
      }
      // |J||x| from below: what the lanes' sums and the pressures' magnitudes come to (neighbouring cells' pressures are
      // alike and cancel). Rows where that stays 2^-kSpare below the largest product of scales may owe their value
      // to terms that the scales cut too short.
      unsigned big[(KD + 1) / 2] = {};
#pragma unroll
      for (int r = 0; r < KD; ++r) {
        const unsigned v = (unsigned)abs((int)(h[r] >> 32)) >> (24 - kSpare - 4);  // 2^(56 - kSpare - 4) makes one
        big[r / 2] |= min(v + __float2uint_rz(fminf(sp[r] * (1.f / (1ll << (56 - kSpare - 4))), 2047.f)), 2047u) << (16 * (r & 1));
      }
#pragma unroll
      for (int off = VL / 2; off >= 1; off >>= 1)
#pragma unroll
        for (int k = 0; k < (KD + 1) / 2; ++k) big[k] += __shfl_xor_sync(0xffffffffu, big[k], off, VL);
      unsigned fail = 0;
#pragma unroll
      for (int r = 0; r < KD; ++r)
        if (plain || (((big[r / 2] >> (16 * (r & 1))) & 0xFFFFu) < 16u && top[r % D] != kNone)) fail |= 1u << r;
      double acc[NAV];
#pragma unroll
      for (int r = 0; r < NAV; ++r) acc[r] = r < KD ? fma((double)h[r], (double)(1ll << kLimbBits), (double)m[r]) : 0.0;
      reduce_scatter<VL, NAV>(acc, lane);
      if (ok && (lane & wmask) == 0) {
#pragma unroll
        for (int q = 0; q < HOLD; ++q) {
          const int r = kv + q;
          if (r < KD && !(fail >> r & 1)) {
            int e = top[0];
#pragma unroll
            for (int l = 1; l < D; ++l)
              if (r % D == l) e = top[l];
            e += __ldg(jexp + D * S::row + r) - 1022 - (2 * kLimbTotal - kLimbBits);
            put(s, (r / D) * s.block + (long long)(r % D) * s.R + i, scale_pow2(acc[q], e));
          }
        }
      }
      if (ok && fail)  // in FP64 from the CSR values, by the lanes of the node
        for (; fail; fail &= fail - 1) {
          const int r = __ffs(fail) - 1;
          const long long row = (r / D) * s.block + (long long)(r % D) * s.R + i, end = s.rowptr[row + 1];
          double t = 0.0;
#pragma unroll 4
          for (long long e = s.rowptr[row] + lane; e < end; e += VL) t = fma(s.val[e], s.x[s.col[e]], t);
#pragma unroll
          for (int off = VL / 2; off >= 1; off >>= 1) t += __shfl_xor_sync(group, t, off, VL);
          if (lane == 0) put(s, row, t);
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

template <int VL, int K>
stm_status launch(const Level& L, LimbArgs& a, cudaStream_t s) {
  static int occ = 0;
  if (!occ) {
    int o = 0;
    STM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_spmv_limbs<VL, K>, 128, 0));
    occ = std::max(o, 1);
  }
  const unsigned npu = (unsigned)(((long long)K * L.C * NP + 31) / 32);
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
  STM_CUDA(cudaLaunchKernelEx(&cfg, k_spmv_limbs<VL, K>, a));
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

template <int K>
stm_status launch_vl(const Level& L, LimbArgs& a, cudaStream_t s) {
  k_cell_exps<K><<<(L.C + 7) / 8, 256, 0, s>>>(L.cell_nodes, a.x, L.C, L.block, L.R, L.cexp);
  note_launch();
  STM_CUDA(cudaGetLastError());
  if constexpr (K < 3)  // 127 positions per lane at most
    if (L.limb_lanes == 8) return launch<8, K>(L, a, s);
  return L.limb_lanes == 16 ? launch<16, K>(L, a, s) : launch<32, K>(L, a, s);
}

}  // namespace

stm_status build_limbs(const Level& L, const double* val, double* nval, short* nexp, cudaStream_t s) {
  const int blocks = (int)std::min<long long>(((long long)L.R * 32 + 255) / 256, sm_count() * 8LL);
  int2* o = reinterpret_cast<int2*>(nval);
#define STM_BUILD(K) \
  k_build_limbs<K><<<blocks, 256, 0, s>>>(L.rowptr, val, L.nbr_ptr, L.ncell, L.lbase, o, nexp, L.block, L.R, L.limb_lanes)
  switch (L.K) {
    case 1: STM_BUILD(1); break;
    case 2: STM_BUILD(2); break;
    default: STM_BUILD(3); break;
  }
#undef STM_BUILD
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

// 3D levels keep limbs whatever their size. Normally distributed x gains 7 to 40 % everywhere; the vectors of V-cycles, which
// send rows to the FP64 sums (us per launch inside FGMRES, FP64 against this): dG(0), 1,024 cells 49 -> 38, 2,048 65 -> 48,
// 4,608 72 -> 70, 16,384 185 -> 187; dG(1), 1,024 cells 69 -> 73, 2,048 95 -> 103, 3,072 160 -> 149, 4,608 183 -> 203, 8,192
// 300 -> 303, 16,384 576 -> 555. 2D levels do not: dG(2) gained 9 % only (544,518 unknowns: 102 -> 93 us), and
// the vectors of its V-cycles sent a third of the rows to the FP64 sums. Lanes per node as in the FP64 product but for
// 3D dG(2) (16 at least: a lane of 8 would see more positions than its sums hold).
int limb_lanes(const Level& L) { return L.dim == 3 ? std::max(node_lanes(L), L.K == 3 ? 16 : 8) : 0; }

size_t limb_node_exps(const Level& L) {
  const int kd = L.K * D;
  return sizeof(short) * (size_t)L.R * (D * (kd + NP) + kd);
}
size_t limb_cell_exps(const Level& L) { return sizeof(short) * (size_t)L.C * (L.K == 1 ? 8 : L.K == 2 ? 16 : 32); }

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
  switch (L.K) {
    case 1: return launch_vl<1>(L, a, s);
    case 2: return launch_vl<2>(L, a, s);
    default: return launch_vl<3>(L, a, s);
  }
}

}  // namespace stm
