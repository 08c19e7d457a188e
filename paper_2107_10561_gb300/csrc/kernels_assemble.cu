// Assembly of the slab Jacobian J_g on the GPU (FP64).
//
// J_g = sum_T R_T^T E_T R_T with the element blocks of Problem 3.1 linearised as in Eq. linNewEq:
//   velocity-velocity (a,l,i; b,m,j): D_ab M_ij d_lm + Mt_ab A_l,ij d_lm + sum_c T_abc N(w^c)_lm,ij
//   velocity-pressure (a,l,i; a,q)  : Mt_aa Bc_l,iq    pressure-velocity (a,q; a,m,j): Mt_aa Br_m,qj
// with A the diffusion + Nitsche operator (Eqs. Def:Ah, Def:B_GamD) and
//   N(w)_lm,ij = ((w . grad) phi_j d_lm + phi_j d_m w_l, phi_i).
// Cells are processed colour by colour (cells of one colour share no node), so every CSR entry
// is updated by at most one thread at a time: no atomics, bitwise reproducible.
#include <cmath>

#include "internal.h"

namespace stm {

// ---------------------------------------------------------------------------------------------
// CSR column indices from the structured pattern
// ---------------------------------------------------------------------------------------------
__global__ void k_fill_colidx(const long long* __restrict__ rowptr, int* __restrict__ colidx,
                              const int* __restrict__ nbr_ptr, const int* __restrict__ nbr,
                              const int* __restrict__ node_cells, const int* __restrict__ cell_nodes,
                              long long N, long long block, int R, int d, int K, int nv, int np,
                              int maxc) {
  const long long warps = (long long)gridDim.x * (blockDim.x / 32);
  const int lane = threadIdx.x & 31;
  for (long long row = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; row < N; row += warps) {
    const int a = (int)(row / block);
    const long long r = row - a * block;
    const long long base = rowptr[row];
    const int len = (int)(rowptr[row + 1] - base);
    if (r < (long long)d * R) {
      const int node = (int)(r % R);
      const int p0 = nbr_ptr[node];
      const int nn = nbr_ptr[node + 1] - p0;
      int nc = 0;
      while (nc < maxc && node_cells[(long long)node * maxc + nc] >= 0) ++nc;
      for (int p = lane; p < len; p += 32) {
        // columns per time block b: d*nn velocity, plus n_p*nc pressure when b == a
        int off = p, b = 0;
        for (; b < K; ++b) {
          const int sz = d * nn + (b == a ? np * nc : 0);
          if (off < sz) break;
          off -= sz;
        }
        long long col;
        if (off < d * nn) {
          const int m = off / nn, j = off - m * nn;
          col = b * block + (long long)m * R + nbr[p0 + j];
        } else {
          const int t = off - d * nn;
          const int ci = t / np, q = t - ci * np;
          col = a * block + (long long)d * R + (long long)node_cells[(long long)node * maxc + ci] * np + q;
        }
        colidx[base + p] = (int)col;
      }
    } else {
      const long long pr = r - (long long)d * R;
      const int c = (int)(pr / np);
      for (int p = lane; p < len; p += 32) {
        const int m = p / nv, j = p - m * nv;
        colidx[base + p] = (int)(a * block + (long long)m * R + cell_nodes[c * nv + j]);
      }
    }
  }
}

stm_status launch_fill_colidx(Level& L, const int* nbr_ptr, const int* nbr, const int* node_cells,
                              cudaStream_t s) {
  const int threads = 256;
  long long warps_needed = L.N;
  int blocks = (int)std::min<long long>((warps_needed + 7) / 8, sm_count() * 64LL);
  k_fill_colidx<<<blocks, threads, 0, s>>>(L.rowptr, L.colidx, nbr_ptr, nbr, node_cells, L.cell_nodes,
                                           L.N, L.block, L.R, L.dim, L.K, L.nv, L.np, 1 << L.dim); note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

// ---------------------------------------------------------------------------------------------
// Linearisation point on every level (injection: coarse nodes are fine nodes)
// ---------------------------------------------------------------------------------------------
__global__ void k_inject(const double* __restrict__ X, double* __restrict__ wnod,
                         const int* __restrict__ inj, int R, int K, int d, long long blockF, int RF) {
  const long long total = (long long)K * d * R;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int node = (int)(e % R);
    const int al = (int)(e / R);  // a * d + l
    const int a = al / d, l = al - a * d;
    wnod[e] = X[a * blockF + (long long)l * RF + inj[node]];
  }
}

stm_status inject_level(const Hierarchy& H, int g, const double* X, double* wnod, cudaStream_t s) {
  const Level& F = H.L.back();
  const Level& L = H.L[g];
  long long total = (long long)L.K * L.dim * L.R;
  int blocks = (int)std::min<long long>((total + 255) / 256, sm_count() * 16LL);
  k_inject<<<std::max(blocks, 1), 256, 0, s>>>(X, wnod, L.inj, L.R, L.K, L.dim, F.block, F.R);
  note_launch();
  STM_CUDA(cudaGetLastError());
  return STM_OK;
}

stm_status inject_linearisation(Hierarchy& H, const double* X, cudaStream_t s) {
  const Level& F = H.L.back();
  for (Level& L : H.L) {
    long long total = (long long)L.K * L.dim * L.R;
    int blocks = (int)std::min<long long>((total + 255) / 256, sm_count() * 16LL);
    k_inject<<<blocks, 256, 0, s>>>(X, L.wnod, L.inj, L.R, L.K, L.dim, F.block, F.R); note_launch();
    STM_CUDA(cudaGetLastError());
  }
  return STM_OK;
}

// ---------------------------------------------------------------------------------------------
// Element assembly
// ---------------------------------------------------------------------------------------------
struct AsmConst {
  double Mt[3][3], D[3][3], T[3][3][3];
  double nu, g1, g2, hT;
  // 1D integrals [axis][s * 9 + i * 3 + j] of the Q2 basis: phi_s phi_i phi_j (times h), phi_s' phi_i phi_j and
  // phi_s phi_i phi_j'
  double c00[3][27], c10[27], c01[27];
};

// One cell per CTA slot (3D: the CTA, 2D: 81 of its threads). On a uniform level the convection blocks
//   N(w)_lm,ij = ((w . grad) phi_j d_lm + phi_j d_m w_l, phi_i)
// are contractions of the cell's nodal velocities with products of 1D integrals, so they are formed axis by
// axis: x and y into shared memory, z (2D: y) by the thread that owns the pair (i, j). That is 36 FMAs per
// pair and time pair (a, b) in 3D, where the quadrature sums took 896 per time node, and the FP64 pipe (2
// FMAs per clock and SM) was what bounded the kernel. The nodal velocities are combined over time first:
// sum_c T_abc w^c, symmetric in a and b. All levels of 2,016 + 252 cells, 3D dG(1): 12.3 -> 2.2 ms; 21,483
// cells, 2D dG(2), twice: 10.5 -> 3.6 ms.
template <int K, int D>
__global__ void __launch_bounds__(256) k_assemble(
    const int* __restrict__ cells, int ncells, const int* __restrict__ cell_nodes,
    const unsigned char* __restrict__ bmask, const unsigned char* __restrict__ rank,
    const unsigned char* __restrict__ cellrank, const int* __restrict__ nn, const int* __restrict__ ncell,
    const long long* __restrict__ rowptr, double* __restrict__ val, const double* __restrict__ wnod,
    const double* __restrict__ ref, RefOffsets ro, const __grid_constant__ AsmConst ac, int R, long long block) {
  constexpr int nv = D == 2 ? 9 : 27, np = D + 1, KD = K * D;
  constexpr int CPB = D == 2 ? 3 : 1, TPC = D == 2 ? 81 : 256;  // cells per CTA, threads per cell
  constexpr int S2 = D == 2 ? 3 : 9;                            // nodes across the x axis
  constexpr int NA = 3 * 9 * S2, NB = D == 2 ? 0 : 4 * 9 * 9 * 3;  // x results (three kinds), y results (four)
  __shared__ double cx[3][27], c10[27], c01[27];
  __shared__ double wall[CPB][K][D][nv], was[CPB][D][nv];
  __shared__ long long rbs[CPB][KD * nv];
  extern __shared__ double dyn[];  // [CPB][D][NA + NB]
  for (int e = threadIdx.x; e < 81; e += 256) cx[e / 27][e % 27] = ac.c00[e / 27][e % 27];
  for (int e = threadIdx.x; e < 27; e += 256) {
    c10[e] = ac.c10[e];
    c01[e] = ac.c01[e];
  }
  const int sub = threadIdx.x / TPC, tid = threadIdx.x - sub * TPC;
  const bool on = sub < CPB;
  const double* Mm = ref + ro.M;
  const double* Ks = ref + ro.Kst;
  const double* Div = ref + ro.Div;
  for (int c0 = blockIdx.x * CPB; c0 < ncells; c0 += gridDim.x * CPB) {
    const bool act = on && c0 + sub < ncells;
    const int c = act ? cells[c0 + sub] : 0;
    const int* cn = cell_nodes + (long long)c * nv;
    const unsigned mask = bmask[c];
    __syncthreads();  // the tables are there; the cell before is done
    if (act) {
      for (int e = tid; e < KD * nv; e += TPC) {
        const int s = e % nv, al = e / nv;
        wall[sub][al / D][al % D][s] = wnod[(long long)al * R + cn[s]];
        rbs[sub][e] = rowptr[(al / D) * block + (long long)(al % D) * R + cn[s]];
      }
    }
    double* A = dyn + (on ? sub : 0) * (D * (NA + NB));
    double* B = A + D * NA;
#pragma unroll 1
    for (int a = 0; a < K; ++a)
#pragma unroll 1
      for (int b = a; b < K; ++b) {
        __syncthreads();
        if (act)
          for (int e = tid; e < D * nv; e += TPC) {
            double v = 0.0;
#pragma unroll
            for (int k = 0; k < K; ++k) v += ac.T[a][b][k] * wall[sub][k][e / nv][e % nv];
            was[sub][e / nv][e % nv] = v;
          }
        __syncthreads();
        // along x: kind 0 phi phi phi, 1 phi_s' phi phi, 2 phi phi phi_j' (component 0 only)
        if (act)
          for (int e = tid; e < D * 9 * S2; e += TPC) {
            const int l = e / (9 * S2), f = e - l * (9 * S2), ij = f / S2, s = f - ij * S2;
            const double* w = &was[sub][l][3 * s];
            double v0 = 0.0, v1 = 0.0, v2 = 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              v0 = fma(cx[0][k * 9 + ij], w[k], v0);
              v1 = fma(c10[k * 9 + ij], w[k], v1);
              if (l == 0) v2 = fma(c01[k * 9 + ij], w[k], v2);
            }
            A[l * NA + f] = v0;
            A[l * NA + 9 * S2 + f] = v1;
            A[l * NA + 18 * S2 + f] = v2;
          }
        __syncthreads();
        if (D == 3) {
          // along y: kinds 0 (d_z), 1 (d_x), 2 (d_y) of the gradient, 3 for the advection by this component
          if (act)
            for (int e = tid; e < D * 243; e += TPC) {
              const int l = e / 243, f = e - l * 243, ij1 = f / 27, g = f - ij1 * 27, ij2 = g / 3, s3 = g - ij2 * 3;
              const double* a0 = A + l * NA + ij1 * S2 + 3 * s3;
              double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
#pragma unroll
              for (int k = 0; k < 3; ++k) {
                const double y = cx[1][k * 9 + ij2], z0 = a0[k];
                v0 = fma(y, z0, v0);
                v1 = fma(y, a0[9 * S2 + k], v1);
                v2 = fma(c10[k * 9 + ij2], z0, v2);
                if (l == 0) v3 = fma(y, a0[18 * S2 + k], v3);
                if (l == 1) v3 = fma(c01[k * 9 + ij2], z0, v3);
              }
              double* o = B + l * NB + f;
              o[0] = v0;
              o[243] = v1;
              o[486] = v2;
              o[729] = l == 2 ? v0 : v3;
            }
          __syncthreads();
        }
        // the last axis, and everything else of the pair's entries (a, l; b, m) and (b, l; a, m)
        if (act)
          for (int e = tid; e < nv * nv; e += TPC) {
            const int i = e / nv, j = e - i * nv;
            const int i1 = i % 3, i2 = (i / 3) % 3, i3 = i / 9, j1 = j % 3, j2 = (j / 3) % 3, j3 = j / 9;
            const int ij1 = i1 * 3 + j1, ij2 = i2 * 3 + j2, ij3 = i3 * 3 + j3;
            double G[D][D], adv = 0.0;
#pragma unroll
            for (int l = 0; l < D; ++l) {
#pragma unroll
              for (int m = 0; m < D; ++m) G[l][m] = 0.0;
#pragma unroll
              for (int k = 0; k < 3; ++k) {
                if (D == 2) {
                  const double* x = A + l * NA + ij1 * S2 + k;
                  const double y = cx[1][k * 9 + ij2];
                  G[l][0] = fma(y, x[9 * S2], G[l][0]);
                  G[l][1] = fma(c10[k * 9 + ij2], x[0], G[l][1]);
                  adv = fma(l == 0 ? y : c01[k * 9 + ij2], l == 0 ? x[18 * S2] : x[0], adv);
                } else {
                  const double* x = B + l * NB + ij1 * 27 + ij2 * 3 + k;
                  const double z = cx[2][k * 9 + ij3];
                  G[l][0] = fma(z, x[243], G[l][0]);
                  G[l][1] = fma(z, x[486], G[l][1]);
                  G[l][D - 1] = fma(c10[k * 9 + ij3], x[0], G[l][D - 1]);
                  adv = fma(l == 2 ? c01[k * 9 + ij3] : z, x[729], adv);
                }
              }
            }
            // diffusion + Nitsche part (identical for all components except the gamma2 normal term)
            double base = ac.nu * Ks[i * nv + j];
            double g2[D];
#pragma unroll
            for (int m = 0; m < D; ++m) g2[m] = 0.0;
            if (mask)
#pragma unroll
              for (int f = 0; f < 2 * D; ++f)
                if (mask & (1u << f)) {
                  const double* F = ref + ro.face0 + f * ro.face_stride;
                  base += -ac.nu * F[ro.fG + i * nv + j] - ac.nu * F[ro.fG + j * nv + i] +
                          ac.g1 * ac.nu / ac.hT * F[ro.fS + i * nv + j];
                  g2[f / 2] += ac.g2 / ac.hT * F[ro.fS + i * nv + j];
                }
            const int node_i = cn[i];
            const int nni = nn[node_i], npc = np * ncell[node_i];
            const int rk = rank[((long long)c * nv + i) * nv + j];
            const double mass = Mm[i * nv + j];
#pragma unroll
            for (int side = 0; side < 2; ++side) {
              if (side == 1 && a == b) break;
              const int ta = side ? b : a, tb = side ? a : b;
#pragma unroll
              for (int l = 0; l < D; ++l) {
                const double diag = ac.D[ta][tb] * mass + ac.Mt[ta][tb] * (base + g2[l]) + adv;
                const long long pb = rbs[sub][(ta * D + l) * nv + i] + tb * D * nni + (tb > ta ? npc : 0) + rk;
#pragma unroll
                for (int m = 0; m < D; ++m) val[pb + m * nni] += G[l][m] + (m == l ? diag : 0.0);
              }
            }
          }
      }
    // pressure couplings (time-diagonal because the Radau-Lagrange time mass is diagonal)
    if (act)
      for (int e = tid; e < KD * nv * np; e += TPC) {
        const int q = e % np, i = (e / np) % nv, l = (e / (np * nv)) % D, a = e / (np * nv * D);
        const double dv = Div[(l * np + q) * nv + i];
        double bc = -dv, br = dv;
        for (int f = 2 * l; f < 2 * l + 2; ++f)
          if (mask & (1u << f)) {
            const double p = (2.0 * (f & 1) - 1.0) * ref[ro.face0 + f * ro.face_stride + ro.fPf + q * nv + i];
            bc += p;
            br -= p;
          }
        const int nni = nn[cn[i]];
        const long long pos = rbs[sub][(a * D + l) * nv + i] + (long long)(a + 1) * D * nni +
                              (long long)cellrank[(long long)c * nv + i] * np + q;
        val[pos] += ac.Mt[a][a] * bc;
        // pressure row (a, q) against velocity (a, l, i): Br_l,qi
        val[rowptr[a * block + (long long)D * R + (long long)c * np + q] + (long long)l * nv + i] += ac.Mt[a][a] * br;
      }
  }
}

template <int K, int D>
static stm_status launch_assemble(Level& L, const AsmConst& ac, cudaStream_t s) {
  constexpr int CPB = D == 2 ? 3 : 1, S2 = D == 2 ? 3 : 9;
  const size_t smem = sizeof(double) * CPB * D * (3 * 9 * S2 + (D == 2 ? 0 : 4 * 243));
  STM_CUDA(cudaFuncSetAttribute(k_assemble<K, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  for (int col = 0; col < (1 << D); ++col) {
    const int nc = L.colour_off[col + 1] - L.colour_off[col];
    if (nc == 0) continue;
    k_assemble<K, D><<<std::min((nc + CPB - 1) / CPB, sm_count() * 8), 256, smem, s>>>(
        L.colour_cells + L.colour_off[col], nc, L.cell_nodes, L.bmask, L.rank, L.cellrank, L.nn, L.ncell, L.rowptr,
        L.val, L.wnod, L.ref, L.ro, ac, L.R, L.block);
    note_launch();
    STM_CUDA(cudaGetLastError());
  }
  return STM_OK;
}

// 1D integrals of products of three Q2 basis functions, by the 4-point Gauss rule (exact to degree 7)
static void triple_products(const Level& L, AsmConst& ac) {
  const double x1 = std::sqrt(3.0 / 7.0 - 2.0 / 7.0 * std::sqrt(6.0 / 5.0)), w1 = (18.0 + std::sqrt(30.0)) / 72.0;
  const double x2 = std::sqrt(3.0 / 7.0 + 2.0 / 7.0 * std::sqrt(6.0 / 5.0)), w2 = (18.0 - std::sqrt(30.0)) / 72.0;
  const double X[4] = {0.5 * (1 - x2), 0.5 * (1 - x1), 0.5 * (1 + x1), 0.5 * (1 + x2)}, W[4] = {w2, w1, w1, w2};
  for (int e = 0; e < 27; ++e) {
    const int s = e / 9, i = (e / 3) % 3, j = e % 3;
    double v = 0.0, d0 = 0.0, d1 = 0.0;
    for (int q = 0; q < 4; ++q) {
      const double x = X[q];
      const double f[3] = {2.0 * (x - 0.5) * (x - 1.0), -4.0 * x * (x - 1.0), 2.0 * x * (x - 0.5)};
      const double g[3] = {4.0 * x - 3.0, -8.0 * x + 4.0, 4.0 * x - 1.0};
      v += W[q] * f[s] * f[i] * f[j];
      d0 += W[q] * g[s] * f[i] * f[j];
      d1 += W[q] * f[s] * f[i] * g[j];
    }
    for (int m = 0; m < 3; ++m) ac.c00[m][e] = v * L.h[m];
    ac.c10[e] = d0;
    ac.c01[e] = d1;
  }
}

stm_status assemble_level(Hierarchy& H, int g, double nu, cudaStream_t s) {
  Level& L = H.L[g];
  STM_CUDA(cudaMemsetAsync(L.val, 0, sizeof(double) * L.nnz, s));
  AsmConst ac;
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) {
      ac.Mt[a][b] = H.Mt[a][b];
      ac.D[a][b] = H.D[a][b];
      for (int c = 0; c < 3; ++c) ac.T[a][b][c] = H.T[a][b][c];
    }
  ac.nu = nu;
  ac.g1 = H.p.gamma1;
  ac.g2 = H.p.gamma2;
  ac.hT = L.hT;
  triple_products(L, ac);
  switch (L.dim * 10 + L.K) {
    case 21: STM_TRY((launch_assemble<1, 2>(L, ac, s))); break;
    case 22: STM_TRY((launch_assemble<2, 2>(L, ac, s))); break;
    case 23: STM_TRY((launch_assemble<3, 2>(L, ac, s))); break;
    case 31: STM_TRY((launch_assemble<1, 3>(L, ac, s))); break;
    case 32: STM_TRY((launch_assemble<2, 3>(L, ac, s))); break;
    default: STM_TRY((launch_assemble<3, 3>(L, ac, s))); break;
  }
  L.jw_current[0] = L.jw_current[1] = false;
  if (L.valT) {
    cudaFree(L.valT);
    L.valT = nullptr;
  }
  if (L.nvalJT) {
    cudaFree(L.nvalJT);
    L.nvalJT = nullptr;
  }
  if (L.nexpJT) {
    cudaFree(L.nexpJT);
    L.nexpJT = nullptr;
  }
  if (L.pvalJT) {
    cudaFree(L.pvalJT);
    L.pvalJT = nullptr;
  }
  STM_TRY(build_nodeblock(L, 0, s));
  // FP32 defect copies follow the new values (J^T's are rebuilt with J^T)
  if (H.p.defect_precision == STM_F32) STM_TRY(build_values_f32(L, 0, s));
  return STM_OK;
}

}  // namespace stm
