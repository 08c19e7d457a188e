// The coarse direct solver's factors (FP64; products and inverses of blocks in kernels_dense.cu).
#include <cfloat>

#include "internal.h"

namespace stm {

// ---------------------------------------------------------------------------------------------
// Coarse level: explicit FP64 inverse of J_0 by Gauss-Jordan with partial pivoting in global memory
// ---------------------------------------------------------------------------------------------
// scal[0] = 1/pivot, scal[1] = old A[k][k]; piv[k] = pivot row
__global__ void k_gj_pivot(double* A, long long n, int k, int* piv, double* scal, int* flag) {
  __shared__ double sb[32];
  __shared__ int si[32];
  double best = -1.0;
  int bi = (int)n;
  for (long long i = k + threadIdx.x; i < n; i += blockDim.x) {
    const double v = fabs(A[i * n + k]);
    if (v > best) { best = v; bi = (int)i; }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const double ob = __shfl_down_sync(0xffffffffu, best, off);
    const int oi = __shfl_down_sync(0xffffffffu, bi, off);
    if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
  }
  if ((threadIdx.x & 31) == 0) { sb[threadIdx.x / 32] = best; si[threadIdx.x / 32] = bi; }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int nw = blockDim.x / 32;
    best = threadIdx.x < nw ? sb[threadIdx.x] : -1.0;
    bi = threadIdx.x < nw ? si[threadIdx.x] : (int)n;
    for (int off = 16; off > 0; off >>= 1) {
      const double ob = __shfl_down_sync(0xffffffffu, best, off);
      const int oi = __shfl_down_sync(0xffffffffu, bi, off);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (threadIdx.x == 0) {
      if (!(best > 0.0) || !(best <= DBL_MAX)) {
        *flag = 1;
        bi = k;
        scal[0] = 0.0;
      } else {
        scal[0] = 1.0 / A[(long long)bi * n + k];
      }
      piv[k] = bi;
      scal[1] = A[(long long)k * n + k];
    }
  }
}

// rows k <-> p for all columns j != k, then scale row k
__global__ void k_gj_swap_scale(double* A, long long n, int k, const int* piv, const double* scal) {
  const int p = piv[k];
  const double pinv = scal[0];
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x) {
    if (j == k) continue;
    const double t = A[(long long)k * n + j];
    const double u = A[(long long)p * n + j];
    A[(long long)p * n + j] = t;
    A[(long long)k * n + j] = u * pinv;
  }
}

// A[i][j] -= A[i][k] A[k][j] for i != k, j != k; column k is still unswapped: row p holds old row k
__global__ void k_gj_update(double* A, long long n, int k, const int* piv, const double* scal) {
  const int p = piv[k];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * n; e += (long long)gridDim.x * blockDim.x) {
    const long long i = e / n, j = e - i * n;
    if (i == k || j == k) continue;
    const double aik = (i == p) ? scal[1] : A[i * n + k];
    A[e] -= aik * A[(long long)k * n + j];
  }
}

__global__ void k_gj_column(double* A, long long n, int k, const int* piv, const double* scal) {
  const int p = piv[k];
  const double pinv = scal[0];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (i == k) {
      A[(long long)k * n + k] = pinv;
    } else {
      const double aik = (i == p) ? scal[1] : A[i * n + k];
      A[i * n + k] = -aik * pinv;
    }
  }
}

__global__ void k_gj_colswap(double* A, long long n, int k, const int* piv) {
  const int p = piv[k];
  if (p == k) return;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double t = A[i * n + k];
    A[i * n + k] = A[i * n + p];
    A[i * n + p] = t;
  }
}

// ---------------------------------------------------------------------------------------------
// Coarse direct solver (Algorithm 1, level 1): the explicit inverse of J_0 from a block LU over
// x-slabs. Velocity DoFs go to the slab of their node's lattice plane (planes 2b, 2b+1 -> slab b,
// the last plane with the last slab), the pressure of cell i to slab i+1 (the last cell's to the
// last slab). A Q2 cell spans the planes 2i..2i+2, so J_0 is block tridiagonal in this order, and
// every slab's pressure is eliminated after the velocities of the cell that carries it, which keeps
// the Schur complements regular (with the pressure of cell b in slab b, S_0 is singular: its
// pressure sees only velocities whose neighbours across the slab face were cut away). Block LU
// without pivoting across slabs, Gauss-Jordan with partial pivoting inside each Schur complement:
//   S_0 = A_00,  S_b = A_bb - A_{b,b-1} W_{b-1},  W_b = S_b^{-1} A_{b,b+1},  G_b = S_b^{-1} A_{b,b-1};
// then the inverse, L^{-1} forward (Z_bb = S_b^{-1}, Z_bj = -G_b Z_{b-1,j}) and U^{-1} backward
// (X_b = Z_b - W_b X_{b+1}), and finally the slab permutation is undone.
// ---------------------------------------------------------------------------------------------

// Dense slab blocks from the CSR of J_0: row r of slab b (permuted index pr = iperm[r]) scatters its
// entries into D_b (same slab), Lo_b (slab b-1) or Up_b (slab b+1); anything else flags an error. Pressure
// rows and columns (from dR on in every time node's block) are scaled.
__global__ void k_slab_blocks(const long long* __restrict__ rowptr, const int* __restrict__ col,
                              const double* __restrict__ val, long long n, const int* __restrict__ iperm,
                              const int* __restrict__ blk, const long long* __restrict__ off,
                              const long long* __restrict__ dpos, const long long* __restrict__ lpos,
                              const long long* __restrict__ upos, double* __restrict__ store, int* flag,
                              long long block, long long dR, double scale) {
  for (long long r = blockIdx.x; r < n; r += gridDim.x) {
    const double fr = r % block >= dR ? scale : 1.0;
    const int pr = iperm[r];
    const int b = blk[pr];
    const long long i = pr - off[b];
    const long long nb = off[b + 1] - off[b];
    for (long long e = rowptr[r] + threadIdx.x; e < rowptr[r + 1]; e += blockDim.x) {
      const int pc = iperm[col[e]];
      const double v = val[e] * (col[e] % block >= dR ? fr * scale : fr);
      const int bc = blk[pc];
      if (bc == b) {
        store[dpos[b] + i * nb + (pc - off[b])] = v;
      } else if (bc == b - 1) {
        store[lpos[b] + i * (off[b] - off[b - 1]) + (pc - off[b - 1])] = v;
      } else if (bc == b + 1) {
        store[upos[b] + i * (off[b + 2] - off[b + 1]) + (pc - off[b + 1])] = v;
      } else {
        atomicExch(flag, 1);
      }
    }
  }
}

// Explicit inverse of a dense n x n block in global memory, one pivot at a time (blocks with more rows
// than a cluster's shared memory holds as one panel, see dense_max_inverse).
static void block_inverse_global(double* M, long long n, int* piv, double* scal, int* flag, cudaStream_t s) {
  const int vb = (int)std::min<long long>((n + 255) / 256, sm_count() * 8LL);
  const int mb = (int)std::min<long long>((n * n + 255) / 256, sm_count() * 32LL);
  for (int k = 0; k < n; ++k) {
    k_gj_pivot<<<1, 1024, 0, s>>>(M, n, k, piv, scal, flag); note_launch();
    k_gj_swap_scale<<<vb, 256, 0, s>>>(M, n, k, piv, scal); note_launch();
    k_gj_update<<<mb, 256, 0, s>>>(M, n, k, piv, scal); note_launch();
    k_gj_column<<<vb, 256, 0, s>>>(M, n, k, piv, scal); note_launch();
  }
  for (int k = (int)n - 1; k >= 0; --k) {
    k_gj_colswap<<<vb, 256, 0, s>>>(M, n, k, piv);
    note_launch();
  }
}

__global__ void k_copy_block(const double* __restrict__ src, long long rows, long long cols, long long lds,
                             double* __restrict__ dst, long long ldd) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < rows * cols;
       e += (long long)gridDim.x * blockDim.x) {
    const long long i = e / cols, j = e - i * cols;
    dst[i * ldd + j] = src[i * lds + j];
  }
}

// cinv[i][j] = Xp[iperm[i]][iperm[j]], the scaling undone
__global__ void k_unpermute(const double* __restrict__ Xp, const int* __restrict__ iperm, long long n,
                            double* __restrict__ out, long long block, long long dR, double scale) {
  for (long long i = blockIdx.y; i < n; i += gridDim.y) {
    const double* src = Xp + (long long)iperm[i] * n;
    const double fi = i % block >= dR ? scale : 1.0;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x)
      out[i * n + j] = src[iperm[j]] * (j % block >= dR ? fi * scale : fi);
  }
}

// dst (cols x rows) = src^T (src rows x cols, both row-major)
__global__ void k_transpose(const double* __restrict__ src, long long rows, long long cols, double* __restrict__ dst) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < rows * cols;
       e += (long long)gridDim.x * blockDim.x) {
    const long long i = e / cols, j = e - i * cols;
    dst[j * rows + i] = src[e];
  }
}
static void transpose_block(const double* src, long long rows, long long cols, double* dst, cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return;
  k_transpose<<<(int)std::min<long long>((rows * cols + 255) / 256, sm_count() * 8LL), 256, 0, s>>>(src, rows, cols, dst);
  note_launch();
}

// Coarse levels from this size on are solved through the twisted slab factors instead of an explicit
// inverse: the dense inverse costs N^2 FP64 FMAs per solve (0.5 ms at 18,000 DoFs), the factors about a
// fifth of that in about nx dependent slab steps.
constexpr long long kCoarseSlabMinDofs = 8000;

// Slab ordering of level 0 (host, once). The pressure of cell i goes to slab i + 1 (the last cell's to the
// last slab) when the slabs are eliminated upwards (i < tw), and to slab i when they are eliminated
// downwards (i >= tw, the lower half of the twisted factorisation): either way it is eliminated after the
// velocities of the cell's far plane, which keeps the Schur complements regular.
static void coarse_slabs(const Level& L, int tw, std::vector<int>& iperm, std::vector<int>& blk,
                         std::vector<long long>& off) {
  const int d = L.dim, nx = L.cells[0];
  const long long n = L.N;
  std::vector<int> slab(n);
  for (int a = 0; a < L.K; ++a) {
    for (int l = 0; l < d; ++l)
      for (int nd = 0; nd < L.R; ++nd) {
        const int lx = L.h_node_lat[nd] % L.lat[0];
        slab[a * L.block + (long long)l * L.R + nd] = std::min(lx / 2, nx - 1);
      }
    for (int c = 0; c < L.C; ++c)
      for (int q = 0; q < L.np; ++q)
        slab[a * L.block + (long long)d * L.R + (long long)c * L.np + q] =
            L.h_cell_xyz[3 * c] < tw ? std::min(L.h_cell_xyz[3 * c] + 1, nx - 1) : L.h_cell_xyz[3 * c];
  }
  off.assign(nx + 2, 0);
  for (long long r = 0; r < n; ++r) off[slab[r] + 1]++;
  for (int b = 0; b < nx; ++b) off[b + 1] += off[b];
  off[nx + 1] = off[nx];
  iperm.assign(n, 0);
  blk.assign(n, 0);
  std::vector<long long> fill(off.begin(), off.begin() + nx);
  for (long long r = 0; r < n; ++r) {
    const long long pr = fill[slab[r]]++;
    iperm[r] = (int)pr;
    blk[pr] = slab[r];
  }
}

// Inverse of one dense FP64 block (Gauss-Jordan, partial pivoting); M is overwritten.
static stm_status invert_block(DenseWork& w, double* M, long long nb, double* out, int* flag, double* scal,
                               cudaStream_t s) {
  if (nb <= dense_max_inverse()) return dense_inverse(w, M, (int)nb, out, flag, s);
  block_inverse_global(M, nb, w.piv, scal, flag, s);
  STM_CUDA(cudaMemcpyAsync(out, M, sizeof(double) * nb * nb, cudaMemcpyDeviceToDevice, s));
  return STM_OK;
}

// Twisted block factorisation of J_0 in slab order, eliminated from both ends towards slab t = nx / 2
// (A_bc the blocks of J_0, nb_b the rows of slab b):
//   top    b < t :  S_b = A_bb - A_{b,b-1} W_{b-1},            W_b = S_b^{-1} A_{b,b+1},  G_b  = S_b^{-1} A_{b,b-1}
//   bottom b > t :  S_b = A_bb - A_{b,b+1} V_{b+1},            V_b = S_b^{-1} A_{b,b-1},  G'_b = S_b^{-1} A_{b,b+1}
//   middle b = t :  S_t = A_tt - A_{t,t-1} W_{t-1} - A_{t,t+1} V_{t+1},  G_t, G'_t as above.
// Then J_0 x = r is z_b = S_b^{-1} r_b (all slabs); y_b = z_b - G_b y_{b-1} (b = 1 .. t-1) together with
// y_b = z_b - G'_b y_{b+1} (b = nx-2 .. t+1); x_t = z_t - G_t y_{t-1} - G'_t y_{t+1}; x_b = y_b - W_b x_{b+1}
// (b = t-1 .. 0) together with x_b = y_b - V_b x_{b-1} (b = t+1 .. nx-1): about half the dependent steps
// of the one-sided block LU. The Schur complements of J_0^T in the same order are the S_b^T, so the
// transposed system needs no inversion of its own: its blocks are S_b^{-T}, (A_{b-1,b} S_b^{-1})^T (lower
// chain, or back-substitution below the twist) and (A_{b+1,b} S_b^{-1})^T (upper chain, or back-
// substitution above the twist). Every block is kept row-major in H.cs_store at cpos[kind][b], kinds
// 0..3 (inverse, lower chain G, upper chain G', back-substitution W or V) for J_0 and 4..7 for J_0^T.
static stm_status twisted_slab_factors(Hierarchy& H, const Level& L, const std::vector<long long>& off,
                                       const std::vector<int>& iperm, double* raw,
                                       const std::vector<long long>& dpos, const std::vector<long long>& lpos,
                                       const std::vector<long long>& upos, double* scal, cudaStream_t s) {
  enum { K_INV = 0, K_LO = 1, K_UP = 2, K_BACK = 3, K_T = 4 };
  const int nx = L.cells[0];
  const long long n = L.N;
  const int t = nx / 2;
  auto rows = [&](int b) { return off[b + 1] - off[b]; };
  std::vector<long long> cpos(8 * (size_t)nx, -1);
  long long ct = 0;
  for (int b = 0; b < nx; ++b) {
    const long long nb = rows(b), npv = b > 0 ? rows(b - 1) : 0, nnx = b + 1 < nx ? rows(b + 1) : 0;
    for (int sys = 0; sys < 2; ++sys) {
      const int k0 = sys * K_T;
      cpos[(k0 + K_INV) * nx + b] = ct; ct += nb * nb;
      if (b >= 1 && b <= t) { cpos[(k0 + K_LO) * nx + b] = ct; ct += nb * npv; }
      if (b >= t && b + 1 < nx) { cpos[(k0 + K_UP) * nx + b] = ct; ct += nb * nnx; }
      if (b < t) { cpos[(k0 + K_BACK) * nx + b] = ct; ct += nb * nnx; }
      if (b > t) { cpos[(k0 + K_BACK) * nx + b] = ct; ct += nb * npv; }
    }
  }
  if ((!H.cs_store && cudaMalloc(&H.cs_store, sizeof(double) * ct)) ||
      (!H.cs_u && cudaMalloc(&H.cs_u, sizeof(double) * n)) || (!H.cs_v && cudaMalloc(&H.cs_v, sizeof(double) * n)) ||
      (!H.cs_off && cudaMalloc(&H.cs_off, sizeof(long long) * (nx + 1))) ||
      (!H.cs_perm && cudaMalloc(&H.cs_perm, sizeof(int) * n))) {
    cudaGetLastError();
    set_error("coarse factorisation: out of device memory");
    return STM_ERR_OOM;
  }
  double* cs = H.cs_store;
  auto at = [&](int kind, int b) { return cs + cpos[kind * nx + b]; };
  const double* D = raw;  // raw blocks: A_bb at dpos, A_{b,b-1} at lpos (b >= 1), A_{b,b+1} at upos (b < nx-1)
  auto Lo = [&](int b) { return D + lpos[b]; };
  auto Up = [&](int b) { return D + upos[b]; };
  // one slab: S_b from A_bb and the neighbours already eliminated, its inverse, then its chain blocks
  auto slab = [&](int b, DenseWork& w, cudaStream_t st) -> stm_status {
    const int nb = (int)rows(b), npv = b > 0 ? (int)rows(b - 1) : 0, nnx = b + 1 < nx ? (int)rows(b + 1) : 0;
    double* Sb = at(K_INV, b);
    const bool below = b > 0 && b <= t, above = b + 1 < nx && b >= t;  // neighbours already eliminated
    const double* W = below ? at(K_BACK, b - 1) : nullptr;
    const double* V = above ? at(K_BACK, b + 1) : nullptr;
    const DenseSlice in[4] = {{2, false, below ? Lo(b) : nullptr, npv, below ? nb : 0, npv},
                              {3, true, W, nb, below ? npv : 0, nb},
                              {4, false, above ? Up(b) : nullptr, nnx, above ? nb : 0, nnx},
                              {5, true, V, nb, above ? nnx : 0, nb}};
    STM_TRY(dense_slice(w, in, 4, H.dflag + 1, st));
    const double* cur = D + dpos[b];
    DenseProduct p;
    p.m = p.n = nb;
    p.ldc0 = p.ldc = nb;
    p.alpha = -1.0;
    p.C = w.tmp;
    if (below) {  // - A_{b,b-1} W_{b-1}
      p.a = 2, p.b = 3, p.k = npv, p.C0 = cur;
      STM_TRY(dense_products(w, &p, 1, st));
      cur = w.tmp;
    }
    if (above) {  // - A_{b,b+1} V_{b+1}
      p.a = 4, p.b = 5, p.k = nnx, p.C0 = cur;
      STM_TRY(dense_products(w, &p, 1, st));
      cur = w.tmp;
    }
    if (cur != w.tmp)
      STM_CUDA(cudaMemcpyAsync(w.tmp, cur, sizeof(double) * (size_t)nb * nb, cudaMemcpyDeviceToDevice, st));
    STM_TRY(invert_block(w, w.tmp, nb, Sb, H.dflag + 1, scal + 2 * (&w - H.dw), st));
    // S_b^{-1} A_{b,b-1}, S_b^{-1} A_{b,b+1}; J_0^T: (A_{b-1,b} S_b^{-1})^T, (A_{b+1,b} S_b^{-1})^T, S_b^{-T}
    const DenseSlice op[6] = {{0, false, Sb, nb, nb, nb},
                              {1, true, Sb, nb, nb, nb},
                              {2, true, b > 0 ? Lo(b) : nullptr, npv, npv ? nb : 0, npv},
                              {3, true, b + 1 < nx ? Up(b) : nullptr, nnx, nnx ? nb : 0, nnx},
                              {4, false, b > 0 ? Up(b - 1) : nullptr, nb, npv, nb},
                              {5, false, b + 1 < nx ? Lo(b + 1) : nullptr, nb, nnx, nb}};
    STM_TRY(dense_slice(w, op, 6, H.dflag + 1, st));
    DenseProduct q[4];
    int nq = 0;
    auto product = [&](int a, int bb, int m, int n, double* C, int trans) {
      DenseProduct& o = q[nq++];
      o.a = a, o.b = bb, o.m = m, o.n = n, o.k = nb;
      o.C = C, o.ldc = trans ? m : n, o.trans = trans;
    };
    if (b > 0) {
      product(0, 2, nb, npv, at(b <= t ? K_LO : K_BACK, b), 0);
      product(4, 1, npv, nb, at(K_T + (b <= t ? K_LO : K_BACK), b), 1);
    }
    if (b + 1 < nx) {
      product(0, 3, nb, nnx, at(b < t ? K_BACK : K_UP, b), 0);
      product(5, 1, nnx, nb, at(K_T + (b < t ? K_BACK : K_UP), b), 1);
    }
    STM_TRY(dense_products(w, q, nq, st));
    transpose_block(Sb, nb, nb, at(K_T + K_INV, b), st);
    return STM_OK;
  };
  // the two chains meet only in slab t: the lower one runs on a stream of its own, with its own work space
  long long maxnb = 0;
  for (int b = 0; b < nx; ++b) maxnb = std::max(maxnb, rows(b));
  for (DenseWork& w : H.dw) {
    w.overlap = true;
    STM_TRY(dense_reserve_inverse(w, maxnb));
    for (int q = 0; q < DenseWork::kSlots; ++q) STM_TRY(dense_reserve(w, q, maxnb, maxnb));
  }
  if (!H.chain_stream) STM_CUDA(cudaStreamCreateWithFlags(&H.chain_stream, cudaStreamNonBlocking));
  for (cudaEvent_t& e : H.chain_ev)
    if (!e) STM_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  STM_CUDA(cudaEventRecord(H.chain_ev[0], s));
  STM_CUDA(cudaStreamWaitEvent(H.chain_stream, H.chain_ev[0], 0));
  stm_status chains = STM_OK;
  for (int i = 0; i < std::max(t, nx - 1 - t) && chains == STM_OK; ++i) {
    if (i < t) chains = slab(i, H.dw[0], s);
    if (chains == STM_OK && nx - 1 - i > t) chains = slab(nx - 1 - i, H.dw[1], H.chain_stream);
  }
  STM_CUDA(cudaEventRecord(H.chain_ev[1], H.chain_stream));
  STM_CUDA(cudaStreamWaitEvent(s, H.chain_ev[1], 0));
  if (chains == STM_OK) chains = slab(t, H.dw[0], s);
  if (chains != STM_OK) {
    cudaStreamSynchronize(s);
    return chains;
  }
  std::vector<long long> hoff(off.begin(), off.begin() + nx + 1);
  cudaMemcpyAsync(H.cs_off, hoff.data(), sizeof(long long) * (nx + 1), cudaMemcpyHostToDevice, s);
  cudaMemcpyAsync(H.cs_perm, iperm.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s);
  H.cs_nx = nx;
  H.cs_t = t;
  H.cs_maxnb = (int)maxnb;
  STM_TRY(coarse_slab_words(H, off, cpos, s));
  const cudaError_t e1 = cudaGetLastError(), e2 = cudaStreamSynchronize(s);
  if (e1 != cudaSuccess || e2 != cudaSuccess) {
    set_error("coarse factorisation: CUDA error");
    return STM_ERR_CUDA;
  }
  H.coarse_slab = true;
  return STM_OK;
}

static stm_status factor_coarse_in(Hierarchy& H, cudaStream_t s);
stm_status factor_coarse(Hierarchy& H, cudaStream_t s) {
  stm_status st = factor_coarse_in(H, s);
  if (st == STM_ERR_OOM) {  // once more without what only saves time
    give_back(H);
    st = factor_coarse_in(H, s);
  }
  return st;
}
static stm_status factor_coarse_in(Hierarchy& H, cudaStream_t s) {
  Level& L = H.L[0];
  const long long n = L.N;
  const int nx = L.cells[0];
  H.N0 = n;
  H.cs_scale = pressure_scale(H, L);
  const bool use_slab = n >= kCoarseSlabMinDofs && nx >= 2;
  std::vector<int> iperm, blk;
  std::vector<long long> off;
  coarse_slabs(L, use_slab ? nx / 2 : nx, iperm, blk, off);
  // dense block storage: D_b, Lo_b (b >= 1), Up_b (b < nx-1), W_b, G_b
  std::vector<long long> dpos(nx), lpos(nx, 0), upos(nx, 0), wpos(nx, 0), gpos(nx, 0);
  long long tot = 0;
  long long maxnb = 0;
  for (int b = 0; b < nx; ++b) {
    const long long nb = off[b + 1] - off[b];
    maxnb = std::max(maxnb, nb);
    dpos[b] = tot; tot += nb * nb;
    if (b > 0) { lpos[b] = tot; tot += nb * (off[b] - off[b - 1]); }
    if (b + 1 < nx) { upos[b] = tot; tot += nb * (off[b + 2] - off[b + 1]); }
  }
  for (int b = 0; b < nx; ++b) {
    const long long nb = off[b + 1] - off[b];
    if (b + 1 < nx) { wpos[b] = tot; tot += nb * (off[b + 2] - off[b + 1]); }
    if (b > 0) { gpos[b] = tot; tot += nb * (off[b] - off[b - 1]); }
  }
  int *d_iperm = nullptr, *d_blk = nullptr;
  long long *d_off = nullptr, *d_dpos = nullptr, *d_lpos = nullptr, *d_upos = nullptr;
  double *Xp = nullptr, *scal = nullptr;
  stm_status st = STM_OK;
  auto fail = [&](stm_status e) { st = e; };
  do {
    if (cudaMalloc(&d_iperm, sizeof(int) * n) || cudaMalloc(&d_blk, sizeof(int) * n) ||
        cudaMalloc(&d_off, sizeof(long long) * (nx + 2)) || cudaMalloc(&d_dpos, sizeof(long long) * nx) ||
        cudaMalloc(&d_lpos, sizeof(long long) * nx) || cudaMalloc(&d_upos, sizeof(long long) * nx) ||
        (!H.cs_raw && cudaMalloc(&H.cs_raw, sizeof(double) * tot)) ||
        (!use_slab && cudaMalloc(&Xp, sizeof(double) * n * n)) || cudaMalloc(&scal, sizeof(double) * 4)) {
      cudaGetLastError();
      set_error("coarse factorisation: out of device memory");
      fail(STM_ERR_OOM);
      break;
    }
    if (!use_slab && !H.cinv && cudaMalloc(&H.cinv, sizeof(double) * n * n)) {
      cudaGetLastError();
      set_error("coarse factorisation: out of device memory");
      fail(STM_ERR_OOM);
      break;
    }
    // the transposed inverse for the adjoint coarse solve
    if (!use_slab && !H.cinvT && cudaMalloc(&H.cinvT, sizeof(double) * n * n)) {
      cudaGetLastError();
      set_error("coarse factorisation: out of device memory");
      fail(STM_ERR_OOM);
      break;
    }
    cudaMemcpyAsync(d_iperm, iperm.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(d_blk, blk.data(), sizeof(int) * n, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(d_off, off.data(), sizeof(long long) * (nx + 2), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(d_dpos, dpos.data(), sizeof(long long) * nx, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(d_lpos, lpos.data(), sizeof(long long) * nx, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(d_upos, upos.data(), sizeof(long long) * nx, cudaMemcpyHostToDevice, s);
    double* store = H.cs_raw;
    cudaMemsetAsync(store, 0, sizeof(double) * tot, s);
    if (Xp) cudaMemsetAsync(Xp, 0, sizeof(double) * n * n, s);
    k_slab_blocks<<<(int)std::min<long long>(n, sm_count() * 32LL), 128, 0, s>>>(L.rowptr, L.colidx, L.val, n, d_iperm, d_blk,
                                                                          d_off, d_dpos, d_lpos, d_upos, store,
                                                                          H.dflag + 1, L.block, (long long)L.dim * L.R, H.cs_scale);
    note_launch();
    if (use_slab) {
      st = twisted_slab_factors(H, L, off, iperm, store, dpos, lpos, upos, scal, s);
      break;
    }
    // C (m x n) = [C0] + alpha A B, ld of each as given
    DenseWork& w = H.dw[0];
    auto product = [&](int m, int n_, int k, double alpha, const double* A, long long lda, const double* B, long long ldb,
                       const double* C0, double* C, long long ldc) -> stm_status {
      const DenseSlice sl[2] = {{2, false, A, lda, m, k}, {3, true, B, ldb, k, n_}};
      STM_TRY(dense_slice(w, sl, 2, H.dflag + 1, s));
      DenseProduct p;
      p.a = 2, p.b = 3, p.m = m, p.n = n_, p.k = k, p.alpha = alpha;
      p.C0 = C0, p.C = C, p.ldc0 = p.ldc = ldc;
      return dense_products(w, &p, 1, s);
    };
    auto build = [&]() -> stm_status {
      STM_TRY(dense_reserve_inverse(w, maxnb));
      STM_TRY(dense_reserve(w, 2, maxnb, maxnb));
      STM_TRY(dense_reserve(w, 3, maxnb, n));
      // forward block LU
      for (int b = 0; b < nx; ++b) {
        const long long nb = off[b + 1] - off[b];
        double* Db = store + dpos[b];
        if (b > 0) {  // S_b = A_bb - A_{b,b-1} W_{b-1}
          const long long np_ = off[b] - off[b - 1];
          STM_TRY(product((int)nb, (int)nb, (int)np_, -1.0, store + lpos[b], np_, store + wpos[b - 1], nb, Db, w.tmp, nb));
        } else {
          STM_CUDA(cudaMemcpyAsync(w.tmp, Db, sizeof(double) * nb * nb, cudaMemcpyDeviceToDevice, s));
        }
        STM_TRY(invert_block(w, w.tmp, nb, Db, H.dflag + 1, scal, s));
        if (b + 1 < nx) {  // W_b = S_b^{-1} A_{b,b+1}
          const long long nn_ = off[b + 2] - off[b + 1];
          STM_TRY(product((int)nb, (int)nn_, (int)nb, 1.0, Db, nb, store + upos[b], nn_, nullptr, store + wpos[b], nn_));
        }
        if (b > 0) {  // G_b = S_b^{-1} A_{b,b-1}
          const long long np_ = off[b] - off[b - 1];
          STM_TRY(product((int)nb, (int)np_, (int)nb, 1.0, Db, nb, store + lpos[b], np_, nullptr, store + gpos[b], np_));
        }
      }
      // Z = L^{-1} (block lower triangular) into the block rows of Xp
      for (int b = 0; b < nx; ++b) {
        const long long nb = off[b + 1] - off[b];
        double* rowb = Xp + off[b] * n;
        k_copy_block<<<(int)std::min<long long>((nb * nb + 255) / 256, sm_count() * 8LL), 256, 0, s>>>(
            store + dpos[b], nb, nb, nb, rowb + off[b], n);
        note_launch();
        if (b > 0) {
          const long long np_ = off[b] - off[b - 1];
          STM_TRY(product((int)nb, (int)off[b], (int)np_, -1.0, store + gpos[b], np_, Xp + off[b - 1] * n, n, nullptr,
                          rowb, n));
        }
      }
      // X = U^{-1} Z, last block row first
      for (int b = nx - 2; b >= 0; --b) {
        const long long nb = off[b + 1] - off[b], nn_ = off[b + 2] - off[b + 1];
        STM_TRY(product((int)nb, (int)n, (int)nn_, -1.0, store + wpos[b], nn_, Xp + off[b + 1] * n, n, Xp + off[b] * n,
                        Xp + off[b] * n, n));
      }
      return STM_OK;
    };
    st = build();
    if (st != STM_OK) {
      cudaStreamSynchronize(s);
      break;
    }
    dim3 ug((unsigned)std::min<long long>((n + 255) / 256, 64), (unsigned)std::min<long long>(n, 65535));
    k_unpermute<<<ug, 256, 0, s>>>(Xp, d_iperm, n, H.cinv, L.block, (long long)L.dim * L.R, H.cs_scale);
    note_launch();
    transpose_block(H.cinv, n, n, H.cinvT, s);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
      set_error("coarse factorisation: CUDA error");
      fail(STM_ERR_CUDA);
    }
  } while (false);
  void* ptrs[] = {d_iperm, d_blk, d_off, d_dpos, d_lpos, d_upos, Xp, scal};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  return st;
}

}  // namespace stm
