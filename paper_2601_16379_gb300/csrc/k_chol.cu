// Batched FP64 factorisations for the least-squares solve (Eq. 3).
//
// pchol_batched  pivoted Cholesky of Hermitian PSD matrices: pivot = largest
//                remaining diagonal, where diagonals within 1e-11 * (largest
//                initial diagonal) of it are ties resolved to the smallest
//                index; stop when it is <= tol * largest initial diagonal.
//                Column j of L is stored as Lt[j][:].
// trinv_batched  W = L_S^{-1} for the kept rows S = perm[:rank] (L_S is lower
//                triangular in pivot order), scattered to Wfull[i][perm[c]] so
//                that xi = Wfull * eta and zeta = Wfull^H * xi give the basic
//                least-squares solution (zeta = 0 on dropped points).
//
// Both take a list of the matrices (q-points) to work on, so that one launch covers the
// scattered representatives of the time-reversal pairs.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"

namespace isdf {

namespace {

constexpr double kTieEps = 1e-11;  // pivot tie window, relative to the largest initial diagonal

// A cluster of C blocks per matrix, one row of L per thread.  What bounds it is the FP64 pipe
// (six operations per complex product, 2 per clock and SM): n r^2 / 2 products are 28 ms on
// one SM at n = 500, r = 270, so the rows are spread over C SMs; the residual diagonals live
// in shared memory, double-buffered, and are read across the cluster.  Rows are written once
// per column and read by their own thread; only the pivot's row of L is gathered per column.
// live != 0: rows that were pivots are skipped from then on (nothing reads their later
// columns); rows from neff on are zero.
constexpr int kBp = 512;  // entries of the pivot's row of L staged at once
__global__ void __launch_bounds__(256) pchol_kernel(const double2* __restrict__ A, int n, int neff, int live,
                                                    const int* __restrict__ qlist, double tol, double2* Lt,
                                                    int32_t* __restrict__ perm, int32_t* __restrict__ rank) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), cr = (int)cl.block_rank();
  const int64_t q = qlist[blockIdx.x / C];
  A += q * n * n;
  Lt += q * n * n;
  perm += q * n;
  const int bd = blockDim.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = bd >> 5;
  const int per = (neff + C - 1) / C, i0 = cr * per, i1 = min(neff, i0 + per);  // rows of this block
  extern __shared__ __align__(16) unsigned char chol_smem[];
  double2* bp = reinterpret_cast<double2*>(chol_smem);           // [kBp] of the pivot's row of L
  double* sd = reinterpret_cast<double*>(bp + kBp);              // [2][per] residual diagonals
  unsigned char* used = reinterpret_cast<unsigned char*>(sd + 2 * per);  // [per]
  __shared__ double sv[8], s_max[2], s_inv;
  __shared__ int si[8], s_idx[2];
  for (int i = i0 + tid; i < i1; i += bd) {
    sd[i - i0] = A[(int64_t)i * n + i].x;
    used[i - i0] = 0;
  }
  __syncthreads();
  double d0 = 0.0;
  int r = 0;
  for (int j = 0; j < neff; ++j) {
    const int cur = j & 1;
    double* d = sd + cur * per;
    double* dn = sd + (cur ^ 1) * per;
    // largest remaining diagonal over unused rows
    double bv = -INFINITY;
    for (int i = i0 + tid; i < i1; i += bd)
      if (!used[i - i0]) bv = fmax(bv, d[i - i0]);
    for (int o = 16; o; o >>= 1) bv = fmax(bv, __shfl_xor_sync(0xffffffffu, bv, o));
    if (lane == 0) sv[w] = bv;
    __syncthreads();
    if (tid == 0) {
      double v = sv[0];
      for (int t = 1; t < nw; ++t) v = fmax(v, sv[t]);
      s_max[cur] = v;
    }
    cl.sync();
    double dmax = -INFINITY;
    for (int c = 0; c < C; ++c) dmax = fmax(dmax, *cl.map_shared_rank(&s_max[cur], c));
    if (j == 0) d0 = dmax;
    if (!(dmax > tol * d0) || !(dmax > 0.0)) break;
    // ties: every unused row within tie_eps * d_max,0 (and >= dmax/2) -> smallest index
    const double thr = fmax(dmax - kTieEps * d0, 0.5 * dmax);
    int bi = n;
    for (int i = i0 + tid; i < i1; i += bd)
      if (!used[i - i0] && d[i - i0] >= thr && i < bi) bi = i;
    for (int o = 16; o; o >>= 1) bi = min(bi, __shfl_xor_sync(0xffffffffu, bi, o));
    if (lane == 0) si[w] = bi;
    __syncthreads();
    if (tid == 0) {
      int ii = si[0];
      for (int t = 1; t < nw; ++t) ii = min(ii, si[t]);
      s_idx[cur] = ii;
    }
    cl.sync();
    int p = n;
    for (int c = 0; c < C; ++c) p = min(p, *cl.map_shared_rank(&s_idx[cur], c));
    if (p >= n) break;  // no finite candidate
    if (tid == 0) {
      const double dp = *cl.map_shared_rank(d + p % per, p / per);
      s_inv = 1.0 / sqrt(dp);
    }
    for (int ib = i0; ib < i1; ib += bd) {
      const int i = ib + tid;
      const bool on = i < i1 && !(live && used[i - i0]);
      double2 acc = on ? A[(int64_t)i * n + p] : make_double2(0.0, 0.0);
      for (int l0 = 0; l0 < j; l0 += kBp) {
        const int nl = min(kBp, j - l0);
        __syncthreads();
        for (int l = tid; l < nl; l += bd) bp[l] = Lt[(int64_t)(l0 + l) * n + p];
        __syncthreads();
        if (!on) continue;
        const double2* Li = Lt + (int64_t)l0 * n + i;
#pragma unroll 8
        for (int l = 0; l < nl; ++l) {
          const double2 a = Li[(int64_t)l * n];
          const double2 b = bp[l];
          // acc -= a * conj(b)
          acc.x -= a.x * b.x + a.y * b.y;
          acc.y -= a.y * b.x - a.x * b.y;
        }
      }
      if (j == 0) __syncthreads();  // s_inv
      if (!on) continue;
      const double inv = s_inv;
      const double2 col = make_double2(acc.x * inv, acc.y * inv);
      Lt[(int64_t)j * n + i] = col;
      dn[i - i0] = d[i - i0] - (col.x * col.x + col.y * col.y);
      if (i == p) used[i - i0] = 1;
    }
    if (cr == 0 && tid == 0) perm[j] = p;
    r = j + 1;
    __syncthreads();
  }
  cl.sync();  // no block leaves while its shared memory may be read
  if (cr == 0 && tid == 0) rank[q] = r;
  // zero what was not computed so that consumers can read a full n x n array
  const int64_t t0 = (int64_t)cr * bd + tid, step = (int64_t)C * bd;
  for (int64_t e = (int64_t)r * n + t0; e < (int64_t)n * n; e += step) Lt[e] = make_double2(0.0, 0.0);
  const int64_t pad = n - neff;
  for (int64_t e = t0; e < (int64_t)r * pad; e += step) Lt[(e / pad) * n + neff + e % pad] = make_double2(0.0, 0.0);
  for (int64_t i = r + t0; i < n; i += step) perm[i] = -1;
}

// work[q][l][i] = L_S[i][l] = Lt[l][perm[i]] for l <= i < r: the rows of the triangular solve,
// contiguous in i.
__global__ void tri_gather_kernel(const double2* __restrict__ Lt, const int32_t* __restrict__ perm,
                                  const int32_t* __restrict__ rank, const int* __restrict__ qlist, int n,
                                  double2* __restrict__ out) {
  const int64_t q = qlist[blockIdx.y];
  const int r = rank[q];
  for (int l = blockIdx.x; l < r; l += gridDim.x)
    for (int i = l + threadIdx.x; i < r; i += blockDim.x)
      out[q * n * n + (int64_t)l * n + i] = Lt[q * n * n + (int64_t)l * n + perm[q * n + i]];
}

// work[q][i][c] = (L_S^{-1})[i][c]: a warp per column c, its entries in shared memory (or, for
// n beyond it, in row c of the scratch array).  Right-looking: entry l is final after l
// updates and is taken from all later ones, which keeps every entry's order of summation
// and leaves one division, not a sum, on the serial chain.
__global__ void __launch_bounds__(256) trinv_kernel(const double2* __restrict__ Lc, const int32_t* __restrict__ rank,
                                                    const int* __restrict__ qlist, int n, int in_smem,
                                                    double2* __restrict__ scratch, double2* __restrict__ work) {
  extern __shared__ __align__(16) unsigned char chol_smem[];
  const int64_t q = qlist[blockIdx.y];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  const int c = blockIdx.x * nwarp + warp;
  const int r = rank[q];
  if (c >= r) return;
  Lc += q * n * n;
  work += q * n * n;
  double2* x = in_smem ? reinterpret_cast<double2*>(chol_smem) + (int64_t)warp * n : scratch + q * n * n + (int64_t)c * n;
  for (int i = c + lane; i < r; i += 32) x[i] = make_double2(i == c ? 1.0 : 0.0, 0.0);
  __syncwarp();
  for (int l = c; l < r; ++l) {
    const double2 acc = x[l], Lii = Lc[(int64_t)l * n + l];
    // acc / Lii
    const double den = __fma_rn(Lii.x, Lii.x, __dmul_rn(Lii.y, Lii.y));
    const double2 wl = make_double2(__ddiv_rn(__fma_rn(acc.x, Lii.x, __dmul_rn(acc.y, Lii.y)), den),
                                    __ddiv_rn(__fma_rn(acc.y, Lii.x, -__dmul_rn(acc.x, Lii.y)), den));
    if (lane == 0) work[(int64_t)l * n + c] = wl;
    for (int i = l + 1 + lane; i < r; i += 32) {
      const double2 Lil = Lc[(int64_t)l * n + i];
      double2 a = x[i];
      // the order of the fused operations is written out: the solve amplifies their rounding
      a.x = __dsub_rn(a.x, __fma_rn(Lil.x, wl.x, -__dmul_rn(Lil.y, wl.y)));
      a.y = __dsub_rn(a.y, __fma_rn(Lil.y, wl.x, __dmul_rn(Lil.x, wl.y)));
      x[i] = a;
    }
    __syncwarp();
  }
}

__global__ void scatter_w_kernel(const double2* __restrict__ work, const int32_t* __restrict__ perm,
                                 const int32_t* __restrict__ rank, const int* __restrict__ qlist, int n, int nq,
                                 double2* __restrict__ W) {
  const int64_t total = (int64_t)nq * n * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = qlist[e / ((int64_t)n * n)];
    const int i = (int)((e / n) % n);
    const int c = (int)(e % n);
    const int r = rank[b];
    if (i < r && c < r) {
      const int col = perm[b * n + c];
      W[b * n * n + (int64_t)i * n + col] = work[b * n * n + (int64_t)i * n + c];
    }
  }
}

__global__ void lt_to_row_kernel(const double2* __restrict__ Lt, const int32_t* __restrict__ rank,
                                 const int* __restrict__ qlist, int n, double2* __restrict__ L) {
  // 32 x 32 tiles transposed through shared memory
  __shared__ double2 t[32][33];
  const int64_t q = qlist[blockIdx.z];
  const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32, r = rank[q];
  Lt += q * n * n;
  L += q * n * n;
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int j = j0 + y, i = i0 + threadIdx.x;
    t[y][threadIdx.x] = (i < n && j < r) ? Lt[(int64_t)j * n + i] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int i = i0 + y, j = j0 + threadIdx.x;
    if (i < n && j < n) L[(int64_t)i * n + j] = t[threadIdx.x][y];
  }
}

// A warp per row.
__global__ void __launch_bounds__(256) row_exp_z_kernel(const double2* __restrict__ A, int n, int rows,
                                                        const int* __restrict__ qlist, int32_t* __restrict__ e) {
  const int64_t q = qlist[blockIdx.y];
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= rows) return;
  const double2* a = A + (q * n + i) * n;
  unsigned m = 0;  // exponent field of the largest component
  for (int c = lane; c < n; c += 32) {
    const double2 v = a[c];
    m = max(m, ((unsigned)__double2hiint(v.x) >> 20) & 0x7FFu);
    m = max(m, ((unsigned)__double2hiint(v.y) >> 20) & 0x7FFu);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) e[q * n + i] = m == 0 || m == 0x7FFu ? 0 : max(-kMaxKexp, min(kMaxKexp, (int)m - 1023));
}

inline int nblocks(int64_t total) {
  int64_t nb = (total + 255) / 256;
  if (nb > 152 * 32) nb = 152 * 32;
  return nb < 1 ? 1 : (int)nb;
}

}  // namespace

cudaError_t pchol_batched(cudaStream_t st, const double2* A, int n, int neff, bool live, const int* qlist, int nq,
                          double tol, double2* Lt, int32_t* perm, int32_t* rank) {
  if (n <= 0 || nq <= 0) return cudaSuccess;
  // blocks per matrix: up to eight (the portable cluster) while they do not fill the SMs
  // four times over and keep a warp of rows each
  int C = 1;
  while (C < 8 && nq * C < 152 * 4 && neff > 32 * C) C *= 2;
  int threads = std::min(256, std::max(32, ((neff + C - 1) / C + 31) / 32 * 32));
  auto smem_of = [&](int c) {
    const size_t per = (size_t)(neff + c - 1) / c;
    return kBp * sizeof(double2) + per * (2 * sizeof(double) + 1);
  };
  const size_t smem = smem_of(C);
  cudaError_t e = allow_smem(pchol_kernel, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(nq * C));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, pchol_kernel, A, n, neff, live ? 1 : 0, qlist, tol, Lt, perm, rank);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

// work holds L_S^{-1} in pivot order (lower triangular, zero outside the rank); tmp: nk n n of scratch.
cudaError_t trinv_batched(cudaStream_t st, const double2* Lt, const int32_t* perm, const int32_t* rank, int n, int nk,
                          const int* qlist, int nq, double2* W, double2* work, double2* tmp) {
  if (n <= 0 || nq <= 0) return cudaSuccess;
  const size_t bytes = sizeof(double2) * (size_t)nk * n * n;
  cudaError_t e = cudaMemsetAsync(work, 0, bytes, st);
  if (e != cudaSuccess) return e;
  tri_gather_kernel<<<dim3((unsigned)std::min(n, 64), nq), 128, 0, st>>>(Lt, perm, rank, qlist, n, tmp);
  count_launch();
  int warps = 8;
  while (warps > 1 && (size_t)warps * n * sizeof(double2) > 64 * 1024) warps /= 2;
  const size_t smem = (size_t)warps * n * sizeof(double2);
  const bool in_smem = smem <= 200 * 1024;
  if (in_smem) e = allow_smem(trinv_kernel, smem);
  if (e != cudaSuccess) return e;
  trinv_kernel<<<dim3((n + warps - 1) / warps, nq), warps * 32, in_smem ? smem : 0, st>>>(tmp, rank, qlist, n, in_smem, W,
                                                                                         work);
  count_launch();
  e = cudaMemsetAsync(W, 0, bytes, st);
  if (e != cudaSuccess) return e;
  scatter_w_kernel<<<nblocks((int64_t)nq * n * n), 256, 0, st>>>(work, perm, rank, qlist, n, nq, W);
  count_launch();
  return cudaGetLastError();
}

cudaError_t row_exponents_z(cudaStream_t st, const double2* A, int n, int rows, const int* qlist, int nq, int32_t* e) {
  if (n <= 0 || rows <= 0 || nq <= 0) return cudaSuccess;
  row_exp_z_kernel<<<dim3((rows + 7) / 8, nq), 256, 0, st>>>(A, n, rows, qlist, e);
  count_launch();
  return cudaGetLastError();
}

cudaError_t lt_to_rowmajor(cudaStream_t st, const double2* Lt, const int32_t* rank, const int* qlist, int nq, int n,
                           double2* L) {
  if (n <= 0 || nq <= 0) return cudaSuccess;
  const unsigned nt = (unsigned)((n + 31) / 32);
  lt_to_row_kernel<<<dim3(nt, nt, nq), dim3(32, 8), 0, st>>>(Lt, rank, qlist, n, L);
  count_launch();
  return cudaGetLastError();
}

}  // namespace isdf
