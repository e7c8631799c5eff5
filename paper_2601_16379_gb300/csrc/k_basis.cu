// Crystalline Gaussian orbitals on the cell grid (Eq. 1) and the
// interpolation-point selection of Section II.A.
//
// ao_eval   Phi^k_mu(r) = sum_T e^{i k.T} phi~_mu(r - T), T over the box
//           |n_i| <= L_i.  For orthorhombic cells the Gaussian and the phase
//           factorise per axis, so the box sum is the product of three 1-D
//           lattice sums S_a(m_a, g_a) per primitive (exactly the same terms as
//           the 3-D box).  Other cells use a direct 3-D sum.
// ip_*      greedy pivoted Cholesky of K(r,r') = D(r,r')^2 with
//           D(r,r') = Re sum_{k,mu} conj(Phi^k_mu(r)) Phi^k_mu(r') (D is real:
//           the k and -k terms are conjugate).  One pivot per ip_step: argmax
//           with ties, column generation, rank-one update.
// ips_*     the same selection for orthorhombic cells (where it is the faster form: ips_supported), in which D
//           factorises as Phi does:
//             D(r,r') = sum_mu sum_{p,p'} c_p c_p' prod_a A_a(g_a, g'_a),
//             A_a(g, g') = sum_{m_a} conj(S_a^p(m_a, g)) S_a^p'(m_a, g')   (real),
//           since the k-mesh is a product of its axes.  A column of D then costs N_AO
//           terms per grid point instead of a pass over Phi.
#include <algorithm>
#include <climits>
#include <cmath>

#include "common.cuh"

namespace isdf {

namespace {

constexpr int KCH = 8;  // k-points per thread in the general path

// --------------------------------------------------------- orthorhombic path
// S[((mu*maxprim + p)*3 + a)*16*64 + m*64 + g] = sum_n e^{2 pi i m n/nk_a} x^l e^{-alpha x^2},
// x = g a_a/n_a - A_a - n a_a.
__global__ void ao_1d_kernel(CellDev c, BasisDev b, double2* __restrict__ S) {
  const int total = b.nao * b.maxprim * 3 * 16 * 64;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int g = e % 64;
    const int m = (e / 64) % 16;
    const int a = (e / (64 * 16)) % 3;
    const int p = (e / (64 * 16 * 3)) % b.maxprim;
    const int mu = e / (64 * 16 * 3 * b.maxprim);
    double2 acc = make_double2(0.0, 0.0);
    const int sh = b.ao_shell[mu];
    const int np = b.sh_off[sh + 1] - b.sh_off[sh];
    if (g < c.mesh[a] && m < c.kmesh[a] && p < np) {
      const double alpha = b.prim_exp[b.sh_off[sh] + p];
      const int l = b.ao_lxyz[mu * 3 + a];
      const double La = c.lat[a * 3 + a];
      const double A = b.coords[b.sh_atom[sh] * 3 + a];
      const double r = (double)g * La / (double)c.mesh[a];
      for (int n = -c.lrange[a]; n <= c.lrange[a]; ++n) {
        const double x = r - A - (double)n * La;
        double v = exp(-alpha * x * x);
        for (int t = 0; t < l; ++t) v *= x;
        // phase e^{2 pi i m n / nk}, angle reduced exactly
        const int nk = c.kmesh[a];
        int mn = (m * n) % nk;
        if (mn < 0) mn += nk;
        double sn, cs;
        sincospi(2.0 * (double)mn / (double)nk, &sn, &cs);
        acc.x += cs * v;
        acc.y += sn * v;
      }
    }
    S[e] = acc;
  }
}

// The two complex products of a value of Phi with the order of their fused operations written
// out: every later step follows the rounding of Phi, so it must not depend on how the
// compiler contracts the expression in its surroundings.
__device__ __forceinline__ double2 phi_xy(double2 a, double2 b) {
  return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(a.y, b.x, __dmul_rn(a.x, b.y)));
}
__device__ __forceinline__ double2 phi_xyz(double2 a, double2 b) {
  return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(a.x, b.y, __dmul_rn(a.y, b.x)));
}

// Phi[k][mu][r] = sum_p c_p (Sx Sy) Sz.  The FP64 pipe bounds it (10 operations per value),
// not the 16 bytes written: a block takes one (k, mu) and forms the products Sx Sy of a
// primitive once per (g0, g1) in shared memory instead of once per grid point, which leaves
// six.  The order of the multiplications is
// that of the direct form, so the values are the same bits.
__global__ void __launch_bounds__(256) ao_combine_kernel(CellDev c, BasisDev b, const double2* __restrict__ S,
                                                         double2* __restrict__ phi, int64_t nblk) {
  const int n1 = c.mesh[1], n2 = c.mesh[2], nxy = c.mesh[0] * n1, ng = nxy * n2;
  __shared__ double2 sxy[256], sz[64];
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    // block: (k, mu) and a run of 256 (g0, g1)
    const int nrun = (nxy + 255) / 256;
    const int run = (int)(blk % nrun), mu = (int)((blk / nrun) % b.nao), k = (int)(blk / ((int64_t)nrun * b.nao));
    const int m2 = k % c.kmesh[2], m1 = (k / c.kmesh[2]) % c.kmesh[1], m0 = k / (c.kmesh[1] * c.kmesh[2]);
    const int sh = b.ao_shell[mu];
    const int np = b.sh_off[sh + 1] - b.sh_off[sh];
    const int x0 = run * 256, cnt = min(256, nxy - x0) * n2;
    double2* out = phi + ((int64_t)k * b.nao + mu) * ng + (int64_t)x0 * n2;
    for (int p = 0; p < np; ++p) {
      const double2* base = S + (int64_t)((mu * b.maxprim + p) * 3) * 16 * 64;
      const double cn = b.prim_norm[mu * b.maxprim + p];
      __syncthreads();
      if (x0 + (int)threadIdx.x < nxy) {
        const int g0 = (x0 + threadIdx.x) / n1, g1 = (x0 + threadIdx.x) % n1;
        sxy[threadIdx.x] = phi_xy(base[m0 * 64 + g0], base[1024 + m1 * 64 + g1]);
      }
      if ((int)threadIdx.x < n2) sz[threadIdx.x] = base[2048 + m2 * 64 + threadIdx.x];
      __syncthreads();
      for (int e = threadIdx.x; e < cnt; e += 256) {
        const double2 t = phi_xyz(sxy[e / n2], sz[e % n2]);
        const double2 acc = p ? out[e] : make_double2(0.0, 0.0);
        out[e] = make_double2(__fma_rn(cn, t.x, acc.x), __fma_rn(cn, t.y, acc.y));
      }
    }
  }
}

// ------------------------------------------------------------- general path
__global__ void ao_general_kernel(CellDev c, BasisDev b, double2* __restrict__ phi) {
  const int ng = c.mesh[0] * c.mesh[1] * c.mesh[2];
  const int nk = c.kmesh[0] * c.kmesh[1] * c.kmesh[2];
  const int nkc = (nk + KCH - 1) / KCH;
  const int64_t total = (int64_t)nkc * b.nao * ng;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e % ng);
    const int mu = (int)((e / ng) % b.nao);
    const int kc = (int)(e / ((int64_t)ng * b.nao));
    const int g2 = r % c.mesh[2], g1 = (r / c.mesh[2]) % c.mesh[1], g0 = r / (c.mesh[1] * c.mesh[2]);
    const double f[3] = {(double)g0 / c.mesh[0], (double)g1 / c.mesh[1], (double)g2 / c.mesh[2]};
    double rc[3];
    for (int x = 0; x < 3; ++x) rc[x] = f[0] * c.lat[0 * 3 + x] + f[1] * c.lat[1 * 3 + x] + f[2] * c.lat[2 * 3 + x];
    const int sh = b.ao_shell[mu];
    const int np = b.sh_off[sh + 1] - b.sh_off[sh];
    const int lx = b.ao_lxyz[mu * 3], ly = b.ao_lxyz[mu * 3 + 1], lz = b.ao_lxyz[mu * 3 + 2];
    const double* A = b.coords + b.sh_atom[sh] * 3;
    double2 acc[KCH];
    int km[KCH][3];
    for (int i = 0; i < KCH; ++i) {
      acc[i] = make_double2(0.0, 0.0);
      const int k = kc * KCH + i;
      const int kk = k < nk ? k : 0;
      km[i][2] = kk % c.kmesh[2];
      km[i][1] = (kk / c.kmesh[2]) % c.kmesh[1];
      km[i][0] = kk / (c.kmesh[1] * c.kmesh[2]);
    }
    for (int n0 = -c.lrange[0]; n0 <= c.lrange[0]; ++n0)
      for (int n1 = -c.lrange[1]; n1 <= c.lrange[1]; ++n1)
        for (int n2 = -c.lrange[2]; n2 <= c.lrange[2]; ++n2) {
          double d[3];
          for (int x = 0; x < 3; ++x)
            d[x] = rc[x] - A[x] - (n0 * c.lat[0 * 3 + x] + n1 * c.lat[1 * 3 + x] + n2 * c.lat[2 * 3 + x]);
          const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
          double poly = 1.0;
          for (int t = 0; t < lx; ++t) poly *= d[0];
          for (int t = 0; t < ly; ++t) poly *= d[1];
          for (int t = 0; t < lz; ++t) poly *= d[2];
          double v = 0.0;
          for (int p = 0; p < np; ++p)
            v += b.prim_norm[mu * b.maxprim + p] * exp(-b.prim_exp[b.sh_off[sh] + p] * r2);
          v *= poly;
          for (int i = 0; i < KCH; ++i) {
            // e^{2 pi i sum_a m_a n_a / nk_a}
            double fr = 0.0;
            const int nn[3] = {n0, n1, n2};
            for (int a = 0; a < 3; ++a) {
              int mn = (km[i][a] * nn[a]) % c.kmesh[a];
              if (mn < 0) mn += c.kmesh[a];
              fr += (double)mn / (double)c.kmesh[a];
            }
            double sn, cs;
            sincospi(2.0 * (fr - floor(fr)), &sn, &cs);
            acc[i].x += cs * v;
            acc[i].y += sn * v;
          }
        }
    for (int i = 0; i < KCH; ++i) {
      const int k = kc * KCH + i;
      if (k < nk) phi[((int64_t)k * b.nao + mu) * ng + r] = acc[i];
    }
  }
}

// ------------------------------------------------------------- IP selection
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// partial[s][r] = sum_{a in split s} Re(conj(F[a][r]) F[a][col]) ; col < 0 -> |F[a][r]|^2
__global__ void ip_partial_kernel(const double2* __restrict__ F, int nkao, int ng,
                                  const int32_t* __restrict__ pcol_ptr, int j, int nsplit,
                                  double* __restrict__ partial, const int32_t* __restrict__ status) {
  if (status && *status != 0) return;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = blockIdx.y;
  if (r >= ng) return;
  const int per = (nkao + nsplit - 1) / nsplit;
  const int a0 = s * per, a1 = min(nkao, a0 + per);
  const int p = pcol_ptr ? pcol_ptr[j] : -1;
  double acc0 = 0.0, acc1 = 0.0;
  int a = a0;
  if (p >= 0) {
    for (; a + 1 < a1; a += 2) {
      const double2 x0 = F[(int64_t)a * ng + r], y0 = F[(int64_t)a * ng + p];
      const double2 x1 = F[(int64_t)(a + 1) * ng + r], y1 = F[(int64_t)(a + 1) * ng + p];
      acc0 = fma(x0.x, y0.x, acc0);
      acc0 = fma(x0.y, y0.y, acc0);
      acc1 = fma(x1.x, y1.x, acc1);
      acc1 = fma(x1.y, y1.y, acc1);
    }
    for (; a < a1; ++a) {
      const double2 x0 = F[(int64_t)a * ng + r], y0 = F[(int64_t)a * ng + p];
      acc0 = fma(x0.x, y0.x, acc0);
      acc0 = fma(x0.y, y0.y, acc0);
    }
  } else {
    for (; a < a1; ++a) {
      const double2 x0 = F[(int64_t)a * ng + r];
      acc0 = fma(x0.x, x0.x, acc0);
      acc0 = fma(x0.y, x0.y, acc0);
    }
  }
  partial[(int64_t)s * ng + r] = acc0 + acc1;
}

__global__ void ip_init_combine_kernel(const double* __restrict__ partial, int nsplit, int ng,
                                       double* __restrict__ d) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= ng) return;
  double D = 0.0;
  for (int s = 0; s < nsplit; ++s) D += partial[(int64_t)s * ng + r];
  d[r] = D * D;
}

// Single block: argmax with the tie rule; writes piv[j], chosen, dp (= d[p]).
__global__ void __launch_bounds__(1024) ip_argmax_kernel(const double* __restrict__ d, int ng, int j,
                                                         int32_t* __restrict__ piv,
                                                         int32_t* __restrict__ chosen,
                                                         uint64_t seed, double tie_eps,
                                                         double chol_tol, double* __restrict__ scal,
                                                         int32_t* __restrict__ status) {
  // scal[0] = d0 (set on j == 0), scal[1] = d[p] of the current pivot
  __shared__ double sv[32];
  __shared__ unsigned long long sh[32];
  __shared__ int si[32];
  __shared__ double s_dmax;
  if (*status != 0) return;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  double m = -INFINITY;
  for (int r = tid; r < ng; r += blockDim.x)
    if (!chosen[r]) m = fmax(m, d[r]);
  for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) sv[w] = m;
  __syncthreads();
  if (w == 0) {
    double v = lane < (int)(blockDim.x >> 5) ? sv[lane] : -INFINITY;
    for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) s_dmax = v;
  }
  __syncthreads();
  const double dmax = s_dmax;
  if (j == 0 && tid == 0) scal[0] = dmax;
  const double d0 = (j == 0) ? dmax : scal[0];
  if (!(dmax >= chol_tol * d0) || !(dmax > 0.0)) {
    if (tid == 0) {
      *status = 1;
      piv[j] = -1;
    }
    return;
  }
  const double thr = fmax(dmax - tie_eps * d0, 0.5 * dmax);
  unsigned long long best = ~0ULL;
  int bi = -1;
  for (int r = tid; r < ng; r += blockDim.x) {
    if (chosen[r] || !(d[r] >= thr)) continue;
    const unsigned long long hsh = splitmix64(seed ^ (uint64_t)r);
    if (hsh < best || (hsh == best && r < bi)) {
      best = hsh;
      bi = r;
    }
  }
  for (int o = 16; o; o >>= 1) {
    const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob < best || (ob == best && oi >= 0 && (bi < 0 || oi < bi))) {
      best = ob;
      bi = oi;
    }
  }
  if (lane == 0) {
    sh[w] = best;
    si[w] = bi;
  }
  __syncthreads();
  if (tid == 0) {
    unsigned long long b = ~0ULL;
    int p = -1;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i)
      if (si[i] >= 0 && (sh[i] < b || (sh[i] == b && si[i] < p))) {
        b = sh[i];
        p = si[i];
      }
    if (p < 0) {
      *status = 2;
      piv[j] = -1;
      return;
    }
    piv[j] = p;
    chosen[p] = 1;
    scal[1] = d[p];
  }
}

// l_r = (D(r,p)^2 - sum_{i<j} Lt[i][r] Lt[i][p]) / sqrt(d_p);  d_r -= l_r^2
__global__ void ip_update_kernel(const double* __restrict__ partial, int nsplit, int ng, int j,
                                 const int32_t* __restrict__ piv, double* __restrict__ Lt,
                                 double* __restrict__ d, const double* __restrict__ scal,
                                 const int32_t* __restrict__ status) {
  if (*status != 0) return;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= ng) return;
  const int p = piv[j];
  double D = 0.0;
  for (int s = 0; s < nsplit; ++s) D += partial[(int64_t)s * ng + r];
  double acc = D * D;
  for (int i = 0; i < j; ++i) acc -= Lt[(int64_t)i * ng + r] * Lt[(int64_t)i * ng + p];
  const double l = acc / sqrt(scal[1]);
  Lt[(int64_t)j * ng + r] = l;
  d[r] -= l * l;
}

// ------------------------------------------- IP selection, orthorhombic cells
// A[term][a][g'][g] (64 x 64 per axis), the factors of one term (mu, p, p'); c_p c_p' is in axis 0.
__global__ void ips_table_kernel(CellDev c, BasisDev b, const double2* __restrict__ S, const int* __restrict__ terms,
                                 int nterm, const int64_t o1, const int64_t o2, double* __restrict__ A) {
  const int n0 = c.mesh[0], n1 = c.mesh[1], n2 = c.mesh[2];
  const int per = n0 * n0 + n1 * n1 + n2 * n2;
  const int64_t total = (int64_t)nterm * per;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int t = (int)(e / per);
    int j = (int)(e % per), a = 0;
    if (j >= n0 * n0) j -= n0 * n0, a = 1;
    if (a == 1 && j >= n1 * n1) j -= n1 * n1, a = 2;
    const int n = c.mesh[a], gp = j / n, g = j % n, mu = terms[3 * t], p = terms[3 * t + 1], pp = terms[3 * t + 2];
    const double2* s = S + (int64_t)((mu * b.maxprim + p) * 3 + a) * 1024 + g;
    const double2* sp = S + (int64_t)((mu * b.maxprim + pp) * 3 + a) * 1024 + gp;
    double acc = 0.0;
    for (int m = 0; m < c.kmesh[a]; ++m) {
      const double2 x = s[m * 64], y = sp[m * 64];
      acc = fma(x.x, y.x, acc);
      acc = fma(x.y, y.y, acc);
    }
    if (a == 0) acc *= b.prim_norm[mu * b.maxprim + p] * b.prim_norm[mu * b.maxprim + pp];
    A[(a == 0 ? 0 : a == 1 ? o1 : o2) + (int64_t)t * n * n + j] = acc;
  }
}

constexpr int kLp = 512;  // entries of the pivot's row staged at once

struct IpsArgs {
  const double* A;  // factor tables: axis 0 at 0, axis 1 at o1, axis 2 at o2
  int64_t o1, o2;
  int nterm, n0, n1, n2, ng;
  int R;            // points per block
  int tile;         // terms whose (g0, g1) products are held at once
  long long* M;     // block maxima of the residual diagonal (order_key), two buffers of gridDim.x
  double* d;        // residual diagonal, two buffers of ng; -inf at the chosen points
  double* Lt;       // [n_p][ng]
  int32_t* piv;
  double* scal;     // scal[0] = d_max,0
  int32_t* status;
  uint64_t seed;
  double tie_eps, chol_tol;
};

// A block has R = a.R points and G groups of R threads; the terms of D and the rows of Lt are
// dealt out to the groups, whose partial sums meet in shared memory: a chain of j loads and
// FP64 FMAs per point would leave the chip waiting (one warp's worth of points per scheduler).

// The FP64 pipe (2 operations per clock and SM) also does comparisons, so maxima are taken on
// order-preserving integers, and what one thread can compute, one thread does.

// Sum over the groups of one value per thread, in the first group.
__device__ __forceinline__ double group_sum(double v, int R, int G, double* red) {
  __syncthreads();
  red[threadIdx.x] = v;
  __syncthreads();
  double s = v;
  if ((int)threadIdx.x < R)
    for (int g = 1; g < G; ++g) s += red[g * R + threadIdx.x];
  return s;
}

// Integer with the order of the double; NaN below everything (as fmax ignores it).
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  if ((b & 0x7FFFFFFFFFFFFFFFLL) > 0x7FF0000000000000LL) return LLONG_MIN;
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ double order_value(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFLL));
}

// D(r, r') for the points r = r0 + threadIdx.x % R: the products of the axes 0 and 1 once per
// (g0, g1) of the block, then one FMA per term.  r' = p, or r' = r (p < 0).
__device__ __forceinline__ double ips_column(const IpsArgs& a, int r0, int p, double* sxy, double* red) {
  const int R = a.R, G = blockDim.x / R, lr = threadIdx.x % R, grp = threadIdx.x / R;
  const int r = r0 + lr, last = min(r0 + R, a.ng) - 1;
  const int x0 = r0 / a.n2, nx = last / a.n2 - x0 + 1;  // (g0, g1) pairs of the block
  const bool in = r < a.ng;
  const int g2 = in ? r % a.n2 : 0, xi = in ? r / a.n2 - x0 : 0;
  const int p0f = p < 0 ? 0 : p / (a.n1 * a.n2), p1f = p < 0 ? 0 : (p / a.n2) % a.n1, p2 = p < 0 ? g2 : p % a.n2;
  double D = 0.0;
  for (int t0 = 0; t0 < a.nterm; t0 += a.tile) {
    const int nt = min(a.tile, a.nterm - t0);
    __syncthreads();
    for (int e = threadIdx.x; e < nt * nx; e += blockDim.x) {
      const int t = t0 + e / nx, x = x0 + e % nx, g0 = x / a.n1, g1 = x % a.n1;
      const int p0 = p < 0 ? g0 : p0f, p1 = p < 0 ? g1 : p1f;
      sxy[e] = a.A[((int64_t)t * a.n0 + p0) * a.n0 + g0] * a.A[a.o1 + ((int64_t)t * a.n1 + p1) * a.n1 + g1];
    }
    __syncthreads();
    const double* A2 = a.A + a.o2 + ((int64_t)t0 * a.n2 + p2) * a.n2 + g2;
#pragma unroll 4
    for (int t = grp; t < nt; t += G) D = fma(sxy[t * nx + xi], A2[(int64_t)t * a.n2 * a.n2], D);
  }
  return group_sum(D, R, G, red);
}

__device__ __forceinline__ long long block_kmax(long long m, long long* sv) {
  for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sv[threadIdx.x >> 5] = m;
  __syncthreads();
  m = sv[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = max(m, sv[i]);
  return m;
}

__global__ void __launch_bounds__(1024) ips_init_kernel(IpsArgs a) {
  extern __shared__ double ips_smem[];
  __shared__ long long sv[32];
  const int r0 = blockIdx.x * a.R, r = r0 + threadIdx.x;
  const double D = ips_column(a, r0, -1, ips_smem + blockDim.x, ips_smem);
  long long v = LLONG_MIN;
  if ((int)threadIdx.x < a.R && r < a.ng) {
    a.d[r] = D * D;
    v = order_key(D * D);
  }
  v = block_kmax(v, sv);
  if (threadIdx.x == 0) a.M[blockIdx.x] = v;
}

// Step j in one launch (the stream order between the steps is the only barrier): every block
// finds the pivot from the block maxima of step j - 1 -- the tie rule looks only into blocks
// whose maximum lies in the window -- then updates its own points and leaves its new maximum.
// The maxima and the diagonal alternate between two buffers, and a step reads piv only below j, so
// that no block reads what another one of its launch writes (scal[0], written at j = 0, is used
// from j = 1 on).  About 150 blocks, more on grids above 152 x 256 points.
__global__ void __launch_bounds__(1024) ips_step_kernel(IpsArgs a, int j) {
  extern __shared__ double ips_smem[];
  __shared__ long long sv[32], s_thr;
  __shared__ unsigned long long sh[32];
  __shared__ int si[32], s_list[32], s_n, s_stop;
  __shared__ double s_inv;
  // a selection that has stopped: piv[j - 1] is -1 from its last step on and fixed for this launch (the
  // status is written by this very launch, so that warps of one block could see it differ)
  if (j > 0 && a.piv[j - 1] < 0) return;
  const int nb = gridDim.x, bd = blockDim.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5, R = a.R, G = bd / R;
  const long long* M = a.M + (j & 1) * nb;
  const double* din = a.d + (int64_t)(j & 1) * a.ng;
  double* dout = a.d + (int64_t)((j & 1) ^ 1) * a.ng;
  if (tid == 0) s_n = 0;
  const double d0r = a.scal[0];
  long long kmax = LLONG_MIN;
  for (int b = tid; b < nb; b += bd) kmax = max(kmax, M[b]);
  kmax = block_kmax(kmax, sv);
  const double dmax = order_value(kmax);
  if (tid == 0) {
    const double d0 = j == 0 ? dmax : d0r;
    s_stop = kmax == LLONG_MIN || !(dmax >= a.chol_tol * d0) || !(dmax > 0.0);
    s_thr = order_key(fmax(dmax - a.tie_eps * d0, 0.5 * dmax));
  }
  __syncthreads();
  if (s_stop) {
    if (blockIdx.x == 0 && tid == 0) {
      *a.status = 1;
      a.piv[j] = -1;
    }
    return;
  }
  const long long thr = s_thr;
  // blocks with candidates (a list of up to 32; beyond it every block is looked at)
  for (int b = tid; b < nb; b += bd)
    if (M[b] >= thr) {
      const int i = atomicAdd(&s_n, 1);
      if (i < 32) s_list[i] = b;
    }
  __syncthreads();
  const int nl = s_n;
  unsigned long long best = ~0ULL;
  int bi = -1;
  for (int i = 0; i < (nl <= 32 ? nl : nb); ++i) {
    const int b = nl <= 32 ? s_list[i] : i;
    for (int x = tid; x < R; x += bd) {
      const int r = b * R + x;
      if (r < a.ng && order_key(din[r]) >= thr) {
        const unsigned long long hsh = splitmix64(a.seed ^ (uint64_t)r);
        if (bi < 0 || hsh < best || (hsh == best && r < bi)) {
          best = hsh;
          bi = r;
        }
      }
    }
  }
  for (int o = 16; o; o >>= 1) {
    const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (oi >= 0 && (bi < 0 || ob < best || (ob == best && oi < bi))) {
      best = ob;
      bi = oi;
    }
  }
  if (lane == 0) {
    sh[w] = best;
    si[w] = bi;
  }
  __syncthreads();
  int p = -1;
  best = ~0ULL;
  for (int i = 0; i < (bd >> 5); ++i)
    if (si[i] >= 0 && (p < 0 || sh[i] < best || (sh[i] == best && si[i] < p))) {
      best = sh[i];
      p = si[i];
    }
  if (p < 0) {  // no finite candidate
    if (blockIdx.x == 0 && tid == 0) {
      *a.status = 2;
      a.piv[j] = -1;
    }
    return;
  }
  if (blockIdx.x == 0 && tid == 0) {
    a.piv[j] = p;
    if (j == 0) a.scal[0] = dmax;
  }
  double* red = ips_smem;                // [bd]
  double* sxy = ips_smem + bd;           // term products, then L[i][p] in pieces of kLp
  const int r0 = blockIdx.x * R, lr = tid % R, grp = tid / R, r = r0 + lr;
  const bool in = r < a.ng;
  const double dr = in ? din[r] : 0.0;
  if (tid == bd - 1) s_inv = 1.0 / sqrt(din[p]);
  const double D = ips_column(a, r0, p, sxy, red);
  const double* Lr = a.Lt + (in ? r : 0);
  double s0 = 0.0, s1 = 0.0;
  for (int i0 = 0; i0 < j; i0 += kLp) {
    const int n = min(kLp, j - i0);
    __syncthreads();
    for (int i = tid; i < n; i += bd) sxy[i] = a.Lt[(int64_t)(i0 + i) * a.ng + p];
    __syncthreads();
    const double* L = Lr + (int64_t)i0 * a.ng;
    int i = grp;
#pragma unroll 4
    for (; i + G < n; i += 2 * G) {
      s0 = fma(L[(int64_t)i * a.ng], sxy[i], s0);
      s1 = fma(L[(int64_t)(i + G) * a.ng], sxy[i + G], s1);
    }
    if (i < n) s0 = fma(L[(int64_t)i * a.ng], sxy[i], s0);
  }
  const double sum = group_sum(s0 + s1, R, G, red);
  long long v = LLONG_MIN;
  if (grp == 0 && in) {
    const double l = (D * D - sum) * s_inv;  // set before the barriers of the sums
    a.Lt[(int64_t)j * a.ng + r] = l;
    const double dn = r == p ? -INFINITY : dr - l * l;
    dout[r] = dn;
    v = order_key(dn);
  }
  v = block_kmax(v, sv);
  if (tid == 0) a.M[((j & 1) ^ 1) * nb + blockIdx.x] = v;
}

__global__ void gather_x_kernel(const double2* __restrict__ phi, int nk, int nao, int ng,
                                const int32_t* __restrict__ ips, int np, double2* __restrict__ X) {
  const int64_t total = (int64_t)nk * np * nao;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int mu = (int)(e % nao);
    const int I = (int)((e / nao) % np);
    const int k = (int)(e / ((int64_t)nao * np));
    X[e] = phi[((int64_t)k * nao + mu) * ng + ips[I]];
  }
}

inline int nblocks(int64_t total, int cap = 152 * 32) {
  int64_t nb = (total + 255) / 256;
  if (nb > cap) nb = cap;
  if (nb < 1) nb = 1;
  return (int)nb;
}

}  // namespace

size_t ao_eval_work_bytes(const CellDev&, const BasisDev& b) {
  return (size_t)b.nao * b.maxprim * 3 * 16 * 64 * sizeof(double2);
}

cudaError_t ao_eval(cudaStream_t st, const CellDev& c, const BasisDev& b, double2* phi, double* work) {
  const int ng = c.mesh[0] * c.mesh[1] * c.mesh[2];
  const int nk = c.kmesh[0] * c.kmesh[1] * c.kmesh[2];
  if (c.orthorhombic) {
    double2* S = reinterpret_cast<double2*>(work);
    const int total1 = b.nao * b.maxprim * 3 * 16 * 64;
    ao_1d_kernel<<<nblocks(total1), 256, 0, st>>>(c, b, S);
    count_launch();
    const int64_t nblk = (int64_t)nk * b.nao * ((c.mesh[0] * c.mesh[1] + 255) / 256);
    ao_combine_kernel<<<(unsigned)std::min<int64_t>(nblk, 152 * 32), 256, 0, st>>>(c, b, S, phi, nblk);
    count_launch();
  } else {
    const int64_t total = (int64_t)((nk + KCH - 1) / KCH) * b.nao * ng;
    ao_general_kernel<<<nblocks(total, 152 * 16), 256, 0, st>>>(c, b, phi);
    count_launch();
  }
  return cudaGetLastError();
}

cudaError_t ip_init(cudaStream_t st, const double2* phi, int nkao, int ng, double* d, double* partial) {
  const int nsplit = 16;
  dim3 g((ng + 255) / 256, nsplit);
  ip_partial_kernel<<<g, 256, 0, st>>>(phi, nkao, ng, nullptr, 0, nsplit, partial, nullptr);
  count_launch();
  ip_init_combine_kernel<<<(ng + 255) / 256, 256, 0, st>>>(partial, nsplit, ng, d);
  count_launch();
  return cudaGetLastError();
}

cudaError_t ip_step(cudaStream_t st, const double2* phi, int nkao, int ng, int j, double* d, double* Lt,
                    int32_t* piv, int32_t* chosen, double* partial, int nsplit, uint64_t seed,
                    double tie_eps, double chol_tol, double* scal, int32_t* status) {
  ip_argmax_kernel<<<1, 1024, 0, st>>>(d, ng, j, piv, chosen, seed, tie_eps, chol_tol, scal, status);
  count_launch();
  dim3 g((ng + 255) / 256, nsplit);
  ip_partial_kernel<<<g, 256, 0, st>>>(phi, nkao, ng, piv, j, nsplit, partial, status);
  count_launch();
  ip_update_kernel<<<(ng + 255) / 256, 256, 0, st>>>(partial, nsplit, ng, j, piv, Lt, d, scal, status);
  count_launch();
  return cudaGetLastError();
}

namespace {
struct IpsLayout {
  int R, G, blocks, tile;  // points per block, thread groups
  size_t table, total;  // doubles
};
IpsLayout ips_layout(const CellDev& c, int nterm) {
  const int ng = c.mesh[0] * c.mesh[1] * c.mesh[2];
  IpsLayout l;
  // one wave: the points spread over the SMs, a warp to eight warps of them each, and up to
  // eight groups of threads on the same points (c5: 9.3 ms, 13.7 with one group)
  l.R = std::min(256, std::max(32, ((ng + 151) / 152 + 31) / 32 * 32));
  l.G = std::max(1, std::min(8, 1024 / l.R));
  l.blocks = (ng + l.R - 1) / l.R;
  const int nx = l.R / c.mesh[2] + 2;
  l.tile = std::max(1, std::min(nterm, 4096 / nx));
  l.table = (size_t)nterm * (c.mesh[0] * c.mesh[0] + c.mesh[1] * c.mesh[1] + c.mesh[2] * c.mesh[2]);
  l.total = l.table + 2 * (size_t)l.blocks + 2 * (size_t)ng;
  return l;
}
constexpr size_t kIpsMaxTable = (size_t)32 << 20;  // doubles (256 MB): beyond it, long contractions, Phi is read instead
}  // namespace

// Whether the separable selection is the faster one.  A step of it takes an FMA per term and grid point, a step
// of the other a pass over Phi (Nk N_AO values per point) and three launches more, so that long contractions
// (the square of the primitives of an AO each) on few k-points belong to the pass.  Nanoseconds per step, fitted to
// runs with 30 to 120 AOs on grids of 16^3 to 40^3.  Separable against the pass over Phi, 120 AOs, 40^3 grid, 300
// points: Nk = 1: 34 / 44 ms with 432 terms, 79 / 44 with 1488; Nk = 8: 81 / 102 with 1488, 116 / 103
// with 2280; 30 AOs, 16^3, Nk = 1, 150 points: 3.3 / 4.4 with 570.
bool ips_supported(const CellDev& c, int nterm, int nao) {
  if (!c.orthorhombic || nterm <= 0 || nterm >= (1 << 20) || ips_layout(c, nterm).table > kIpsMaxTable) return false;
  const double ng = (double)c.mesh[0] * c.mesh[1] * c.mesh[2], nk = (double)c.kmesh[0] * c.kmesh[1] * c.kmesh[2];
  return nterm * std::max(19.0, 2.1e-3 * ng) <= 15000.0 + (0.75 + 3.4e-3 * nk * nao) * ng;
}
size_t ips_work_bytes(const CellDev& c, int nterm) { return ips_layout(c, nterm).total * sizeof(double); }

// The separable selection.  Measured on GB300 (Phi and points together, 300 points, 24^3 grid,
// Nk = 1000, N_AO = 26): 9.3 ms, against 478 ms with one pass over Phi per pivot.
cudaError_t ips_select(cudaStream_t st, const CellDev& c, const BasisDev& b, const double* ao_work, const int* terms,
                       int nterm, int n_p, double* work, double* Lt, int32_t* piv, uint64_t seed, double tie_eps,
                       double chol_tol, double* scal, int32_t* status) {
  const IpsLayout l = ips_layout(c, nterm);
  IpsArgs a;
  a.A = work;
  a.o1 = (int64_t)nterm * c.mesh[0] * c.mesh[0];
  a.o2 = a.o1 + (int64_t)nterm * c.mesh[1] * c.mesh[1];
  a.nterm = nterm;
  a.n0 = c.mesh[0];
  a.n1 = c.mesh[1];
  a.n2 = c.mesh[2];
  a.ng = a.n0 * a.n1 * a.n2;
  a.R = l.R;
  a.tile = l.tile;
  a.M = reinterpret_cast<long long*>(work + l.table);
  a.d = work + l.table + 2 * (size_t)l.blocks;
  a.Lt = Lt;
  a.piv = piv;
  a.scal = scal;
  a.status = status;
  a.seed = seed;
  a.tie_eps = tie_eps;
  a.chol_tol = chol_tol;
  ips_table_kernel<<<nblocks((int64_t)l.table), 256, 0, st>>>(c, b, reinterpret_cast<const double2*>(ao_work), terms,
                                                              nterm, a.o1, a.o2, work);
  count_launch();
  const int threads = l.R * l.G;
  const size_t smem = sizeof(double) * (threads + std::max<size_t>(kLp, (size_t)l.tile * (l.R / a.n2 + 2)));
  ips_init_kernel<<<l.blocks, threads, smem, st>>>(a);
  count_launch();
  for (int j = 0; j < n_p; ++j) {
    ips_step_kernel<<<l.blocks, threads, smem, st>>>(a, j);
    count_launch();
  }
  return cudaGetLastError();
}

cudaError_t gather_x(cudaStream_t st, const double2* phi, int nk, int nao, int ng, const int32_t* ips,
                     int np, double2* X) {
  gather_x_kernel<<<nblocks((int64_t)nk * np * nao), 256, 0, st>>>(phi, nk, nao, ng, ips, np, X);
  count_launch();
  return cudaGetLastError();
}

}  // namespace isdf
