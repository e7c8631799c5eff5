// Tensor-core (tcgen05) kernels of the fragment ERIs, Eq. 19:
//     E = sum_q B^q B^q^H   with  B^q = M^q L^q   (V^q = L^q L^q^H).
// syrk_tc_kernel forms E (below); mlgemm_tc_kernel forms B (further down, with
// three slices).
//
// Structural zeros of L^q.  Pi^q is factorised with truncation to rank r_q
// (pivots perm_q[0..r_q)), W = L_S^{-1} is nonzero only in the columns
// perm_q[c], and V_xi = L_xi L_xi^H has rank n_q <= r_q, so L^q = W^T L_xi is
// nonzero only in the rows perm_q[c], c < r_q, and the columns J < n_q.
// B^q = M^q L^q therefore contracts over the r_q gathered columns of M^q and
// has n_J = max_q n_q columns; nothing else of L^q is touched.
//
// E as a real symmetric matrix.  The AO basis is real and the k-mesh
// Gamma-centred, so V^{-q} = conj(V^q) and M^{-q}_{(qp)} = conj(M^q_{(pq)}), hence
// E_{s(a) s(b)} = conj(E_ab) with s((pq)) = (qp).  That antiunitary symmetry fixes
// the basis  u_(pq) = e_(pq) + e_(qp),  v_(pq) = i (e_(pq) - e_(qp))  (p < q)  and
// e_(pp), so E is real in it.  The pair products are formed in that basis
// (rows u: 2 Re(conj(t_p) t_q), v: 2 Im(conj(t_p) t_q), pp: |t_p|^2, all real), so
// the rows R^q of M^q and B^q = M^q L^q are already those of the basis, with
// M^{-q} = conj(M^q); E' = sum_{all q} R^q R^q^H is real, i.e.
//     E' = c sum_{q in S} [Re R^q, Im R^q] [Re R^q, Im R^q]^T
// (c = 2 over the half set S of the time-reversal pairing, c = 1 over every q).
// One real SYRK of n_f^2 rows replaces the complex HERK: half its real
// products.  Only lower-triangle tiles are formed; the finish maps E' to E.
//
// Precision.  Each real row of R is scaled by a power of two 2^e so that its
// largest entry lies in [64, 128), and every scaled value x is written as two
// fp16 slices
//     x = s1 + s2 + d,   s1 = rint(x) (an integer, |s1| <= 128),  s2 = fp16(x - s1) (|s2| <= 1/2),
// so that |d| <= 2^-12 |s2| (19 significant bits, against 24 in FP32).  The
// tcgen05.mma kind::f16 products feed two FP32 TMEM accumulators:
//     g0 = S1.T1   (integers of magnitude <= 2^14),
//     g1 = S1.T2 + S2.T1 + S2.T2   (magnitude <= 2^6 + 2^-2 per product).
// g0 carries the bulk of E' and must be exact: a chunk of 1024 k-steps keeps
// its partial sums integers of magnitude at most 2^24, so the FP32
// accumulation is exact whatever its rounding.  g1 is not exact, but its
// products are 2^-7 of g0's and of either sign (s2 is a rounding remainder),
// so the truncation of tcgen05's FP32 accumulation over two chunks enters at
// ~2^-30 of |R_a||R_b|.  Both accumulators are double-buffered, g0 drained every
// chunk and g1 every second chunk (overlapping the next chunk's MMAs), into
// float-float (TwoSum) running sums held in the drain warps' registers.  Four products per useful
// product (the three-slice form with the same accuracy target needs six); the
// representation error d is random in sign off the diagonal, and the slicing
// kernel sums each row's sum of x^2 - (s1 + s2)^2 in FP64 so that the finish
// makes the diagonal exact.  Simulated on the c2 and c4 k-mesh data against the
// exact FP64 products: ERIs within ~1e-9 Ha, E_J within ~3e-8 Ha.
//
// Kernel roles (576 threads): warp 0 issues TMA loads, warp 1 allocates TMEM
// and issues the MMAs, warps 2-17 drain TMEM into the float-float sums.
// Every wait is bounded: on expiry the CTA records an error code and exits.
#include <cuda.h>
#include <cuda_fp16.h>

#include <cstring>
#include <vector>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace isdf {

namespace tc {

constexpr int BM = 128;        // A' rows per tile (64 complex rows of E)
constexpr int BN = 128;        // B' rows per tile (complex columns of E)
constexpr int BK = 64;         // fp16 per row per stage (one 128-byte swizzle row)
constexpr int NSLICE = 2;                   // fp16 slices per value in E': s1 (integer), s2 (remainder)
constexpr int TMEM_COLS = 512;              // g0 and g1, each two 128-column FP32 buffers
// E' kernel: warp 0 TMA, warp 1 MMA, 16 drain warps (TMEM lane quarter warp % 4, 32 of
// the 128 columns each), whose registers hold the tile's float-float running sums
constexpr int kSyrkThreads = 576, kDrainWarps = 16, kDrainCols = 32;
constexpr int kP1 = 2;                      // chunks per g1 drain
// Instruction descriptor of kind::f16: FP32 accumulate, fp16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

struct TileArgs {
  const int2* tiles;   // (ti, tj) per CTA
  float* ws_hi;        // [tile][BN][BM] float-float sums, high part
  float* ws_lo;        // low part
  int nkb;             // k-blocks of BK
  int accumulate;      // 1: add to the workspace of an earlier launch (K chunks)
  int* err;            // device error word
};

// Pipeline variants: BKt fp16 of K per stage row (64: 128-byte swizzle, 32: 64-byte
// swizzle) and NST stages; a 1024-element exact chunk of g0 is 1024 / BKt k-blocks.
// TMEM columns: g0 of chunk c at (c & 1) BN, g1 of chunk c at (2 + (c / kP1 & 1)) BN.
template <int BKt, int NST>
__global__ void __launch_bounds__(kSyrkThreads, 1)
    syrk_tc_kernel(const __grid_constant__ CUtensorMap mS1, const __grid_constant__ CUtensorMap mS2, TileArgs args) {
  constexpr int kA = BM * BKt * 2, kB = BN * BKt * 2, kStage = NSLICE * (kA + kB);
  constexpr int kChunk = 1024 / BKt;  // k-blocks per exact g0 chunk
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 1024-byte alignment of the shared-window address (swizzle atoms)
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NST * kStage);
  uint64_t* full = bars;                // [NST]
  uint64_t* empty = bars + NST;         // [NST]
  uint64_t* accf = bars + 2 * NST;      // [2] chunk accumulated (per buffer pair)
  uint64_t* acce = bars + 2 * NST + 2;  // [2] g0 buffer drained
  uint64_t* acce1 = bars + 2 * NST + 4; // [2] g1 buffer drained
  uint64_t* done = bars + 2 * NST + 6;  // settle
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* s_err = reinterpret_cast<volatile int*>(s_tmem + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int2 tile = args.tiles[blockIdx.x];
  const int nkb = args.nkb;
  const int nchunks = (nkb + kChunk - 1) / kChunk;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], kDrainWarps);
      mbar_init(&acce1[b], kDrainWarps);
    }
    mbar_init(done, 1);
    *s_err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;

  int fills = 0;  // stages filled so far (thread 0)
  if (warp == 0) {
    if (lane == 0) {
      // stage layout: S1 rows of A, S2 rows of A, S1 rows of B, S2 rows of B
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % NST, r = kb / NST;
        if (!mbar_wait(&empty[s], (r & 1) ^ 1, s_err, args.err, 1)) break;
        uint8_t* st = smem + s * kStage;
        mbar_expect_tx(&full[s], kStage);
        const int x = kb * BKt;
        tma_load_2d(st, &mS1, &full[s], x, tile.x * BM);
        tma_load_2d(st + kA, &mS2, &full[s], x, tile.x * BM);
        tma_load_2d(st + 2 * kA, &mS1, &full[s], x, tile.y * BN);
        tma_load_2d(st + 2 * kA + kB, &mS2, &full[s], x, tile.y * BN);
        ++fills;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % NST, r = kb / NST;
        const int c = kb / kChunk;
        const bool first_in_chunk = (kb % kChunk) == 0;
        const int p = c / kP1;  // g1 period
        const bool first_in_period = first_in_chunk && (c % kP1) == 0;
        if (first_in_chunk) {
          // g0 buffer (c & 1) was last used by chunk c - 2, g1 buffer (p & 1) by period p - 2
          if (c >= 2 && !mbar_wait(&acce[c & 1], ((c >> 1) - 1) & 1, s_err, args.err, 2)) break;
          if (first_in_period && p >= 2 && !mbar_wait(&acce1[p & 1], ((p >> 1) - 1) & 1, s_err, args.err, 5))
            break;
          tc_fence_after();
        }
        if (!mbar_wait(&full[s], r & 1, s_err, args.err, 3)) break;
        tc_fence_after();
        const uint8_t* st = smem + s * kStage;
        const uint64_t a1 = sdesc_k<BKt>(st), a2 = sdesc_k<BKt>(st + kA);
        const uint64_t b1 = sdesc_k<BKt>(st + 2 * kA), b2 = sdesc_k<BKt>(st + 2 * kA + kB);
        const uint32_t g0 = tmem_base + (uint32_t)((c & 1) * BN), g1 = tmem_base + (uint32_t)((2 + (p & 1)) * BN);
#pragma unroll
        for (int kk = 0; kk < BKt / 16; ++kk) {
          const uint64_t off = (uint64_t)(kk * 32) >> 4;  // 16 fp16 = 32 bytes along K
          const uint32_t acc0 = (first_in_chunk && kk == 0) ? 0u : 1u;
          const uint32_t acc1 = (first_in_period && kk == 0) ? 0u : 1u;
          umma_f16(g0, a1 + off, b1 + off, kIdesc, acc0);
          umma_f16(g1, a1 + off, b2 + off, kIdesc, acc1);
          umma_f16(g1, a2 + off, b1 + off, kIdesc, 1u);
          umma_f16(g1, a2 + off, b2 + off, kIdesc, 1u);
        }
        umma_commit(&empty[s]);
        if ((kb % kChunk) == kChunk - 1 || kb == nkb - 1) umma_commit(&accf[c & 1]);
      }
    }
  } else {
    // drain warps 2..17: TMEM lane quarter warp % 4 (a hardware rule), 32 columns each;
    // the tile's float-float sums stay in registers until the last chunk
    const int q = warp & 3, cblk = (warp - 2) >> 2;
    const int row = q * 32 + lane, col0 = cblk * kDrainCols;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    float* __restrict__ wh = args.ws_hi + (size_t)blockIdx.x * BN * BM;
    float* __restrict__ wl = args.ws_lo + (size_t)blockIdx.x * BN * BM;
    float H[kDrainCols], L[kDrainCols];
#pragma unroll
    for (int j = 0; j < kDrainCols; ++j) {
      H[j] = args.accumulate ? wh[(size_t)(col0 + j) * BM + row] : 0.f;
      L[j] = args.accumulate ? wl[(size_t)(col0 + j) * BM + row] : 0.f;
    }
    bool ok = true;
    for (int c = 0; c < nchunks; ++c) {
      ok = __all_sync(0xffffffffu, mbar_wait(&accf[c & 1], (c >> 1) & 1, s_err, args.err, 4));
      if (!ok) break;
      tc_fence_after();
      const int p = c / kP1;
      const bool drain1 = (c % kP1) == kP1 - 1 || c == nchunks - 1;
      const uint32_t t0 = tmem_base + lane_off + (uint32_t)((c & 1) * BN + col0);
      const uint32_t t1 = tmem_base + lane_off + (uint32_t)((2 + (p & 1)) * BN + col0);
#pragma unroll
      for (int cb = 0; cb < kDrainCols / 4; ++cb) {
        uint32_t v0[4], v1[4];
        tmem_ld4(t0 + cb * 4, v0);
        if (drain1) tmem_ld4(t1 + cb * 4, v1);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int jj = cb * 4 + j;
          const float a0 = __uint_as_float(v0[j]);
          // (H, L) += a0 with TwoSum on the high part; g1 into the low part
          const float S = H[jj] + a0;
          const float bp = S - H[jj];
          const float e = (H[jj] - (S - bp)) + (a0 - bp);
          H[jj] = S;
          float l = L[jj] + e;
          if (drain1) l += __uint_as_float(v1[j]);
          L[jj] = l;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&acce[c & 1]);
        if (drain1) mbar_arrive(&acce1[p & 1]);
      }
    }
    if (ok) {
#pragma unroll
      for (int j = 0; j < kDrainCols; ++j) {
        wh[(size_t)(col0 + j) * BM + row] = H[j];
        wl[(size_t)(col0 + j) * BM + row] = L[j];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*s_err) settle(full, NST, fills, done);  // a wait expired: wait for what is in flight
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS)
                 : "memory");
  }
}

// ----------------------------------------------------------------- helpers
// B is addressed as element (a, k), k = Q nJ + J, at B[slot(Q) sQ + a sA + J]
// (J < nJ), slot(Q) = qmap[Q], or Q without a map.
struct BView {
  const float2* p;
  int64_t sQ, sA, nJ;
  const int* qmap;
  __device__ __forceinline__ float2 at(int64_t a, int64_t k) const {
    const int64_t Q = k / nJ, J = k - Q * nJ;
    const int64_t slot = qmap ? (int64_t)__ldg(qmap + Q) : Q;
    return p[slot * sQ + a * sA + J];
  }
};

__device__ __forceinline__ float amax2(float2 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }
// Exponent e with m 2^e in [64, 128) (0 for a zero or non-finite maximum).
__device__ __forceinline__ int slice_exp(float m) { return (m > 0.f && isfinite(m)) ? 6 - ilogbf(m) : 0; }

template <typename T>
__device__ __forceinline__ T block_max(T v, T* sm) {
  for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  T m = sm[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = max(m, sm[i]);
  __syncthreads();
  return m;
}

// Row exponents of R over the whole sum (one block per row).  The rows of B^q
// are those of the time-reversal basis: pair o = (p < q) -> rows 2o (u) and
// 2o + 1 (v), diagonal p -> row 2P + p; R^q = [Re B^q, Im B^q].
__global__ void rrow_scale_kernel(BView B, int64_t K, int* __restrict__ row_exp) {
  const int64_t a = blockIdx.x;
  float m = 0.f;
  for (int64_t k = threadIdx.x; k < K; k += blockDim.x) m = fmaxf(m, amax2(B.at(a, k)));
  __shared__ float sm[32];
  m = block_max(m, sm);
  if (threadIdx.x == 0) row_exp[a] = min(slice_exp(m), 127);
}

// rint(x) for |x| < 2^22 by two additions (the conversion pipe runs at an eighth of their rate).
__device__ __forceinline__ float rint_small(float x) { return __fadd_rn(__fadd_rn(x, 12582912.f), -12582912.f); }
__device__ __forceinline__ uint32_t half2_bits(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Two slices of x = v 2^e (|x| < 128), the integer s1 = rint(x) and the fp16 remainder s2 = fp16(x - s1), with
// dd = x - s1 - s2 exactly (FP32), of the R rows for the sum positions j0 .. j0 + nq - 1, one block per
// row a: columns 2 (jl nJ + J) and + 1 hold the (re, im) of B at (position
// j0 + jl, J); columns beyond 2 nq nJ (up to the padded width K2) are zero.
// With corr, the block also adds to corr[a] the part of E'_aa (in slice units)
// that the slices do not represent, sum of x^2 - (s1 + s2)^2 = dd (2 x - dd), so
// that the finish makes the diagonal exact; off the diagonal the representation
// error is of either sign and averages out.
// A row's values of one position are contiguous: a warp takes a position at a time.
__global__ void __launch_bounds__(256) rsplit_kernel(BView B, int64_t j0, int nq, int64_t K2,
                                                     const int* __restrict__ row_exp, __half* __restrict__ S1,
                                                     __half* __restrict__ S2, double* __restrict__ corr) {
  const int64_t a = blockIdx.x;
  const int ex = row_exp[a], nJ = (int)B.nJ, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float sc = ldexpf(1.f, ex);
  float d = 0.f;
  auto put = [&](float2 v, int64_t at) {
    const float x = v.x * sc, y = v.y * sc, r1 = rint_small(x), i1 = rint_small(y), rx = x - r1, ry = y - i1;
    const __half2 h2 = __floats2half2_rn(rx, ry);
    const float2 f2 = __half22float2(h2);
    const float rd = rx - f2.x, id = ry - f2.y;
    *reinterpret_cast<uint32_t*>(S1 + at) = half2_bits(r1, i1);
    *reinterpret_cast<__half2*>(S2 + at) = h2;
    d += rd * (2.f * x - rd) + id * (2.f * y - id);
  };
  for (int jl = warp; jl < nq; jl += 8) {
    const int64_t slot = B.qmap ? (int64_t)__ldg(B.qmap + j0 + jl) : j0 + jl;
    const float2* p = B.p + slot * B.sQ + a * B.sA;
    const int64_t at = a * K2 + 2 * (int64_t)jl * nJ;
#pragma unroll 4
    for (int J = lane; J < nJ; J += 32) put(p[J], at + 2 * J);
  }
  for (int64_t c = 2 * (int64_t)nq * nJ + threadIdx.x; c < K2; c += 256) S1[a * K2 + c] = S2[a * K2 + c] = __half(0.f);
  if (!corr) return;
  __shared__ double sd[8];
  double v = d;
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sd[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sd[w];
    corr[a] += t;
  }
}

// The E' -> E map fused with the chemist's permutation and the traces, so that E
// is never stored.  Orbit o1 (a pair p < q: rows u = 2 o1, v = 2 o1 + 1; or a
// diagonal p: one row) and orbit o2 (x < y or x) span a block of E':
// U = E'(u1, u2), X = E'(u1, v2), Y = E'(v1, u2), Z = E'(v1, v2).  Its ERIs are
//   pair-pair:  (pq|yx) = [(U+Z) + i(Y-X)]/4,  (pq|xy) = [(U-Z) + i(X+Y)]/4,
//               (qp|yx) = conj (pq|xy),       (qp|xy) = conj (pq|yx);
//   pair-diag:  (pq|xx) = (U + iY)/2,  (qp|xx) = conj;
//   diag-pair:  (pp|yx) = (U - iX)/2,  (pp|xy) = conj;     diag-diag: (pp|xx) = U.
// For a Hermitian gamma the four terms of a block in E_J = 1/2 sum gamma_pq gamma_rs (pq|rs)
// and E_K = -1/4 sum gamma_ps gamma_rq (pq|rs) pair up into real parts:
//   J_block = U Re A Re B - Z Im A Im B + X Re A Im B - Y Im A Re B   (A = gamma_pq, B = gamma_yx),
//   K_block = 2 Re(gamma_px gamma_yq (pq|yx)) + 2 Re(gamma_py gamma_xq (pq|xy)),
// and the pair-diagonal and diagonal cases likewise, so the traces take a few
// real FP64 operations per block instead of complex ones per ERI.  Each thread
// takes one block with o1 >= o2 (consecutive threads: consecutive o1, so the
// workspace reads of the lower triangle are contiguous) and its mirror (o2, o1),
// whose values are (U, Y, X, Z).  Values are formed in float-float, the ERIs
// written as complex64 (mixed) or complex128 (FP64_TC); eri may be NULL, and
// gamma NULL skips the traces.  Per-block partials go to part[blk] (J) and
// part[gridDim.x + blk] (K); the fixed grid keeps the sums reproducible.
// part[2 gridDim.x].x: whether gamma is Hermitian (gamma_herm_kernel).
__device__ __forceinline__ ffloat ep_ff(const float* __restrict__ wh, const float* __restrict__ wl,
                                        const int* __restrict__ tile_of, int nt, int64_t i, int64_t j,
                                        const int* __restrict__ row_exp, ffloat sc) {
  if (i < j) {
    const int64_t t = i;
    i = j;
    j = t;
  }
  const int t = tile_of[(i / BM) * nt + (j / BN)];
  const size_t base = ((size_t)t * BN + (size_t)(j % BN)) * BM + (size_t)(i % BM);
  const ffloat v = ff_two_sum(wh[base], wl[base]);
  return ff_ldexp(v, -(row_exp[i] + row_exp[j])) * sc;
}

struct BlockVals {
  double U, X, Y, Z;
};

// Trace terms of the block (row orbit (p, q), column orbit (x, y)); a diagonal orbit has q == p
// (resp. y == x).  (r1, i1) = (pq|yx), (r2, i2) = (pq|xy) as in the table above.
__device__ __forceinline__ void block_traces(const double2* __restrict__ g, int nf, int p, int q, int x, int y,
                                             const BlockVals& b, double r1, double i1, double r2, double i2,
                                             double& aj, double& ak) {
  auto gm = [&](int i, int j) { return g[(int64_t)i * nf + j]; };
  if (p != q && x != y) {
    const double2 A = gm(p, q), B = gm(y, x);
    aj += b.U * A.x * B.x - b.Z * A.y * B.y + b.X * A.x * B.y - b.Y * A.y * B.x;
    const double2 w1 = cmul(gm(p, x), gm(y, q)), w2 = cmul(gm(p, y), gm(x, q));
    ak += 2.0 * (w1.x * r1 - w1.y * i1 + w2.x * r2 - w2.y * i2);
  } else if (p != q) {
    const double2 A = gm(p, q), w = cmul(gm(p, x), gm(x, q));
    aj += gm(x, x).x * (A.x * b.U - A.y * b.Y);
    ak += 2.0 * (w.x * r1 - w.y * i1);
  } else if (x != y) {
    const double2 B = gm(y, x), w = cmul(gm(p, x), gm(y, p));
    aj += gm(p, p).x * (B.x * b.U + B.y * b.X);
    ak += 2.0 * (w.x * r1 - w.y * i1);
  } else {
    const double2 w = gm(p, x);
    aj += gm(p, p).x * gm(x, x).x * b.U;
    ak += (w.x * w.x + w.y * w.y) * b.U;
  }
}

__device__ __forceinline__ void put_part(float& o, double v) { o = ffloat(v).hi; }
__device__ __forceinline__ void put_part(double& o, double v) { o = v; }

// ERIs and trace terms of the block (o1, o2) and, with mirror, of (o2, o1).  The FP64 pipe bounds
// this (two operations a clock and SM): the mirrored block has the same four numbers up to
// conjugation, so each is formed and narrowed once; and for a Hermitian gamma its trace terms
// equal the block's (A' = conj B, B' = conj A; the exchange products conjugate along with
// their integrals), so they count twice instead of being formed twice.
template <typename TO>
__device__ __forceinline__ void emit_block(TO* __restrict__ eri, const double2* __restrict__ g, int nf, int p,
                                           int q, int x, int y, const BlockVals& b, bool mirror, bool herm,
                                           double& aj, double& ak) {
  const bool pr = p != q, pc = x != y;
  double r1, i1, r2 = 0.0, i2 = 0.0;
  if (pr && pc) {
    r1 = 0.25 * (b.U + b.Z), i1 = 0.25 * (b.Y - b.X), r2 = 0.25 * (b.U - b.Z), i2 = 0.25 * (b.X + b.Y);
  } else if (pr || pc) {
    r1 = 0.5 * b.U, i1 = pr ? 0.5 * b.Y : -0.5 * b.X;
  } else {
    r1 = b.U, i1 = 0.0;
  }
  if (eri) {
    auto at = [&](int i0, int i1, int i2, int i3) { return eri + (((int64_t)i0 * nf + i1) * nf + i2) * nf + i3; };
    auto cj = [](TO v) {
      v.y = -v.y;
      return v;
    };
    TO z1, z2;
    put_part(z1.x, r1);
    put_part(z1.y, i1);
    if (pr && pc) {
      put_part(z2.x, r2);
      put_part(z2.y, i2);
      *at(p, q, y, x) = z1;
      *at(p, q, x, y) = z2;
      *at(q, p, y, x) = cj(z2);
      *at(q, p, x, y) = cj(z1);
      if (mirror) {  // (xy|qp) = conj (pq|yx)^(X <-> Y) and so on
        *at(x, y, q, p) = cj(z1);
        *at(x, y, p, q) = z2;
        *at(y, x, q, p) = cj(z2);
        *at(y, x, p, q) = z1;
      }
    } else if (pr) {
      *at(p, q, x, x) = z1;
      *at(q, p, x, x) = cj(z1);
      if (mirror) {
        *at(x, x, q, p) = cj(z1);
        *at(x, x, p, q) = z1;
      }
    } else if (pc) {
      *at(p, p, y, x) = z1;
      *at(p, p, x, y) = cj(z1);
      if (mirror) {
        *at(x, y, p, p) = cj(z1);
        *at(y, x, p, p) = z1;
      }
    } else {
      *at(p, p, x, x) = z1;
      if (mirror) *at(x, x, p, p) = z1;
    }
  }
  if (!g) return;
  double tj = 0.0, tk = 0.0;
  block_traces(g, nf, p, q, x, y, b, r1, i1, r2, i2, tj, tk);
  if (mirror && herm) {
    tj += tj;
    tk += tk;
  } else if (mirror) {
    block_traces(g, nf, x, y, p, q, BlockVals{b.U, b.Y, b.X, b.Z}, r1, -i1, r2, i2, tj, tk);
  }
  aj += tj;
  ak += tk;
}

// flag = gamma is Hermitian to 2^-44 of its mean modulus, the rounding of a C n C^H (one block)
__global__ void __launch_bounds__(1024) gamma_herm_kernel(const double2* __restrict__ g, int nf,
                                                          double2* __restrict__ flag) {
  __shared__ double sm[32], sd[32];
  double m = 0.0, d = 0.0;
  for (int e = threadIdx.x; e < nf * nf; e += blockDim.x) {
    const double2 u = g[e], v = g[(e % nf) * nf + e / nf];
    m += fabs(u.x) + fabs(u.y);
    d = fmax(d, fabs(u.x - v.x) + fabs(u.y + v.y));
    if (!(fabs(u.x) + fabs(u.y) <= 1e300)) d = INFINITY;
  }
  m /= (double)nf * nf;
  for (int o = 16; o; o >>= 1) {
    m += __shfl_xor_sync(0xffffffffu, m, o);
    d = fmax(d, __shfl_xor_sync(0xffffffffu, d, o));
  }
  if ((threadIdx.x & 31) == 0) {
    sm[threadIdx.x >> 5] = m;
    sd[threadIdx.x >> 5] = d;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) {
      sm[0] += sm[w];
      sd[0] = fmax(sd[0], sd[w]);
    }
    *flag = make_double2(sd[0] <= sm[0] * 0x1p-44 ? 1.0 : 0.0, 0.0);
  }
}

template <typename TO>
__global__ void __launch_bounds__(256) syrk_eri_kernel(const float* __restrict__ wh, const float* __restrict__ wl,
                                                       const int* __restrict__ tile_of, int nt,
                                                       const int2* __restrict__ orb, int nf,
                                                       const int* __restrict__ row_exp, const double* __restrict__ corr,
                                                       double scale, TO* __restrict__ eri,
                                                       const double2* __restrict__ gam, double2* __restrict__ part,
                                                       int tested) {
  const int no = nf * (nf + 1) / 2, P = nf * (nf - 1) / 2;
  const int nch = (no + 255) / 256;
  const int64_t ntask = (int64_t)no * nch;
  const ffloat sc(scale);
  const bool herm = gam && tested && part[2 * gridDim.x].x != 0.0;
  double aj = 0.0, ak = 0.0;
  for (int64_t task = blockIdx.x; task < ntask; task += gridDim.x) {
    const int o2 = (int)(task / nch), o1 = (int)(task % nch) * 256 + (int)threadIdx.x;
    if (o1 < o2 || o1 >= no) continue;
    const int2 r = orb[o1], c = orb[o2];
    const bool pr = o1 < P, pc = o2 < P;
    const int64_t u1 = pr ? 2 * (int64_t)o1 : 2 * (int64_t)P + (o1 - P);
    const int64_t u2 = pc ? 2 * (int64_t)o2 : 2 * (int64_t)P + (o2 - P);
    BlockVals b{0.0, 0.0, 0.0, 0.0};
    b.U = ep_ff(wh, wl, tile_of, nt, u1, u2, row_exp, sc).to_double();
    if (pc) b.X = ep_ff(wh, wl, tile_of, nt, u1, u2 + 1, row_exp, sc).to_double();
    if (pr) b.Y = ep_ff(wh, wl, tile_of, nt, u1 + 1, u2, row_exp, sc).to_double();
    if (pr && pc) b.Z = ep_ff(wh, wl, tile_of, nt, u1 + 1, u2 + 1, row_exp, sc).to_double();
    if (o1 == o2 && corr) {
      // the diagonal's products left out of the contraction (slice units)
      b.U += ldexp(corr[u1], -2 * row_exp[u1]) * scale;
      if (pr) b.Z += ldexp(corr[u1 + 1], -2 * row_exp[u1 + 1]) * scale;
    }
    emit_block<TO>(eri, gam, nf, r.x, r.y, c.x, c.y, b, o1 != o2, herm, aj, ak);
  }
  if (!gam) return;
  __shared__ double sj[256], sk[256];
  sj[threadIdx.x] = aj;
  sk[threadIdx.x] = ak;
  __syncthreads();
  for (int o = 128; o; o >>= 1) {
    if ((int)threadIdx.x < o) {
      sj[threadIdx.x] += sj[threadIdx.x + o];
      sk[threadIdx.x] += sk[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[blockIdx.x] = make_double2(sj[0], 0.0);
    part[gridDim.x + blockIdx.x] = make_double2(sk[0], 0.0);
  }
}

// out4 = (E_J, E_K, Im E_J, Im E_K) from the per-block partials (one block, fixed order).
__global__ void __launch_bounds__(256) eri_traces_final_kernel(const double2* __restrict__ part, int nblk,
                                                               double* __restrict__ out4) {
  __shared__ double2 sj[256], sk[256];
  double2 aj = make_double2(0.0, 0.0), ak = make_double2(0.0, 0.0);
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
    aj = cadd(aj, part[i]);
    ak = cadd(ak, part[nblk + i]);
  }
  sj[threadIdx.x] = aj;
  sk[threadIdx.x] = ak;
  __syncthreads();
  for (int o = 128; o; o >>= 1) {
    if ((int)threadIdx.x < o) {
      sj[threadIdx.x] = cadd(sj[threadIdx.x], sj[threadIdx.x + o]);
      sk[threadIdx.x] = cadd(sk[threadIdx.x], sk[threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out4[0] = 0.5 * sj[0].x;
    out4[1] = -0.25 * sk[0].x;
    out4[2] = 0.5 * sj[0].y;
    out4[3] = -0.25 * sk[0].y;
  }
}

// ---------------------------------------------------------------------------
// B^q = M^q L^q on the tensor cores with three slices per operand.
//
// Only the structural nonzeros of L^q enter (see the top of the file): the
// contraction runs over c < r_q with M^q's column perm_q[c] and L^q's row
// perm_q[c], and the output has n_J columns.  Real form: one A' row per row of M,
// P_a = (Re M_a,perm(c), Im M_a,perm(c))_c, and two B' rows per column of L,
// R_J = (Re L_perm(c)J, -Im L_perm(c)J)_c and I_J = (Im L_perm(c)J, Re L_perm(c)J)_c,
// so P_a.R_J = Re B_aJ and P_a.I_J = Im B_aJ (the complex embedding sits on the
// small operand; the slices of M are written and streamed once).  M rows are
// scaled by 2^e_a (largest gathered
// component over the q of the sum in [64, 128)), L columns by 2^f_qJ per q; both
// are cut into an integer and two fp16 remainders,
//     x = s1 + s2 + s3 + d,  s1 = rint(x),  s2 = fp16(x - s1),  s3 = fp16(x - s1 - s2),
// about 30 significant bits (B = M W^T L_xi carries the cancellation of the
// ill-conditioned W, so 19 bits measurably degrade the traces).  Six fp16
// products feed three groups
//   g0 = S1T1, g1 = S1T2 + S2T1, g2 = S1T3 + S2T2 + S3T1;
// with K' = 2 r <= kMlMaxK every partial sum of g0 is an integer of magnitude
// below 2^24, so its FP32 TMEM accumulation is exact; g1 and g2 are 2^-7 and
// 2^-18 of it and accumulate in FP32 over at most kMlMaxK terms.  The epilogue
// forms g0 + (g1 + g2) once and rescales.  Simulated on the c2 data against the
// exact products: E_J within ~1e-9 Ha (four 7-bit slices with ten products: ~2e-8).
//
// One kernel slices M and multiplies.  What bounds the product is the tensor pipe (six
// products) as long as M is read once and B written once; slices of M in memory would cost
// 12 + 12 bytes per value on top of the 8 + 8 (measured: the separate slicing pass and the
// GEMM on 128 x 64 tiles took 27 ms at Nk = 1000, 16,000 rows, r = 128).  So a persistent
// CTA takes 128 rows of one q: producer warps load the gathered columns of M, cut them and
// write the slices in the MMA's shared-memory layout, the slices of L come by TMA (a q's
// stay in L2 while its row blocks pass), and passes of up to 64 complex columns (N = 128: an
// MMA of 128 x N x 16 takes N/2 clocks only from N = 128 on) accumulate in three 128-column
// TMEM groups.  The next pass's MMAs wait only for the TMEM reads of the one before.
// The epilogue also leaves the rows' largest entries for the slicing of B.
//
// Kernel roles (704 threads): warp 0 TMA, warp 1 TMEM and MMAs, warps 2-13 producers (three groups
// that take the k-blocks in turn, each with its next one in flight), warps 14-21 epilogue.
constexpr int MSL = 3;                                     // slices per operand
constexpr int MBJ = 32;                                    // columns of L are padded to a multiple of it
constexpr int MBK = 32;                                    // fp16 of K per stage row (64-byte swizzle)
constexpr int MPN = 128;                                   // B' rows per pass (64 complex columns)
constexpr int MA_BYTES = BM * MBK * 2;                     // 8 KB per slice
constexpr int MB_BYTES = MPN * MBK * 2;                    // 8 KB per slice
constexpr int MBOX = 64 * MBK * 2;                         // bytes of one TMA box (64 rows)
constexpr int MSTAGE_BYTES = MSL * (MA_BYTES + MB_BYTES);  // 48 KB
constexpr int MSTAGES = 3;
constexpr int MGROUPS = 3;                                 // producer groups of four warps
constexpr int MTHREADS = 64 + 128 * MGROUPS + 256;
constexpr int MEPI = 8;                                    // epilogue warps
constexpr int kMlPitch = MPN + 2;                          // floats per staged row (bank-conflict padding)
constexpr int kMlOut = BM * kMlPitch * 4;
constexpr int kMlTmem = 512;                               // three 128-column groups
constexpr int kMlMaxK = 640;                               // K' bound for exact accumulation
constexpr uint32_t kIdescMl = (1u << 4) | ((uint32_t)(BM >> 4) << 24);  // N >> 3 at bit 17 is added per pass

struct MlArgs {
  const float2* M;      // gathered: element (a, c) of sum position j at M[j sqM + a pm + c], c < r_q
  float2* B;            // element (a, J) of position j at B[j sqB + a nj + J]
  const int* row_exp;   // e_a, [rows]
  const float* col_scale;  // 2^-f_qJ, [position][nj_pad], zero for J >= nj
  const int* qmap;      // q of each sum position
  const int* rank;      // r_q by q
  unsigned* bmax;       // [rows]: bits of the largest |component| of the rows of B
  int64_t sqM, sqB;
  int pm, rows, nj, nj_pad, mt, nkb, npass;
  int64_t units;        // mt x positions
  int* err;
};

__device__ __forceinline__ float round_int(float x) { return rintf(x); }
__device__ __forceinline__ double round_int(double x) { return rint(x); }

// Three slices of v (|v| < 128): the integer s1 = rint(v) and the fp16 remainders
// s2 = fp16(v - s1), s3 = fp16(v - s1 - s2).
template <typename R>
__device__ __forceinline__ void slice3r(R v, __half& h1, __half& h2, __half& h3) {
  const R s1 = round_int(v);
  const R r1 = v - s1;
  h2 = __float2half_rn((float)r1);
  const R r2 = r1 - (R)__half2float(h2);
  h1 = __float2half_rn((float)s1);
  h3 = __float2half_rn((float)r2);
}

// slice3r of two values, packed by slice.
__device__ __forceinline__ void slice3_pair(float x, float y, uint32_t (&out)[3]) {
  const float sx = rint_small(x), sy = rint_small(y), rx = x - sx, ry = y - sy;
  const __half2 h2 = __floats2half2_rn(rx, ry);
  const float2 f2 = __half22float2(h2);
  out[0] = half2_bits(sx, sy);
  out[1] = *reinterpret_cast<const uint32_t*>(&h2);
  out[2] = half2_bits(rx - f2.x, ry - f2.y);
}

__device__ __forceinline__ uint32_t pack2(__half a, __half b) {
  const __half2 h = __halves2half2(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

__global__ void __launch_bounds__(MTHREADS, 1)
    mlgemm_tc_kernel(const __grid_constant__ CUtensorMap mB1, const __grid_constant__ CUtensorMap mB2,
                     const __grid_constant__ CUtensorMap mB3, MlArgs args) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  float* tileS = reinterpret_cast<float*>(smem + MSTAGES * MSTAGE_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + MSTAGES * MSTAGE_BYTES + kMlOut);
  uint64_t* full = bars;                 // [MSTAGES] slices of L landed, four producer warps done
  uint64_t* empty = bars + MSTAGES;      // [MSTAGES] read by the MMAs
  uint64_t* accf = bars + 2 * MSTAGES;   // pass accumulated
  uint64_t* drained = accf + 1;          // pass read out of TMEM
  uint64_t* done = drained + 1;          // settle
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* s_err = reinterpret_cast<volatile int*>(s_tmem + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = args.nkb, npass = args.npass;

  if (threadIdx.x == 0) {
    for (int s = 0; s < MSTAGES; ++s) {
      mbar_init(&full[s], 1 + 4);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accf, 1);
    mbar_init(drained, MEPI);
    mbar_init(done, 1);
    *s_err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                 "r"(kMlTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  // B' rows of pass p: 128, or 64 where at most 32 complex columns are left
  auto pass_n = [&](int p) { return args.nj_pad - p * (MPN / 2) > MPN / 4 ? MPN : MPN / 2; };

  int64_t fills = 0;  // stages filled so far (thread 0)
  if (warp == 0) {
    if (lane == 0) {
      const CUtensorMap* mb[MSL] = {&mB1, &mB2, &mB3};
      int64_t& it = fills;
      bool ok = true;
      for (int64_t u = blockIdx.x; u < args.units && ok; u += gridDim.x) {
        const int pos = (int)(u / args.mt);
        for (int p = 0; p < npass && ok; ++p) {
          const int boxes = pass_n(p) / 64, brow = pos * 2 * args.nj_pad + p * MPN;
          for (int kb = 0; kb < nkb; ++kb, ++it) {
            const int s = (int)(it % MSTAGES);
            if (!mbar_wait(&empty[s], (uint32_t)((it / MSTAGES) & 1) ^ 1, s_err, args.err, 11)) {
              ok = false;
              break;
            }
            uint8_t* st = smem + s * MSTAGE_BYTES + MSL * MA_BYTES;
            mbar_expect_tx(&full[s], MSL * boxes * MBOX);
            for (int i = 0; i < MSL; ++i)
              for (int b = 0; b < boxes; ++b)
                tma_load_2d(st + i * MB_BYTES + b * MBOX, mb[i], &full[s], kb * MBK, brow + b * 64);
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int64_t it = 0, ps = 0;
      bool ok = true;
      for (int64_t u = blockIdx.x; u < args.units && ok; u += gridDim.x)
        for (int p = 0; p < npass && ok; ++p, ++ps) {
          const uint32_t idesc = kIdescMl | ((uint32_t)(pass_n(p) >> 3) << 17);
          const uint32_t g0 = tmem_base, g1 = tmem_base + MPN, g2 = tmem_base + 2 * MPN;
          if (ps > 0 && !mbar_wait(drained, (uint32_t)((ps - 1) & 1), s_err, args.err, 14)) {
            ok = false;
            break;
          }
          tc_fence_after();
          for (int kb = 0; kb < nkb; ++kb, ++it) {
            const int s = (int)(it % MSTAGES);
            if (!mbar_wait(&full[s], (uint32_t)((it / MSTAGES) & 1), s_err, args.err, 12)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint8_t* st = smem + s * MSTAGE_BYTES;
            uint64_t dA[MSL], dB[MSL];
#pragma unroll
            for (int i = 0; i < MSL; ++i) {
              dA[i] = sdesc_k<MBK>(st + i * MA_BYTES);
              dB[i] = sdesc_k<MBK>(st + MSL * MA_BYTES + i * MB_BYTES);
            }
#pragma unroll
            for (int kk = 0; kk < MBK / 16; ++kk) {
              const uint64_t off = (uint64_t)(kk * 32) >> 4;
              const uint32_t acc = (kb == 0 && kk == 0) ? 0u : 1u;
              umma_f16(g0, dA[0] + off, dB[0] + off, idesc, acc);
              umma_f16(g1, dA[0] + off, dB[1] + off, idesc, acc);
              umma_f16(g1, dA[1] + off, dB[0] + off, idesc, 1u);
              umma_f16(g2, dA[0] + off, dB[2] + off, idesc, acc);
              umma_f16(g2, dA[1] + off, dB[1] + off, idesc, 1u);
              umma_f16(g2, dA[2] + off, dB[0] + off, idesc, 1u);
            }
            umma_commit(&empty[s]);
          }
          if (ok) umma_commit(accf);
        }
    }
  } else if (warp < 2 + 4 * MGROUPS) {
    // producers: group g takes the stages it = g, g + MGROUPS, ...; lanes 8 per row, two complex values
    // each, so that a warp's load covers four 128-byte runs of M and its store whole rows of the
    // swizzled layout.  A group's next block is in flight while the others' are cut.
    const int grp = (warp - 2) >> 2, t = ((warp - 2) & 3) * 32 + lane, l8 = t & 7, rr = t >> 3;
    const int per_unit = npass * nkb;
    // the unit the loads are in: its row of this thread, its rank, rows left
    int64_t lu = blockIdx.x;
    const float2* lm = nullptr;
    int lr = 0, lrows = 0, lrem = grp, lkb = 0;
    auto enter = [&]() {
      if (lu >= args.units) return;
      const int pos = (int)(lu / args.mt), ti = (int)(lu % args.mt);
      lr = __ldg(args.rank + __ldg(args.qmap + pos));
      lrows = args.rows - ti * BM;
      lm = args.M + (int64_t)pos * args.sqM + ((int64_t)ti * BM + rr) * args.pm + l8 * 2;
    };
    auto forward = [&]() {  // brings lrem below per_unit
      if (lrem >= per_unit) {
        do {
          lrem -= per_unit;
          lu += gridDim.x;
        } while (lrem >= per_unit);
        enter();
      }
      lkb = lrem % nkb;
    };
    float4 x[8];
    auto load = [&]() {
      const int col = lkb * (MBK / 2) + l8 * 2, rows = col < lr ? lrows : 0;
      const float2* m = lm + lkb * (MBK / 2);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i * 16 + rr < rows) {
          x[i] = __ldg(reinterpret_cast<const float4*>(m + (int64_t)i * 16 * args.pm));
          if (col + 1 >= lr) x[i].z = x[i].w = 0.f;  // beyond the rank: not written
        }
      }
    };
    float sc[8];
    int64_t it = grp, su = -1;
    enter();
    forward();
    if (lu < args.units) load();
    while (lu < args.units) {
      if (su != lu) {
        su = lu;
        const int a0 = (int)(lu % args.mt) * BM + rr;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int ex = a0 + i * 16 < args.rows ? __ldg(args.row_exp + a0 + i * 16) : 0;  // -121 .. 127
          sc[i] = __int_as_float((ex + 127) << 23);
        }
      }
      const int s = (int)(it % MSTAGES);
      if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], (uint32_t)((it / MSTAGES) & 1) ^ 1, s_err, args.err, 15))) break;
      uint8_t* st = smem + s * MSTAGE_BYTES;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int row = i * 16 + rr;
        uint32_t h[3], g[3];
        slice3_pair(x[i].x * sc[i], x[i].y * sc[i], h);
        slice3_pair(x[i].z * sc[i], x[i].w * sc[i], g);
        uint8_t* d = st + row * (MBK * 2) + (((l8 >> 1) ^ ((row >> 1) & 3)) << 4) + (l8 & 1) * 8;
#pragma unroll
        for (int k = 0; k < MSL; ++k) *reinterpret_cast<uint2*>(d + k * MA_BYTES) = make_uint2(h[k], g[k]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
      it += MGROUPS;
      lrem += MGROUPS;
      forward();
      if (lu < args.units) load();
    }
  } else {
    // epilogue: TMEM lane quarter warp % 4; the two warps of a quarter take half of the pass's columns
    // each.  Lane r is row a of M, TMEM column n is B' row n: complex column n / 2, part n % 2.
    const int q = warp & 3, half = (warp - 2 - 4 * MGROUPS) >> 2, r = q * 32 + lane;
    int64_t ps = 0;
    bool ok = true;
    for (int64_t u = blockIdx.x; u < args.units; u += gridDim.x) {
      const int pos = (int)(u / args.mt), ti = (int)(u % args.mt), a = ti * BM + r;
      const float rs = a < args.rows ? ldexpf(1.f, -args.row_exp[a]) : 0.f;
      float m = 0.f;
      for (int p = 0; p < npass; ++p, ++ps) {
        const int N = pass_n(p), n0 = half * (N / 2);
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(accf, (uint32_t)(ps & 1), s_err, args.err, 13));
        if (ok) {
          tc_fence_after();
          // 2^-f_qJ, zero for J >= nj
          const float* fcol = args.col_scale + (int64_t)pos * args.nj_pad + p * (MPN / 2);
#pragma unroll 1
          for (int cb = n0; cb < n0 + N / 2; cb += 8) {
            uint32_t v0[8], v1[8], v2[8];
            const uint32_t lo = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)cb;
            tmem_ld8(lo, v0);
            tmem_ld8(lo + MPN, v1);
            tmem_ld8(lo + 2 * MPN, v2);
            const float4 f = __ldg(reinterpret_cast<const float4*>(fcol + (cb >> 1)));
            const float fs[4] = {f.x, f.y, f.z, f.w};
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float x = __uint_as_float(v0[2 * j]) + (__uint_as_float(v1[2 * j]) + __uint_as_float(v2[2 * j]));
              const float y =
                  __uint_as_float(v0[2 * j + 1]) + (__uint_as_float(v1[2 * j + 1]) + __uint_as_float(v2[2 * j + 1]));
              const float2 z = make_float2(x * rs * fs[j], y * rs * fs[j]);
              m = fmaxf(m, fmaxf(fabsf(z.x), fabsf(z.y)));
              *reinterpret_cast<float2*>(tileS + r * kMlPitch + cb + 2 * j) = z;
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(drained);
        }
        // a warp whose wait expired keeps the barriers below company, without storing
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (ok) {
          const int lg = N == MPN ? 6 : 5, t = threadIdx.x - (MTHREADS - 256), Jl = t & ((1 << lg) - 1), rstep = 256 >> lg;
          if (p * (MPN / 2) + Jl < args.nj) {
            const float* src = tileS + (t >> lg) * kMlPitch + 2 * Jl;
            float2* out = args.B + (int64_t)pos * args.sqB + (int64_t)(ti * BM + (t >> lg)) * args.nj + p * (MPN / 2) + Jl;
            const int last = min(BM, args.rows - ti * BM);
#pragma unroll 8
            for (int ar = t >> lg; ar < last; ar += rstep) {
              *out = *reinterpret_cast<const float2*>(src);
              out += (int64_t)rstep * args.nj;
              src += rstep * kMlPitch;
            }
          }
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
      }
      if (ok && a < args.rows) {
        const unsigned bits = __float_as_uint(m);
        if (bits > args.bmax[a]) atomicMax(args.bmax + a, bits);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*s_err) settle(full, MSTAGES, fills, done);  // a wait expired: wait for what is in flight
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kMlTmem)
                 : "memory");
  }
}

// Row exponents from the bits of the rows' largest entries.
__global__ void row_exp_kernel(const unsigned* __restrict__ mx, int64_t rows, int* __restrict__ row_exp) {
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // at most 2^127, a float (rows below 2^-121 keep fewer digits of what is subnormal anyway)
  if (a < rows) row_exp[a] = min(slice_exp(__uint_as_float(mx[a])), 127);
}

// inv[j][I] = c where perm_q[c] = I, c < r_q (q = qmap[j]), else -1.
__global__ void inv_perm_kernel(const int* __restrict__ qmap, const int* __restrict__ perm, const int* __restrict__ rank,
                                int np, int16_t* __restrict__ inv) {
  const int j = blockIdx.x, q = qmap[j], r = rank[q];
  for (int I = threadIdx.x; I < np; I += blockDim.x) inv[(int64_t)j * np + I] = -1;
  __syncthreads();
  for (int c = threadIdx.x; c < r; c += blockDim.x) inv[(int64_t)j * np + perm[(int64_t)q * np + c]] = (int16_t)c;
}

// B' slices of w_q^{1/2} L^q for the positions of the sum: block (32 columns J, position), row = 2 J + part, is
// R_J = (Re L, -Im L) (part 0) or I_J = (Im L, Re L) (part 1) over the gathered rows perm_q(c) of column J,
// scaled by 2^f_qJ (largest component of the column in [64, 128)); columns J >= nj,
// c >= r_q and beyond 2 r_q are zero.  Layout [position][2 nj_pad][Kp] per slice; the inverse scales
// [position][nj_pad].  Rows of L are read along J and the slices written along c, through shared memory.
// A block takes CW values of c at a time.  Bound by the FP64 pipe (~40 operations per value at two a
// clock and SM, ~10 us per 32 x 32 values): where the blocks of 32 columns do not fill the SMs, the
// values of c are split over blockIdx.z too, each block finding the scales anew in integers
// (5 positions, rank ~70: 39 -> 13.5 us; 20 positions, rank ~100: 46 -> 32).
template <int CW>
__global__ void __launch_bounds__(256) lslice_kernel(const double2* __restrict__ L, const double* __restrict__ sw, int np,
                                                     const int* __restrict__ qmap, const int* __restrict__ perm,
                                                     const int* __restrict__ rank, int nj, int nj_pad, int Kp,
                                                     __half* __restrict__ S1, __half* __restrict__ S2,
                                                     __half* __restrict__ S3, float* __restrict__ col_scale) {
  const int j = blockIdx.y, q = qmap[j], J0 = blockIdx.x * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const double w = sw[q];
  const int r = rank[q], J = J0 + tx;
  const double2* Lq = L + (int64_t)q * np * np;
  const int* pq = perm + (int64_t)q * np;
  __shared__ unsigned long long sm[8][32];
  __shared__ uint32_t sd[3][32][CW + 1];
  constexpr unsigned long long kAbs = 0x7FFFFFFFFFFFFFFFULL, kInf = 0x7FF0000000000000ULL;
  unsigned long long mb = 0;  // bits of the largest |component| of the column, NaN left out
  if (J < nj)
    for (int c = ty; c < r; c += 8) {
      const double2 v = Lq[(int64_t)pq[c] * np + J];
      const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & kAbs;
      const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & kAbs;
      if (a <= kInf) mb = max(mb, a);
      if (b <= kInf) mb = max(mb, b);
    }
  sm[ty][tx] = mb;
  __syncthreads();
  for (int i = 0; i < 8; ++i) mb = max(mb, sm[i][tx]);
  const double m = __longlong_as_double((long long)mb) * w;  // w >= 0: the largest |component| w
  // within what a float's power of two holds
  const int ex = (m > 0.0 && isfinite(m)) ? max(-126, min(126, 6 - ilogb(m))) : 0;
  if (ty == 0 && blockIdx.z == 0) col_scale[(int64_t)j * nj_pad + J] = J < nj ? ldexpf(1.f, -ex) : 0.f;
  __half* const S[3] = {S1, S2, S3};
  for (int c0 = blockIdx.z * CW; c0 < Kp / 2; c0 += gridDim.z * CW) {
    __syncthreads();
    for (int cc = ty; cc < CW; cc += 8) {
      const int c = c0 + cc;
      double lr = 0.0, li = 0.0;
      if (J < nj && c < r) {
        const double2 v = Lq[(int64_t)pq[c] * np + J];
        lr = ldexp(v.x * w, ex);
        li = ldexp(v.y * w, ex);
      }
      __half a1, a2, a3, b1, b2, b3;
      slice3r<double>(lr, a1, a2, a3);
      slice3r<double>(li, b1, b2, b3);
      sd[0][tx][cc] = pack2(a1, b1);
      sd[1][tx][cc] = pack2(a2, b2);
      sd[2][tx][cc] = pack2(a3, b3);
    }
    __syncthreads();
    // row 2 Jl + part of the block, lanes along c
    for (int t = threadIdx.x; t < 64 * CW; t += 256) {
      const int e = t / CW, Jl = e >> 1, part = e & 1, cc = t % CW, c = c0 + cc;
      if (c >= Kp / 2) continue;
      const int64_t at = ((int64_t)j * 2 * nj_pad + 2 * (J0 + Jl) + part) * Kp + 2 * c;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const uint32_t x = sd[i][Jl][cc];
        // (re, -im) or (im, re); the slices of -x are those of x negated
        const uint32_t y = part ? (x >> 16) | (x << 16) : x ^ 0x80000000u;
        *reinterpret_cast<uint32_t*>(S[i] + at) = y;
      }
    }
  }
}

inline int64_t round_up(int64_t x, int64_t m) { return ((x + m - 1) / m) * m; }

}  // namespace tc

// ---- E = sum_q B^q B^q^H in the real symmetric form (host side)
void pair_orbits(int nf, std::vector<int2>& orb) {
  orb.clear();
  for (int p = 0; p < nf; ++p)
    for (int q = p + 1; q < nf; ++q) orb.push_back(make_int2(p, q));
  for (int p = 0; p < nf; ++p) orb.push_back(make_int2(p, p));
}

size_t syrk_tc_split_bytes(int64_t n2, int64_t kcols) {
  return (size_t)tc::NSLICE * n2 * tc::round_up(2 * kcols, tc::BK) * sizeof(__half) + 256;
}

// Lower-triangle tiles (ti >= tj) of the n2 x n2 E' in launch order, and their
// index by (ti, tj).  Every CTA streams the whole K extent of its row blocks and
// about one CTA per SM is resident, so the order decides what L2 can share:
// tiles go in bands of `band` row blocks, and within a band column by column,
// so that the ~150 CTAs of a wave read about band + 150/band row blocks instead
// of ~150.
void syrk_tc_tiles(int64_t n2, std::vector<int2>& tiles, std::vector<int>& tile_of, int band) {
  const int64_t kGroupA = band < 1 ? 1 : band;
  tiles.clear();
  const int64_t nt = (n2 + tc::BM - 1) / tc::BM;
  tile_of.assign(nt * nt, -1);
  for (int64_t t0 = 0; t0 < nt; t0 += kGroupA)
    for (int64_t tj = 0; tj < nt; ++tj)
      for (int64_t ti = t0; ti < std::min(nt, t0 + kGroupA); ++ti)
        if (ti >= tj) {
          tile_of[ti * nt + tj] = (int)tiles.size();
          tiles.push_back(make_int2((int)ti, (int)tj));
        }
}

size_t syrk_tc_ws_bytes(int64_t ntiles) { return (size_t)ntiles * tc::BN * tc::BM * 2 * sizeof(float); }

cudaError_t syrk_tc_rowscale(cudaStream_t st, const float2* B, int64_t sQ, int64_t sA, int64_t nJ, const int* qmap,
                             int nS, int64_t n2, int* row_exp) {
  tc::BView bv{B, sQ, sA, nJ, qmap};
  tc::rrow_scale_kernel<<<(unsigned)n2, 256, 0, st>>>(bv, (int64_t)nS * nJ, row_exp);
  count_launch();
  return cudaGetLastError();
}

namespace {
template <int BKt, int NST>
cudaError_t syrk_launch(cudaStream_t st, __half* const sl[tc::NSLICE], int64_t n2, int64_t K2, const int2* tiles_d,
                        int ntiles, void* ws, int accumulate, int* err) {
  using namespace tc;
  CUtensorMap m[NSLICE];
  for (int i = 0; i < NSLICE; ++i)
    if (!make_map(&m[i], sl[i], K2, n2, K2, BM, BKt)) return cudaErrorInvalidValue;
  const size_t smem = (size_t)NST * NSLICE * (BM + BN) * BKt * 2 + 1024 + 256;
  cudaError_t e = cudaFuncSetAttribute(syrk_tc_kernel<BKt, NST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  float* wh = reinterpret_cast<float*>(ws);
  float* wl = wh + (size_t)ntiles * BN * BM;
  TileArgs args{tiles_d, wh, wl, (int)(K2 / BKt), accumulate, err};
  syrk_tc_kernel<BKt, NST><<<ntiles, kSyrkThreads, smem, st>>>(m[0], m[1], args);
  count_launch();
  return cudaGetLastError();
}
}  // namespace

cudaError_t syrk_tc_chunk(cudaStream_t st, const float2* B, int64_t sQ, int64_t sA, int64_t nJ, const int* qmap,
                          int64_t n2, int j0, int nq, const int* row_exp, void* split, const int2* tiles_d, int ntiles,
                          void* ws, int accumulate, int* err, int cfg) {
  cudaError_t e = syrk_tc_split(st, B, sQ, sA, nJ, qmap, n2, j0, nq, row_exp, split, nullptr);
  if (e != cudaSuccess) return e;
  return syrk_tc_mma(st, split, n2, nq, nJ, tiles_d, ntiles, ws, accumulate, err, cfg);
}

cudaError_t syrk_tc_split(cudaStream_t st, const float2* B, int64_t sQ, int64_t sA, int64_t nJ, const int* qmap,
                          int64_t n2, int j0, int nq, const int* row_exp, void* split, double* corr) {
  using namespace tc;
  if (n2 <= 0 || nq <= 0) return cudaSuccess;
  if (n2 > 2147483647LL) return cudaErrorInvalidValue;
  const int64_t K2 = round_up(2 * (int64_t)nq * nJ, BK);
  __half* S1 = reinterpret_cast<__half*>(split);
  __half* S2 = S1 + (size_t)n2 * K2;
  BView bv{B, sQ, sA, nJ, qmap};
  rsplit_kernel<<<(unsigned)n2, 256, 0, st>>>(bv, j0, nq, K2, row_exp, S1, S2, corr);
  count_launch();
  return cudaGetLastError();
}

cudaError_t syrk_tc_mma(cudaStream_t st, void* split, int64_t n2, int nq, int64_t nJ, const int2* tiles_d,
                        int ntiles, void* ws, int accumulate, int* err, int cfg) {
  using namespace tc;
  if (n2 <= 0 || nq <= 0 || ntiles <= 0) return cudaSuccess;
  const int64_t K2 = round_up(2 * (int64_t)nq * nJ, BK);
  __half* S1 = reinterpret_cast<__half*>(split);
  __half* const sl[tc::NSLICE] = {S1, S1 + (size_t)n2 * K2};
  return cfg == 1 ? syrk_launch<32, 6>(st, sl, n2, K2, tiles_d, ntiles, ws, accumulate, err)
                  : syrk_launch<64, 3>(st, sl, n2, K2, tiles_d, ntiles, ws, accumulate, err);
}

// The test of gamma takes 13 us (one block) and saves an eighth of a finish of ~30 us at 33 orbitals,
// ~750 us on average over 23 to 120.
constexpr int kHermMin = 48;
constexpr int kEriBlocks = 152 * 16;  // fixed grid of the fused finish (reproducible traces)
size_t syrk_tc_eri_part_count() { return 2 * (size_t)kEriBlocks + 1; }  // partials, Hermitian flag

template <typename TO>
static cudaError_t finish_eri_impl(cudaStream_t st, const void* ws, int ntiles, const int* tile_of_d,
                                   const int2* orb, int nf, const int* row_exp, const double* corr, double scale,
                                   TO* eri, const double2* gamma, double2* part, double* out4) {
  using namespace tc;
  if (!eri && !gamma) return cudaSuccess;
  const float* wh = reinterpret_cast<const float*>(ws);
  const float* wl = wh + (size_t)ntiles * BN * BM;
  const int64_t n2 = (int64_t)nf * nf, nt = (n2 + BM - 1) / BM;
  const int tested = gamma && nf >= kHermMin;
  if (tested) {
    gamma_herm_kernel<<<1, 1024, 0, st>>>(gamma, nf, part + 2 * kEriBlocks);
    count_launch();
  }
  syrk_eri_kernel<TO><<<kEriBlocks, 256, 0, st>>>(wh, wl, tile_of_d, (int)nt, orb, nf, row_exp, corr, scale, eri,
                                                  gamma, part, tested);
  count_launch();
  if (gamma) {
    eri_traces_final_kernel<<<1, 256, 0, st>>>(part, kEriBlocks, out4);
    count_launch();
  }
  return cudaGetLastError();
}
cudaError_t syrk_tc_finish_eri(cudaStream_t st, const void* ws, int ntiles, const int* tile_of_d, const int2* orb,
                               int nf, const int* row_exp, const double* corr, double scale, float2* eri,
                               const double2* gamma, double2* part, double* out4) {
  return finish_eri_impl<float2>(st, ws, ntiles, tile_of_d, orb, nf, row_exp, corr, scale, eri, gamma, part, out4);
}
cudaError_t syrk_tc_finish_eri_z(cudaStream_t st, const void* ws, int ntiles, const int* tile_of_d, const int2* orb,
                                 int nf, const int* row_exp, const double* corr, double scale, double2* eri,
                                 const double2* gamma, double2* part, double* out4) {
  return finish_eri_impl<double2>(st, ws, ntiles, tile_of_d, orb, nf, row_exp, corr, scale, eri, gamma, part, out4);
}

cudaError_t row_exponents(cudaStream_t st, const unsigned* mx, int64_t rows, int* row_exp) {
  if (rows <= 0) return cudaSuccess;
  tc::row_exp_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(mx, rows, row_exp);
  count_launch();
  return cudaGetLastError();
}

// ---- B = M L on the tensor cores, three slices (host side)
int mlgemm_tc_kp(int rp) { return (int)tc::round_up(2 * (int64_t)rp, tc::BK); }
int mlgemm_tc_nj_pad(int nj) { return (int)tc::round_up(nj, tc::MBJ); }
bool mlgemm_tc_supported(int rp) { return rp > 0 && mlgemm_tc_kp(rp) <= tc::kMlMaxK; }
size_t mlgemm_tc_lslice_bytes(int nS, int rp, int nj) {
  return (size_t)tc::MSL * nS * (2 * mlgemm_tc_nj_pad(nj)) * mlgemm_tc_kp(rp) * sizeof(__half) + 256;
}

cudaError_t mlgemm_tc_prepare(cudaStream_t st, const double2* L, const double* sw, int np, const int* qmap, int nS,
                              const int* perm, const int* rank, int rp, int nj, void* lsl, float* col_scale, int16_t* inv) {
  using namespace tc;
  if (np > 32767) return cudaErrorInvalidValue;
  const int Kp = mlgemm_tc_kp(rp), njp = mlgemm_tc_nj_pad(nj);
  const size_t per = (size_t)nS * 2 * njp * Kp;
  __half* S1 = reinterpret_cast<__half*>(lsl);
  // below two blocks per SM the values of c are split over blocks too
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if ((int64_t)(njp / 32) * nS < 2 * sms)
    lslice_kernel<8><<<dim3(njp / 32, nS, (Kp / 2 + 7) / 8), 256, 0, st>>>(L, sw, np, qmap, perm, rank, nj, njp, Kp, S1,
                                                                           S1 + per, S1 + 2 * per, col_scale);
  else
    lslice_kernel<32><<<dim3(njp / 32, nS), 256, 0, st>>>(L, sw, np, qmap, perm, rank, nj, njp, Kp, S1, S1 + per,
                                                          S1 + 2 * per, col_scale);
  count_launch();
  inv_perm_kernel<<<nS, 128, 0, st>>>(qmap, perm, rank, np, inv);
  count_launch();
  return cudaGetLastError();
}

cudaError_t mlgemm_tc(cudaStream_t st, const float2* M, int pm, float2* B, const int* qmap, int nS, int64_t rows,
                      const int* rank, int rp, int nj, const int* row_exp, const void* lsl, const float* col_scale,
                      unsigned* bmax, int* err) {
  using namespace tc;
  if (rows <= 0 || nS <= 0) return cudaSuccess;
  if (!mlgemm_tc_supported(rp) || pm < rp || pm % 2 != 0 || rows > 2147483647LL - BM) return cudaErrorInvalidValue;
  const int Kp = mlgemm_tc_kp(rp), njp = mlgemm_tc_nj_pad(nj);
  const size_t pb = (size_t)nS * 2 * njp * Kp;
  const __half* L1 = reinterpret_cast<const __half*>(lsl);
  CUtensorMap mB[MSL];
  for (int i = 0; i < MSL; ++i)
    if (!make_map(&mB[i], L1 + i * pb, Kp, (int64_t)nS * 2 * njp, Kp, 64, MBK)) return cudaErrorInvalidValue;
  const size_t smem = (size_t)MSTAGES * MSTAGE_BYTES + kMlOut + 1024 + 256;
  cudaError_t e = cudaFuncSetAttribute(mlgemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  MlArgs a{};
  a.M = M;
  a.B = B;
  a.row_exp = row_exp;
  a.col_scale = col_scale;
  a.qmap = qmap;
  a.rank = rank;
  a.bmax = bmax;
  a.sqM = rows * pm;
  a.sqB = rows * nj;
  a.pm = pm;
  a.rows = (int)rows;
  a.nj = nj;
  a.nj_pad = njp;
  a.mt = (int)((rows + BM - 1) / BM);
  a.nkb = Kp / MBK;
  a.npass = (njp + MPN / 2 - 1) / (MPN / 2);
  a.units = (int64_t)a.mt * nS;
  a.err = err;
  mlgemm_tc_kernel<<<(unsigned)std::min<int64_t>(a.units, sms), MTHREADS, smem, st>>>(mB[0], mB[1], mB[2], a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace isdf
