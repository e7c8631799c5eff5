// FP64-accurate batched complex GEMM on the tensor cores (tcgen05):
//     C_b = alpha op(A_b) op(B_b),   op in {N, T, C, R}, complex128, row-major.
// It carries the complex128 products of the library but those that the mixed and FP64_TC paths keep as FMA
// chains (k_gemm.cu): the fit (Eqs. 3-5), the FP64
// Coulomb metric (Eq. 6), the FP64 fragment contractions (Eq. 19), exchange (Eq. 10),
// AO integrals (Eq. 9) and the polarisability (Eqs. 12-15).
//
// Why not FMA: this GPU's FP64 pipe runs 2 FMA per clock and SM (1.2 TFLOP/s over the
// chip), 1/64 of FP32, and conversions or additions in FP64 cost the same.  So nothing
// here touches it per element: slicing and the final sums are integer arithmetic.
//
// Error-free slicing (Ozaki, Ogita, Oishi & Rump, 2012).  Each row of op(A) and each
// column of op(B) is scaled by a power of two so that its largest component lies in
// [32, 64) and rounded once to a 63-bit integer F (v 2^56), whose signed base-256 digits
//     v = s_0 + s_1/2^8 + ... + s_7/2^56,   |s_0| <= 64, -128 <= s_i <= 127
// are stored as fp16 integers, real and imaginary parts in rows of their own.  A tile
// is 64 x 32 complex entries of C: the 128 rows [Re a; Im a] of 64 rows of op(A) times the 64
// columns [Re b, Im b] of 32 columns of op(B) give the four real products of the complex one,
// which are combined with their signs at the end, as integers.  The products S_a T_b with
// a + b <= 7 (36 of them) feed eight groups g = a + b of 64 FP32 accumulator columns: all 512
// TMEM columns.  Over a chunk of 144 k every partial sum is an integer of magnitude at most
// 144 * (2 * 64 * 128 + 6 * 128 * 128) < 2^24, so the FP32 accumulation is exact whatever its
// rounding; each chunk is drained into 64-bit integers (groups 0-3 and 4-7), exact up to
// K = 2^21, and rounded once to FP64 at the end.
//
// What is lost is the rounding of F (2^-62 of the row's largest entry; none for entries above 2^-9 of
// it) and the products with a + b >= 8: per term ~2^-60 max|a_i| max|b_j|, where an FP64 FMA chain
// loses up to 2^-53 of each partial sum.  So operands whose rows are graded lose nothing either until
// max|a_i| max|b_j| exceeds the sums by 2^7 or so.  Base-128 digits (chunks of 384 k, 2^-56) were below
// the chain's error for most products, but not where the order of k grades both operands:
// there the caller gives powers of two for the contraction index (ZOpt::kexp), column k of op(A) times
// 2^-d_k and row k of op(B) times 2^d_k, which is exact.  Largest error over the largest entry,
// against 80-bit sums (26 AOs, 8 k-points, 12^3 grid, n_p = 150, rank 119), FMA chain / base 128 / this:
//   G 4.4e-16 / 1.1e-16 / 9e-17,  xi = W eta 1.1e-12 / 3.8e-13 / 2.1e-14,  V_xi 5.0e-15 / 2.6e-15 / 2.2e-16,
//   B = M L 1.6e-15 / 1.8e-15 / 1e-16,  E = B B^H 1.7e-15 / 1.9e-16 / 4e-17,
//   L = W^T L_xi 1.9e-16 / 1.5e-14 / 1.4e-15, with kexp 5e-17.
//
// The tile shape: an MMA of 128 x N x 16 takes N/2 clocks from N = 128 on, but 55 at N = 64
// and 49 at N = 32 (measured), so N = 64 costs 36 x 55 clocks per 16 k (58 % of the peak).
// N = 128 would need the accumulators of two passes, whose 64-bit sums (16 bytes per entry)
// would fill the register file.
//
// Seven slices (K <= 64): the form in which the mixed and FP64_TC paths have their g and T, with
// ~2^-48 of the rows' largest entries; digits and sums are those of that form bit for bit, on
// the same kernel.
//
// A row (column) with an infinity or NaN gives NaN in its whole row (column) of C.
//
// Layout of the slices.  The slicing kernels write them in the exact order in which the
// GEMM wants them in shared memory, so that a stage is fetched by bulk copies without a
// tensor map: [batch][32-row block][16-k block][slice][re, im][8-row group][k half][row % 8]
// [k % 8], i.e. K-major core matrices of 8 rows x 16 bytes (no swizzle), 16 KB per (row block,
// k block).  One layout serves both sides, so a product of a matrix with itself is sliced
// once.  Rows beyond the matrix are left unwritten: they only reach entries of C that are
// not stored.  k beyond K is zero.
//
// The drain of groups 0-3 runs while the MMAs of groups 4-7 of the chunk's last k block do, and that of
// groups 4-7 under those of groups 0-3 of the next chunk: two pairs of barriers (K <= 32 and seven slices: one
// chunk and one drain, where a second wait per tile cost 4 to 11 % of the kernel).  With the chunks of
// 384 k of base-128 digits and one drain per chunk, 320 x 320 x K in a batch of 200 took 671 us at K = 64,
// 1149 at 128, 2055 at 256 and 2955 at 384; it takes 649, 1078, 2064 and 3041.
//
// Kernel roles (576 threads, one CTA per SM, persistent over the tiles): warp 0 copies,
// warp 1 allocates TMEM and issues the MMAs, warps 2-17 drain and store.  Every wait is
// bounded.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace isdf {

namespace ztc {

using namespace tc;

constexpr int RB = 32;                       // rows per block of the slices
constexpr int BM = 64, BN = 32, BK = 16;     // tile rows, columns, k per stage (complex)
constexpr int kSlice = 2 * RB * BK;          // fp16 of one slice of a block: re rows, im rows (2 KB)
// of one (row block, k block) for NS slices: 16 KB at eight
template <int NS>
struct Blk {
  static constexpr int kElems = NS * kSlice;
  static constexpr int kBytesA = 2 * kElems * 2;      // two row blocks
  static constexpr int kBytesB = kElems * 2;
  static constexpr int kStage = kBytesA + kBytesB;    // 48 KB at eight slices
};
constexpr int NST = 3;                       // stages
constexpr int kChunk = 9;                    // k blocks per exact chunk (144 k)
constexpr int kShortK = 32;                  // K up to which every group stays below 2^22 (32 * 114688)
constexpr int kOutBytes = 65536;             // exchange of the partial sums, then the tile of C on its way out
constexpr int NT = 576;
constexpr int kDrainWarps = 16;
constexpr int kDrainCols = 16;               // accumulator columns per drain warp
constexpr int kTmem = 512;                   // 8 groups x 64 columns
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)((2 * BN) >> 3) << 17) | ((uint32_t)((2 * BM) >> 4) << 24);
constexpr int kBadExp = INT_MIN;            // row or column with a non-finite entry

// K-major descriptor of 8 x 16-byte core matrices: the two core matrices of a 16-k row
// are 128 bytes apart, 8-row groups 256 bytes.
__device__ __forceinline__ uint64_t sdesc_core(uint32_t a) {
  return (uint64_t)((a & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) |
         ((uint64_t)1 << 46);
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

struct Args {
  const __half *SA, *SB;    // slices
  const int *eA, *eB;       // exponents [batch][rows]
  double2* C;
  int64_t ldc, sC;
  double alpha;
  int scale;                // alpha != 1 (the FP64 pipe is kept out of the loop)
  int m, n, nkb;            // nkb: 16-k blocks
  int mt, nt, mb, nb;       // tiles of 64 rows and 32 columns; 32-row blocks per batch entry of A and B
  int64_t ntiles;
  int lower;                // op(A) lower triangular: k < m0 + 64 only
  const int* qmap;          // batch entry -> matrix (or NULL)
  const int32_t* krank;     // by matrix: op(A) is zero from row and column krank on (or NULL)
  int neg_ri, neg_ir, neg_ii;  // signs of re x im, im x re, im x im
  int* err;
};

__device__ __noinline__ double scale_slow(unsigned long long T, int e) { return ldexp((double)T, e); }

// +-(hi 2^-24 + lo 2^-56) (exact integers), times 2^e, rounded to FP64 in integer arithmetic.
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, bool flip, int e) {
  long long H = hi + (lo >> 32);
  uint32_t l = (uint32_t)lo;  // value = (H 2^32 + l) 2^-56
  const bool neg = H < 0;
  if (neg) {
    H = (l == 0) ? -H : -H - 1;
    l = 0u - l;
  }
  unsigned long long T;
  int top;  // exponent of T's leading bit
  if (H != 0) {
    const int z = __clzll(H);
    // the leading bits of H:l in 64 bits (z >= 1 as H > 0)
    T = ((unsigned long long)H << z) | (((unsigned long long)l << 32) >> (64 - z));
    top = 63 - z + 32 - 56 + e;
  } else if (l != 0) {
    const int z = __clzll((long long)l);
    T = (unsigned long long)l << z;
    top = 63 - z - 56 + e;
  } else {
    return 0.0;
  }
  const unsigned long long r = (T >> 11) + ((T >> 10) & 1);  // 53 bits, rounded; bit 52 adds to the exponent
  const int be = 1022 + top;
  unsigned long long v = r + ((unsigned long long)(unsigned)be << 52);
  if ((unsigned)be >= 2045u) v = (unsigned long long)__double_as_longlong(scale_slow(T, top - 63));  // subnormal, overflow
  if (neg != flip) v |= 1ULL << 63;
  return __longlong_as_double((long long)v);
}

// T rounded to `keep` leading bits, half to even (its low bits zero).
__device__ __forceinline__ unsigned long long round_even(unsigned long long T, int drop) {
  if (drop <= 0) return T;
  const unsigned long long r = T >> drop, rem = T & ((1ULL << drop) - 1), half = 1ULL << (drop - 1);
  return (r + (rem > half || (rem == half && (r & 1)))) << drop;
}

__device__ __noinline__ double seven_slow(long long T1, int v0, int e) {
  // the magnitudes at which a sum of 64-bit integers could wrap, or an exponent range end
  return ldexp(fma((double)v0, 4398046511104.0, (double)T1), e - 42);
}

// The seven-slice form: groups g = 0..6 of weight 2^{-7 g} summed in FP64 from the smallest to the
// largest, acc = fma(v_g, 2^{-7 g}, acc).  The sum is exact up to group 2, so that it is
// T1 = sum_{g>=1} v_g 2^{7 (6 - g)} rounded to 53 bits, plus v0 2^42, rounded to 53 bits; times
// 2^(e - 42).
__device__ __forceinline__ double seven_to_double(long long T1, int v0, bool flip, int e) {
  unsigned long long m = (unsigned long long)(T1 < 0 ? -T1 : T1);
  if (m >> 53) {
    m = round_even(m, 64 - __clzll((long long)m) - 53);
    T1 = T1 < 0 ? -(long long)m : (long long)m;
  }
  unsigned long long v;
  const bool wide = v0 >= (1 << 20) || v0 <= -(1 << 20);
  const long long X = T1 + (long long)((unsigned long long)(long long)v0 << 42);
  m = (unsigned long long)(X < 0 ? -X : X);
  if (m == 0 && !wide) return 0.0;
  const int z = __clzll((long long)m);
  const unsigned long long T = m << z;
  unsigned long long r = T >> 11;
  const unsigned rem = (unsigned)T & 0x7FFu;
  r += (rem + 0x3FFu + ((unsigned)r & 1u)) >> 11;
  const int be = 1022 + 63 - z + e - 42;
  v = r + ((unsigned long long)(unsigned)be << 52);
  if (X < 0) v |= 1ULL << 63;
  if (wide || (unsigned)be >= 2045u) v = (unsigned long long)__double_as_longlong(seven_slow(T1, v0, e));
  if (flip) v ^= 1ULL << 63;
  return __longlong_as_double((long long)v);
}

// NS = 8: the exact sum of the groups, rounded once.  NS = 7: see seven_to_double.
template <int NS, bool kShort>
__global__ void __launch_bounds__(NT, 1) zgemm_tc_kernel(Args args) {
  constexpr int kBlk = Blk<NS>::kElems, kABytes = Blk<NS>::kBytesA, kStage = Blk<NS>::kStage;
  constexpr int kHalves = kShort ? 1 : 2;  // parts of a drain: all groups, or groups 0-3 and 4-7
  constexpr int kGrp = kShort ? NS : 4;    // groups of a part
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* outS = smem + NST * kStage;
  uint64_t* bars = reinterpret_cast<uint64_t*>(outS + kOutBytes);
  uint64_t* full = bars;             // [NST] stage landed
  uint64_t* empty = bars + NST;      // [NST] stage read by the MMAs
  uint64_t* accf = bars + 2 * NST;   // [2] chunk accumulated: groups 0-3, the others
  uint64_t* drained = accf + 2;      // [2] and drained
  uint64_t* done = drained + 2;      // settle
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* s_err = reinterpret_cast<volatile int*>(s_tmem + 1);
  volatile int64_t* s_fills = reinterpret_cast<volatile int64_t*>(s_tmem + 2);  // stages filled by thread 0
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&accf[i], 1);
      mbar_init(&drained[i], kDrainWarps);
    }
    mbar_init(done, 1);
    *s_err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                 "r"(kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  const int64_t per_batch = (int64_t)args.mt * args.nt;
  // the column tiles of one row block are adjacent, so the CTAs of a wave share it through L2
  auto tile_of = [&](int64_t t, int& b, int& ti, int& tj) {
    b = (int)(t / per_batch);
    const int rem = (int)(t % per_batch);
    ti = rem / args.nt;
    tj = rem % args.nt;
  };
  auto kblocks = [&](int b, int ti) {
    int nk = args.lower ? min(args.nkb, (ti + 1) * (BM / BK)) : args.nkb;
    if (args.krank) {
      const int r = args.krank[args.qmap ? args.qmap[b] : b];
      nk = r > ti * BM ? min(nk, (r + BK - 1) / BK) : 0;
    }
    return nk;
  };

  if (warp == 0) {
    if (lane == 0) {
      int64_t it = 0;  // stages filled so far
      bool ok = true;
      for (int64_t t = blockIdx.x; t < args.ntiles && ok; t += gridDim.x) {
        int b, ti, tj;
        tile_of(t, b, ti, tj);
        const int nk = kblocks(b, ti);
        const __half* a0 = args.SA + ((int64_t)b * args.mb + 2 * ti) * args.nkb * kBlk;
        // the second row block of the last tile may not exist: its rows are not stored
        const __half* a1 = (2 * ti + 1 < args.mb) ? a0 + (int64_t)args.nkb * kBlk : a0;
        const __half* bb = args.SB + ((int64_t)b * args.nb + tj) * args.nkb * kBlk;
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = (int)(it % NST);
          if (!mbar_wait(&empty[s], (uint32_t)((it / NST) & 1) ^ 1, s_err, args.err, 41)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + s * kStage;
          mbar_expect_tx(&full[s], kStage);
          bulk_load(st + kABytes, bb + (int64_t)kb * kBlk, Blk<NS>::kBytesB, &full[s]);
          // per slice the two row blocks of A side by side
#pragma unroll
          for (int i = 0; i < NS; ++i) {
            bulk_load(st + (2 * i) * kSlice * 2, a0 + (int64_t)kb * kBlk + i * kSlice, kSlice * 2, &full[s]);
            bulk_load(st + (2 * i + 1) * kSlice * 2, a1 + (int64_t)kb * kBlk + i * kSlice, kSlice * 2, &full[s]);
          }
        }
      }
      *s_fills = it;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int64_t it = 0, ch = 0;  // stages and chunks so far
      bool ok = true;
      for (int64_t t = blockIdx.x; t < args.ntiles && ok; t += gridDim.x) {
        int b, ti, tj;
        tile_of(t, b, ti, tj);
        const int nk = kblocks(b, ti);
        for (int kb = 0; kb < nk && ok; ++kb, ++it) {
          const bool first = (kb % kChunk) == 0, last = (kb % kChunk) == kChunk - 1 || kb == nk - 1;
          const int s = (int)(it % NST);
          if (!mbar_wait(&full[s], (uint32_t)((it / NST) & 1), s_err, args.err, 43)) {
            ok = false;
            break;
          }
          const uint32_t st = smem_u32(smem + s * kStage);
          const uint64_t dA = sdesc_core(st), dB = sdesc_core(st + kABytes);
          constexpr uint64_t oA = (2 * kSlice * 2) >> 4, oB = (kSlice * 2) >> 4;  // slice strides of the descriptors
#pragma unroll
          for (int gh = 0; gh < kHalves; ++gh) {
            if (first && ch > 0 && !mbar_wait(&drained[gh], (uint32_t)((ch - 1) & 1), s_err, args.err, 42)) {
              ok = false;
              break;
            }
            tc_fence_after();
#pragma unroll
            for (int i = 0; i < NS; ++i)
#pragma unroll
              for (int c = 0; c < NS - i; ++c)
                if (kShort || (i + c >= 4) == (gh == 1))
                  umma_f16(tmem + (uint32_t)((i + c) * 2 * BN), dA + i * oA, dB + c * oB, kIdesc,
                           (first && i == 0) ? 0u : 1u);
            if (last) umma_commit(&accf[gh]);
          }
          if (!ok) break;
          umma_commit(&empty[s]);
          if (last) ++ch;
        }
      }
    }
  } else {
    // drain: TMEM lane quarter q = warp % 4 (a hardware rule): row block q / 2, Re a (q even) or
    // Im a (q odd); 16 columns: half 0 (Re b) or 1 (Im b) of the 64, sub-block 0 or 1 of the half
    constexpr int kKeep = kDrainCols / 2;
    const int q = warp & 3, cblk = (warp - 2) >> 2, half = cblk >> 1, sub = cblk & 1, odd = q & 1;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cblk * kDrainCols);
    const int part = odd ^ half;  // what this warp's products go to: Re c or Im c
    // signs of this warp's products and of its partner's
    const bool neg = odd ? (half ? args.neg_ii : args.neg_ir) : (half ? args.neg_ri : 0);
    const bool pneg = odd ? (half ? 0 : args.neg_ri) : (half ? args.neg_ir : args.neg_ii);
    const long long pm = (neg != pneg) ? -1LL : 0LL;
    // the two warps of a part exchange half of their columns: even q keeps the first eight, odd q
    // the others.  Registers 0-7 hold the kept ones.
    const uint32_t keep = (uint32_t)(odd * kKeep);
    ulonglong2* xmine = reinterpret_cast<ulonglong2*>(outS) + (size_t)(q + 4 * cblk) * kKeep * 32 + lane;
    const ulonglong2* xother =
        reinterpret_cast<const ulonglong2*>(outS) + (size_t)((q ^ 1) + 4 * (cblk ^ 2)) * kKeep * 32 + lane;
    const int row = (q >> 1) * 32 + lane, col0 = sub * kDrainCols + odd * kKeep;
    double* out = reinterpret_cast<double*>(outS);
    int64_t ch = 0;
    bool ok = true;
    for (int64_t t = blockIdx.x; t < args.ntiles; t += gridDim.x) {
      int b, ti, tj;
      tile_of(t, b, ti, tj);
      const int nch = (kblocks(b, ti) + kChunk - 1) / kChunk;
      long long hi[kDrainCols], lo[kDrainCols];
#pragma unroll
      for (int j = 0; j < kDrainCols; ++j) hi[j] = lo[j] = 0;
      for (int c = 0; c < nch && ok; ++c, ++ch) {
#pragma unroll
        for (int gh = 0; gh < kHalves; ++gh) {
          if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&accf[gh], (uint32_t)(ch & 1), s_err, args.err, 44));
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int cb = 0; cb < kDrainCols / 4; ++cb) {
            uint32_t v[kGrp][4];
#pragma unroll
            for (int g = 0; g < kGrp; ++g)
              tmem_ld4(tbase + (uint32_t)((gh * 4 + g) * 2 * BN) + ((uint32_t)(cb * 4) ^ keep), v[g]);
            tmem_wait_ld();
            if (cb == kDrainCols / 4 - 1) {  // the last read: the MMAs may go on
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&drained[gh]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              int w[kGrp];
#pragma unroll
              for (int g = 0; g < kGrp; ++g) {
                const float f = __uint_as_float(v[g][j]);
                // exact integers; below 2^22 the addition of 1.5 2^23 puts them into the low bits
                w[g] = kShort ? __float_as_int(f + 12582912.f) - 0x4B400000 : __float2int_rn(f);
              }
              long long &h = hi[cb * 4 + j], &l = lo[cb * 4 + j];
              if constexpr (NS == 7) {
                // groups 1-6 below 2^22 (64 * 36864): weights 2^35 .. 1 in hi; group 0 apart
                const int a0 = w[1] * 128 + w[2], a1 = w[3] * 128 + w[4], a2 = w[5] * 128 + w[6];
                h += (long long)a0 * (1 << 28) + (long long)a1 * (1 << 14) + a2;
                l += w[0];
              } else {
                // |w_0| <= 144 * 2^12 and |w_2| <= 144 * 2^15: 256 w_g + w_(g+1) fits 32 bits
                constexpr int o = kShort ? 4 : 0;  // group 4 among the part's
                if (gh == 0) h += (long long)(w[0] * 256 + w[1]) * 65536 + (w[2] * 256 + w[3]);
                if (kShort || gh == 1)
                  l += (long long)w[o] * (1 << 24) + (long long)w[o + 1] * 65536 + ((long long)w[o + 2] * 256 + w[o + 3]);
              }
            }
          }
        }
        if (!ok) break;
      }
      // a warp whose wait expired keeps the barriers below company, without storing
      const int r = ti * BM + row, n0 = tj * BN;
      const int ea = r < args.m ? args.eA[(int64_t)b * args.m + r] : 0;
      const int* eb = args.eB + (int64_t)b * args.n;
#pragma unroll
      for (int j = 0; j < kKeep; ++j) {
        xmine[j * 32] = make_ulonglong2((unsigned long long)hi[kKeep + j], (unsigned long long)lo[kKeep + j]);
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
      double x[kKeep];
#pragma unroll
      for (int j = 0; j < kKeep; ++j) {
        const ulonglong2 o = xother[j * 32];
        const int n = n0 + col0 + j;
        const int eb1 = n < args.n ? __ldg(eb + n) : 0;
        // own +- the partner's, negated as a whole if the own sign is
        const long long h = hi[j] + (((long long)o.x ^ pm) - pm), l = lo[j] + (((long long)o.y ^ pm) - pm);
        x[j] = NS == 7 ? seven_to_double(h, (int)l, neg, -(ea + eb1)) : fixed_to_double(h, l, neg, -(ea + eb1));
        if (ea == kBadExp || eb1 == kBadExp) x[j] = __longlong_as_double(0x7FF8000000000000LL);
        if (args.scale) x[j] *= args.alpha;
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
      // staged with the columns rotated by the row, so that lanes (rows) hit different banks
#pragma unroll
      for (int j = 0; j < kKeep; ++j) out[(row * BN + ((col0 + j) ^ lane)) * 2 + part] = x[j];
      asm volatile("bar.sync 1, 512;" ::: "memory");
      if (ok) {
        double2* C = args.C + (int64_t)(args.qmap ? args.qmap[b] : b) * args.sC;
        const int wv = warp - 2, n = n0 + lane;
        const double2* o2 = reinterpret_cast<const double2*>(outS);
#pragma unroll 4
        for (int i = 0; i < BM / kDrainWarps; ++i) {
          const int rr = wv * (BM / kDrainWarps) + i, gr = ti * BM + rr;
          if (gr < args.m && n < args.n) C[(int64_t)gr * args.ldc + n] = o2[rr * BN + (lane ^ (rr & 31))];
        }
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*s_err) settle(full, NST, *s_fills, done);  // a wait expired: wait for what is in flight
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmem) : "memory");
  }
}

// ---------------------------------------------------------------- slicing
// Exponent ex with max 2^ex in [32, 64) (NS = 8) or [64, 128) (NS = 7) from the bits of the largest magnitude.
template <int NS>
__device__ __forceinline__ int exp_of(unsigned long long mx) {
  constexpr int kTop = NS == 8 ? 5 : 6;
  if (mx == 0) return 0;
  // the sign of a NaN may have come through: the compiler may clear sign bits by abs.f64, which keeps it
  const int f = (int)(mx >> 52) & 0x7FF;
  if (f == 0x7FF) return kBadExp;
  return f ? kTop - (f - 1023) : kTop - (63 - __clzll((long long)mx) - 1074);
}

// The 63-bit integer rint(x 2^(ex + 56)) plus 128 at each of the lower seven digits, so that
// digit i is bits [8 (7 - i), +8) minus 128 (i >= 1) and s_0 the bits from 56 on.
__device__ __forceinline__ long long digits_of(double x, int ex) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int f = (int)((u >> 52) & 0x7FF);
  unsigned long long m = u & 0xFFFFFFFFFFFFFULL;
  if (f) m |= 1ULL << 52;
  const int s = (f ? f : 1) - 1019 + ex;  // <= 9 for normal rows
  unsigned long long F;
  if (s >= 0)
    F = m << s;
  else
    F = s > -55 ? (m + (1ULL << (-s - 1))) >> -s : 0ULL;
  long long v = (long long)u < 0 ? -(long long)F : (long long)F;
  return v + 0x0080808080808080LL;
}

// Slices of eight consecutive k of one row, part re or im of the chunk at dst (16 bytes per slice).
// Digits as fp16 pairs: 1024 + u has the bits 0x6400 | u (u < 1024), minus 1024 + 128.
__device__ __forceinline__ void store_planes(const long long (&F)[8], int part, __half* dst) {
  constexpr int NS = 8;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (s == 0) {
        const __half2 h = __floats2half2_rn((float)(int)(F[2 * i] >> 56), (float)(int)(F[2 * i + 1] >> 56));
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
      } else {
        const uint32_t u0 = (uint32_t)(F[2 * i] >> (8 * (NS - 1 - s))) & 255u;
        const uint32_t u1 = (uint32_t)(F[2 * i + 1] >> (8 * (NS - 1 - s))) & 255u;
        const uint32_t p = 0x64006400u | u0 | (u1 << 16);
        const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&p), __floats2half2_rn(1152.f, 1152.f));
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
      }
    }
    *reinterpret_cast<uint4*>(dst + s * kSlice + part * (RB * BK)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// The seven-slice form takes the digits one after the other, each the nearest integer (half to
// even) of what is left: |s_i| <= 64.  x 2^ex as a 62-bit integer (v 2^55), a last bit that
// stands for anything below it.
__device__ __forceinline__ long long digits7_of(double x, int ex) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int f = (int)((u >> 52) & 0x7FF);
  unsigned long long m = u & 0xFFFFFFFFFFFFFULL;
  if (f) m |= 1ULL << 52;
  const int s = (f ? f : 1) - 1020 + ex;  // <= 9 for normal rows
  unsigned long long F;
  if (s >= 0)
    F = m << s;
  else if (s > -63)
    F = (m >> -s) | ((m & ((1ULL << -s) - 1)) != 0);
  else
    F = m != 0;
  return (long long)u < 0 ? -(long long)F : (long long)F;
}

__device__ __forceinline__ void store_planes7(long long (&F)[8], int part, __half* dst) {
#pragma unroll
  for (int s = 0; s < 7; ++s) {
    const int pos = 55 - 7 * s;
    const long long half = 1LL << (pos - 1);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const long long t = F[i] + half;
      long long q = t >> pos;
      if ((t & ((1LL << pos) - 1)) == 0) q &= ~1LL;  // a tie: to even
      F[i] -= q << pos;
      const uint32_t h = 0x6400u | ((uint32_t)((int)q + 128) & 1023u);
      if (i & 1)
        w[i >> 1] |= h << 16;
      else
        w[i >> 1] = h;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w[i]), __floats2half2_rn(1152.f, 1152.f));
      w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(dst + s * kSlice + part * (RB * BK)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

template <int NS>
__device__ __forceinline__ void emit_chunk(const double2 (&x)[8], int ex, __half* dst) {
  long long F[8];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const double v = p ? x[i].y : x[i].x;
      F[i] = NS == 7 ? digits7_of(v, ex) : digits_of(v, ex);
    }
    if constexpr (NS == 7)
      store_planes7(F, p, dst);
    else
      store_planes(F, p, dst);
  }
}

__device__ __forceinline__ unsigned long long amax_bits(double2 v) {
  constexpr long long kAbs = 0x7FFFFFFFFFFFFFFFLL;
  const unsigned long long a = (unsigned long long)(__double_as_longlong(v.x) & kAbs);
  const unsigned long long b = (unsigned long long)(__double_as_longlong(v.y) & kAbs);
  return a > b ? a : b;
}

// Powers of two by k: entry k times 2^(sgn d[k]) (exact; |d| <= kMaxKexp).
struct KScale {
  const int32_t* d;
  int64_t stride;  // by matrix
  int sgn;
  template <bool kOn>
  __device__ __forceinline__ double2 of(double2 v, int k) const {
    if constexpr (!kOn) return v;
    const double f = __longlong_as_double((long long)(1023 + sgn * __ldg(d + k)) << 52);
    return make_double2(v.x * f, v.y * f);
  }
};

// Where chunk kc (eight k) of row r goes.
template <int NS>
__device__ __forceinline__ int64_t slot_of(int r, int kc, int nkb) {
  return ((int64_t)(r / RB) * nkb + (kc >> 1)) * Blk<NS>::kElems + ((r % RB) >> 3) * (2 * 64) + (kc & 1) * 64 + (r & 7) * 8;
}

// Rows stored contiguously along k: a block takes eight rows, one warp per row for the
// largest entry, then eight lanes per 128-byte line of the slices.
template <int NS, bool kOn>
__global__ void __launch_bounds__(256) zslice_rows_kernel(const double2* __restrict__ X, int64_t ld, int64_t sX, int rows,
                                                          int K, int nkb, int nblk, const int* __restrict__ qmap,
                                                          KScale ks, __half* __restrict__ S, int* __restrict__ ex) {
  const int b = blockIdx.y, r0 = blockIdx.x * 8, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qb = qmap ? qmap[b] : b;
  X += (int64_t)qb * sX;
  if constexpr (kOn) ks.d += (int64_t)qb * ks.stride;
  S += (int64_t)b * nblk * nkb * Blk<NS>::kElems;
  __shared__ int se[8];
  {
    const int r = r0 + warp;
    unsigned long long m = 0;
    if (r < rows)
      for (int k = lane; k < K; k += 32) m = max(m, amax_bits(ks.of<kOn>(X[(int64_t)r * ld + k], k)));
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
      const int e = exp_of<NS>(m);
      se[warp] = e;
      if (r < rows) ex[(int64_t)b * rows + r] = e;
    }
  }
  __syncthreads();
  const int r = r0 + (threadIdx.x & 7);
  if (r >= rows) return;
  const int e = se[threadIdx.x & 7];
  const double2* row = X + (int64_t)r * ld;
  for (int kc = threadIdx.x >> 3; kc < nkb * 2; kc += 32) {
    double2 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = (kc * 8 + i < K && e != kBadExp) ? ks.of<kOn>(row[kc * 8 + i], kc * 8 + i) : make_double2(0.0, 0.0);
    emit_chunk<NS>(x, e, S + slot_of<NS>(r, kc, nkb));
  }
}

// Rows stored with stride ld along k (columns of the array), optionally gathered
// (k -> idx[k], none where negative): a block takes 32 rows, lanes along them.
template <int NS, bool kOn>
__global__ void __launch_bounds__(256) zslice_cols_kernel(const double2* __restrict__ X, int64_t ld, int64_t sX, int rows,
                                                          int K, int nkb, int nblk, const int32_t* __restrict__ idx,
                                                          int64_t sIdx, const int* __restrict__ qmap, KScale ks,
                                                          __half* __restrict__ S, int* __restrict__ ex) {
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = blockIdx.x * 32 + lane;
  const int qb = qmap ? qmap[b] : b;
  X += (int64_t)qb * sX + r;
  S += (int64_t)b * nblk * nkb * Blk<NS>::kElems;
  if (idx) idx += (int64_t)qb * sIdx;
  if constexpr (kOn) ks.d += (int64_t)qb * ks.stride;
  const bool in = r < rows;
  auto at = [&](int k) {
    const int kk = idx ? __ldg(idx + k) : k;
    return (in && kk >= 0) ? ks.of<kOn>(X[(int64_t)kk * ld], k) : make_double2(0.0, 0.0);
  };
  __shared__ unsigned long long sm[8][32];
  unsigned long long m = 0;
#pragma unroll 4
  for (int k = warp; k < K; k += 8) m = max(m, amax_bits(at(k)));
  sm[warp][lane] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) m = max(m, sm[w][lane]);
  const int e = exp_of<NS>(m);
  if (!in) return;
  if (warp == 0) ex[(int64_t)b * rows + r] = e;
  for (int kc = warp; kc < nkb * 2; kc += 8) {
    double2 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = (kc * 8 + i < K && e != kBadExp) ? at(kc * 8 + i) : make_double2(0.0, 0.0);
    emit_chunk<NS>(x, e, S + slot_of<NS>(r, kc, nkb));
  }
}

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
inline size_t slice_bytes(int slices, int rows, int k, int nb) {
  return (size_t)nb * cdiv(rows, RB) * cdiv(k, BK) * slices * kSlice * 2;
}

// Slices of op(X) by rows (side A) or of op(X)^T (side B): `cols` when the wanted rows run
// along the fast index of the array.
template <int NS, bool kOn>
void slice_launch(cudaStream_t st, bool cols, const double2* X, int64_t ld, int64_t sX, int rows, int K, int batch,
                  const int32_t* idx, int64_t sIdx, const int* qmap, const KScale& ks, __half* S, int* ex) {
  const int nkb = (int)cdiv(K, BK), nblk = (int)cdiv(rows, RB);
  if (cols)
    zslice_cols_kernel<NS, kOn><<<dim3((unsigned)cdiv(rows, 32), batch), 256, 0, st>>>(X, ld, sX, rows, K, nkb, nblk, idx,
                                                                                       sIdx, qmap, ks, S, ex);
  else
    zslice_rows_kernel<NS, kOn><<<dim3((unsigned)cdiv(rows, 8), batch), 256, 0, st>>>(X, ld, sX, rows, K, nkb, nblk, qmap,
                                                                                      ks, S, ex);
}
template <int NS>
cudaError_t slice(cudaStream_t st, bool cols, const double2* X, int64_t ld, int64_t sX, int rows, int K, int batch,
                  const int32_t* idx, int64_t sIdx, const int* qmap, const KScale& ks, __half* S, int* ex) {
  if (NS == 8 && ks.d)
    slice_launch<8, true>(st, cols, X, ld, sX, rows, K, batch, idx, sIdx, qmap, ks, S, ex);
  else
    slice_launch<NS, false>(st, cols, X, ld, sX, rows, K, batch, idx, sIdx, qmap, ks, S, ex);
  count_launch();
  return cudaGetLastError();
}

}  // namespace ztc

size_t zgemm_tc_work_bytes(int slices, int m, int n, int k, int nb, bool same) {
  return ztc::slice_bytes(slices, m, k, nb) + (same ? 0 : ztc::slice_bytes(slices, n, k, nb)) +
         sizeof(int) * (size_t)nb * (m + n) + 256;
}

template <int NS>
static cudaError_t zgemm_tc_impl(cudaStream_t st, char opA, char opB, int m, int n, int k, double alpha, const double2* A,
                     int64_t lda, int64_t sA, const double2* B, int64_t ldb, int64_t sB, double2* C, int64_t ldc,
                     int64_t sC, int batch, const ZOpt& o, void* work, size_t work_bytes, int* err) {
  using namespace ztc;
  if (m <= 0 || n <= 0 || k <= 0 || batch <= 0) return cudaSuccess;
  if (o.brow && opB != 'N') return cudaErrorInvalidValue;
  if (k > kZgemm8MaxK || (NS == 7 && o.kexp)) return cudaErrorInvalidValue;
  const bool aT = opA == 'T' || opA == 'C', aC = opA == 'C' || opA == 'R';
  const bool bT = opB == 'T' || opB == 'C', bC = opB == 'C' || opB == 'R';
  const bool same = !o.brow && !o.kexp && zgemm_tc_same(opA, opB, m, n, A, lda, sA, B, ldb, sB);
  const size_t per = slice_bytes(NS, m, k, 1) + (same ? 0 : slice_bytes(NS, n, k, 1)) + sizeof(int) * (size_t)(m + n);
  if (work_bytes < per + 256) return cudaErrorInvalidValue;
  const int nbc = (int)std::min<size_t>((size_t)std::min(batch, 65535), (work_bytes - 256) / per);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  constexpr size_t smem = (size_t)NST * Blk<NS>::kStage + kOutBytes + 128;
  const bool ks = NS == 7 || k <= kShortK;
  e = cudaFuncSetAttribute(ks ? zgemm_tc_kernel<NS, true> : zgemm_tc_kernel<NS, NS == 7>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  for (int b0 = 0; b0 < batch; b0 += nbc) {
    const int nb = std::min(nbc, batch - b0);
    __half* SA = reinterpret_cast<__half*>(work);
    __half* SB = same ? SA : SA + slice_bytes(NS, m, k, nb) / 2;
    int* eA = reinterpret_cast<int*>(SB + slice_bytes(NS, n, k, nb) / 2);  // n = m where SB is SA
    int* eB = same ? eA : eA + (size_t)nb * m;
    // with a map the arrays stay where they are and the map moves on
    const int* qm = o.qmap ? o.qmap + b0 : nullptr;
    const int64_t s0 = qm ? 0 : b0;
    const int32_t* kx = o.kexp ? o.kexp + s0 * o.sExp : nullptr;
    e = slice<NS>(st, aT, A + s0 * sA, lda, sA, m, k, nb, nullptr, 0, qm, KScale{kx, o.sExp, o.kneg ? 1 : -1}, SA, eA);
    if (e == cudaSuccess && !same)
      e = slice<NS>(st, !bT, B + s0 * sB, ldb, sB, n, k, nb, o.brow ? o.brow + s0 * o.sIdx : nullptr, o.sIdx, qm,
                    KScale{kx, o.sExp, o.kneg ? -1 : 1}, SB, eB);
    if (e != cudaSuccess) return e;
    Args a{};
    a.SA = SA;
    a.SB = SB;
    a.eA = eA;
    a.eB = eB;
    a.C = C + s0 * sC;
    a.ldc = ldc;
    a.sC = sC;
    a.alpha = alpha;
    a.scale = alpha != 1.0;
    a.m = m;
    a.n = n;
    a.nkb = (int)cdiv(k, BK);
    a.mt = (int)cdiv(m, BM);
    a.nt = (int)cdiv(n, BN);
    a.mb = (int)cdiv(m, RB);
    a.nb = (int)cdiv(n, RB);
    a.ntiles = (int64_t)nb * a.mt * a.nt;
    a.lower = o.lowerA;
    a.qmap = qm;
    a.krank = o.krank ? o.krank + s0 : nullptr;
    // a = ar + i ca ai, b = br + i cb bi:  Re = ar br - ca cb ai bi,  Im = cb ar bi + ca ai br
    a.neg_ri = bC;
    a.neg_ir = aC;
    a.neg_ii = (aC == bC);
    a.err = err;
    const unsigned grid = (unsigned)std::min<int64_t>(a.ntiles, sms);
    if (ks)
      zgemm_tc_kernel<NS, true><<<grid, NT, smem, st>>>(a);
    else
      zgemm_tc_kernel<NS, NS == 7><<<grid, NT, smem, st>>>(a);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t zgemm_tc(cudaStream_t st, char opA, char opB, int m, int n, int k, double alpha, const double2* A,
                     int64_t lda, int64_t sA, const double2* B, int64_t ldb, int64_t sB, double2* C, int64_t ldc,
                     int64_t sC, int batch, const ZOpt& o, void* work, size_t work_bytes, int* err) {
  if (o.slices == 7) {
    if (k > kZgemm7MaxK) return cudaErrorInvalidValue;
    return zgemm_tc_impl<7>(st, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, C, ldc, sC, batch, o, work, work_bytes,
                            err);
  }
  return zgemm_tc_impl<8>(st, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, C, ldc, sC, batch, o, work, work_bytes,
                          err);
}

}  // namespace isdf
