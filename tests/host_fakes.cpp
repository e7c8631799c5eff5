// Fakes of the CUDA runtime calls and of the kernels that isdf_api.cu uses, for tests of its host side
// without a GPU: device memory is host memory with a capacity, the kernels do nothing but what the
// host reads back, and the calls of interest are counted.
#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include "common.cuh"

namespace {
std::map<void*, size_t> g_live;
size_t g_cap = ~(size_t)0, g_used = 0, g_peak = 0;
int g_rank = 4, g_nulls = 0, g_arm = -1, g_n_tc = 0, g_n_fma = 0, g_ml_rp = 0, g_ml_rank = 0, g_n_kexp = 0;
size_t g_last_work = 0;
void used(const void* p) { g_nulls += p == nullptr; }
}  // namespace

extern "C" {
// ---- controls of the tests
void fake_reset() {
  g_cap = ~(size_t)0;
  g_peak = g_used;
  g_rank = 4;
  g_nulls = g_n_kexp = g_n_tc = g_n_fma = g_ml_rp = g_ml_rank = 0;
  g_arm = -1;
}
void fake_capacity(size_t b) { g_cap = b; }
size_t fake_used() { return g_used; }
size_t fake_peak() { return g_peak; }
void fake_peak_reset() { g_peak = g_used; }
void fake_rank(int r) { g_rank = r; }
int fake_nulls() { return g_nulls; }
void fake_arm(int n) { g_arm = n; }  // the n-th complex128 tensor-core product from now on times out
int fake_tc_calls() { return g_n_tc; }
int fake_fma_calls() { return g_n_fma; }
int fake_ml_rp() { return g_ml_rp; }
int fake_ml_rank() { return g_ml_rank; }
int fake_kexp_calls() { return g_n_kexp; }
size_t fake_last_work() { return g_last_work; }
int isdf_eri_traces_noalloc(const void*, int, const void*, double*, double*, void*) { return 0; }

// ---- runtime
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_used + n > g_cap) return cudaErrorMemoryAllocation;
  void* m = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (m == MAP_FAILED) return cudaErrorMemoryAllocation;
  g_live[m] = n;
  g_used += n;
  if (g_used > g_peak) g_peak = g_used;
  *p = m;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  auto it = g_live.find(p);
  if (it == g_live.end()) return cudaSuccess;
  munmap(p, it->second);
  g_used -= it->second;
  g_live.erase(it);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *t = g_cap;
  *f = g_cap > g_used ? g_cap - g_used : 0;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  used(d), used(s);
  if (d && s && n < ((size_t)64 << 20)) memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  used(d);
  if (d && n < ((size_t)1 << 20)) memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemset2DAsync(void* d, size_t, int, size_t, size_t, cudaStream_t) {
  used(d);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = nullptr;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
}  // extern "C"

namespace isdf {
typedef cudaStream_t S;
typedef const double2* cz;
#define NOP(name, ...) \
  cudaError_t name(__VA_ARGS__) { return cudaSuccess; }

// ---- points, fit and metric
size_t ao_eval_work_bytes(const CellDev&, const BasisDev&) { return 64; }
cudaError_t ao_eval(S, const CellDev&, const BasisDev&, double2* phi, double*) {
  used(phi);
  return cudaSuccess;
}
bool ips_supported(const CellDev&, int, int) { return true; }
size_t ips_work_bytes(const CellDev&, int) { return 64; }
NOP(ips_select, S, const CellDev&, const BasisDev&, const double*, const int*, int, int, double*, double*, int32_t*,
    uint64_t, double, double, double*, int32_t*)
NOP(ip_init, S, cz, int, int, double*, double*)
NOP(ip_step, S, cz, int, int, int, double*, double*, int32_t*, int32_t*, double*, int, uint64_t, double, double, double*,
    int32_t*)
cudaError_t gather_x(S, cz phi, int, int, int, const int32_t*, int, double2* X) {
  used(phi), used(X);
  return cudaSuccess;
}
void grid_twiddles(const int*, double2*) {}
cudaError_t zgemm(S, char, char, int, int, int, double, cz A, int64_t, int64_t, cz B, int64_t, int64_t, double2* C,
                  int64_t, int64_t, int, const ZOpt&) {
  used(A), used(B), used(C);
  ++g_n_fma;
  return cudaSuccess;
}
size_t zgemm_tc_work_bytes(int slices, int m, int n, int k, int nb, bool same) {
  return (size_t)nb * ((size_t)m + (same ? 0 : n)) * ((k + 15) / 16 * 16) * slices * 4 + 256;
}
cudaError_t zgemm_tc(S, char, char, int, int, int, double, cz A, int64_t, int64_t, cz B, int64_t, int64_t, double2* C,
                     int64_t, int64_t, int, const ZOpt& o, void* work, size_t wb, int* err) {
  used(A), used(B), used(C), used(work), used(err);
  ++g_n_tc;
  g_last_work = wb;
  g_n_kexp += o.kexp != nullptr;
  if (g_arm >= 0 && g_arm-- == 0) *err = 41;
  return cudaSuccess;
}
NOP(kdft_cols, S, double2* d, int64_t, KMesh, int, int, int, double, bool)
NOP(kdft_cols_f, S, float2*, int64_t, KMesh, int, int, int, float)
NOP(kdft_cols_ff, S, ffcomplex*, int64_t, KMesh, int, int, int, double)
NOP(kdft_cols_zff, S, double2*, int64_t, KMesh, int, int, int, double)
cudaError_t pchol_batched(S, cz A, int n, int neff, bool, const int* qlist, int nq, double, double2* Lt, int32_t* perm,
                          int32_t* rank) {
  used(A), used(Lt);
  const int r = neff < g_rank ? neff : g_rank;
  for (int i = 0; i < nq; ++i) {
    rank[qlist[i]] = r;
    for (int c = 0; c < n; ++c) perm[(int64_t)qlist[i] * n + c] = c < r ? c : -1;
  }
  return cudaSuccess;
}
NOP(trinv_batched, S, cz, const int32_t*, const int32_t*, int, int, const int*, int, double2*, double2*, double2*)
NOP(row_exponents_z, S, cz, int, int, const int*, int, int32_t*)
NOP(lt_to_rowmajor, S, cz, const int32_t*, const int*, int, int, double2*)
size_t grid_coulomb_work_bytes(int, const CellDev&) { return 64; }
cudaError_t grid_coulomb_fft(S, double2* x, int, int, int, const CellDev&, cz, void*, bool) {
  used(x);
  return cudaSuccess;
}
cudaError_t grid_coulomb_fft_ff(S, ffcomplex* x, int, int, int, const CellDev&, cz, void*) {
  used(x);
  return cudaSuccess;
}
cudaError_t z2ff(S, cz in, ffcomplex* out, int64_t) {
  used(in), used(out);
  return cudaSuccess;
}
int vxi_tc_chunk(int, int, size_t) { return 1; }
size_t vxi_tc_work_bytes(int, int, int) { return 64; }
NOP(vxi_tc, S, const ffcomplex*, int64_t, int, int, int, double, double2*, int64_t, int64_t, void*, int, int*)
cudaError_t mirror_conj(S, double2* x, int64_t, const int2*, int) {
  used(x);
  return cudaSuccess;
}
cudaError_t mirror_copy(S, int32_t* x, int64_t per, const int2* pairs, int n) {
  for (int i = 0; i < n; ++i) memcpy(x + pairs[i].x * per, x + pairs[i].y * per, sizeof(int32_t) * per);
  return cudaSuccess;
}
cudaError_t z2c(S, cz in, float2* out, int64_t) {
  used(in), used(out);
  return cudaSuccess;
}

// ---- fragments
NOP(cgemm, S, char, char, int, int, int, float2, const float2*, int64_t, int64_t, const float2*, int64_t, int64_t,
    float2, float2*, int64_t, int64_t, int)
NOP(kdft_real_f, S, const float*, float2*, int64_t, KMesh, int, float, const int*, const KeepCols&)
NOP(kdft_real_ff, S, const ffloat*, ffcomplex*, int64_t, KMesh, int, double, const int*)
NOP(pair_products, S, cz, int, int, int, double2*)
NOP(pair_products_real_f, S, const float2*, int, int, int, float*, int64_t, int64_t)
NOP(pair_products_real_ff, S, const ffcomplex*, int, int, int, ffloat*, int64_t, int64_t)
NOP(eri_permute, S, cz, int, double, double2*)
NOP(eri_traces, S, cz, int, double, cz, double*, double2*)
NOP(eri_swapconj_sym, S, double2*, int)
NOP(scale_blocks, S, cz, int64_t, int, const double*, double2*)
NOP(scale_blocks_f, S, cz, int64_t, int, const double*, float2*)
void pair_orbits(int, std::vector<int2>& orb) { orb.assign(1, make_int2(0, 0)); }
size_t syrk_tc_split_bytes(int64_t n2, int64_t kcols) { return (size_t)n2 * kcols * 8; }
void syrk_tc_tiles(int64_t, std::vector<int2>& t, std::vector<int>& o, int) {
  t.assign(1, make_int2(0, 0));
  o.assign(1, 0);
}
size_t syrk_tc_ws_bytes(int64_t n) { return (size_t)n * 131072; }
size_t syrk_tc_eri_part_count() { return 2 * 2432 + 1; }
NOP(syrk_tc_rowscale, S, const float2*, int64_t, int64_t, int64_t, const int*, int, int64_t, int*)
NOP(syrk_tc_chunk, S, const float2*, int64_t, int64_t, int64_t, const int*, int64_t, int, int, const int*, void*,
    const int2*, int, void*, int, int*, int)
NOP(syrk_tc_split, S, const float2*, int64_t, int64_t, int64_t, const int*, int64_t, int, int, const int*, void*, double*)
NOP(syrk_tc_mma, S, void*, int64_t, int, int64_t, const int2*, int, void*, int, int*, int)
NOP(syrk_tc_finish_eri, S, const void*, int, const int*, const int2*, int, const int*, const double*, double, float2*, cz,
    double2*, double*)
NOP(syrk_tc_finish_eri_z, S, const void*, int, const int*, const int2*, int, const int*, const double*, double, double2*,
    cz, double2*, double*)
size_t syrk4_tc_split_bytes(int64_t n2, int64_t kcols) { return (size_t)n2 * kcols * 16; }
NOP(syrk4_tc_rowscale, S, const ffcomplex*, int64_t, int64_t, int64_t, int, int64_t, int*)
NOP(syrk4_tc_split, S, const ffcomplex*, int64_t, int64_t, int64_t, int64_t, int, int, const int*, void*, double*)
NOP(syrk4_tc_mma, S, void*, int64_t, int, int64_t, const int2*, int, void*, int, int*)
int mlgemm5_tc_nj_pad(int nj) { return (nj + 95) / 96 * 96; }
bool mlgemm5_tc_supported(int rp) { return 2 * rp <= 576; }
size_t mlgemm5_tc_lslice_bytes(int, int, int) { return 64; }
size_t mlgemm5_tc_split_bytes(int64_t, int, int) { return 64; }
cudaError_t mlgemm5_tc_prepare(S, cz, const double*, int, int, const int*, const int* rank, int rp, int, void*, int*) {
  g_ml_rp = rp;
  g_ml_rank = rank[0];
  return cudaSuccess;
}
NOP(mlgemm5_tc_rowscale, S, const ffcomplex*, int64_t, int, const int*, int, const int*, const int*, int, int64_t, int*)
NOP(mlgemm5_tc_chunk, S, ffcomplex*, int64_t, const int*, int64_t, int, const int*, const int*, int, int, int, int,
    const int*, void*, const void*, const int*, int, int*)
int mlgemm_tc_nj_pad(int nj) { return (nj + 31) / 32 * 32; }
bool mlgemm_tc_supported(int rp) { return 2 * rp <= 640; }
size_t mlgemm_tc_lslice_bytes(int, int, int) { return 64; }
cudaError_t mlgemm_tc_prepare(S, cz, const double*, int, const int*, int, const int*, const int* rank, int rp, int, void*,
                              float*, int16_t*) {
  g_ml_rp = rp;
  g_ml_rank = rank[0];
  return cudaSuccess;
}
NOP(mlgemm_tc, S, const float2*, int, float2*, const int*, int, int64_t, const int*, int, int, const int*, const void*,
    const float*, unsigned*, int*)
NOP(row_exponents, S, const unsigned*, int64_t, int*)

// ---- the other calls
NOP(ao_pairs, S, cz, cz, int, int, double2*)
NOP(scale_cols, S, cz, int, int, int, int, int, const double*, double, double2*)
NOP(sos_trace_parts, S, cz, cz, const int*, int, double*)
NOP(hadamard_t, S, cz, cz, int, int, double2*)
const char* noalloc_last_error() { return ""; }
}  // namespace isdf
