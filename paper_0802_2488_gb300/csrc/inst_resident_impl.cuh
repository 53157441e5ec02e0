// Instantiation of the resident schedule (resident.cuh) for one real type
// EPFFT_REAL, tilings 0 and 1.
#pragma once
#include "launch.cuh"
#include "resident.cuh"

namespace epfft {

// Sides and tilings, X(L, V).  FP64 to L = 128 (above, the FP64 pipe binds
// both forms: L = 256 takes 54 us an iteration here and 48 in the loop); FP32
// tiling 1 to L = 512.  Tiling 0 where its column pass is the Stockham one
// (its register-staged column pass from L = 128 on is another kernel) and the
// compiler forms the same fused multiply-adds in both inlinings (not at
// L = 8 and 16), so that a solve has the same bits on either schedule;
// tests/test_gpu_resident.py holds every entry to that.
#define EPFFT_RES_double(X) \
  X(8, 0) X(16, 0) X(32, 0) X(64, 0) X(128, 0) X(8, 1) X(16, 1) X(32, 1) X(64, 1) X(128, 1)
#define EPFFT_RES_float(X) X(32, 0) X(64, 0) X(8, 1) X(16, 1) X(32, 1) X(64, 1) X(128, 1) X(256, 1) X(512, 1)
#define EPFFT_RES_CAT(T) EPFFT_RES_##T
#define EPFFT_RES_LIST(T) EPFFT_RES_CAT(T)

template <typename T, int L, int V>
static cudaError_t res_prepare(int* per_sm) {
  using R = ResCfg<T, L, V>;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(solve_resident<T, L, V, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)R::SMEM)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(solve_resident<T, L, V, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)R::SMEM)) != cudaSuccess) return e;
  int a = 0, b = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, solve_resident<T, L, V, false>, R::NT, R::SMEM)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, solve_resident<T, L, V, true>, R::NT, R::SMEM)) != cudaSuccess) return e;
  *per_sm = a < b ? a : b;
  return cudaSuccess;
}

template <typename T, int L, int V>
static cudaError_t res_launch(int g, int nb, cudaStream_t s, Solve* solves, BatchCtl* bc, double* part2,
                              unsigned* bars, const void* tw, const void* ktab, int general) {
  using R = ResCfg<T, L, V>;
  const C2<T>* tw_ = reinterpret_cast<const C2<T>*>(tw);
  const C2<T>* k_ = reinterpret_cast<const C2<T>*>(ktab);
  void* args[] = {&solves, &bc, &part2, &bars, &tw_, &k_};
  const void* f = general ? (const void*)solve_resident<T, L, V, true> : (const void*)solve_resident<T, L, V, false>;
  return cudaLaunchCooperativeKernel(f, dim3(g, nb), dim3(R::NT), args, R::SMEM, s);
}

template <>
bool resident_supported<EPFFT_REAL>(int L, int var) {
#define X(n, v) if (L == n && var == v) return true;
  EPFFT_RES_LIST(EPFFT_REAL)(X)
#undef X
  return false;
}

template <>
cudaError_t prepare_resident<EPFFT_REAL>(int L, int var, int* per_sm) {
#define X(n, v) if (L == n && var == v) return res_prepare<EPFFT_REAL, n, v>(per_sm);
  EPFFT_RES_LIST(EPFFT_REAL)(X)
#undef X
  return cudaErrorInvalidValue;
}

template <>
cudaError_t launch_resident<EPFFT_REAL>(int L, int var, int g, int nb, cudaStream_t s, Solve* solves, BatchCtl* bc,
                                        double* part2, unsigned* bars, const void* tw, const void* ktab, int general) {
#define X(n, v) \
  if (L == n && var == v) return res_launch<EPFFT_REAL, n, v>(g, nb, s, solves, bc, part2, bars, tw, ktab, general);
  EPFFT_RES_LIST(EPFFT_REAL)(X)
#undef X
  return cudaErrorInvalidValue;
}

template <>
cudaError_t check_record_resident<EPFFT_REAL>(void** out) {
#ifdef EPFFT_CHECKS
  return cudaGetSymbolAddress(out, g_check);
#else
  *out = nullptr;
  return cudaSuccess;
#endif
}

template <>
cudaError_t read_check_resident<EPFFT_REAL>(CheckRec* out) {
#ifdef EPFFT_CHECKS
  cudaError_t e = cudaMemcpyFromSymbol(out, g_check, sizeof(CheckRec));
  if (e != cudaSuccess || out->code == 0) return e;  // a clear record needs no clearing
  CheckRec z = {};
  return cudaMemcpyToSymbol(g_check, &z, sizeof(CheckRec));
#else
  *out = CheckRec{};
  return cudaSuccess;
#endif
}

}  // namespace epfft
