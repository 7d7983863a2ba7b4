// Launchers of the symmetric CUDA-core stage, instantiated per precision in
// sym_f32.cu and sym_f64.cu.
#pragma once
#include "sym_body.cuh"

namespace wadg {

template <typename Real, int N, int G, bool KAPPA>
__global__ void __launch_bounds__(kSymThreads, SymTile<Real, N, G, KAPPA>::min_blocks)
sym_stage_kernel(const StageParams<Real> P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  sym_body<Real, N, G, KAPPA>(P, smem_raw, blockIdx.x, gridDim.x);
}

template <typename Real, int N, int G, bool KAPPA>
cudaError_t sym_configure_one() {
  using ST = SymTile<Real, N, G, KAPPA>;
  const size_t a = ST::bytes(ST::T, ST::S0), b = ST::bytes(ST::tile_max(ST::SS), ST::SS);
  return cudaFuncSetAttribute(sym_stage_kernel<Real, N, G, KAPPA>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(a > b ? a : b));
}

inline int sm_count() {
  static const int sms = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
  }();
  return sms;
}

// Elements per tile: the largest, or, where that leaves SMs without a tile,
// as many as give every SM one.
inline int sym_tile(int tmax, int64_t n, int sms) {
  const int64_t per = (n + sms - 1) / sms;
  return (int)(per < 1 ? 1 : per < tmax ? per : tmax);
}

template <typename Real, int N, int G, bool KAPPA>
cudaError_t sym_launch_one(const StageParams<Real>& P, int nb, cudaStream_t s) {
  using ST = SymTile<Real, N, G, KAPPA>;
  if (P.n_elem <= 0) return cudaSuccess;
  StageParams<Real> Q = P;
  Q.nb = nb;
  const int S = P.split > ST::S0 ? P.split : ST::S0;
  int te = sym_tile(ST::tile_max(S), (int64_t)P.n_elem * nb, sm_count());
  if (P.tile_elems > 0 && P.tile_elems < te) te = P.tile_elems;
  Q.tile_elems = te;
  const size_t smem = ST::bytes(te, S);
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, sym_stage_kernel<Real, N, G, KAPPA>, kSymThreads, smem);
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)((P.n_elem + te - 1) / te) * nb;
  const int grid = (int)std::min<long long>(tiles, (long long)std::max(per_sm, 1) * sm_count());
  sym_stage_kernel<Real, N, G, KAPPA><<<grid, kSymThreads, smem, s>>>(Q);
  return cudaGetLastError();
}

template <typename Real, int N>
cudaError_t sym_configure_n() {
  cudaError_t e = sym_configure_one<Real, N, 0, false>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 2, false>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 2, true>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 4, false>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 4, true>();
  return e;
}

template <typename Real, int N>
cudaError_t sym_launch_n(int G, bool kappa, const StageParams<Real>& P, int nb, cudaStream_t s) {
  if (G == 0) return sym_launch_one<Real, N, 0, false>(P, nb, s);
  if (G == 2)
    return kappa ? sym_launch_one<Real, N, 2, true>(P, nb, s)
                 : sym_launch_one<Real, N, 2, false>(P, nb, s);
  return kappa ? sym_launch_one<Real, N, 4, true>(P, nb, s)
               : sym_launch_one<Real, N, 4, false>(P, nb, s);
}

template <typename Real, int N, int G, bool KAPPA>
int sym_split_one(int64_t n) {
  using ST = SymTile<Real, N, G, KAPPA>;
  return n < (int64_t)ST::T * sm_count() ? ST::SS : ST::S0;
}
template <typename Real, int N>
int sym_split_n(int G, bool kappa, int64_t n) {
  if (G == 0) return sym_split_one<Real, N, 0, false>(n);
  if (G == 2)
    return kappa ? sym_split_one<Real, N, 2, true>(n) : sym_split_one<Real, N, 2, false>(n);
  return kappa ? sym_split_one<Real, N, 4, true>(n) : sym_split_one<Real, N, 4, false>(n);
}

#define WADG_SYM_SWITCH(call)        \
  switch (N) {                       \
    case 1: return call(1);          \
    case 2: return call(2);          \
    case 3: return call(3);          \
    case 4: return call(4);          \
    case 5: return call(5);          \
    default: break;                  \
  }

#define WADG_SYM_INSTANTIATE(Real)                                                      \
  template <>                                                                           \
  cudaError_t configure_sym_kernels<Real>(int N) {                                      \
    auto f = [](auto n) { return sym_configure_n<Real, decltype(n)::value>(); };        \
    WADG_SYM_SWITCH(WADG_SYM_CALL)                                                      \
    return cudaErrorInvalidValue;                                                       \
  }                                                                                     \
  template <>                                                                           \
  cudaError_t launch_sym<Real>(int N, int G, bool kappa, const StageParams<Real>& P,    \
                               int nb, cudaStream_t s) {                                \
    auto f = [&](auto n) {                                                              \
      return sym_launch_n<Real, decltype(n)::value>(G, kappa, P, nb, s);                \
    };                                                                                  \
    WADG_SYM_SWITCH(WADG_SYM_CALL)                                                      \
    return cudaErrorInvalidValue;                                                       \
  }                                                                                     \
  template <>                                                                           \
  int sym_split<Real>(int N, int G, bool kappa, int64_t n) {                            \
    auto f = [&](auto k) { return sym_split_n<Real, decltype(k)::value>(G, kappa, n); }; \
    WADG_SYM_SWITCH(WADG_SYM_CALL)                                                      \
    return 1;                                                                           \
  }
#define WADG_SYM_CALL(k) f(std::integral_constant<int, k>{})

}  // namespace wadg
