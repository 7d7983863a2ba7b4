// Launchers of the symmetric CUDA-core stage, instantiated per precision in
// sym_f32.cu and sym_f64.cu.
#pragma once
#include "sym_body.cuh"

namespace wadg {

template <typename Real, int N, int G, bool KAPPA>
__global__ void __launch_bounds__(SymTile<Real, N, G, KAPPA>::NT, SymTile<Real, N, G, KAPPA>::min_blocks)
sym_stage_kernel(const StageParams<Real> P,
                 const __grid_constant__ SymCoef<SymTile<Real, N, G, KAPPA>::coefs> C) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  sym_body<Real, N, G, KAPPA>(P, C, smem_raw, blockIdx.x, gridDim.x);
}

template <typename Real, int N, int G, bool KAPPA>
cudaError_t sym_configure_one() {
  using ST = SymTile<Real, N, G, KAPPA>;
  cudaError_t e = cudaFuncSetAttribute(sym_stage_kernel<Real, N, G, KAPPA>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)ST::max_bytes());
  // the driver's own choice left room for two of three blocks
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sym_stage_kernel<Real, N, G, KAPPA>,
                             cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  return e;
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

// Elements per tile of a class of n elements (times excitations): tmax at
// most, and no more than spreads the class evenly over the waves of `blocks`
// resident blocks that tiles of tmax would take (a last wave of a few tiles
// costs a whole tile's time).
inline int sym_tile(int tmax, int64_t n, int blocks) {
  const int64_t full = (int64_t)tmax * blocks, waves = (n + full - 1) / full;
  const int64_t per = (n + waves * blocks - 1) / (waves * blocks);
  return (int)(per < 1 ? 1 : per < tmax ? per : tmax);
}

// The same for the PML class in FP64, whose pipe serves an SM's warps one
// instruction at a time whatever lanes they use: the tile that leaves the
// fewest warps' rows on an SM, plus half a warp's worth for what a tile costs
// besides (rows: threads per element).
inline int sym_tile64(int tmax, int rows, int64_t n) {
  int64_t best = -1;
  int bt = 1;
  for (int te = 1; te <= tmax; ++te) {
    const int64_t waves = (n + (int64_t)te * sm_count() - 1) / ((int64_t)te * sm_count());
    const int64_t cost = waves * (2 * ((te * rows + 31) / 32) + 1);
    if (best < 0 || cost <= best) {
      best = cost;
      bt = te;
    }
  }
  return bt;
}

template <typename Real, int N, int G, bool KAPPA>
cudaError_t sym_launch_one(const StageParams<Real>& P, const float* coef, int nb,
                           cudaStream_t s) {
  using ST = SymTile<Real, N, G, KAPPA>;
  if (P.n_elem <= 0) return cudaSuccess;
  StageParams<Real> Q = P;
  Q.nb = nb;
  const int S = P.split > ST::S0 ? P.split : ST::S0;
  // resident blocks with the largest tile; a smaller tile may allow more
  auto resident = [&](int te, int* n) {
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        n, sym_stage_kernel<Real, N, G, KAPPA>, ST::NT, ST::bytes(te, S));
    if (*n < 1) *n = 1;
    return e;
  };
  int per_sm = 1;
  cudaError_t e = resident(ST::tile_max(S), &per_sm);
  if (e != cudaSuccess) return e;
  int te = sizeof(Real) == 8 && ST::PML
               ? sym_tile64(ST::tile_max(S), 12 * S, (int64_t)P.n_elem * nb)
               : sym_tile(ST::tile_max(S), (int64_t)P.n_elem * nb, per_sm * sm_count());
  if (P.tile_elems > 0 && P.tile_elems < te) te = P.tile_elems;
  Q.tile_elems = te;
  const size_t smem = ST::bytes(te, S);
  if ((e = resident(te, &per_sm)) != cudaSuccess) return e;
  const long long tiles = (long long)((P.n_elem + te - 1) / te) * nb;
  const int grid = (int)std::min<long long>(tiles, (long long)per_sm * sm_count());
  const auto C = sym_coef<ST>(coef, P.ngroups);
  sym_stage_kernel<Real, N, G, KAPPA><<<grid, ST::NT, smem, s>>>(Q, C);
  return cudaGetLastError();
}

template <typename Real, int N>
cudaError_t sym_configure_n() {
  cudaError_t e = sizeof(Real) == 4 ? upload_sym_constants(N) : cudaSuccess;
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 0, false>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 2, false>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 2, true>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 4, false>();
  if (e == cudaSuccess) e = sym_configure_one<Real, N, 4, true>();
  return e;
}

template <typename Real, int N>
cudaError_t sym_launch_n(int G, bool kappa, const StageParams<Real>& P, const float* coef, int nb,
                         cudaStream_t s) {
  if (G == 0) return sym_launch_one<Real, N, 0, false>(P, coef, nb, s);
  if (G == 2)
    return kappa ? sym_launch_one<Real, N, 2, true>(P, coef, nb, s)
                 : sym_launch_one<Real, N, 2, false>(P, coef, nb, s);
  return kappa ? sym_launch_one<Real, N, 4, true>(P, coef, nb, s)
               : sym_launch_one<Real, N, 4, false>(P, coef, nb, s);
}

template <typename Real, int N, int G, bool KAPPA>
int sym_split_one(int64_t n) {
  using ST = SymTile<Real, N, G, KAPPA>;
  return ST::split_for((int)std::min<int64_t>(ST::T, (n + sm_count() - 1) / sm_count()));
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
                               const float* coef, int nb, cudaStream_t s) {             \
    auto f = [&](auto n) {                                                              \
      return sym_launch_n<Real, decltype(n)::value>(G, kappa, P, coef, nb, s);          \
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
