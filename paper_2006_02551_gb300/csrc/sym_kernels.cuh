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

// both classes of a stage: blocks below n0 the non-PML class, the others the PML
// class.  On a small mesh a stage is a few microseconds, of which the fork and
// join of two launches took as much again.  Taken only where every tile of both
// classes has a block at once: beyond that the two launches' own tile sizes and
// registers are better (N = 4 spills here).  The next stage's blocks start
// their set-up (operators, first face tables) while the last ones of this stage
// run.  3,072 tets, N = 2, FP32, 10 steps: 873 -> 583 us; 384 tets, N = 3,
// FP64, 200 steps: 47.0 -> 42.9 ms.
template <typename Real, int N, int G, bool KAPPA>
__global__ void __launch_bounds__(SymTile<Real, N, G, KAPPA>::NT, SymTile<Real, N, G, KAPPA>::min_blocks)
sym_both_kernel(const __grid_constant__ StageParams<Real> A,
                const __grid_constant__ StageParams<Real> B,
                const __grid_constant__ SymCoef<SymTile<Real, N, G, KAPPA>::coefs> C, int n0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if ((int)blockIdx.x < n0)
    sym_body<Real, N, 0, false>(A, SymCoef<1>{}, smem_raw, blockIdx.x, n0);
  else
    sym_body<Real, N, G, KAPPA>(B, C, smem_raw, blockIdx.x - n0, gridDim.x - n0);
}

template <typename Real, int N, int G, bool KAPPA>
cudaError_t sym_configure_one() {
  using ST = SymTile<Real, N, G, KAPPA>;
  cudaError_t e = cudaFuncSetAttribute(sym_stage_kernel<Real, N, G, KAPPA>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)ST::max_bytes());
  if constexpr (ST::PML) {
    // the driver's own choice left room for two of three blocks (the non-PML
    // class asks for it per launch: sym_launch_one)
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(sym_stage_kernel<Real, N, G, KAPPA>,
                               cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
    constexpr size_t other = SymTile<Real, N, 0>::max_bytes();
    const size_t most = ST::max_bytes() > other ? ST::max_bytes() : other;
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(sym_both_kernel<Real, N, G, KAPPA>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(sym_both_kernel<Real, N, G, KAPPA>,
                               cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
  }
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
                           cudaStream_t s, DensePml beside) {
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
  // beside a dense PML launch that takes longer: as few blocks as do it, since
  // they only have to end before the other's (and each one delays a block of it)
  int te = beside == DensePml::longer ? ST::tile_max(S)
           : sizeof(Real) == 8 && ST::PML
               ? sym_tile64(ST::tile_max(S), 12 * S, (int64_t)P.n_elem * nb)
               : sym_tile(ST::tile_max(S), (int64_t)P.n_elem * nb, per_sm * sm_count());
  if (P.tile_elems > 0 && P.tile_elems < te) te = P.tile_elems;
  Q.tile_elems = te;
  const size_t smem = ST::bytes(te, S);
  if ((e = resident(te, &per_sm)) != cudaSuccess) return e;
  const long long tiles = (long long)((P.n_elem + te - 1) / te) * nb;
  const int grid = (int)std::min<long long>(tiles, (long long)per_sm * sm_count());
  const auto C = sym_coef<ST>(coef, P.ngroups);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(ST::NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  // room for several blocks, except beside a dense PML launch, which reads its
  // operators through L1 and would lose that on every SM (stored scheme, N = 3,
  // 24,576 tets, a stage: 170 us without this preference, 196 with it)
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  at.val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
  cfg.attrs = &at;
  cfg.numAttrs = ST::PML || beside != DensePml::none ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, sym_stage_kernel<Real, N, G, KAPPA>, Q, C);
}

template <typename Real, int N, int G, bool KAPPA>
cudaError_t sym_both_one(const StageParams<Real>& A, const StageParams<Real>& B, const float* coef,
                         int nb, bool chained, cudaStream_t s, bool* done) {
  using S0 = SymTile<Real, N, 0>;
  using S1 = SymTile<Real, N, G, KAPPA>;
  static_assert(S0::NT == S1::NT, "one block size for both classes");
  const int sp0 = A.split > S0::S0 ? A.split : S0::S0, sp1 = B.split > S1::S0 ? B.split : S1::S0;
  const int t0 = S0::tile_max(sp0), t1 = S1::tile_max(sp1);
  const int64_t n0 = (int64_t)A.n_elem * nb, n1 = (int64_t)B.n_elem * nb;
  auto tiles = [&](int64_t n, int te, int tmax) {
    const int t = te < tmax ? te : tmax;
    return (n / nb + t - 1) / t * nb;
  };
  // the smallest tile (of both classes, up to each one's largest) at which
  // every tile has a block at once
  for (int te = 1; te <= (t0 > t1 ? t0 : t1); ++te) {
    const int e0 = te < t0 ? te : t0, e1 = te < t1 ? te : t1;
    const size_t b0 = S0::bytes(e0, sp0), b1 = S1::bytes(e1, sp1), smem = b0 > b1 ? b0 : b1;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, sym_both_kernel<Real, N, G, KAPPA>, S1::NT, smem);
    if (e != cudaSuccess) return e;
    const int64_t g0 = tiles(n0, te, t0), g1 = tiles(n1, te, t1);
    if (g0 + g1 > (int64_t)per_sm * sm_count()) continue;
    StageParams<Real> P = A, Q = B;
    P.nb = Q.nb = nb;
    P.tile_elems = e0;
    Q.tile_elems = e1;
    const auto C = sym_coef<S1>(coef, B.ngroups);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(g0 + g1));
    cfg.blockDim = dim3(S1::NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    *done = true;
    return cudaLaunchKernelEx(&cfg, sym_both_kernel<Real, N, G, KAPPA>, P, Q, C, (int)g0);
  }
  return cudaSuccess;
}
template <typename Real, int N>
cudaError_t sym_both_n(int G, bool kappa, const StageParams<Real>& A, const StageParams<Real>& B,
                       const float* coef, int nb, bool chained, cudaStream_t s, bool* done) {
  // (every block at once: more elements than blocks of the largest tiles never fit)
  if ((int64_t)(A.n_elem + B.n_elem) * nb > (int64_t)6 * 21 * sm_count()) return cudaSuccess;
  if (G == 2)
    return kappa ? sym_both_one<Real, N, 2, true>(A, B, coef, nb, chained, s, done)
                 : sym_both_one<Real, N, 2, false>(A, B, coef, nb, chained, s, done);
  return kappa ? sym_both_one<Real, N, 4, true>(A, B, coef, nb, chained, s, done)
               : sym_both_one<Real, N, 4, false>(A, B, coef, nb, chained, s, done);
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
                         cudaStream_t s, DensePml beside) {
  if (G == 0) return sym_launch_one<Real, N, 0, false>(P, coef, nb, s, beside);
  if (G == 2)
    return kappa ? sym_launch_one<Real, N, 2, true>(P, coef, nb, s, beside)
                 : sym_launch_one<Real, N, 2, false>(P, coef, nb, s, beside);
  return kappa ? sym_launch_one<Real, N, 4, true>(P, coef, nb, s, beside)
               : sym_launch_one<Real, N, 4, false>(P, coef, nb, s, beside);
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
                               const float* coef, int nb, cudaStream_t s, DensePml beside) { \
    auto f = [&](auto n) {                                                              \
      return sym_launch_n<Real, decltype(n)::value>(G, kappa, P, coef, nb, s, beside);  \
    };                                                                                  \
    WADG_SYM_SWITCH(WADG_SYM_CALL)                                                      \
    return cudaErrorInvalidValue;                                                       \
  }                                                                                     \
  template <>                                                                           \
  cudaError_t launch_sym_both<Real>(int N, int G, bool kappa, const StageParams<Real>& A, \
                                    const StageParams<Real>& B, const float* coef, int nb, \
                                    bool chained, cudaStream_t s, bool* done) {         \
    auto f = [&](auto n) {                                                              \
      return sym_both_n<Real, decltype(n)::value>(G, kappa, A, B, coef, nb, chained, s, done); \
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
