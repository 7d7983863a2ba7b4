// Grouped launch of the CUDA-core stage (FP32): several contexts' element
// classes advanced with one launch per (order, element class) variant and
// Runge-Kutta stage.
#include "sym_body.cuh"

namespace wadg {

// ------------------------------------------------------------ grouped launch
// A grouped stage advances every element class of every context of a group
// by one stage (FP32) with one launch per (order, element class) variant
// present.  A variant's kernel is the single-context stage kernel of that
// variant (the symmetric stage, same body and block shape) with a dynamic
// tile schedule over the variant's items; the host issues a stage's variant
// launches on parallel branches of the step graph, so one variant's blocks
// take the SMs that another's leave as its tiles run out.

template <int N, bool PML, bool KAPPA>
using GTile = SymTile<float, N, PML ? 2 : 0, KAPPA>;

// every block starts on the item of the variant that the static split gives
// it, takes that item's tiles from its counter, then moves on to the
// variant's items that still have tiles
template <int N, bool PML, bool KAPPA>
__global__ void __launch_bounds__(GTile<N, PML, KAPPA>::NT, GTile<N, PML, KAPPA>::min_blocks)
group_stage_kernel(const GroupParams G,
                   const __grid_constant__ SymCoef<GTile<N, PML, KAPPA>::coefs> C) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ StageParams<float> P;
  __shared__ int start;
  __shared__ int go;
  if (threadIdx.x == 0) {
    int it = 0;
    while (it + 1 < G.nitems && (int)blockIdx.x >= G.first[it + 1]) ++it;
    start = it;
  }
  for (int k = 0; k < G.nitems; ++k) {
    __syncthreads();   // start is set; the previous item's body is done with P and go
    const int it = (start + k) % G.nitems;
    // one thread decides whether the item still has tiles, so that the whole
    // block takes the same path through the barriers
    if (threadIdx.x == 0) {
      go = *reinterpret_cast<volatile const int*>(G.counter + it) < G.ntiles[it];
      if (go) P = G.p[it];
    }
    __syncthreads();
    if (!go) continue;
    if (!sym_body<float, N, PML ? 2 : 0, KAPPA>(P, C, smem_raw, 0, 1, G.counter + it)) return;
  }
}

// f receives the kernel of a variant code and its tile plan
template <typename F>
auto with_variant(int code, F&& f) -> decltype(f(group_stage_kernel<1, false, false>,
                                                 GTile<1, false, false>{})) {
#define WADG_GROUP_CASE(NN)                                                                 \
  case NN * 4 + 0: return f(group_stage_kernel<NN, false, false>, GTile<NN, false, false>{}); \
  case NN * 4 + 1: return f(group_stage_kernel<NN, true, false>, GTile<NN, true, false>{});   \
  case NN * 4 + 2: return f(group_stage_kernel<NN, true, true>, GTile<NN, true, true>{});
  switch (code) {
    WADG_GROUP_CASE(1)
    WADG_GROUP_CASE(2)
    WADG_GROUP_CASE(3)
    WADG_GROUP_CASE(4)
    WADG_GROUP_CASE(5)
    default: return {};
  }
#undef WADG_GROUP_CASE
}

int group_tile_max(int code, int split) {
  return with_variant(code, [&](auto, auto t) {
    using ST = decltype(t);
    return ST::tile_max(split > ST::S0 ? split : ST::S0);
  });
}

size_t group_smem_bytes(int code, int tile, int split) {
  return with_variant(code, [&](auto, auto t) {
    using ST = decltype(t);
    return ST::bytes(tile, split > ST::S0 ? split : ST::S0);
  });
}

cudaError_t configure_group_kernel() {
  for (int N = 1; N <= 5; ++N) {
    cudaError_t e = upload_sym_constants(N);
    if (e != cudaSuccess) return e;
    for (int v = 0; v < 3; ++v) {
      e = with_variant(N * 4 + v, [&](auto k, auto t) {
        using ST = decltype(t);
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)ST::max_bytes());
      });
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

int group_threads(int) { return GTile<1, true, false>::NT; }

int group_blocks_per_sm(int code, size_t smem) {
  int nb = 0;
  cudaError_t e = with_variant(code, [&](auto k, auto) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, (GTile<1, true, false>::NT), smem);
  });
  if (e != cudaSuccess || nb < 1) nb = 1;
  return nb;
}

cudaError_t launch_group_stage(int code, const GroupParams& G, int nblocks, size_t smem,
                               const float* coef, int ngroups, cudaStream_t s) {
  if (nblocks <= 0 || G.nitems <= 0) return cudaSuccess;
  if (code / 4 < 1 || code / 4 > 5 || code % 4 > 2) return cudaErrorInvalidValue;
  with_variant(code, [&](auto k, auto t) {
    k<<<nblocks, (GTile<1, true, false>::NT), smem, s>>>(G, sym_coef<decltype(t)>(coef, ngroups));
    return cudaSuccess;
  });
  return cudaGetLastError();
}

}  // namespace wadg
