// Body of the symmetric CUDA-core DGTD stage (FP64 and FP32): the stage of
// stage_body.cuh with every reference operator in the block form of
// sym_tables.hpp, which takes a quarter of the dense products' multiplications
// (half for V_q and P_q of a conical-product rule).
//
// What bounds the dense body: in FP64 the FP64 pipe (two lanes per SM and
// cycle), in FP32 the issue slots and shared-memory loads of 160 kflop per
// PML element (N = 4).  Here, per tile of up to 16 elements and 192 threads:
//   copies   E,H, P, sigma and geometry by bulk copies; face constants
//   flux     one thread per (element, orbit of four face nodes, one on each
//            face): upwind flux at the four nodes, adapted sums over them;
//            and per (element, field, node orbit) the covariant components
//            u_a = X_a . F, X_a = dx/dxi_a, in adapted values: the curl
//            J'^-1 sum_a X_a (d_b u_c - d_c u_b) then takes two reference
//            derivatives per component instead of three
//   curl     one thread per (element, field, character[, row]): derivative
//            and LIFT blocks, back to Cartesian components (all adapted
//            values: element-constant factors commute with the node sums)
//   PML      one thread per (element, component of E,H or of P^E,P^H): its
//            row's adapted values in registers; per orbit of four points the
//            V_q coefficients come by broadcast loads, the field and
//            auxiliary threads of a component trade their four point values
//            by shuffles, apply eq. 9 and add the orbit's share of P_q
//   update   nodal right-hand sides in shared memory, Runge-Kutta update in
//            memory order
// Reference coefficients are the same for all lanes of a warp (rows are the
// lanes), so each is one broadcast load for 32 rows.
//
// Measured, a step against the dense stage: FP32, 384,000 tets, N = 4, compact
// rule: 17.6 -> 5.9 ms; FP64, 48,000 tets, N = 4: 33.3 -> 12.9 ms (the FP64
// pipe bounds both); FP32, 162,000 tets, N = 3, 16 excitations: 59 -> 22.9 ms;
// FP64, 384 tets, N = 3, (N+1)^3 rule: 1.16 -> 0.28 ms (mostly the smaller
// tiles); kappa = 2, 29,478 tets, N = 4: 1.78 -> 0.73 ms.
#pragma once
#include "kernels.cuh"
#include "stage_body.cuh"
#include "sym_tables.hpp"
#include "tc_ptx.cuh"

namespace wadg {

constexpr int kSymThreads = 192;

// shared-memory plan (in Reals) of a tile of TE elements; G: symmetry of the
// volume rule (4, 2), or 0 for the non-PML class
template <typename Real, int N, int G, bool KAPPA = false>
struct SymTile {
  using B = Blocks<N, 4>;
  using L = SymLayout<N>;
  static constexpr int Np = B::Np, Nfp = L::Nfp, NF = 4 * Nfp;
  static constexpr bool PML = G != 0;
  static constexpr int NG = PML ? sym_groups(N, G) : 0;        // groups of four points, at most
  static constexpr int CP = PML ? sym_cp(Np, G) : 0;
  static constexpr int RS = (int)sizeof(Real);
  WADG_HD static constexpr int al(int x) { return (x * RS + 15) / 16 * 16 / RS; }
  static constexpr int ops = al(L::oV + 2 * NG * CP);
  // element strides of the covariant / right-hand-side rows and of the flux,
  // odd so that lanes over (element, field) fall on distinct banks
  static constexpr int UST = 3 * Np | 1, FST = 3 * NF | 1;
  static constexpr int NOB = B::NFul + 3 * B::NH + B::NS;      // node orbits
  static constexpr int TAB = 8 * Nfp + 4 * B::NFul + 8;        // symmetry tables (bytes)
  static constexpr int tabB = (TAB + NF + 96 * Nfp + 15) & ~15;
  WADG_HD static constexpr int cov(int te) { return al(te * 6 * Np) + 16 / RS; }   // staged fields
  WADG_HD static constexpr int fieldsR(int te) { return (PML ? 2 : 1) * cov(te); }
  WADG_HD static constexpr int sigR(int te) { return (KAPPA ? 2 : 1) * te * NG * 12; }
  WADG_HD static constexpr int reals(int te, int s) {
    return ops + fieldsR(te) + sigR(te) + te * 12 + te * 32 + al(te * 2 * UST) +
           al(te * 2 * FST) + (s - 1) * te * 12 * Np;
  }
  // + neighbours and codes, source list, tables, barrier
  WADG_HD static constexpr size_t bytes(int te, int s) {
    return (size_t)reals(te, s) * RS + te * 32 + 256 + tabB + 64;
  }
  static constexpr size_t kMax = 226 * 1024;
  // elements of a tile (T) and threads that share a row's point groups (S0):
  // as many of the block's threads as shared memory allows, then the largest
  // tile (16 and 1 except in FP64 at N = 5)
  static constexpr int pick(bool tile) {
    int bt = 1, bs = 1, best = -1;
    for (int s = 1; s <= 4; ++s)
      for (int t = 16 / s; t >= 1; --t)
        if (bytes(t, s) <= kMax && 100 * t * s + t > best) {
          best = 100 * t * s + t;
          bt = t;
          bs = s;
        }
    return tile ? bt : bs;
  }
  static constexpr int T = pick(true), S0 = pick(false);
  // a class too small to fill the device with tiles of T: tiles of at most
  // four elements whose rows' point groups are shared by four threads
  static constexpr int SS = PML && !KAPPA && S0 < 4 && bytes(T < 4 ? T : 4, 4) <= kMax ? 4 : S0;
  WADG_HD static constexpr int tile_max(int s) { return 16 / s < T ? 16 / s : T; }
  // FP32: two blocks per SM where a tile fits half of the shared memory
  static constexpr int min_blocks = RS == 4 && bytes(T, S0) <= 113 * 1024 ? 2 : 1;
  static_assert(bytes(T, S0) <= kMax && bytes(tile_max(SS), SS) <= kMax, "shared memory");
};

// butterflies between nodal values f and adapted values (sums forward, no
// scaling either way)
template <typename Real, int N, int G>
struct Fly {
  using B = Blocks<N, G>;
  __device__ static __forceinline__ void had4(Real& a, Real& b, Real& c, Real& d) {
    const Real p = a + b, m = a - b, q = c + d, n = c - d;
    a = p + q; b = p - q; c = m + n; d = m - n;
  }
  __device__ static __forceinline__ void forward(const Real* f, Real* s) {
    constexpr NodeOrbits<N> O{};
    if constexpr (G == 4) {
#pragma unroll
      for (int o = 0; o < B::NFul; ++o) {
        Real v[4] = {f[O.ful[o][0]], f[O.ful[o][1]], f[O.ful[o][2]], f[O.ful[o][3]]};
        had4(v[0], v[1], v[2], v[3]);
#pragma unroll
        for (int x = 0; x < 4; ++x) s[B::off(x) + o] = v[x];
      }
      if constexpr (B::NH) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const Real p = f[O.hal[a][0]], q = f[O.hal[a][1]];
          s[B::NFul + a] = p + q;
          s[B::off(a + 1) + B::NFul] = p - q;
        }
      }
      if constexpr (B::NS) s[B::D0 - 1] = f[O.sin];
    } else {
#pragma unroll
      for (int o = 0; o < B::NFul; ++o) {
        s[o] = f[O.pr[o][0]] + f[O.pr[o][1]];
        s[B::D0 + o] = f[O.pr[o][0]] - f[O.pr[o][1]];
      }
#pragma unroll
      for (int o = 0; o < B::NS; ++o) s[B::NFul + o] = f[O.fx[o]];
    }
  }
  // values at the nodes from adapted coefficients; put(node, value)
  template <typename Put>
  __device__ static __forceinline__ void inverse(const Real* t, Put put) {
    constexpr NodeOrbits<N> O{};
    if constexpr (G == 4) {
#pragma unroll
      for (int o = 0; o < B::NFul; ++o) {
        Real v[4] = {t[o], t[B::off(1) + o], t[B::off(2) + o], t[B::off(3) + o]};
        had4(v[0], v[1], v[2], v[3]);
#pragma unroll
        for (int y = 0; y < 4; ++y) put(O.ful[o][y], v[y]);
      }
      if constexpr (B::NH) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const Real p = t[B::NFul + a], q = t[B::off(a + 1) + B::NFul];
          put(O.hal[a][0], p + q);
          put(O.hal[a][1], p - q);
        }
      }
      if constexpr (B::NS) put(O.sin, t[B::D0 - 1]);
    } else {
#pragma unroll
      for (int o = 0; o < B::NFul; ++o) {
        put(O.pr[o][0], t[o] + t[B::D0 + o]);
        put(O.pr[o][1], t[o] - t[B::D0 + o]);
      }
#pragma unroll
      for (int o = 0; o < B::NS; ++o) put(O.fx[o], t[B::NFul + o]);
    }
  }
};

// n consecutive shared-memory values, by the widest loads the row allows (VW:
// values per aligned load)
template <int n, int VW, typename Real>
__device__ __forceinline__ void load_row(const Real* p, Real* v) {
#pragma unroll
  for (int i = 0; i < n; i += VW) {
    if constexpr (VW == 4) lds4(p + i, v + i);
    else if constexpr (VW == 2) lds2(p + i, v + i);
    else v[i] = p[i];
  }
}
// n values of a coefficient column that starts on a 16-byte boundary
template <int n>
__device__ __forceinline__ void load_col(const float* p, float* v) {
#pragma unroll
  for (int i = 0; i + 4 <= n; i += 4) lds4(p + i, v + i);
  constexpr int r = n & ~3;
  if constexpr (n - r >= 2) lds2(p + r, v + r);
  if constexpr ((n - r) & 1) v[n - 1] = p[n - 1];
}
template <int n>
__device__ __forceinline__ void load_col(const double* p, double* v) {
#pragma unroll
  for (int i = 0; i < n; ++i) v[i] = p[i];
}

// rows [r0, r0 + RW) of character x of the right-hand side of one field of
// one element: curl of the covariant components u, LIFT of the flux fl,
// scaled by sc; res[3][RW]
template <typename Real, int N, int RW>
__device__ __forceinline__ void sym_curl_rows(const Real* ops, int x, int r0, const Real* u,
                                              const Real* fl, const Real* gx, Real sc,
                                              Real* res) {
  using L = SymLayout<N>;
  using B = Blocks<N, 4>;
  constexpr int Np = B::Np, Nfp = L::Nfp, NF = 4 * Nfp;
  const int rp = L::RP(x);
  Real w[3][RW];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < RW; ++r) w[c][r] = 0;
  const Real* D = ops + (x == 0 ? 0 : L::DX0 + (x - 1) * L::DX1) + r0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int b = (a + 1) % 3, c = (a + 2) % 3;
    const int xi = x ^ (a + 1), nj = B::dim(xi);
    const Real* ub = u + b * Np + B::off(xi);
    const Real* uc = u + c * Np + B::off(xi);
#pragma unroll 4
    for (int j = 0; j < nj; ++j) {
      Real k[RW];
      load_col<RW>(D + j * rp, k);
      const Real vb = ub[j], vc = uc[j];
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        w[c][r] += k[r] * vb;
        w[b][r] -= k[r] * vc;
      }
    }
    D += nj * rp;
  }
  // Cartesian components of sum_a X_a w_a / J'
  const Real iJ = gx[9];
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    const Real w0 = w[0][r] * iJ, w1 = w[1][r] * iJ, w2 = w[2][r] * iJ;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      w[c][r] = gx[3 * c] * w0 + gx[3 * c + 1] * w1 + gx[3 * c + 2] * w2;
  }
  const Real* Lx = ops + L::l_off(x) + r0;
  const Real* f = fl + x * Nfp;
#pragma unroll 5
  for (int m = 0; m < Nfp; ++m) {
    Real k[RW];
    load_col<RW>(Lx + m * rp, k);
    const Real f0 = f[m], f1 = f[NF + m], f2 = f[2 * NF + m];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      w[0][r] += k[r] * f0;
      w[1][r] += k[r] * f1;
      w[2][r] += k[r] * f2;
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < RW; ++r) res[c * RW + r] = sc * w[c][r];
}

// point values of a group of four volume points from a row's adapted values
template <typename Real, int N, int G>
__device__ __forceinline__ void sym_interp(const Real* coef, const Real* s, Real* v) {
  using B = Blocks<N, G>;
  constexpr int Np = B::Np, CP = sym_cp(Np, G);
  Real c[CP];
#pragma unroll
  for (int i = 0; i < CP; i += 4) lds4(coef + i, c + i);
#pragma unroll
  for (int o = 0; o < 4 / G; ++o) {
#pragma unroll
    for (int x = 0; x < G; ++x) {
      Real a = 0;
#pragma unroll
      for (int j = B::off(x); j < B::off(x) + B::dim(x); ++j) a += c[o * Np + j] * s[j];
      v[G * o + x] = a;
    }
    if constexpr (G == 4) {
      Fly<Real, N, 4>::had4(v[0], v[1], v[2], v[3]);
    } else {
      const Real p = v[2 * o], q = v[2 * o + 1];
      v[2 * o] = p + q;
      v[2 * o + 1] = p - q;
    }
  }
}
// the group's share of P_q: adapted sums of the point values, into acc
template <typename Real, int N, int G>
__device__ __forceinline__ void sym_project(const Real* coef, Real* v, Real* acc) {
  using B = Blocks<N, G>;
  constexpr int Np = B::Np, CP = sym_cp(Np, G);
  Real c[CP];
#pragma unroll
  for (int i = 0; i < CP; i += 4) lds4(coef + i, c + i);
#pragma unroll
  for (int o = 0; o < 4 / G; ++o) {
    if constexpr (G == 4) {
      Fly<Real, N, 4>::had4(v[0], v[1], v[2], v[3]);
    } else {
      const Real p = v[2 * o], q = v[2 * o + 1];
      v[2 * o] = p + q;
      v[2 * o + 1] = p - q;
    }
#pragma unroll
    for (int x = 0; x < G; ++x)
#pragma unroll
      for (int j = B::off(x); j < B::off(x) + B::dim(x); ++j)
        acc[j] += c[o * Np + j] * v[G * o + x];
  }
}

// One element class of one context; smem_raw is the block's dynamic shared
// memory.  Tiles by a static schedule, or from the counter *dyn (grouped
// launch), as stage_body.
template <typename Real, int N, int G, bool KAPPA>
__device__ __forceinline__ void sym_body(const StageParams<Real>& P, unsigned char* smem_raw,
                                         int bid, int nblk, int* dyn = nullptr) {
  using ST = SymTile<Real, N, G, KAPPA>;
  using B = Blocks<N, 4>;
  using L = SymLayout<N>;
  constexpr int Np = ST::Np, Nfp = ST::Nfp, NF = ST::NF, UST = ST::UST, FST = ST::FST;
  constexpr int NT = kSymThreads, CP = ST::CP;
  constexpr bool PML = ST::PML;
  const int S = P.split > ST::S0 ? P.split : ST::S0;
  const int TM = ST::tile_max(S);
  const int TE = P.tile_elems > 0 && P.tile_elems < TM ? P.tile_elems : TM;
  const int ng = P.ngroups;
  Real* ops = reinterpret_cast<Real*>(smem_raw);
  Real* QB = ops + ST::ops;                       // E,H, as the cover of the global block
  Real* PB = QB + ST::cov(TE);                    // P (PML)
  Real* SG = QB + ST::fieldsR(TE);                // sigma [TE][ng][3][4], then kappa
  Real* GX = SG + ST::sigR(TE);                   // [TE][12]: X [3][3], 1/J', 1/eps, 1/mu
  Real* FC = GX + TE * 12;                        // [TE][4][8]: normal, flux factors
  Real* U = FC + TE * 32;                         // [TE][2][UST]
  Real* FL = U + ST::al(TE * 2 * UST);            // [TE][2][FST]; then P's right-hand side
  Real* PS = FL + ST::al(TE * 2 * FST);           // [S - 1][TE * 12][Np] partial sums
  int* nbr = reinterpret_cast<int*>(ops + ST::reals(TE, S));   // [TE][4]
  int* cod = nbr + TE * 4;
  int* srcl = cod + TE * 4;                       // [64]
  unsigned char* tab = reinterpret_cast<unsigned char*>(srcl + 64);
  uint64_t* bar = reinterpret_cast<uint64_t*>(tab + ST::tabB);
  const unsigned char* t_fm = tab;                // [Nfp][4] face node
  const unsigned char* t_fn = tab + 4 * Nfp;      // [Nfp][4] volume node
  const unsigned char* t_or = tab + 8 * Nfp;      // node orbits
  const unsigned char* fperm = tab + ST::TAB + NF;
  __shared__ int nsl, dyn_tile;
  const int tid = threadIdx.x;

  for (int i = tid; i < ST::ops / 2; i += NT) {
    ops[2 * i] = P.symops[2 * i];
    ops[2 * i + 1] = P.symops[2 * i + 1];
  }
  for (int i = tid; i < ST::TAB; i += NT) tab[i] = P.symtab[i];
  for (int i = tid; i < 100 * Nfp; i += NT) tab[ST::TAB + i] = P.tabs[i];
  const uint32_t mb = tc::saddr(bar);
  if (tid == 0) {
    tc::mbar_init(mb, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  const double tbase = P.t_dev ? *P.t_dev : P.t;
  const double tst = tbase + P.rk_c * P.dt;
  const Real rka = (Real)P.rk_a, rkb = (Real)P.rk_b, rdt = (Real)P.dt;
  const int tiles_per_batch = (P.n_elem + TE - 1) / TE;
  const int ntiles = tiles_per_batch * P.nb;
  int claimed = 0;
  auto claim = [&]() {
    if (dyn && tid == 0) claimed = atomicAdd(dyn, 1);
  };
  auto next_tile = [&](int cur) -> int {
    if (!dyn) return cur < 0 ? bid : cur + nblk;
    __syncthreads();   // every thread has read the previous value
    if (tid == 0) dyn_tile = claimed;
    __syncthreads();
    return dyn_tile;
  };
  uint32_t phase = 0;
  bool failed = false;
  claim();
  for (int tile = next_tile(-1); tile < ntiles; tile = next_tile(tile)) {
    claim();
    const int b = tile / tiles_per_batch;
    const int t0 = (tile - b * tiles_per_batch) * TE;
    const int ne = min(TE, P.n_elem - t0);
    const int eg0 = P.e_begin + t0;
    const int64_t oq = (int64_t)b * P.strideQ + (int64_t)eg0 * 6 * Np;
    const int64_t op = (int64_t)b * P.strideP + (int64_t)(eg0 - P.K0) * 6 * Np;
    const Real* qin = P.qin + (int64_t)b * P.strideQ;
    const Real* QS = QB + (reinterpret_cast<uintptr_t>(P.qin + oq) & 15) / sizeof(Real);
    const Real* PQ =
        PML ? PB + (reinterpret_cast<uintptr_t>(P.p + op) & 15) / sizeof(Real) : nullptr;
    __syncthreads();   // the shared buffers are free (and, first, the barrier ready)

    // ---- copies of the tile's blocks (16-byte covers)
    if (tid == 0) {
      nsl = 0;
      const void* src[5] = {P.qin + oq, P.geox + (int64_t)eg0 * 12, nullptr, nullptr, nullptr};
      uint32_t len[5] = {(uint32_t)(ne * 6 * Np * sizeof(Real)),
                         (uint32_t)(ne * 12 * sizeof(Real)), 0, 0, 0};
      uint32_t dst[5] = {tc::saddr(QB), tc::saddr(GX), 0, 0, 0};
      int n = 2;
      if constexpr (PML) {
        const int64_t os = (int64_t)(eg0 - P.K0) * ng * 12;
        src[n] = P.p + op; len[n] = len[0]; dst[n++] = tc::saddr(PB);
        src[n] = P.sig + os; len[n] = (uint32_t)(ne * ng * 12 * sizeof(Real));
        dst[n++] = tc::saddr(SG);
        if constexpr (KAPPA) {
          src[n] = P.kap + os; len[n] = len[n - 1]; dst[n++] = tc::saddr(SG + TE * ng * 12);
        }
      }
      uint32_t total = 0;
      for (int a = 0; a < n; ++a) {
        const uint32_t lo = (uint32_t)(reinterpret_cast<uintptr_t>(src[a]) & 15);
        len[a] = (lo + len[a] + 15) & ~15u;
        src[a] = static_cast<const unsigned char*>(src[a]) - lo;
        total += len[a];
      }
      tc::fence_async_smem();   // earlier reads of the buffers come before the copies
      tc::mbar_expect_tx(mb, total);
      for (int a = 0; a < n; ++a) tc::bulk_g2s(dst[a], src[a], len[a], mb);
      // the registers the update reads, and the next tile, into L2 meanwhile
      auto pre = [&](const Real* p, int n_) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(p) & ~uintptr_t(15);
        const uint32_t l = (uint32_t)((reinterpret_cast<uintptr_t>(p) + n_ * sizeof(Real) + 15 - a) &
                                      ~uintptr_t(15));
        tc::bulk_prefetch_l2(reinterpret_cast<const void*>(a), l);
      };
      pre(P.resq + oq, ne * 6 * Np);
      if (PML) pre(P.resp + op, ne * 6 * Np);
      const int nx = tile + nblk;
      if (!dyn && nx < ntiles) {
        const int b2 = nx / tiles_per_batch, t2 = (nx - b2 * tiles_per_batch) * TE;
        const int n2 = min(TE, P.n_elem - t2);
        pre(P.qin + (int64_t)b2 * P.strideQ + (int64_t)(P.e_begin + t2) * 6 * Np, n2 * 6 * Np);
        if constexpr (PML) {
          pre(P.p + (int64_t)b2 * P.strideP + (int64_t)(P.e_begin + t2 - P.K0) * 6 * Np,
              n2 * 6 * Np);
          pre(P.sig + (int64_t)(P.e_begin + t2 - P.K0) * ng * 12, n2 * ng * 12);
        }
      }
    }
    // ---- per face: normal, flux factors, neighbour
    for (int idx = tid; idx < ne * 4; idx += NT) {
      const int e = eg0 + (idx >> 2);
      Real n4[4];
      ld4(P.fnrm + (int64_t)e * 16 + (idx & 3) * 4, n4);
      const int nb = P.nbr[e * 4 + (idx & 3)];
      const int cd = nb >= 0 ? P.code[e * 4 + (idx & 3)] : 0;
      const bool ok = nb >= 0 && WADG_INDEX_OK(nb < P.strideQ / (6 * Np) && cd < 24, P.err);
      nbr[idx] = ok ? nb : -1;
      cod[idx] = cd;
      const Real ZM = P.mat[e * 3 + 2], ZP = ok ? P.mat[nb * 3 + 2] : ZM;
      const Real iz = n4[3] / (ZM + ZP), al = (Real)P.alpha;
      Real* fc = FC + idx * 8;
      fc[0] = n4[0]; fc[1] = n4[1]; fc[2] = n4[2];
      fc[3] = ZP * iz;            // on n x dH          (drives E)
      fc[4] = al * iz;            // on n (n . dE) - dE
      fc[5] = ZM * iz;            // on n x dE          (drives H): Y+ / (Y- + Y+)
      fc[6] = al * ZM * ZP * iz;  // on n (n . dH) - dH: 1 / (Y- + Y+)
    }
    const bool landed = tc::mbar_wait_sleep(mb, phase);
    phase ^= 1;
    if (!__syncthreads_and(landed)) { failed = true; break; }
    for (int s = tid; s < P.nsrc; s += NT) {
      const SrcDev& sd = P.src[s];
      if (sd.batch == b && sd.elem >= eg0 && sd.elem < eg0 + ne) {
        const int slot = atomicAdd(&nsl, 1);
        if (slot < 64) srcl[slot] = s;
      }
    }

    // ---- upwind flux at the four nodes of a face-node orbit, adapted sums
    for (int idx = tid; idx < ne * Nfp; idx += NT) {
      const int e = idx / Nfp, m = idx - e * Nfp;
      const Real* qe = QS + e * 6 * Np;
      constexpr int fy[4] = {0, 1, 3, 2};
      Real X[4][6];
#pragma unroll
      for (int y = 0; y < 4; ++y) {   // neighbour traces (all in flight at once)
        const int nb = nbr[e * 4 + fy[y]];
#pragma unroll
        for (int c = 0; c < 6; ++c) X[y][c] = 0;
        if (nb >= 0) {
          const int mm = t_fm[m * 4 + y] - fy[y] * Nfp;
          const int np2 = fperm[(fy[y] * 24 + cod[e * 4 + fy[y]]) * Nfp + mm];
          if (WADG_INDEX_OK(np2 < Np, P.err)) {
            const Real* qn = qin + (int64_t)nb * 6 * Np + np2;
#pragma unroll
            for (int c = 0; c < 6; ++c) X[y][c] = qn[c * Np];
          }
        }
      }
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int f = fy[y], ni = t_fn[m * 4 + y];
        const bool pec = nbr[e * 4 + f] < 0;
        const Real* fc = FC + (e * 4 + f) * 8;
        const Real nx = fc[0], ny = fc[1], nz = fc[2];
        const Real c3 = fc[3], c4 = fc[4], c5 = fc[5], c6 = fc[6];
        Real d[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          const Real v = qe[c * Np + ni];
          // perfect electric conductor: mirror state, dE = -2 E, dH = 0
          d[c] = pec ? (c < 3 ? Real(-2) * v : Real(0)) : X[y][c] - v;
        }
        const Real ndE = nx * d[0] + ny * d[1] + nz * d[2];
        const Real ndH = nx * d[3] + ny * d[4] + nz * d[5];
        X[y][0] = c3 * (ny * d[5] - nz * d[4]) - c4 * (nx * ndE - d[0]);
        X[y][1] = c3 * (nz * d[3] - nx * d[5]) - c4 * (ny * ndE - d[1]);
        X[y][2] = c3 * (nx * d[4] - ny * d[3]) - c4 * (nz * ndE - d[2]);
        X[y][3] = c5 * (ny * d[2] - nz * d[1]) + c6 * (nx * ndH - d[3]);
        X[y][4] = c5 * (nz * d[0] - nx * d[2]) + c6 * (ny * ndH - d[4]);
        X[y][5] = c5 * (nx * d[1] - ny * d[0]) + c6 * (nz * ndH - d[5]);
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        Fly<Real, N, 4>::had4(X[0][c], X[1][c], X[2][c], X[3][c]);
        Real* fl = FL + (e * 2 + c / 3) * FST + (c % 3) * NF + m;
#pragma unroll
        for (int x = 0; x < 4; ++x) fl[x * Nfp] = X[x][c];
      }
    }
    // ---- covariant components of E and H, adapted.  The derivatives of a
    // constant vanish, so each component is taken relative to its value at the
    // node nearest the centroid: the adapted sums then round at the size of the
    // field's variation over the element instead of the field's own (FP32 curl
    // of a plane wave at N = 4: relative error 9.7e-7, 2.9e-6 without the
    // subtraction, 1.8e-6 by dense Cartesian derivatives)
    const int nc = t_or[4 * B::NFul + 7];
    for (int idx = tid; idx < ne * 2 * B::NFul; idx += NT) {
      const int ef = idx / B::NFul, o = idx - ef * B::NFul;
      const Real* g = GX + (ef >> 1) * 12;
      const Real* q = QS + ef * 3 * Np;   // e * 6 + field * 3
      Real* u = U + ef * UST + o;
      const Real r0 = q[nc], r1 = q[Np + nc], r2 = q[2 * Np + nc];
      Real v[3][4];
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int n = t_or[4 * o + y];
        const Real f0 = q[n] - r0, f1 = q[Np + n] - r1, f2 = q[2 * Np + n] - r2;
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a][y] = g[a] * f0 + g[3 + a] * f1 + g[6 + a] * f2;
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        Fly<Real, N, 4>::had4(v[a][0], v[a][1], v[a][2], v[a][3]);
#pragma unroll
        for (int x = 0; x < 4; ++x) u[a * Np + B::off(x)] = v[a][x];
      }
    }
    if constexpr (B::NH + B::NS > 0) {
      constexpr int NR = 3 * B::NH + B::NS;
      for (int idx = tid; idx < ne * 2 * NR; idx += NT) {
        const int ef = idx / NR, o = idx - ef * NR;
        const Real* g = GX + (ef >> 1) * 12;
        const Real* q = QS + ef * 3 * Np;
        Real* u = U + ef * UST;
        const bool one = o == 3 * B::NH;
        const int n0 = t_or[4 * B::NFul + 2 * o], n1 = t_or[4 * B::NFul + 2 * o + (one ? 0 : 1)];
        const Real r0 = q[nc], r1 = q[Np + nc], r2 = q[2 * Np + nc];
        const Real f0 = q[n0] - r0, f1 = q[Np + n0] - r1, f2 = q[2 * Np + n0] - r2;
        const Real h0 = q[n1] - r0, h1 = q[Np + n1] - r1, h2 = q[2 * Np + n1] - r2;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const Real p = g[a] * f0 + g[3 + a] * f1 + g[6 + a] * f2;
          const Real r = g[a] * h0 + g[3 + a] * h1 + g[6 + a] * h2;
          u[a * Np + B::NFul + o] = one ? p : p + r;
          if (!one) u[a * Np + B::off(1) + o * B::D1 + B::NFul] = p - r;
        }
      }
    }
    __syncthreads();

    // ---- curl and LIFT in adapted values; results stay in registers until
    // every thread has read U, which then holds them: [TE][E, H][3][Np]
    // FP64: one row per task (the FP64 pipe bounds it, so the finest split
    // balances best); FP32: all rows of a character, for fewer loads per
    // multiplication, one character per warp
    if constexpr (sizeof(Real) == 8) {
      constexpr int MT = (ST::T * 2 * Np + NT - 1) / NT;
      Real res[MT][3];
#pragma unroll
      for (int k = 0; k < MT; ++k) {
        const int idx = tid + k * NT;
        if (idx >= ne * 2 * Np) continue;
        const int row = idx / (ne * 2), ef = idx - row * (ne * 2), f = ef & 1;
        int x = 0;
        if (row >= B::D0) x = 1 + (row - B::D0) / B::D1;
        const Real* g = GX + (ef >> 1) * 12;
        sym_curl_rows<Real, N, 1>(ops, x, row - B::off(x), U + ef * UST, FL + (ef ^ 1) * FST, g,
                                  f ? g[10] : -g[11], res[k]);
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < MT; ++k) {
        const int idx = tid + k * NT;
        if (idx >= ne * 2 * Np) continue;
        const int row = idx / (ne * 2), ef = idx - row * (ne * 2);
#pragma unroll
        for (int c = 0; c < 3; ++c) U[(ef ^ 1) * UST + c * Np + row] = res[k][c];
      }
    } else {
      Real res[3 * B::D0];
      const int x = tid / (2 * TE), ef = tid - x * 2 * TE, f = ef & 1;
      const bool act = x < 4 && ef < 2 * ne;
      if (act) {
        const Real* g = GX + (ef >> 1) * 12;
        const Real sc = f ? g[10] : -g[11];
        if (x == 0)
          sym_curl_rows<Real, N, B::D0>(ops, 0, 0, U + ef * UST, FL + (ef ^ 1) * FST, g, sc, res);
        else
          sym_curl_rows<Real, N, B::D1>(ops, x, 0, U + ef * UST, FL + (ef ^ 1) * FST, g, sc, res);
      }
      __syncthreads();
      if (act) {
        Real* u = U + (ef ^ 1) * UST + B::off(x);
        if (x == 0) {
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int r = 0; r < B::D0; ++r) u[c * Np + r] = res[c * B::D0 + r];
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int r = 0; r < B::D1; ++r) u[c * Np + r] = res[c * B::D1 + r];
        }
      }
    }
    const int nsrc_l = min(nsl, 64);
    __syncthreads();
    if (nsrc_l) {   // dipole sources: adapted coefficients of M_k^-1 l(r_s)
      for (int k = 0; k < nsrc_l; ++k) {
        const SrcDev& sd = P.src[srcl[k]];
        const int e = sd.elem - eg0;
        const Real jt = (Real)dipole_current(sd, tst) * GX[e * 12 + 10];
        for (int i = tid; i < 3 * Np; i += NT) {
          const int c = i / Np;
          U[e * 2 * UST + i] -= jt * (Real)sd.dir[c] * P.src_ws[srcl[k] * Np + i - c * Np];
        }
        __syncthreads();
      }
    }

    if constexpr (!PML) {
      // ---- back to nodal values, in place
      for (int idx = tid; idx < ne * 6; idx += NT) {
        Real* u = U + (idx / 3) * UST + (idx % 3) * Np;
        Real t[Np];
#pragma unroll
        for (int i = 0; i < Np; ++i) t[i] = u[i];
        Fly<Real, N, 4>::inverse(t, [&](int n, Real v) { u[n] = v; });
      }
    } else {
      // ---- eqs. 26-29.  Thread (part, e, c, role): component c of E,H (role
      // 0) or of P (role 1); the S parts share the row's point groups
      const int TE12 = TE * 12;
      const int warp0 = tid & ~31;
      if (warp0 < TE12 * S) {
        const int part_ = tid / TE12, row = tid - part_ * TE12;
        const int part = part_ < S ? part_ : 0;   // spare lanes repeat part 0, and write nothing
        const int e = row / 12, c = (row >> 1) - e * 6, role = row & 1;
        const bool act = part_ < S && e < ne;
        const int u = c % 3, v_ = (u + 1) % 3, w_ = (u + 2) % 3;
        constexpr int VW = Np % 4 == 0 && sizeof(Real) == 4 ? 4 : (Np % 2 == 0 ? 2 : 1);
        Real s[Np], acc[Np];
        {
          Real f[Np];
          load_row<Np, VW>((role ? PQ : QS) + (e * 6 + c) * Np, f);
          Fly<Real, N, G>::forward(f, s);
        }
#pragma unroll
        for (int i = 0; i < Np; ++i) acc[i] = 0;
        const Real* sg = SG + e * ng * 12;
        const Real* Vc = ops + L::oV;
        const Real* Pc = Vc + ng * CP;
#pragma unroll 1
        for (int g0 = 0; g0 < ng; g0 += S) {   // as many rounds in every lane
          const bool on = g0 + part < ng;
          const int g = on ? g0 + part : ng - 1;
          Real v[4], o[4], su[4], sv[4], sw[4];
          sym_interp<Real, N, G>(Vc + g * CP, s, v);
          lds4(sg + g * 12 + u * 4, su);
          lds4(sg + g * 12 + v_ * 4, sv);
          lds4(sg + g * 12 + w_ * 4, sw);
#pragma unroll
          for (int k = 0; k < 4; ++k) o[k] = __shfl_xor_sync(0xffffffffu, v[k], 1);
          if constexpr (!KAPPA) {
            // eq. 9 with kappa = 1 (samples are sigma / eps0): a = 1,
            // b = sv + sw - su, c = sv sw - b su, d = su
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const Real bc = sv[k] + sw[k] - su[k];
              const Real cc = sv[k] * sw[k] - bc * su[k];
              const Real k1 = role ? -su[k] : bc, k2 = role ? Real(1) : cc;
              v[k] = k1 * v[k] + k2 * o[k];
            }
          } else {
            Real ku[4], kv[4], kw[4];
            const Real* kp = sg + TE * ng * 12 + g * 12;
            lds4(kp + u * 4, ku);
            lds4(kp + v_ * 4, kv);
            lds4(kp + w_ * 4, kw);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const Real ki = Real(1) / ku[k];
              const Real a = kv[k] * kw[k] * ki;
              const Real bc = (sv[k] * kw[k] + sw[k] * kv[k] - a * su[k]) * ki;
              const Real cc = sv[k] * sw[k] - bc * su[k];
              const Real k1 = role ? -su[k] * ki : bc, k2 = role ? ki : cc;
              v[k] = k1 * v[k] + k2 * o[k];
            }
          }
          if (!on) v[0] = v[1] = v[2] = v[3] = 0;
          sym_project<Real, N, G>(Pc + g * CP, v, acc);
        }
        if (S > 1) {   // the parts' sums, in order
          if (part_ > 0 && part_ < S) {
            Real* ps = PS + ((part_ - 1) * TE12 + row) * Np;
#pragma unroll
            for (int i = 0; i < Np; ++i) ps[i] = acc[i];
          }
        }
        // the rows' own threads continue below, once all sums are there
        if (S > 1) tc::nbar_sync(1, (TE12 * S + 31) & ~31);
        const bool own = part_ == 0 && act;
        if (own && S > 1) {
          for (int p = 1; p < S; ++p) {
            const Real* ps = PS + ((p - 1) * TE12 + row) * Np;
#pragma unroll
            for (int i = 0; i < Np; ++i) acc[i] += ps[i];
          }
        }
        Real* rq = U + (e * 2 + c / 3) * UST + u * Np;       // adapted curl and LIFT
        Real* rp = FL + e * 2 * FST + c * Np;                 // the flux is spent
        if constexpr (!KAPPA) {
          if (own) {
            if constexpr (G == 4) {
              if (!role) {
#pragma unroll
                for (int i = 0; i < Np; ++i) acc[i] = rq[i] - acc[i];
              }
              Real* r = role ? rp : rq;
              Fly<Real, N, 4>::inverse(acc, [&](int n, Real v) { r[n] = v; });
            } else if (role) {
              Fly<Real, N, G>::inverse(acc, [&](int n, Real v) { rp[n] = v; });
            } else {
              Real t[Np], f[Np];
#pragma unroll
              for (int i = 0; i < Np; ++i) t[i] = rq[i];
              Fly<Real, N, G>::inverse(acc, [&](int n, Real v) { f[n] = v; });
              Fly<Real, N, 4>::inverse(t, [&](int n, Real v) { rq[n] = v - f[n]; });
            }
          }
        } else {
          // P_q a^-1 V_q of the E,H rows: the two threads of a component
          // share its point groups (S = 1)
          if (own && role) Fly<Real, N, G>::inverse(acc, [&](int n, Real v) { rp[n] = v; });
          if constexpr (G == 4) {
#pragma unroll
            for (int i = 0; i < Np; ++i) s[i] = rq[i] - acc[i];
          } else {
            Real t[Np], f[Np];
#pragma unroll
            for (int i = 0; i < Np; ++i) t[i] = rq[i];
            Fly<Real, N, G>::inverse(acc, [&](int n, Real v) { f[n] = v; });
            Fly<Real, N, 4>::inverse(t, [&](int n, Real v) { f[n] = v - f[n]; });
            Fly<Real, N, G>::forward(f, s);
          }
          // role 0 holds the row: sums forward again (G = 4: rescaled below)
          if constexpr (G == 4) {
            // adapted coefficients -> adapted sums: times the orbit size
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
              for (int j = 0; j < B::dim(x); ++j)
                s[B::off(x) + j] *=
                    j < B::NFul ? Real(4) : (x == 0 && j == 3 * B::NH + B::NFul ? Real(1) : Real(2));
          }
#pragma unroll
          for (int i = 0; i < Np; ++i) {
            s[i] = __shfl_sync(0xffffffffu, s[i], tid & 30);
            acc[i] = 0;
          }
#pragma unroll 1
          for (int g = 0; g < ng; g += 2) {
            const int gg = g + role < ng ? g + role : g;
            Real v[4], ku[4], kv[4], kw[4];
            sym_interp<Real, N, G>(Vc + gg * CP, s, v);
            const Real* kp = sg + TE * ng * 12 + gg * 12;
            lds4(kp + u * 4, ku);
            lds4(kp + v_ * 4, kv);
            lds4(kp + w_ * 4, kw);
            const bool on = g + role < ng;
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = on ? ku[k] / (kv[k] * kw[k]) * v[k] : Real(0);
            sym_project<Real, N, G>(Pc + gg * CP, v, acc);
          }
#pragma unroll
          for (int i = 0; i < Np; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 1);
          __syncwarp();
          if (own && !role) Fly<Real, N, G>::inverse(acc, [&](int n, Real v) { rq[n] = v; });
        }
      }
    }
    __syncthreads();

    // ---- Runge-Kutta update, two consecutive values per task
    for (int idx = tid; idx < ne * 3 * Np; idx += NT) {
      const int li = 2 * idx, ef = li / (3 * Np);
      const Real* r = U + li + ef * (UST - 3 * Np);
      Real res[2], q[2] = {QS[li], QS[li + 1]};
      lds2(P.resq + oq + li, res);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        res[k] = rka * res[k] + rdt * r[k];
        q[k] += rkb * res[k];
      }
      sts2(P.resq + oq + li, res);
      sts2(P.qout + oq + li, q);
    }
    if constexpr (PML) {
      Real* pout = P.pout ? P.pout : P.p;
      for (int idx = tid; idx < ne * 3 * Np; idx += NT) {
        const int li = 2 * idx, e = li / (6 * Np);
        const Real* r = FL + li + e * (2 * FST - 6 * Np);
        Real res[2], q[2] = {PQ[li], PQ[li + 1]};
        lds2(P.resp + op + li, res);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          res[k] = rka * res[k] + rdt * r[k];
          q[k] += rkb * res[k];
        }
        sts2(P.resp + op + li, res);
        sts2(pout + op + li, q);
      }
    }
  }
  if (failed) {
    // a copy that did not land in time: report it, and wait once more (bounded)
    // so that it does not land in memory given away
    if (tid == 0) {
      atomicExch(P.err, 1);
      tc::mbar_wait_sleep(mb, phase ^ 1);
    }
  }
  __syncthreads();
  if (tid == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mb) : "memory");
  __syncthreads();
}

}  // namespace wadg
