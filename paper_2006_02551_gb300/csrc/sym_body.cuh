// Body of the symmetric CUDA-core DGTD stage (FP64 and FP32): the stage of
// stage_body.cuh with every reference operator in the block form of
// sym_tables.hpp, which takes a quarter of the dense products' multiplications
// (half for V_q and P_q of a conical-product rule).
//
// What bounds the dense body: in FP64 the FP64 pipe (two lanes per SM and
// cycle), in FP32 the issue slots and shared-memory loads of 160 kflop per
// PML element (N = 4).  Here, per tile (FP32: up to 16 elements and 192 threads, two
// blocks per SM; FP64: 21 and 256, so that the PML rows fill eight warps, two
// per scheduler):
//   copies   E,H, P, sigma, geometry and face factors by bulk copies
//   flux     one thread per (element, orbit of four face nodes, one on each
//            face): upwind flux at the four nodes, adapted sums over them;
//            and per (element, field, node orbit) the adapted values of E and H;
//            in FP64 of the covariant components u_a = X_a . F, X_a = dx/dxi_a:
//            the curl J'^-1 sum_a X_a (d_b u_c - d_c u_b) takes two reference
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
// lanes): one broadcast load each in FP64; in FP32, where those loads were the
// bound, constant-bank operands for V_q and P_q (N <= 4) and, at N <= 2, for the
// derivative and LIFT blocks.
//
// What bounds it now: FP64 the FP64 pipe; FP32 the barriers between phases of
// unequal warps, instruction fetch and shared-memory loads (issue slots 39 %
// busy, load path 50 %, DRAM 25 %: ncu, PML class, 82,944 tets, N = 4).
//
// Measured, a step against the dense stage: FP32, 384,000 tets, N = 4, compact
// rule: 17.6 -> 4.7 ms; FP32, 162,000 tets, N = 3, 16 excitations: 59 -> 18.5
// ms; FP64, 48,000 tets, N = 4: 33.3 -> 12.5 ms; FP64, 384 tets, N = 3, (N+1)^3
// rule: 1.16 -> 0.21 ms (mostly the smaller tiles, then
// sym_both_kernel); kappa = 2, 29,478 tets, N =
// 4: 1.78 -> 0.74 ms.  Of the FP32 step, the first version (scalar
// multiplications, face factors computed in the kernel, the update's registers
// loaded one by one) took 5.9 ms; the update's loads were 9,500 of a PML tile's
// 32,000 cycles.  Measured and not kept: 256 threads and 21 elements in FP32
// (3.48 against 3.03 ns per PML element at N = 4: 128 registers spill), 128
// threads and 10 elements (3.72), one thread doing V_q and P_q of both rows
// (3.6: 144 registers of rows and sums spill), the derivative and LIFT blocks
// from constant memory above N = 2 (curl 1.73 -> 2.34 ns per element at N = 4:
// 6 kB of coefficients walked by four warps miss the constant cache; at N = 2
// 0.87 -> 0.61).
#pragma once
#include "kernels.cuh"
#include "refelem.hpp"
#include "stage_body.cuh"
#include "sym_tables.hpp"
#include "tc_ptx.cuh"

namespace wadg {

// FP32 derivative and LIFT blocks (they depend on the order alone) of N <= 2 in
// constant memory: a warp's coefficient comes through the constant cache to the
// uniform registers, where a broadcast from shared memory takes a cycle of the
// SM's load path per coefficient.  Above N = 2 they miss the constant cache
// (N = 4: 2.34 against 1.74 ns per non-PML element) and stay in shared memory.
// One copy per translation unit, written by upload_sym_constants.
static __constant__ float c_sym1[SymLayout<1>::oV], c_sym2[SymLayout<2>::oV];
template <int N>
__device__ __forceinline__ const float* sym_const() {
  static_assert(N <= 2, "orders in constant memory");
  if constexpr (N == 1) return c_sym1;
  else return c_sym2;
}
// this translation unit's copy for order N on the current device (the same
// bytes whenever it is written)
inline cudaError_t upload_sym_constants(int N) {
  if (N > 2) return cudaSuccess;
  const std::vector<float>& h = sym_constants(N);
  const size_t n = h.size() * sizeof(float);
  return N == 1 ? cudaMemcpyToSymbol(c_sym1, h.data(), n) : cudaMemcpyToSymbol(c_sym2, h.data(), n);
}

// V_q and P_q coefficients of a volume rule (n each) as a kernel parameter,
// for the same reason: they reach the multiplications through the constant
// bank
template <int n>
struct SymCoef {
  float v[n], p[n];
};

// shared-memory plan (in Reals) of a tile of TE elements; G: symmetry of the
// volume rule (4, 2), or 0 for the non-PML class
template <typename Real, int N, int G, bool KAPPA = false>
struct SymTile {
  using B = Blocks<N, 4>;
  using L = SymLayout<N>;
  static constexpr int Np = B::Np, Nfp = L::Nfp, NF = 4 * Nfp;
  static constexpr bool PML = G != 0;
  static constexpr int NG = PML ? sym_groups(N, G) : 0;        // groups of four points, at most
  static constexpr int CP = PML ? sym_cp(N, G) : 0;
  static constexpr int RS = (int)sizeof(Real);
  static constexpr int NT = RS == 8 ? 256 : 192;   // threads of a block
  static constexpr int TM = NT / 12;               // elements of a tile at most
  // BOTH: half of the block interpolates (one thread per component, with its
  // E,H row and its P row in registers, so that each coefficient load serves
  // both) and the other half projects the point values of the previous CG
  // groups; the point values pass through shared memory.  (One thread doing
  // both needs 144 registers for the rows and sums alone and spilled.)  Where
  // two rows are too many registers (FP64, N = 5), a thread per row does both
  // in turn.
  static constexpr bool BOTH = PML && RS == 4 && N <= 4;
  static constexpr int CG = N >= 3 ? 2 : 1;
  WADG_HD static constexpr int al(int x) { return (x * RS + 15) / 16 * 16 / RS; }
  // which coefficients come through the constant bank (CC: derivative and LIFT
  // blocks, VC: V_q and P_q) instead of shared memory
  static constexpr bool CC = RS == 4 && N <= 2, VC = BOTH;
  static constexpr int oV = CC ? 0 : L::oV;
  static constexpr int ops = al(oV + (VC ? 0 : 2 * NG * CP));
  static constexpr int coefs = VC ? NG * CP : 1;
  // element strides of the covariant / right-hand-side rows and of the flux,
  // odd so that lanes over (element, field) fall on distinct banks
  static constexpr int UST = 3 * Np | 1, FST = 3 * NF | 1;
  static constexpr int NOB = B::NFul + 3 * B::NH + B::NS;      // node orbits
  static constexpr int TAB = 8 * Nfp + 4 * B::NFul + 8;        // symmetry tables (bytes)
  static constexpr int tabB = (TAB + NF + 96 * Nfp + 15) & ~15;
  WADG_HD static constexpr int cov(int te) { return al(te * 6 * Np) + 16 / RS; }   // staged fields
  WADG_HD static constexpr int fieldsR(int te) { return (PML ? 2 : 1) * cov(te); }
  WADG_HD static constexpr int sigR(int te) { return (KAPPA ? 2 : 1) * te * NG * 12; }
  // flux; then the point values in transit (two buffers of CG groups)
  WADG_HD static constexpr int fluxR(int te) {
    return al(te * (BOTH && 2 * CG * 48 > 2 * FST ? 2 * CG * 48 : 2 * FST));
  }
  WADG_HD static constexpr int reals(int te, int s) {
    return ops + fieldsR(te) + te * 12 + te * 64 + al(te * 2 * UST) + fluxR(te) + sigR(te) +
           (s - 1) * te * 12 * Np;
  }
  // + neighbours, tables, barriers
  WADG_HD static constexpr size_t bytes(int te, int s) {
    return (size_t)reals(te, s) * RS + te * 32 + tabB + 64;
  }
  static constexpr size_t kMax = 226 * 1024;
  static constexpr int blocks(int te) {   // that fit an SM, of the two wanted
    return bytes(te, 1) <= 113 * 1024 ? 2 : 1;
  }
  // elements of a tile (T) and threads that share a row's point groups (S0):
  // TM / S0 at most, where the PML rows fill the block.  FP32 with BOTH, and
  // the FP32 non-PML class: the most elements per SM, since these kernels live
  // on the other block's work while one waits.  FP64 and N = 5: as many of the
  // block's threads as shared memory allows, then the largest tile.
  static constexpr bool MANY = RS == 4 && (BOTH || !PML);
  static constexpr int pick(bool tile) {
    int bt = 1, bs = 1, best = -1;
    for (int s = 1; s <= (MANY || !PML || KAPPA ? 1 : 4); ++s)
      for (int t = TM / s; t >= 1; --t) {
        const int v = MANY ? blocks(t) * t : 100 * t * s + t;
        if (bytes(t, s) <= kMax && v > best) {
          best = v;
          bt = t;
          bs = s;
        }
      }
    return tile ? bt : bs;
  }
  static constexpr int T = pick(true), S0 = pick(false);
  WADG_HD static constexpr int tile_max(int s) {
    int t = TM / s < T ? TM / s : T;
    while (t > 1 && bytes(t, s) > kMax) --t;
    return t;
  }
  // a class too small to fill the device with tiles of T: the threads that
  // share a row's groups where an SM gets te elements, for the fewest warp
  // rounds over the groups (an SM's FP64 pipe takes a warp at a time, so what
  // counts is full lanes; each part also transforms the row, hence the third)
  static constexpr bool SPLITS = PML && !KAPPA && !BOTH;
  WADG_HD static constexpr int split_for(int te) {
    if (!SPLITS || te >= T) return S0;
    int bs = S0, best = 1 << 30;
    for (int s = S0; s <= TM / te && s <= 8; ++s) {
      const int cost = (12 * te * s + 31) / 32 * (3 * ((NG + s - 1) / s) + 1);
      if (bytes(te, s) <= kMax && cost < best) {
        best = cost;
        bs = s;
      }
    }
    return bs;
  }
  static constexpr size_t max_bytes() {   // of any tile and split
    size_t m = bytes(T, S0);
    for (int te = 1; te < T; ++te) {
      const size_t b = bytes(tile_max(split_for(te)), split_for(te));
      if (b > m) m = b;
    }
    return m;
  }
  static constexpr int min_blocks = MANY ? blocks(T) : 1;
  static_assert(max_bytes() <= kMax && 12 * T * S0 <= NT, "plan");
};

// the coefficients of a rule of ng groups (host: V_q [ng][CP], then P_q)
template <typename ST>
SymCoef<ST::coefs> sym_coef(const float* h, int ng) {
  SymCoef<ST::coefs> C{};
  if (ST::VC && h) {
    const int n = ng * ST::CP;
    std::copy(h, h + n, C.v);
    std::copy(h + n, h + 2 * n, C.p);
  }
  return C;
}

// butterflies between nodal values f and adapted values (sums forward, no
// scaling either way)
template <typename Real, int N, int G>
struct Fly {
  using B = Blocks<N, G>;
  __device__ static __forceinline__ void had4(Real& a, Real& b, Real& c, Real& d) {
    const Real p = a + b, m = a - b, q = c + d, n = c - d;
    a = p + q; b = p - q; c = m + n; d = m - n;
  }
  // the butterfly over one point orbit's G values
  __device__ static __forceinline__ void group(Real* v) {
    if constexpr (G == 4) {
      had4(v[0], v[1], v[2], v[3]);
    } else {
      const Real p = v[0], q = v[1];
      v[0] = p + q;
      v[1] = p - q;
    }
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

// Pairs of FP32 values: one instruction multiplies and adds both (each as an
// FMA rounds), which halves the issue slots of the contractions.
using pair2 = unsigned long long;
__device__ __forceinline__ pair2 pack2(float a, float b) {
  pair2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(pair2 p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ void fma2(pair2& d, pair2 a, pair2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
// n coefficient pairs: from the constant bank (CB), or from shared memory by
// 16-byte broadcasts (an even number readable)
template <int n, bool CB>
__device__ __forceinline__ void load_pairs(const float* p, pair2* v) {
  if constexpr (CB) {
#pragma unroll
    for (int i = 0; i < n; ++i) v[i] = pack2(p[2 * i], p[2 * i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < n; i += 2) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p + 2 * i);
      v[i] = t.x;
      if (i + 1 < n) v[i + 1] = t.y;
    }
  }
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

// The same in FP32 for all rows of character X, in pairs of rows, from the
// Cartesian components F (u) and the metric g_a = grad xi_a (gx): curl F =
// sum_a g_a x d_a F.  Three derivatives per component instead of two, but none
// of the covariant form's roundings before the derivative, which FP32 notices
// (curl of a plane wave, N = 3: relative error 3.4e-7 against 4.2e-7; 4.1e-7
// dense).
// (X: 0, or 1 for any other character x: two instances keep the code small)
template <int N, int X, bool CB>
__device__ __forceinline__ void sym_curl_pairs(const float* ops, int x, const float* u,
                                               const float* fl, const float* gx, float sc,
                                               float* out) {
  using L = SymLayout<N>;
  using B = Blocks<N, 4>;
  constexpr int Np = B::Np, Nfp = L::Nfp, NF = 4 * Nfp;
  constexpr int RW = B::dim(X), rp = L::RP(X);
  constexpr int R2 = (RW + 1) / 2;   // the padding rows' coefficients are zero
  if constexpr (CB) ops = sym_const<N>();
  const float* D = ops + (X ? L::DX0 + (x - 1) * L::DX1 : 0);
  pair2 w[3][R2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < R2; ++r) w[c][r] = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int xi = x ^ (a + 1), nj = X ? B::dim(xi) : B::D1;
    const float* f = u + B::off(xi);
    pair2 d[3][R2];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < R2; ++r) d[c][r] = 0;
#pragma unroll 4
    for (int j = 0; j < nj; ++j) {
      pair2 k[R2];
      load_pairs<R2, CB>(D + j * rp, k);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float v = f[c * Np + j];
        const pair2 pv = pack2(v, v);
#pragma unroll
        for (int r = 0; r < R2; ++r) fma2(d[c][r], k[r], pv);
      }
    }
    D += nj * rp;
    pair2 g[3], m[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float v = gx[3 * a + i];
      g[i] = pack2(v, v);
      m[i] = pack2(-v, -v);
    }
#pragma unroll
    for (int r = 0; r < R2; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        fma2(w[c][r], g[(c + 1) % 3], d[(c + 2) % 3][r]);
        fma2(w[c][r], m[(c + 2) % 3], d[(c + 1) % 3][r]);
      }
  }
  const float* Lx = ops + L::l_off(X ? x : 0);
  const float* f = fl + x * Nfp;
#pragma unroll 5
  for (int m = 0; m < Nfp; ++m) {
    pair2 k[R2];
    load_pairs<R2, CB>(Lx + m * rp, k);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float v = f[c * NF + m];
      const pair2 pv = pack2(v, v);
#pragma unroll
      for (int r = 0; r < R2; ++r) fma2(w[c][r], k[r], pv);
    }
  }
  __syncthreads();   // every thread has read u, which takes the results
  if (out) {
    out += B::off(X ? x : 0);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < R2; ++r) {
        float p, q;
        unpack2(w[c][r], p, q);
        out[c * Np + 2 * r] = sc * p;
        if (2 * r + 1 < RW) out[c * Np + 2 * r + 1] = sc * q;
      }
  }
}

// point values of a group of four volume points from a row's adapted values
template <typename Real, int N, int G>
__device__ __forceinline__ void sym_interp(const Real* coef, const Real* s, Real* v) {
  using B = Blocks<N, G>;
  constexpr int PO = B::PO, CP = B::CP;
  Real c[CP];
#pragma unroll
  for (int i = 0; i < CP; i += 4) lds4(coef + i, c + i);
#pragma unroll
  for (int o = 0; o < 4 / G; ++o) {
#pragma unroll
    for (int x = 0; x < G; ++x) {
      Real a = 0;
#pragma unroll
      for (int j = 0; j < B::dim(x); ++j) a += c[o * PO + B::poff(x) + j] * s[B::off(x) + j];
      v[G * o + x] = a;
    }
    Fly<Real, N, G>::group(v + G * o);
  }
}
// the group's share of P_q: adapted sums of the point values, into acc
template <typename Real, int N, int G>
__device__ __forceinline__ void sym_project(const Real* coef, Real* v, Real* acc) {
  using B = Blocks<N, G>;
  constexpr int PO = B::PO, CP = B::CP;
  Real c[CP];
#pragma unroll
  for (int i = 0; i < CP; i += 4) lds4(coef + i, c + i);
#pragma unroll
  for (int o = 0; o < 4 / G; ++o) {
    Fly<Real, N, G>::group(v + G * o);
#pragma unroll
    for (int x = 0; x < G; ++x)
#pragma unroll
      for (int j = 0; j < B::dim(x); ++j)
        acc[B::off(x) + j] += c[o * PO + B::poff(x) + j] * v[G * o + x];
  }
}

// adapted values <-> pairs in the padded order of the coefficients
template <int N, int G>
__device__ __forceinline__ void to_pairs(const float* s, pair2* p) {
  using B = Blocks<N, G>;
#pragma unroll
  for (int x = 0; x < G; ++x)
#pragma unroll
    for (int j = 0; j < B::dim(x); j += 2)
      p[(B::poff(x) + j) / 2] =
          pack2(s[B::off(x) + j], j + 1 < B::dim(x) ? s[B::off(x) + j + 1] : 0.f);
}
template <int N, int G>
__device__ __forceinline__ void from_pairs(const pair2* p, float* s) {
  using B = Blocks<N, G>;
#pragma unroll
  for (int x = 0; x < G; ++x)
#pragma unroll
    for (int j = 0; j < B::dim(x); j += 2) {
      float a, b;
      unpack2(p[(B::poff(x) + j) / 2], a, b);
      s[B::off(x) + j] = a;
      if (j + 1 < B::dim(x)) s[B::off(x) + j + 1] = b;
    }
}
// point values of a group for a component's two rows
template <int N, int G, bool CB>
__device__ __forceinline__ void sym_interp2(const float* coef, const pair2* s, const pair2* p,
                                            float* v, float* w) {
  using B = Blocks<N, G>;
  constexpr int PO = B::PO, CP = B::CP;
  pair2 c[CP / 2];
  load_pairs<CP / 2, CB>(coef, c);
#pragma unroll
  for (int o = 0; o < 4 / G; ++o) {
#pragma unroll
    for (int x = 0; x < G; ++x) {
      pair2 a = 0, b = 0;
#pragma unroll
      for (int j = B::poff(x) / 2; j < (B::poff(x) + B::dim(x) + 1) / 2; ++j) {
        fma2(a, c[o * PO / 2 + j], s[j]);
        fma2(b, c[o * PO / 2 + j], p[j]);
      }
      float a0, a1, b0, b1;
      unpack2(a, a0, a1);
      unpack2(b, b0, b1);
      v[G * o + x] = a0 + a1;
      w[G * o + x] = b0 + b1;
    }
    Fly<float, N, G>::group(v + G * o);
    Fly<float, N, G>::group(w + G * o);
  }
}
// P_q of a group's adapted point sums for both rows
template <int N, int G, bool CB>
__device__ __forceinline__ void sym_add2(const float* coef, const float* v, const float* w,
                                         pair2* a, pair2* b) {
  using B = Blocks<N, G>;
  constexpr int PO = B::PO, CP = B::CP;
  pair2 c[CP / 2];
  load_pairs<CP / 2, CB>(coef, c);
#pragma unroll
  for (int o = 0; o < 4 / G; ++o)
#pragma unroll
    for (int x = 0; x < G; ++x) {
      const pair2 tv = pack2(v[G * o + x], v[G * o + x]);
      const pair2 tw = pack2(w[G * o + x], w[G * o + x]);
#pragma unroll
      for (int j = B::poff(x) / 2; j < (B::poff(x) + B::dim(x) + 1) / 2; ++j) {
        fma2(a[j], c[o * PO / 2 + j], tv);
        fma2(b[j], c[o * PO / 2 + j], tw);
      }
    }
}
// the same for one row (constant-bank coefficients)
template <int N, int G>
__device__ __forceinline__ void sym_add1(const float* coef, const float* v, float* acc) {
  using B = Blocks<N, G>;
#pragma unroll
  for (int o = 0; o < 4 / G; ++o)
#pragma unroll
    for (int x = 0; x < G; ++x)
#pragma unroll
      for (int j = 0; j < B::dim(x); ++j)
        acc[B::off(x) + j] += coef[o * B::PO + B::poff(x) + j] * v[G * o + x];
}
// V4-adapted coefficients -> adapted sums: times the orbits' sizes
template <typename Real, int N>
__device__ __forceinline__ void sym_to_sums(Real* s) {
  using B = Blocks<N, 4>;
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int j = 0; j < B::dim(x); ++j)
      s[B::off(x) + j] *=
          j < B::NFul ? Real(4) : (x == 0 && j == 3 * B::NH + B::NFul ? Real(1) : Real(2));
}

// Dipole sources of a tile (s0 .. s1 of the table): the currents of the first 32
// from s0 on by one warp, in double, scaled by 1/eps; and all of them, adapted
// coefficients of M_k^-1 l(r_s), into the adapted right-hand sides U.  Every thread
// evaluating every current took 2 us a source; in FP32 a warp that has no part in
// the curl evaluates them meanwhile (evaluated after it, one source prolonged the
// stage: kappa = 2, 29,478 tets, 10 steps 7.53 against 7.42 ms).  Not inlined: few
// tiles have sources, and the others fetch less code.
template <typename Real>
__device__ __noinline__ void sym_currents(const SrcDev* src, int s0, int s1, int eg0, double t,
                                          const Real* GX, Real* cur) {
  const int k = threadIdx.x & 31;
  if (s0 + k < s1) {
    const SrcDev& sd = src[s0 + k];
    cur[k] = (Real)dipole_current(sd, t) * GX[(sd.elem - eg0) * 12 + 10];
  }
}
// (the first 32 currents are there)
template <typename Real, int Np, int UST, int NT>
__device__ __noinline__ void sym_sources(const SrcDev* src, const Real* src_ws, int s0, int s1,
                                         int eg0, double t, const Real* GX, Real* cur, Real* U) {
  const int tid = threadIdx.x;
  for (int sb = s0; sb < s1; sb += 32) {
    if (sb > s0) {
      if (tid < 32) sym_currents(src, sb, s1, eg0, t, GX, cur);
      __syncthreads();
    }
    for (int s = sb; s < min(s1, sb + 32); ++s) {   // (a thread keeps its values of an element)
      const SrcDev& sd = src[s];
      const int e = sd.elem - eg0;
      const Real jt = cur[s - sb];
      for (int i = tid; i < 3 * Np; i += NT) {
        const int c = i / Np;
        U[e * 2 * UST + i] -= jt * (Real)sd.dir[c] * src_ws[(int64_t)s * Np + i - c * Np];
      }
    }
    __syncthreads();
  }
}

// One element class of one context; smem_raw is the block's dynamic shared
// memory.  Tiles by a static schedule, or from the counter *dyn (grouped
// launch).  False where a copy did not land in time: the block then takes no
// more tiles.
template <typename Real, int N, int G, bool KAPPA, typename ST = SymTile<Real, N, G, KAPPA>>
__device__ __forceinline__ bool sym_body(const StageParams<Real>& P, const SymCoef<ST::coefs>& C,
                                         unsigned char* smem_raw, int bid, int nblk,
                                         int* dyn = nullptr) {
  using B = Blocks<N, 4>;
  using L = SymLayout<N>;
  constexpr int Np = ST::Np, Nfp = ST::Nfp, NF = ST::NF, UST = ST::UST, FST = ST::FST;
  constexpr int NT = ST::NT, CP = ST::CP;
  constexpr bool PML = ST::PML;
  const int S = P.split > ST::S0 ? P.split : ST::S0;
  const int TX = ST::tile_max(S);
  const int TE = P.tile_elems > 0 && P.tile_elems < TX ? P.tile_elems : TX;
  const int ng = P.ngroups;
  Real* ops = reinterpret_cast<Real*>(smem_raw);
  Real* QB = ops + ST::ops;                       // E,H, as the cover of the global block
  Real* PB = QB + ST::cov(TE);                    // P (PML)
  // [TE][12]: FP64 X [3][3], 1/J'; FP32 grad xi_a [3][3]; 1/eps, 1/mu
  Real* GX = QB + ST::fieldsR(TE);
  Real* FC2 = GX + TE * 12;                       // 2 x [TE][4][8]: normal, flux factors, code
  Real* U = FC2 + TE * 64;                        // [TE][2][UST]
  // flux [TE][2][FST]; then point values in transit; then P's right-hand side
  // [TE][6][Np]
  Real* FL = U + ST::al(TE * 2 * UST);
  Real* SG = FL + ST::fluxR(TE);                  // sigma [TE][ng][3][4], then kappa
  Real* PS = SG + ST::sigR(TE);                   // [S - 1][TE * 12][Np] partial sums
  int* nbr2 = reinterpret_cast<int*>(ops + ST::reals(TE, S));   // 2 x [TE][4]
  unsigned char* tab = reinterpret_cast<unsigned char*>(nbr2 + TE * 8);
  uint64_t* bar = reinterpret_cast<uint64_t*>(tab + ST::tabB);
  const unsigned char* t_fm = tab;                // [Nfp][4] face node
  const unsigned char* t_fn = tab + 4 * Nfp;      // [Nfp][4] volume node
  const unsigned char* t_or = tab + 8 * Nfp;      // node orbits
  const unsigned char* fperm = tab + ST::TAB + NF;
  __shared__ int nsl, src0, dyn_tile;   // the tile's sources: count, first of the table
  __shared__ Real cur[32];
  const int tid = threadIdx.x;

  for (int i = tid; i < ST::ops / 2; i += NT) {
    const Real* src = P.symops + (L::oV - ST::oV) + 2 * i;   // (oV = 0: from V_q on)
    ops[2 * i] = src[0];
    ops[2 * i + 1] = src[1];
  }
  for (int i = tid; i < ST::TAB; i += NT) tab[i] = P.symtab[i];
  for (int i = tid; i < 100 * Nfp; i += NT) tab[ST::TAB + i] = P.tabs[i];
  const uint32_t mb = tc::saddr(bar), mf = tc::saddr(bar + 1);
  if (tid == 0) {
    tc::mbar_init(mb, 1);
    tc::mbar_init(mf, 1);
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
  // copies of n global blocks (16-byte covers) completing on barrier m
  // (withheld: bytes that the barrier waits for and no copy brings)
  auto copy_in = [&](const void* const* src, const uint32_t* len, const uint32_t* dst, int n,
                     uint32_t m, uint32_t withheld) {
    uint32_t total = withheld;
    for (int a = 0; a < n; ++a)
      total += ((uint32_t)(reinterpret_cast<uintptr_t>(src[a]) & 15) + len[a] + 15) & ~15u;
    tc::fence_async_smem();   // earlier reads of the buffers come before the copies
    tc::mbar_expect_tx(m, total);
    for (int a = 0; a < n; ++a) {
      const uint32_t lo = (uint32_t)(reinterpret_cast<uintptr_t>(src[a]) & 15);
      tc::bulk_g2s(dst[a], static_cast<const unsigned char*>(src[a]) - lo,
                   (lo + len[a] + 15) & ~15u, m);
    }
  };
  // a tile's neighbours and face factors into buffer fb
  auto faces_in = [&](int tile, int fb) {
    const int t0 = tile % tiles_per_batch * TE, n = min(TE, P.n_elem - t0);
    const int64_t e0 = P.e_begin + t0;
    const void* src[2] = {P.nbr + e0 * 4, P.facex + e0 * 32};
    const uint32_t len[2] = {(uint32_t)(n * 16), (uint32_t)(n * 32 * sizeof(Real))};
    const uint32_t dst[2] = {tc::saddr(nbr2 + fb * TE * 4), tc::saddr(FC2 + fb * TE * 32)};
    copy_in(src, len, dst, 2, mf, 0);
  };
  uint32_t phase = 0;   // tiles done: the barriers' parities
  bool failed = false, ahead = !dyn && bid < ntiles;   // ahead: this tile's faces are on their way
  if (ahead && tid == 0) faces_in(bid, 0);
  // in a chained launch: the next stage may start its set-up, and this one's
  // reads of the state wait for the last stage's writes (no-ops otherwise)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  claim();
  for (int tile = next_tile(-1); tile < ntiles; tile = next_tile(tile), ++phase) {
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

    // ---- copies of the tile's blocks; the faces' were issued a tile ahead
    // where the schedule is known
    const int nx = dyn ? ntiles : tile + nblk;
    const int fb = phase & 1;
    if (tid == 0) {
      nsl = 0;
      src0 = P.nsrc;
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
      if (!ahead) faces_in(tile, fb);
      copy_in(src, len, dst, n, mb, wadg_take_request(P.inject, kRequestStage) ? 16 : 0);
      // the registers the update reads, and the next tile, into L2 meanwhile
      auto pre = [&](const Real* p, int n_) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(p) & ~uintptr_t(15);
        const uint32_t l = (uint32_t)((reinterpret_cast<uintptr_t>(p) + n_ * sizeof(Real) + 15 - a) &
                                      ~uintptr_t(15));
        tc::bulk_prefetch_l2(reinterpret_cast<const void*>(a), l);
      };
      pre(P.resq + oq, ne * 6 * Np);
      if (PML) pre(P.resp + op, ne * 6 * Np);
      if (nx < ntiles) {
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
    bool landed = tc::mbar_wait_sleep(mf, phase & 1);
    const int* nbr = nbr2 + fb * TE * 4;
    const Real* FC = FC2 + fb * TE * 32;

    // ---- neighbour traces into registers while the tile's own blocks land.
    // A task is an orbit of four face nodes, one on each face; FP32 a thread
    // per orbit (24 gathers in flight), FP64 four lanes per orbit (four times
    // the tasks: a small tile's 15 orbits per element left the FP64 pipe to a
    // warp or two)
    constexpr int FO = sizeof(Real) == 8 ? 1 : 4;   // nodes of a task
    constexpr int FR = (ST::T * Nfp * (4 / FO) + NT - 1) / NT;   // tasks of a thread
    Real X[FR][FO][6];
#pragma unroll
    for (int r = 0; r < FR; ++r) {
      const int idx = tid + r * NT;
      const bool act = landed && idx < ne * Nfp * (4 / FO);
      if (!act) continue;
      const int em = idx / (4 / FO), y0 = FO == 4 ? 0 : idx & 3;
      const int e = em / Nfp, m = em - e * Nfp;
#pragma unroll
      for (int k = 0; k < FO; ++k) {
        const int y = y0 + k, f = y < 2 ? y : 5 - y;   // face of g_y: 0, 1, 3, 2
        const int nb = nbr[e * 4 + f];
        const int mm = t_fm[m * 4 + y] - f * Nfp, cd = (int)FC[(e * 4 + f) * 8 + 7];
        const bool in = nb >= 0 && WADG_INDEX_OK(nb < P.strideQ / (6 * Np) && cd < 24, P.err);
        const int np2 = in ? fperm[(f * 24 + cd) * Nfp + mm] : 0;
        // (zeros stay where there is no neighbour: the flux mirrors the state)
#pragma unroll
        for (int c = 0; c < 6; ++c) X[r][k][c] = 0;
        if (in && WADG_INDEX_OK(np2 < Np, P.err)) {
          const Real* qn = qin + (int64_t)nb * 6 * Np + np2;
#pragma unroll
          for (int c = 0; c < 6; ++c) X[r][k][c] = qn[c * Np];
        }
      }
    }
    landed = tc::mbar_wait_sleep(mb, phase & 1) && landed;
    ahead = false;
    if (!__syncthreads_and(landed)) { failed = true; break; }
    // every thread is past its wait for this tile's faces (a phase completed
    // while a thread still waited for the one before would be lost on it): the
    // next tile's may come
    ahead = nx < ntiles;
    if (ahead && tid == 0) faces_in(nx, fb ^ 1);
    for (int s = tid; s < P.nsrc; s += NT) {
      const SrcDev& sd = P.src[s];
      if (sd.batch == b && sd.elem >= eg0 && sd.elem < eg0 + ne) {
        atomicAdd(&nsl, 1);
        atomicMin(&src0, s);
      }
    }

    // ---- upwind flux at the orbit's nodes, adapted sums over them (FP64: two
    // shuffles and a signed sum per value)
#pragma unroll
    for (int r = 0; r < FR; ++r) {
      const int idx = tid + r * NT;
      const bool act = idx < ne * Nfp * (4 / FO);
      // (with shuffles a warp goes on while any of its lanes has a task)
      if (FO == 4 ? !act : (idx & ~31) >= ne * Nfp * 4) continue;
      const int em = act ? idx / (4 / FO) : 0, y0 = FO == 4 ? 0 : idx & 3;
      const int e = em / Nfp, m = em - e * Nfp;
      const Real* qe = QS + e * 6 * Np;
#pragma unroll
      for (int k = 0; k < FO; ++k) {
        const int y = y0 + k, f = y < 2 ? y : 5 - y, ni = t_fn[m * 4 + y];
        const Real* fc = FC + (e * 4 + f) * 8;
        // perfect electric conductor: mirror state E+ = -E-, H+ = H-
        const bool pec = nbr[e * 4 + f] < 0;
        const Real nx = fc[0], ny = fc[1], nz = fc[2];
        const Real c3 = fc[3], c4 = fc[4], c5 = fc[5], c6 = fc[6];
        Real d[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          const Real v = qe[c * Np + ni];
          d[c] = (pec ? (c < 3 ? -v : v) : X[r][k][c]) - v;
        }
        const Real ndE = nx * d[0] + ny * d[1] + nz * d[2];
        const Real ndH = nx * d[3] + ny * d[4] + nz * d[5];
        X[r][k][0] = c3 * (ny * d[5] - nz * d[4]) - c4 * (nx * ndE - d[0]);
        X[r][k][1] = c3 * (nz * d[3] - nx * d[5]) - c4 * (ny * ndE - d[1]);
        X[r][k][2] = c3 * (nx * d[4] - ny * d[3]) - c4 * (nz * ndE - d[2]);
        X[r][k][3] = c5 * (ny * d[2] - nz * d[1]) + c6 * (nx * ndH - d[3]);
        X[r][k][4] = c5 * (nz * d[0] - nx * d[2]) + c6 * (ny * ndH - d[4]);
        X[r][k][5] = c5 * (nx * d[1] - ny * d[0]) + c6 * (nz * ndH - d[5]);
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        Real* fl = FL + (e * 2 + c / 3) * FST + (c % 3) * NF + m;
        if constexpr (FO == 4) {
          Fly<Real, N, 4>::had4(X[r][0][c], X[r][1][c], X[r][2][c], X[r][3][c]);
#pragma unroll
          for (int x = 0; x < 4; ++x) fl[x * Nfp] = X[r][x][c];
        } else {
          // lane y: after the exchanges with y xor 1 and y xor 2 it holds the
          // signed sum (-1)^(y . z) over z, the character `ch` of its y
          Real v = X[r][0][c];
          const Real p = __shfl_xor_sync(0xffffffffu, v, 1);
          v = y0 & 1 ? p - v : v + p;
          const Real q = __shfl_xor_sync(0xffffffffu, v, 2);
          v = y0 & 2 ? q - v : v + q;
          const int ch = y0 == 0 ? 0 : (y0 == 1 ? 2 : (y0 == 2 ? 1 : 3));
          if (act) fl[ch * Nfp] = v;
        }
      }
    }
    // ---- E and H adapted: in FP64 their covariant components u_a = X_a . F
    // (fewer FP64 operations), in FP32 the Cartesian ones.  The derivatives of
    // a constant vanish, so each component is taken relative to its value at
    // the node nearest the centroid: the adapted sums then round at the size
    // of the field's variation over the element instead of the field's own
    // (without it the FP32 curl's error is half as large again at N = 3, and
    // two and a half times at N = 4).
    constexpr bool COV = sizeof(Real) == 8;
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
        for (int a = 0; a < 3; ++a)
          v[a][y] = COV ? g[a] * f0 + g[3 + a] * f1 + g[6 + a] * f2 : (a == 0 ? f0 : a == 1 ? f1 : f2);
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
          const Real p = COV ? g[a] * f0 + g[3 + a] * f1 + g[6 + a] * f2 : (a == 0 ? f0 : a == 1 ? f1 : f2);
          const Real r = COV ? g[a] * h0 + g[3 + a] * h1 + g[6 + a] * h2 : (a == 0 ? h0 : a == 1 ? h1 : h2);
          u[a * Np + B::NFul + o] = one ? p : p + r;
          if (!one) u[a * Np + B::off(1) + o * B::D1 + B::NFul] = p - r;
        }
      }
    }
    __syncthreads();

    const int sb0 = src0, sb1 = sb0 + nsl;   // the tile's sources
    // ---- curl and LIFT in adapted values; results stay in registers until
    // every thread has read U, which then holds them: [TE][E, H][3][Np]
    // FP64: one row per task (the FP64 pipe bounds it, so the finest split
    // balances best); FP32: all rows of a character, for fewer loads per
    // multiplication, one character per warp
    if constexpr (sizeof(Real) == 8) {
      if (sb1 > sb0 && tid < 32) sym_currents(P.src, sb0, sb1, eg0, tst, GX, cur);
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
      // warps 0-3: characters 0-3, a lane per (element, field)
      static_assert(2 * ST::T <= 32, "a warp holds the tile's rows of a character");
      const int x = (tid >> 5) & 3, ef = tid & 31, f = ef & 1;
      const bool act = tid < 128 && ef < 2 * ne;
      const int r = act ? ef : 0;   // spare lanes repeat row 0 and write nothing
      const Real* g = GX + (r >> 1) * 12;
      const Real sc = f ? g[10] : -g[11];
      Real* out = act ? U + (ef ^ 1) * UST : nullptr;
      const Real* uu = U + r * UST;
      const Real* ff = FL + (r ^ 1) * FST;
      if (tid >= 128) {
        if (sb1 > sb0 && tid < 160) sym_currents(P.src, sb0, sb1, eg0, tst, GX, cur);
        __syncthreads();
      } else if (x == 0) {
        sym_curl_pairs<N, 0, ST::CC>(ops, 0, uu, ff, g, sc, out);
      } else {
        sym_curl_pairs<N, 1, ST::CC>(ops, x, uu, ff, g, sc, out);
      }
    }
    __syncthreads();
    if (sb1 > sb0)
      sym_sources<Real, Np, UST, NT>(P.src, P.src_ws, sb0, sb1, eg0, tst, GX, cur, U);

    if constexpr (!PML) {
      // ---- back to nodal values, in place
      for (int idx = tid; idx < ne * 6; idx += NT) {
        Real* u = U + (idx / 3) * UST + (idx % 3) * Np;
        Real t[Np];
#pragma unroll
        for (int i = 0; i < Np; ++i) t[i] = u[i];
        Fly<Real, N, 4>::inverse(t, [&](int n, Real v) { u[n] = v; });
      }
    } else if constexpr (ST::BOTH) {
      // ---- eqs. 26-29.  Thread (half, e, c): component c of E,H and of P.  The
      // first half interpolates and applies eq. 9 to CG groups of points while
      // the second projects the CG groups before
      constexpr int HT = NT / 2, CG = ST::CG;
      const int half = tid / HT, row = tid - half * HT, R = TE * 6;
      const int e = row / 6, c = row - e * 6;
      const bool on = row < R;
      const int u = c % 3, v_ = (u + 1) % 3, w_ = (u + 2) % 3;
      constexpr int VW = Np % 4 == 0 ? 4 : (Np % 2 == 0 ? 2 : 1);
      const float* Vc = ST::VC ? C.v : ops + ST::oV;
      const float* Pc = ST::VC ? C.p : Vc + ng * CP;
      const Real* sg = SG + e * ng * 12;
      Real* rq = U + (e * 2 + c / 3) * UST + u * Np;   // adapted curl and LIFT
      Real* tz = FL + row;                             // [2][CG][8][R]
      constexpr int NP2 = Blocks<N, G>::PO / 2;
      pair2 a[NP2], b_[NP2];   // first half: adapted rows; second half: sums
#pragma unroll
      for (int i = 0; i < NP2; ++i) a[i] = b_[i] = 0;
      if (on && !half) {
        Real f[Np], s[Np];
        load_row<Np, VW>(QS + row * Np, f);
        Fly<Real, N, G>::forward(f, s);
        to_pairs<N, G>(s, a);
        load_row<Np, VW>(PQ + row * Np, f);
        Fly<Real, N, G>::forward(f, s);
        to_pairs<N, G>(s, b_);
      }
      const int nk = (ng + CG - 1) / CG;
#pragma unroll 1
      for (int k = 0; k <= nk; ++k) {
        if (on && !half) {
#pragma unroll 1
          for (int g = k * CG; g < min(ng, (k + 1) * CG); ++g) {
            Real v[4], o[4], su[4], sv[4], sw[4];
            sym_interp2<N, G, ST::VC>(Vc + g * CP, a, b_, v, o);
            lds4(sg + g * 12 + u * 4, su);
            lds4(sg + g * 12 + v_ * 4, sv);
            lds4(sg + g * 12 + w_ * 4, sw);
            if constexpr (!KAPPA) {
              // eq. 9 with kappa = 1 (samples are sigma / eps0): a = 1,
              // b = sv + sw - su, c = sv sw - b su, d = su
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const Real bc = sv[i] + sw[i] - su[i];
                const Real cc = sv[i] * sw[i] - bc * su[i];
                const Real t = bc * v[i] + cc * o[i];
                o[i] = v[i] - su[i] * o[i];
                v[i] = t;
              }
            } else {
              Real ku[4], kv[4], kw[4];
              const Real* kp = sg + TE * ng * 12 + g * 12;
              lds4(kp + u * 4, ku);
              lds4(kp + v_ * 4, kv);
              lds4(kp + w_ * 4, kw);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const Real ki = Real(1) / ku[i];
                const Real aa = kv[i] * kw[i] * ki;
                const Real bc = (sv[i] * kw[i] + sw[i] * kv[i] - aa * su[i]) * ki;
                const Real cc = sv[i] * sw[i] - bc * su[i];
                const Real t = bc * v[i] + cc * o[i];
                o[i] = ki * v[i] - su[i] * ki * o[i];
                v[i] = t;
              }
            }
            Real* z = tz + ((k & 1) * CG + g - k * CG) * 8 * R;
#pragma unroll
            for (int x = 0; x < 4; x += G) {
              Fly<Real, N, G>::group(v + x);
              Fly<Real, N, G>::group(o + x);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              z[i * R] = v[i];
              z[(4 + i) * R] = o[i];
            }
          }
        } else if (on && k > 0) {
#pragma unroll 1
          for (int g = (k - 1) * CG; g < min(ng, k * CG); ++g) {
            const Real* z = tz + (((k - 1) & 1) * CG + g - (k - 1) * CG) * 8 * R;
            Real v[4], o[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              v[i] = z[i * R];
              o[i] = z[(4 + i) * R];
            }
            sym_add2<N, G, ST::VC>(Pc + g * CP, v, o, a, b_);
          }
        }
        __syncthreads();
      }
      if (on && half) {
        Real* xp = FL + row * Np;   // every point value is spent
        Real t[Np], d[Np];
        from_pairs<N, G>(b_, d);
        Fly<Real, N, G>::inverse(d, [&](int n, Real v) { xp[n] = v; });
        from_pairs<N, G>(a, d);
#pragma unroll
        for (int i = 0; i < Np; ++i) t[i] = rq[i];
        if constexpr (G == 4) {
#pragma unroll
          for (int i = 0; i < Np; ++i) t[i] -= d[i];
          if constexpr (!KAPPA) {
            Fly<Real, N, 4>::inverse(t, [&](int n, Real v) { rq[n] = v; });
          } else {
            sym_to_sums<Real, N>(t);
#pragma unroll
            for (int i = 0; i < Np; ++i) rq[i] = t[i];
          }
        } else {
          Real f[Np];
          Fly<Real, N, G>::inverse(d, [&](int n, Real v) { f[n] = v; });
          Fly<Real, N, 4>::inverse(t, [&](int n, Real v) { f[n] = v - f[n]; });
          if constexpr (KAPPA) {
            Fly<Real, N, G>::forward(f, t);
#pragma unroll
            for (int i = 0; i < Np; ++i) f[i] = t[i];
          }
#pragma unroll
          for (int i = 0; i < Np; ++i) rq[i] = f[i];
        }
      }
      if constexpr (KAPPA) {
        // P_q a^-1 V_q of the E,H rows (their adapted sums are in rq), the two
        // halves of the block sharing each row's groups; the second half's
        // sums pass through the sigma buffer, which is spent
        __syncthreads();
        Real* xf = SG + row * Np;
        static_assert(!PML || 6 * Np <= 2 * 12 * ST::NG, "exchange rows");
        Real s[Np], d[Np];
#pragma unroll
        for (int i = 0; i < Np; ++i) {
          s[i] = on ? rq[i] : Real(0);
          d[i] = 0;
        }
        if (on) {
#pragma unroll 1
          for (int g = half; g < ng; g += 2) {
            Real v[4], ku[4], kv[4], kw[4];
            sym_interp<Real, N, G>(Vc + g * CP, s, v);
            const Real* kp = sg + TE * ng * 12 + g * 12;
            lds4(kp + u * 4, ku);
            lds4(kp + v_ * 4, kv);
            lds4(kp + w_ * 4, kw);
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] *= ku[i] / (kv[i] * kw[i]);
            sym_project<Real, N, G>(Pc + g * CP, v, d);
          }
        }
        __syncthreads();
        if (on && half) {
#pragma unroll
          for (int i = 0; i < Np; ++i) xf[i] = d[i];
        }
        __syncthreads();
        if (on && !half) {
#pragma unroll
          for (int i = 0; i < Np; ++i) d[i] += xf[i];
          Fly<Real, N, G>::inverse(d, [&](int n, Real v) { rq[n] = v; });
        }
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
        const Real* Vc = ops + ST::oV;
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
        Real* rp = FL + (e * 6 + c) * Np;                     // the flux is spent
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
          if constexpr (G == 4) sym_to_sums<Real, N>(s);   // role 0 holds the row
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
    // ---- Runge-Kutta update, two consecutive values per task; a thread's
    // register values are all loaded before the barrier, so that their latency
    // is paid once per tile (one load and store at a time: 9,500 of the 32,000
    // cycles of a PML tile at N = 4)
    constexpr int UT = (ST::T * 3 * Np + NT - 1) / NT;   // tasks of a thread
    const int nu = ne * 3 * Np;
    Real r1[UT][2], r2[PML ? UT : 1][2];
#pragma unroll
    for (int k = 0; k < UT; ++k)
      if (tid + k * NT < nu) {
        lds2(P.resq + oq + 2 * (tid + k * NT), r1[k]);
        if constexpr (PML) lds2(P.resp + op + 2 * (tid + k * NT), r2[k]);
      }
    __syncthreads();
    Real* pout = P.pout ? P.pout : P.p;
#pragma unroll
    for (int k = 0; k < UT; ++k) {
      const int li = 2 * (tid + k * NT);
      if (li >= 2 * nu) continue;
      const Real* r = U + li + li / (3 * Np) * (UST - 3 * Np);
      Real q[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        r1[k][i] = rka * r1[k][i] + rdt * r[i];
        q[i] = QS[li + i] + rkb * r1[k][i];
      }
      sts2(P.resq + oq + li, r1[k]);
      sts2(P.qout + oq + li, q);
      if constexpr (PML) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          r2[k][i] = rka * r2[k][i] + rdt * FL[li + i];
          q[i] = PQ[li + i] + rkb * r2[k][i];
        }
        sts2(P.resp + op + li, r2[k]);
        sts2(pout + op + li, q);
      }
    }
  }
  if (failed && tid == 0) {
    // a copy that did not land in time: report it, and wait once more (bounded)
    // so that it does not land in memory given away
    atomicExch(P.err, 1);
    tc::mbar_wait_sleep(mb, phase & 1);
    tc::mbar_wait_sleep(mf, phase & 1);
    if (ahead) tc::mbar_wait_sleep(mf, (phase & 1) ^ 1);
  }
  __syncthreads();
  if (tid == 0) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mb) : "memory");
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mf) : "memory");
  }
  __syncthreads();
  return !failed;
}

}  // namespace wadg
