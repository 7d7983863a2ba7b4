// Reverse Runge-Kutta stage (adjoint.cu's definitions) in FP32 with the
// reference operators in the block form of sym_tables.hpp.  The transposes act
// on adapted values as the operators do (A^T g has the sums of g as input and
// the same butterflies), so LIFT^T, curl^T, P_q^T and V_q^T take a quarter of
// the dense products' multiplications (V_q^T, P_q^T half for a conical rule).
//
// The dense kernel spent its time on those products (PML class, N = 3: 379 us a
// launch on 48,000 elements) and on the forward curl of H for dJ/deps_k.  That
// term needs no forward derivative: with a_E = mu_E / eps,
//   <a_E, curl H + LIFT f> = <curl^T a_E, H> + <LIFT^T a_E, f>,
// and both transposes are at hand.  What bounds it now: the gathers of the
// traces and the phases' barriers, as the forward stage.  Gradient of 40 steps,
// 82,944 tets, N = 3: 193 -> 130 ms with these kernels (and one allocation for
// the call's states instead of two hundred); 303 ms with the dense forward
// stage as well.
#include "sym_body.cuh"

namespace wadg {

namespace {

constexpr int kSaThreads = 192;

// shared-memory plan in floats, per tile of T elements
template <int N, int G>
struct SaTile {
  using B = Blocks<N, 4>;
  using L = SymLayout<N>;
  static constexpr int Np = B::Np, Nfp = L::Nfp, NF = 4 * Nfp;
  static constexpr bool PML = G != 0;
  static constexpr int NG = PML ? sym_groups(N, G) : 0, CP = PML ? sym_cp(N, G) : 0;
  static constexpr int UST = 3 * Np | 1;
  static constexpr int DT = L::oL;            // transposed derivative blocks
  // Low parts of P_q's coefficients (what FP32 rounds off), in the place of the
  // derivative blocks once these are spent.  A V4 rule's P_q has a few hundred
  // coefficients, whose roundings every element repeats, so that they add up over
  // a mesh in the profile derivatives: median relative error of dJ/dsigma_max, N =
  // 4, 16,464 tets, 8.3e-7 without the low parts, 3.8e-7 with them, 3.3e-7 in the
  // dense kernel with its 48 times 35 coefficients (N = 5, 6,000 tets: 3.3e-6,
  // 2.3e-6, 2.3e-6).  A gradient takes 1.2 % longer for them (N = 3, 82,944
  // tets, 40 steps: 129.9 -> 131.5 ms).  Z2 rules have several times as many
  // coefficients and the dense kernel's errors.
  static constexpr int LO = G == 4 ? NG * CP : 0, LOT = (LO + kSaThreads - 1) / kSaThreads;
  static_assert(LO <= DT, "low parts of P_q");
  static constexpr int TAB = 8 * Nfp + 4 * B::NFul + 8 + 3 * Np;
  static constexpr int tabB = (TAB + NF + 192 * Nfp + 15) & ~15;
  WADG_HD static constexpr int al(int x) { return (x + 3) & ~3; }
  WADG_HD static constexpr int cov(int te) { return al(te * 6 * Np) + 4; }
  WADG_HD static constexpr int floats(int te) {
    return al(DT) + (PML ? 2 : 1) * (cov(te) + al(te * 6 * Np)) + te * (12 + 32) +
           al(te * 2 * UST) + al(te * 6 * NF) + te * NG * 12 + te * NG * 48 + al(te);
  }
  WADG_HD static constexpr size_t bytes(int te) {
    return (size_t)floats(te) * 4 + te * 16 + tabB + 64;
  }
  static constexpr int fit() {   // two blocks per SM; one where four elements need it
    for (int t = 16; t > 4; --t)
      if (bytes(t) <= 113 * 1024) return t;
    for (int t = 16; t > 1; --t)
      if (bytes(t) <= 226 * 1024) return t;
    return 1;
  }
  static constexpr int T = fit();
  static constexpr int min_blocks = bytes(T) <= 113 * 1024 ? 2 : 1;
};

// ------------------------------------------------------------------- lift
template <int N>
struct SaLift {
  using B = Blocks<N, 4>;
  using L = SymLayout<N>;
  static constexpr int Np = B::Np, Nfp = L::Nfp, NF = 4 * Nfp, RM = (Nfp + 3) & ~3;
  static constexpr int LT = Np * RM;          // LIFT^T blocks: [character][i][RM]
  static constexpr int UST = 3 * Np | 1, FST = 3 * NF | 1;
  static constexpr int T = N == 5 ? 8 : 16, NT = 128;
  static constexpr int TAB = 8 * Nfp + 4 * B::NFul + 8;
  static constexpr size_t bytes =
      (size_t)(LT + ((T * 6 * Np + 3) & ~3) + ((T * 2 * UST + 3) & ~3) + T * 2 * FST) * 4 + TAB;
};

// adapted sums of the rows [e][6][Np] in `rows`, per (element, field, orbit),
// into u [e * 2 + field][3][Np] (element stride 2 UST)
template <int N, int UST>
__device__ __forceinline__ void adapt_rows(const float* rows, const unsigned char* t_or, float* u,
                                           int ne, int tid, int nt) {
  using B = Blocks<N, 4>;
  constexpr int Np = B::Np;
  for (int idx = tid; idx < ne * 6 * B::NFul; idx += nt) {
    const int row = idx / B::NFul, o = idx - row * B::NFul;
    const float* q = rows + row * Np;
    float* d = u + (row / 3) * UST + (row % 3) * Np + o;
    float v[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) v[y] = q[t_or[4 * o + y]];
    Fly<float, N, 4>::had4(v[0], v[1], v[2], v[3]);
#pragma unroll
    for (int x = 0; x < 4; ++x) d[B::off(x)] = v[x];
  }
  if constexpr (B::NH + B::NS > 0) {
    constexpr int NR = 3 * B::NH + B::NS;
    for (int idx = tid; idx < ne * 6 * NR; idx += nt) {
      const int row = idx / NR, o = idx - row * NR;
      const float* q = rows + row * Np;
      float* d = u + (row / 3) * UST + (row % 3) * Np;
      const bool one = o == 3 * B::NH;
      const float p = q[t_or[4 * B::NFul + 2 * o]];
      const float r = one ? 0.f : q[t_or[4 * B::NFul + 2 * o + 1]];
      d[B::NFul + o] = p + r;
      if (!one) d[B::off(1) + o * B::D1 + B::NFul] = p - r;
    }
  }
}

// G[b][e][fm][0..2] = Fscale LIFT^T (mu_E / eps), [3..5] = Fscale LIFT^T (-mu_H / mu)
template <int N>
__global__ void __launch_bounds__(SaLift<N>::NT) sym_lift_kernel(const AdjParams<float> A) {
  using SL = SaLift<N>;
  using B = Blocks<N, 4>;
  constexpr int Np = SL::Np, Nfp = SL::Nfp, NF = SL::NF, T = SL::T, NT = SL::NT, RM = SL::RM;
  constexpr int UST = SL::UST, FST = SL::FST;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* ops = reinterpret_cast<float*>(smem_raw);          // LIFT^T blocks
  float* rows = ops + SL::LT;                               // [T][6][Np]
  float* U = rows + ((T * 6 * Np + 3) & ~3);                // [T][2][UST]
  float* FA = U + ((T * 2 * UST + 3) & ~3);                 // [T][2][FST]: [3][character][Nfp]
  unsigned char* tab = reinterpret_cast<unsigned char*>(FA + T * 2 * FST);
  const int tid = threadIdx.x, b = blockIdx.y, e0 = blockIdx.x * T;
  const int ne = min(T, A.K - e0);
  const float* src = A.symadj + SymLayout<N>::oL;
  for (int i = tid; i < SL::LT; i += NT) ops[i] = src[i];
  for (int i = tid; i < SL::TAB; i += NT) tab[i] = A.symtab[i];
  const int64_t o = (int64_t)b * A.strideQ + (int64_t)e0 * 6 * Np;
  for (int idx = tid; idx < ne * 3 * Np; idx += NT) {
    const int li = 2 * idx;
    float r[2], l[2];
    lds2(A.rho_q + o + li, r);
    lds2(A.lam_q + o + li, l);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int e = (li + k) / (6 * Np), c = (li + k - e * 6 * Np) / Np;
      const float s = c < 3 ? A.geox[(int64_t)(e0 + e) * 12 + 10] : -A.geox[(int64_t)(e0 + e) * 12 + 11];
      rows[li + k] = (r[k] + A.rk_b_r * l[k]) * s;
    }
  }
  __syncthreads();
  adapt_rows<N, UST>(rows, tab + 8 * Nfp, U, ne, tid, NT);
  __syncthreads();
  for (int t = tid; t < 8 * 16; t += NT) {   // (character, element, field): one character per warp
    const int x = t >> 5, ef = t & 31;
    if (ef >= 2 * ne) continue;
    const float* u = U + ef * UST + B::off(x);
    const float* c = ops + B::off(x) * RM;
    pair2 w[3][RM / 2];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int m = 0; m < RM / 2; ++m) w[k][m] = 0;
    for (int i = 0; i < B::dim(x); ++i) {
      pair2 k2[RM / 2];
      load_pairs<RM / 2, false>(c + i * RM, k2);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const pair2 v = pack2(u[k * Np + i], u[k * Np + i]);
#pragma unroll
        for (int m = 0; m < RM / 2; ++m) fma2(w[k][m], k2[m], v);
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int m = 0; m < RM / 2; ++m) {
        float p, q;
        unpack2(w[k][m], p, q);
        float* d = FA + ef * FST + k * NF + x * Nfp + 2 * m;
        if (2 * m < Nfp) d[0] = p;
        if (2 * m + 1 < Nfp) d[1] = q;
      }
  }
  __syncthreads();
  float* Gb = A.G + ((int64_t)b * A.K + e0) * NF * 6;
  for (int idx = tid; idx < ne * Nfp; idx += NT) {
    const int e = idx / Nfp, m = idx - e * Nfp;
    float v[6][4];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const float* d = FA + (e * 2 + c / 3) * FST + (c % 3) * NF + m;
#pragma unroll
      for (int x = 0; x < 4; ++x) v[c][x] = d[x * Nfp];
      Fly<float, N, 4>::had4(v[c][0], v[c][1], v[c][2], v[c][3]);
    }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int f = y < 2 ? y : 5 - y;
      const float s = A.fnrm[(int64_t)(e0 + e) * 16 + f * 4 + 3];
      float* g = Gb + ((int64_t)e * NF + tab[4 * m + y]) * 6;
#pragma unroll
      for (int c = 0; c < 6; c += 2) {
        const float p[2] = {s * v[c][y], s * v[c + 1][y]};
        sts2(g + c, p);
      }
    }
  }
}

// ------------------------------------------------------------------- main
// curl^T of one field of one element for the output rows of character y (Y: 0,
// or 1 for any other): sum_a D_a^T a x g_a, a's adapted sums in u; the block's
// barrier is inside, since the results take u's place
template <int N, int Y>
__device__ __forceinline__ void sym_curlt_pairs(const float* ops, int y, const float* u,
                                                const float* gx, float* out) {
  using L = SymLayout<N>;
  using B = Blocks<N, 4>;
  constexpr int Np = B::Np, RW = B::dim(Y), R2 = (RW + 1) / 2;
  const int rp = L::RP(Y);
  pair2 w[3][R2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < R2; ++r) w[c][r] = 0;
  const float* D = ops + (Y ? L::DX0 + (y - 1) * L::DX1 : 0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int xi = y ^ (a + 1), ni = Y ? B::dim(xi) : B::D1;
    const float* f = u + B::off(xi);
    pair2 d[3][R2];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < R2; ++r) d[c][r] = 0;
#pragma unroll 4
    for (int i = 0; i < ni; ++i) {
      pair2 k[R2];
      load_pairs<R2, false>(D + i * rp, k);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const pair2 v = pack2(f[c * Np + i], f[c * Np + i]);
#pragma unroll
        for (int r = 0; r < R2; ++r) fma2(d[c][r], k[r], v);
      }
    }
    D += ni * rp;
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
      for (int c = 0; c < 3; ++c) {   // (d x g)_c
        fma2(w[c][r], d[(c + 1) % 3][r], g[(c + 2) % 3]);
        fma2(w[c][r], d[(c + 2) % 3][r], m[(c + 1) % 3]);
      }
  }
  __syncthreads();
  if (out) {
    out += B::off(Y ? y : 0);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < R2; ++r) {
        float p, q;
        unpack2(w[c][r], p, q);
        out[c * Np + 2 * r] = p;
        if (2 * r + 1 < RW) out[c * Np + 2 * r + 1] = q;
      }
  }
}

template <int N, int G>
__global__ void __launch_bounds__(kSaThreads, SaTile<N, G>::min_blocks)
sym_adj_kernel(const AdjParams<float> A,
               const __grid_constant__ SymCoef<SaTile<N, G>::PML ? SaTile<N, G>::NG * SaTile<N, G>::CP : 1> C) {
  using ST = SaTile<N, G>;
  using B = Blocks<N, 4>;
  using L = SymLayout<N>;
  constexpr int Np = ST::Np, Nfp = ST::Nfp, NF = ST::NF, UST = ST::UST, NT = kSaThreads;
  constexpr bool PML = ST::PML;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int TE = A.tile;
  const int ng = A.nsl / 4;
  float* ops = reinterpret_cast<float*>(smem_raw);          // transposed derivative blocks
  float* QB = ops + ST::al(ST::DT);                         // stage input E,H (cover)
  float* PB = QB + ST::cov(TE);                             // P (cover), later its adjoint
  float* MQ = QB + (PML ? 2 : 1) * ST::cov(TE);             // mu [TE][6][Np]
  float* MP = MQ + ST::al(TE * 6 * Np);
  float* GX = MQ + (PML ? 2 : 1) * ST::al(TE * 6 * Np);     // [TE][12] metric, 1/eps, 1/mu
  float* FC = GX + TE * 12;                                 // [TE][4][8]
  float* U = FC + TE * 32;                                  // [TE][2][UST]
  float* X = U + ST::al(TE * 2 * UST);                      // [TE][6][NF] transposed traces
  float* SG = X + ST::al(TE * 6 * NF);                      // [TE][ng][3][4]
  float* ZV = SG + TE * ST::NG * 12;                        // [ng][8][6 TE] point values
  float* GE = ZV + TE * ST::NG * 48;                        // [TE] dJ/deps_k
  int* nbr = reinterpret_cast<int*>(smem_raw + (size_t)ST::floats(TE) * 4);
  unsigned char* tab = reinterpret_cast<unsigned char*>(nbr + TE * 4);
  uint64_t* bar = reinterpret_cast<uint64_t*>(tab + ST::tabB);
  const unsigned char* t_or = tab + 8 * Nfp;
  const unsigned char* t_nf = tab + 8 * Nfp + 4 * B::NFul + 8;   // [Np][3] face nodes, NF: none
  const unsigned char* Fmask = tab + ST::TAB;
  const unsigned char* fperm = Fmask + NF;
  const unsigned char* fmap = fperm + 96 * Nfp;
  __shared__ int nsl, src0;   // the tile's sources: count, first of the table
  __shared__ double red[6][NT / 32];
  const int tid = threadIdx.x;
  const uint32_t mb = tc::saddr(bar);
  const int tiles_per_batch = (A.n_elem + TE - 1) / TE;
  const int tile = blockIdx.x;
  const int b = tile / tiles_per_batch, t0 = (tile - b * tiles_per_batch) * TE;
  const int ne = min(TE, A.n_elem - t0);
  const int eg0 = A.e_begin + t0, ep0 = eg0 - A.K0;
  const int64_t oq = (int64_t)b * A.strideQ + (int64_t)eg0 * 6 * Np;
  const int64_t op = (int64_t)b * A.strideP + (int64_t)ep0 * 6 * Np;
  const float* qin = A.q_in + (int64_t)b * A.strideQ;
  const float* Gb = A.G + (int64_t)b * A.K * NF * 6;
  const float* QS = QB + (reinterpret_cast<uintptr_t>(A.q_in + oq) & 15) / 4;
  float* PQ = PML ? PB + (reinterpret_cast<uintptr_t>(A.p_in + op) & 15) / 4 : nullptr;
  if (tid == 0) {
    tc::mbar_init(mb, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    nsl = 0;
    src0 = A.nsrc;
    const void* src[6] = {A.nbr + (int64_t)eg0 * 4, A.facex + (int64_t)eg0 * 32, A.q_in + oq,
                          A.geox + (int64_t)eg0 * 12, nullptr, nullptr};
    uint32_t len[6] = {(uint32_t)ne * 16, (uint32_t)ne * 128, (uint32_t)(ne * 6 * Np * 4),
                       (uint32_t)ne * 48, 0, 0};
    uint32_t dst[6] = {tc::saddr(nbr), tc::saddr(FC), tc::saddr(QB), tc::saddr(GX), 0, 0};
    int n = 4;
    if constexpr (PML) {
      src[n] = A.p_in + op; len[n] = len[2]; dst[n++] = tc::saddr(PB);
      src[n] = A.sig + (int64_t)ep0 * ng * 12; len[n] = (uint32_t)ne * ng * 48;
      dst[n++] = tc::saddr(SG);
    }
    uint32_t total = wadg_take_request(A.inject, kRequestReverse) ? 16 : 0;
    for (int a = 0; a < n; ++a) {
      const uint32_t lo = (uint32_t)(reinterpret_cast<uintptr_t>(src[a]) & 15);
      len[a] = (lo + len[a] + 15) & ~15u;
      src[a] = static_cast<const unsigned char*>(src[a]) - lo;
      total += len[a];
    }
    tc::mbar_expect_tx(mb, total);
    for (int a = 0; a < n; ++a) tc::bulk_g2s(dst[a], src[a], len[a], mb);
  }
  for (int i = tid; i < ST::DT; i += NT) ops[i] = A.symadj[i];
  float low[ST::LOT ? ST::LOT : 1];
#pragma unroll
  for (int k = 0; k < ST::LOT; ++k) {
    const int i = tid + k * NT;
    low[k] = i < ng * ST::CP ? A.symadj[L::oL + Np * ((Nfp + 3) & ~3) + i] : 0.f;
  }
  for (int i = tid; i < ST::TAB; i += NT) tab[i] = A.symtab[i];
  for (int i = tid; i < NF + 192 * Nfp; i += NT) tab[ST::TAB + i] = A.tabs[i];
  for (int i = tid; i < TE; i += NT) GE[i] = 0.f;
  // ---- mu = rho + B lambda
  for (int idx = tid; idx < ne * 3 * Np; idx += NT) {
    float r[2], l[2];
    lds2(A.rho_q + oq + 2 * idx, r);
    lds2(A.lam_q + oq + 2 * idx, l);
    MQ[2 * idx] = r[0] + A.rk_b_r * l[0];
    MQ[2 * idx + 1] = r[1] + A.rk_b_r * l[1];
    if constexpr (PML) {
      lds2(A.rho_p + op + 2 * idx, r);
      lds2(A.lam_p + op + 2 * idx, l);
      MP[2 * idx] = r[0] + A.rk_b_r * l[0];
      MP[2 * idx + 1] = r[1] + A.rk_b_r * l[1];
    }
  }
  __syncthreads();   // the barrier and the tables are there
  const bool landed = tc::mbar_wait_sleep(mb, 0);
  if (!__syncthreads_and(landed)) {
    if (tid == 0) {
      atomicExch(A.err, 1);
      tc::mbar_wait_sleep(mb, 0);
    }
    return;
  }
  for (int s = tid; s < A.nsrc; s += NT) {
    const SrcDev& sd = A.src[s];
    if (sd.batch == b && sd.elem >= eg0 && sd.elem < eg0 + ne) {
      atomicAdd(&nsl, 1);
      atomicMin(&src0, s);
    }
  }
  // ---- traces: the transposed upwind flux of both sides of each face node,
  // and the flux terms of dJ/deps_k (alpha = 1; h = 1/(Z- + Z+))
  for (int idx = tid; idx < ne * NF; idx += NT) {
    const int e = idx / NF, fm = idx - e * NF, f = fm / Nfp, m = fm - f * Nfp;
    const int ni = Fmask[fm], nb = nbr[e * 4 + f];
    const float* fc = FC + (e * 4 + f) * 8;
    const float n[3] = {fc[0], fc[1], fc[2]};
    const float* qe = QS + e * 6 * Np + ni;
    const float* g1 = Gb + ((int64_t)(eg0 + e) * NF + fm) * 6;
    float gH[3], gE[3], gH2[3] = {0, 0, 0}, gE2[3] = {0, 0, 0}, dE[3], dH[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      gH[c] = g1[c];
      gE[c] = g1[3 + c];
    }
    if (nb >= 0) {
      const int code = (int)fc[7], k = (f * 24 + code) * Nfp + m;
      const float* qn = qin + (int64_t)nb * 6 * Np + fperm[k];
      const float* g2 = Gb + ((int64_t)nb * NF + (code / 6) * Nfp + fmap[k]) * 6;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dE[c] = qn[c * Np] - qe[c * Np];
        dH[c] = qn[(3 + c) * Np] - qe[(3 + c) * Np];
        gH2[c] = g2[c];
        gE2[c] = g2[3 + c];
      }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dE[c] = -2.f * qe[c * Np];
        dH[c] = 0.f;
      }
    }
    // fc[3..6] are Fscale times Z+ h, h, Z- h, Z- Z+ h; Fscale is in g already
    const float is = 1.f / (fc[3] + fc[5]);   // Z+ h + Z- h = 1
    const float zp = fc[3] * is, h = fc[4] * is, zm = fc[5] * is, zz = fc[6] * is;
    const float ndE = n[0] * dE[0] + n[1] * dE[1] + n[2] * dE[2];
    const float ndH = n[0] * dH[0] + n[1] * dH[1] + n[2] * dH[2];
    float nxdE[3], nxdH[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int p = (c + 1) % 3, q = (c + 2) % 3;
      nxdE[c] = n[p] * dE[q] - n[q] * dE[p];
      nxdH[c] = n[p] * dH[q] - n[q] * dH[p];
    }
    const float ie = GX[e * 12 + 10];
    const float ZM = fc[6] / fc[3];             // Z- Z+ h / (Z+ h)
    const float dZ = -0.5f * ZM * ie, dY = 0.5f * ie / ZM;
    float ge = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float tE = n[c] * ndE - dE[c], tH = n[c] * ndH - dH[c];
      const float fCH = zp * nxdH[c] - h * tE, fCE = zm * nxdE[c] + zz * tH;
      // d/deps_k of mu_E . LIFT f / eps_k, then through Z- and Y-
      ge -= gH[c] * fCH * (ie + h * dZ) + gE[c] * fCE * (zz * dY);
      if (nb >= 0) {   // the neighbour's flux: normal -n, jumps -dE, -dH, its Z+ is Z_k
        const float fCH2 = zm * nxdH[c] + h * tE, fCE2 = zp * nxdE[c] - zz * tH;
        ge += gH2[c] * (nxdH[c] - fCH2) * (h * dZ) + gE2[c] * (nxdE[c] - fCE2) * (zz * dY);
      } else {         // Z+ = Z-
        ge += gH[c] * (nxdH[c] - fCH) * (h * dZ) + gE[c] * (nxdE[c] - fCE) * (zz * dY);
      }
    }
    atomicAdd(&GE[e], ge);
    // adjoint of the traces: E: h (n n.g - g) over g = gH - gH2, + n x (zm gE + zp gE2);
    // H: n x (zp gH + zm gH2) - zz (n n.g - g) over g = gE - gE2
    float* xo = X + e * 6 * NF + fm;
    float aH[3], aE[3], xE[3], xH[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      aH[c] = gH[c] - gH2[c];
      aE[c] = gE[c] - gE2[c];
      xE[c] = zm * gE[c] + zp * gE2[c];
      xH[c] = zp * gH[c] + zm * gH2[c];
    }
    const float naH = n[0] * aH[0] + n[1] * aH[1] + n[2] * aH[2];
    const float naE = n[0] * aE[0] + n[1] * aE[1] + n[2] * aE[2];
    const float pe = nb >= 0 ? 1.f : 2.f, ph = nb >= 0 ? 1.f : 0.f;   // PEC: dE = -2 E-, dH = 0
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int p = (c + 1) % 3, q = (c + 2) % 3;
      xo[c * NF] = pe * (h * (n[c] * naH - aH[c]) + n[p] * xE[q] - n[q] * xE[p]);
      xo[(3 + c) * NF] = ph * (n[p] * xH[q] - n[q] * xH[p] - zz * (n[c] * naE - aE[c]));
    }
  }
  // ---- adapted sums of mu (scaled by 1/eps, -1/mu below: element constants)
  adapt_rows<N, UST>(MQ, t_or, U, ne, tid, NT);
  __syncthreads();
  const int sb0 = src0, sb1 = sb0 + nsl;
  // ---- curl^T: warps 0-3 take the four characters; E rows act on H and H
  // rows on E (TE <= 16: one lane per element and field)
  {
    const int y = (tid >> 5) & 3, ef = tid & 31, f = ef & 1;
    const bool act = tid < 128 && ef < 2 * ne;
    const int r = act ? ef : 0;
    const float* g = GX + (r >> 1) * 12;
    const float sc = f ? -g[11] : g[10];
    float gs[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) gs[i] = sc * g[i];
    float* out = act ? U + (ef ^ 1) * UST : nullptr;
    if (tid >= 128) __syncthreads();
    else if (y == 0) sym_curlt_pairs<N, 0>(ops, 0, U + r * UST, gs, out);
    else sym_curlt_pairs<N, 1>(ops, y, U + r * UST, gs, out);
  }
#pragma unroll
  for (int k = 0; k < ST::LOT; ++k)   // (the derivative blocks are spent)
    if (tid + k * NT < ST::LO) ops[tid + k * NT] = low[k];
  __syncthreads();
  float gp[6] = {0, 0, 0, 0, 0, 0};   // d/dsigma_max[3], d/dp_sigma[3] (this thread's points)
  const int R = TE * 6;
  if constexpr (PML) {
    // ---- at the points: v = V_q q, w = P_q^T mu, eqs. 26-29 transposed, the
    // profile derivatives.  Thread (part, e, c): component c of E,H and of P,
    // every second group of points
    constexpr int NP2 = Blocks<N, G>::PO / 2, CP = ST::CP;
    constexpr int VW = Np % 4 == 0 ? 4 : (Np % 2 == 0 ? 2 : 1);
    const int part = tid / R, row = tid - part * R;
    const int e = row / 6, c = row - e * 6;
    const int u = c % 3, v_ = (u + 1) % 3, w_ = (u + 2) % 3;
    const bool live = part < 2 && e < ne;
    if (live) {
      pair2 s[NP2], p[NP2];
      float f[Np], t[Np];
      load_row<Np, VW>(QS + row * Np, f);
      Fly<float, N, G>::forward(f, t);
      to_pairs<N, G>(t, s);
      load_row<Np, VW>(PQ + row * Np, f);
      Fly<float, N, G>::forward(f, t);
      to_pairs<N, G>(t, p);
#pragma unroll 1
      for (int g = part; g < ng; g += 2) {
        float v[4], o[4];
        sym_interp2<N, G, true>(C.v + g * CP, s, p, v, o);
        float* z = ZV + g * 8 * R + row;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          z[i * R] = v[i];
          z[(4 + i) * R] = o[i];
        }
      }
      load_row<Np, 1>(MQ + row * Np, f);
      Fly<float, N, G>::forward(f, t);
      to_pairs<N, G>(t, s);
      load_row<Np, 1>(MP + row * Np, f);
      Fly<float, N, G>::forward(f, t);
      to_pairs<N, G>(t, p);
      const float* sg = SG + e * ng * 12;
      const float e0 = A.eps0_r, ie0 = A.inv_eps0_r;
#pragma unroll 1
      for (int g = part; g < ng; g += 2) {
        float w[4], o[4], su[4], sv[4], sw[4];
        sym_interp2<N, G, true>(C.p + g * CP, s, p, w, o);
        if constexpr (ST::LO) {
          sym_interp2<N, G, false>(ops + g * CP, s, p, su, sv);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            w[i] += su[i];
            o[i] += sv[i];
          }
        }
        lds4(sg + g * 12 + u * 4, su);
        lds4(sg + g * 12 + v_ * 4, sv);
        lds4(sg + g * 12 + w_ * 4, sw);
        float* z = ZV + g * 8 * R + row;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float vF = z[i * R], vP = z[(4 + i) * R];
          const float wF = w[i], wP = o[i];
          const float bc = sv[i] + sw[i] - su[i];
          const float cc = sv[i] * sw[i] - bc * su[i];
          w[i] = wP - bc * wF;
          o[i] = -cc * wF - su[i] * wP;
          // derivatives of mu . f with respect to s_u, s_v, s_w (b, c, d of
          // eq. 9), scaled by ds/dsigma_max and ds/dp_sigma
          const float a0 = wF * vF, a1 = wF * vP;
          const float du = a0 - (su[i] - bc) * a1 - wP * vP;
          const float dv = -a0 - (sw[i] - su[i]) * a1, dw = -a0 - (sv[i] - su[i]) * a1;
          const float ss[3] = {su[i], sv[i], sw[i]}, dd[3] = {du, dv, dw};
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const int ax = k == 0 ? u : (k == 1 ? v_ : w_);
            const float x = ss[k] * e0 * A.inv_sigma_max[ax];
            const bool on = ss[k] > 0.f && x > 0.f;
            const float d1 = on ? x * ie0 * dd[k] : 0.f;
            const float d2 = on ? ss[k] * __logf(x) * A.inv_p_sigma[ax] * dd[k] : 0.f;
#pragma unroll
            for (int q = 0; q < 3; ++q) {   // (static register index)
              gp[q] += ax == q ? d1 : 0.f;
              gp[3 + q] += ax == q ? d2 : 0.f;
            }
          }
        }
#pragma unroll
        for (int x = 0; x < 4; x += G) {
          Fly<float, N, G>::group(w + x);
          Fly<float, N, G>::group(o + x);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          z[i * R] = w[i];
          z[(4 + i) * R] = o[i];
        }
      }
    }
    __syncthreads();
  }
  // ---- rows back to the nodes: V_q^T of the point sums (PML), curl^T; and
  // <curl^T a_E, H> of dJ/deps_k from the H rows.  Thread (e, row of E,H or P)
  {
    const int row = tid < R ? tid : tid - R, e = row / 6, c = row - e * 6;
    const bool isP = tid >= R, live = tid < (PML ? 2 : 1) * R && e < ne;
    if (live) {
      float t[Np];
      if constexpr (PML) {
        constexpr int CP = ST::CP;
        float acc[Np];
#pragma unroll
        for (int i = 0; i < Np; ++i) acc[i] = 0.f;
#pragma unroll 1
        for (int g = 0; g < ng; ++g) {
          float z[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) z[i] = ZV[(g * 8 + (isP ? 4 : 0) + i) * R + row];
          sym_add1<N, G>(C.v + g * CP, z, acc);
        }
        if (isP) {   // P's adjoint, over its spent stage input
          float* d = PQ + row * Np;
          Fly<float, N, G>::inverse(acc, [&](int n, float v) { d[n] = v; });
        } else {
          Fly<float, N, G>::inverse(acc, [&](int n, float v) { t[n] = v; });
        }
      }
      if (!isP) {
        float* d = U + (e * 2 + c / 3) * UST + (c % 3) * Np;
        float k[Np];
#pragma unroll
        for (int i = 0; i < Np; ++i) k[i] = d[i];
        float f[Np];
        Fly<float, N, 4>::inverse(k, [&](int n, float v) { f[n] = v; });
        if (c >= 3) {
          const float* h = QS + row * Np;
          float s = 0.f;
#pragma unroll
          for (int i = 0; i < Np; ++i) s += f[i] * h[i];
          atomicAdd(&GE[e], -GX[e * 12 + 10] * s);
        }
#pragma unroll
        for (int i = 0; i < Np; ++i) d[i] = PML ? f[i] + t[i] : f[i];
      }
    }
  }
  // source term of dJ/deps_k: + mu_E . J / eps^2
  // (a warp per source)
  for (int s = sb0 + (tid >> 5); s < sb1; s += NT / 32) {
    const SrcDev& sd = A.src[s];
    const int e = sd.elem - eg0;
    const float ie = GX[e * 12 + 10];
    const float jt = (float)dipole_current(sd, A.t) * ie * ie;
    float g = 0.f;
    for (int i = tid & 31; i < 3 * Np; i += 32)
      g += (float)sd.dir[i / Np] * A.src_w[(int64_t)s * Np + i % Np] * MQ[e * 6 * Np + i];
    atomicAdd(&GE[e], jt * g);
  }
  // ---- lambda_in = lambda_out + dt L^T mu, rho_prev = A_i mu (all loads first)
  constexpr int UT = (ST::T * 3 * Np + NT - 1) / NT;
  const int nu = ne * 3 * Np;
  float lq[UT][2], lp[PML ? UT : 1][2];
#pragma unroll
  for (int k = 0; k < UT; ++k)
    if (tid + k * NT < nu) {
      lds2(A.lam_q + oq + 2 * (tid + k * NT), lq[k]);
      if constexpr (PML) lds2(A.lam_p + op + 2 * (tid + k * NT), lp[k]);
    }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < UT; ++k) {
    const int li = 2 * (tid + k * NT);
    if (li >= 2 * nu) continue;
    float r[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int x = li + i, er = x / Np, n = x - er * Np;   // er = e * 6 + component
      float a = U[x + x / (3 * Np) * (UST - 3 * Np)];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int fm = t_nf[3 * n + j];
        if (fm < NF) a += X[er * NF + fm];
      }
      lq[k][i] += A.dt_r * a;
      r[i] = A.rk_a_r * MQ[x];
    }
    sts2(A.lam_q + oq + li, lq[k]);
    sts2(A.rho_q + oq + li, r);
    if constexpr (PML) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        lp[k][i] += A.dt_r * PQ[li + i];
        r[i] = A.rk_a_r * MP[li + i];
      }
      sts2(A.lam_p + op + li, lp[k]);
      sts2(A.rho_p + op + li, r);
    }
  }
  for (int e = tid; e < ne; e += NT)
    A.grad_eps[(int64_t)b * A.K + eg0 + e] += (double)A.dt_r * (double)GE[e];
  if constexpr (PML) {
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      float v = gp[k];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[k][wid] = (double)v;
    }
    __syncthreads();
    if (tid < 6) {
      double s = 0;
      for (int w = 0; w < NT / 32; ++w) s += red[tid][w];
      atomicAdd(&A.grad_prof[b * 6 + tid], (double)A.dt_r * s);
    }
  }
}

// the rule's coefficients are a kernel parameter: N = 5 with the (N+1)^3 rule has
// too many (48 kB of the 32 kB allowed) and runs the dense kernel
template <int N, int G>
constexpr bool sa_built = !(N == 5 && G == 2);

template <int N, int G>
cudaError_t sa_configure() {
  using ST = SaTile<N, G>;
  cudaError_t e = cudaFuncSetAttribute(
      sym_adj_kernel<N, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ST::bytes(ST::T));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sym_adj_kernel<N, G>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  return e;
}

template <int N, int G>
cudaError_t sa_main(const AdjParams<float>& P, const float* coef, int nb, cudaStream_t s) {
  using ST = SaTile<N, G>;
  if (P.n_elem <= 0) return cudaSuccess;
  AdjParams<float> Q = P;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t per = ((int64_t)P.n_elem * nb + sms - 1) / std::max(sms, 1);
  Q.tile = (int)std::max<int64_t>(1, std::min<int64_t>(per, ST::T));   // every SM a tile
  SymCoef<ST::PML ? ST::NG * ST::CP : 1> C{};
  if (ST::PML) {
    const int n = P.nsl / 4 * ST::CP;
    std::copy(coef, coef + n, C.v);
    std::copy(coef + n, coef + 2 * n, C.p);
  }
  const unsigned grid = (unsigned)((P.n_elem + Q.tile - 1) / Q.tile * (int64_t)nb);
  sym_adj_kernel<N, G><<<grid, kSaThreads, ST::bytes(Q.tile), s>>>(Q, C);
  return cudaGetLastError();
}

template <int N>
cudaError_t sa_main_g(int G, const AdjParams<float>& P, const float* coef, int nb,
                      cudaStream_t s) {
  if (G == 0) return sa_main<N, 0>(P, coef, nb, s);
  if (G == 4) return sa_main<N, 4>(P, coef, nb, s);
  if constexpr (sa_built<N, 2>) return sa_main<N, 2>(P, coef, nb, s);
  return cudaErrorInvalidValue;
}

template <int N>
cudaError_t sa_lift(const AdjParams<float>& P, int nb, cudaStream_t s) {
  using SL = SaLift<N>;
  sym_lift_kernel<N><<<dim3((P.K + SL::T - 1) / SL::T, nb), SL::NT, SL::bytes, s>>>(P);
  return cudaGetLastError();
}

template <int N>
cudaError_t sa_configure_n() {
  cudaError_t e = cudaFuncSetAttribute(
      sym_lift_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SaLift<N>::bytes);
  if (e == cudaSuccess) e = sa_configure<N, 0>();
  if constexpr (sa_built<N, 2>)
    if (e == cudaSuccess) e = sa_configure<N, 2>();
  if (e == cudaSuccess) e = sa_configure<N, 4>();
  return e;
}

}  // namespace

#define WADG_SA_SWITCH(call)                \
  switch (N) {                              \
    case 1: return call(1);                 \
    case 2: return call(2);                 \
    case 3: return call(3);                 \
    case 4: return call(4);                 \
    case 5: return call(5);                 \
    default: return cudaErrorInvalidValue;  \
  }

bool sym_adjoint_built(int N, int G) { return !(N == 5 && G == 2); }

cudaError_t configure_sym_adjoint(int N) {
#define WADG_SA_C(n) sa_configure_n<n>()
  WADG_SA_SWITCH(WADG_SA_C)
}

cudaError_t launch_sym_lift(int N, const AdjParams<float>& P, int nb, cudaStream_t s) {
#define WADG_SA_L(n) sa_lift<n>(P, nb, s)
  WADG_SA_SWITCH(WADG_SA_L)
}

cudaError_t launch_sym_adjoint(int N, int G, const AdjParams<float>& P, const float* coef, int nb,
                               cudaStream_t s) {
#define WADG_SA_M(n) sa_main_g<n>(G, P, coef, nb, s)
  WADG_SA_SWITCH(WADG_SA_M)
}

}  // namespace wadg
