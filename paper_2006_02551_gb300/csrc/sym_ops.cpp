// Symmetry-adapted reference operators (host, FP64): detection of a volume
// rule's symmetry and the tables of the symmetric CUDA-core stage.
#include <cmath>
#include <utility>
#include <vector>

#include "refelem.hpp"
#include "sym_tables.hpp"

namespace wadg {

namespace {

using Signed = std::vector<std::pair<int, int>>;   // (point, sign)

// adapted values of the nodes as signed sums, in the order of Blocks<N, 4>
template <int N>
std::vector<Signed> node_sums_v4() {
  const NodeOrbits<N> O{};
  constexpr int NH = Blocks<N, 4>::NH;
  std::vector<Signed> t;
  for (int x = 0; x < 4; ++x) {
    for (int o = 0; o < O.nful; ++o) {
      Signed s;
      for (int y = 0; y < 4; ++y) s.push_back({O.ful[o][y], v4_sign(x, y)});
      t.push_back(s);
    }
    for (int a = 0; a < 3; ++a)
      if (NH && (x == 0 || x == a + 1))
        t.push_back({{O.hal[a][0], 1}, {O.hal[a][1], x == 0 ? 1 : -1}});
    if (x == 0 && O.sin >= 0) t.push_back({{O.sin, 1}});
  }
  return t;
}

template <int N>
std::vector<Signed> node_sums_z2() {
  const NodeOrbits<N> O{};
  std::vector<Signed> t;
  for (int x = 0; x < 2; ++x) {
    for (int o = 0; o < O.npr; ++o) t.push_back({{O.pr[o][0], 1}, {O.pr[o][1], x ? -1 : 1}});
    if (x == 0)
      for (int o = 0; o < O.nfx; ++o) t.push_back({{O.fx[o], 1}});
  }
  return t;
}

template <int N>
void tables(const RefOps& R, const SymRule& S, std::vector<double>& ops,
            std::vector<unsigned char>& tabs) {
  using L = SymLayout<N>;
  using B = Blocks<N, 4>;
  const int Np = R.Np, Nfp = R.Nfp, NF = 4 * Nfp;
  const auto T = node_sums_v4<N>();
  ops.assign(L::oV, 0.0);
  // d/dxi_a in terms of d/dr, d/ds, d/dt
  const double mix[3][3] = {{0.5, -0.5, -0.5}, {-0.5, 0.5, -0.5}, {-0.5, -0.5, 0.5}};
  for (int x = 0; x < 4; ++x)
    for (int a = 1; a <= 3; ++a)
      for (int j = 0; j < B::dim(x ^ a); ++j)
        for (int i = 0; i < B::dim(x); ++i) {
          const Signed& to = T[B::off(x) + i];
          const Signed& ti = T[B::off(x ^ a) + j];
          double v = 0.0;
          for (const auto& p : to)
            for (const auto& q : ti) {
              const int k = p.first * Np + q.first;
              v += p.second * q.second *
                   (mix[a - 1][0] * R.Dr[k] + mix[a - 1][1] * R.Ds[k] + mix[a - 1][2] * R.Dt[k]);
            }
          ops[L::d_off(x, a) + j * L::RP(x) + i] = v / (double)(to.size() * ti.size());
        }
  // face nodes: node m of face 0 and its images (face of g_y: 0, 1, 3, 2)
  tabs.assign(8 * Nfp, 0);
  const int fy[4] = {0, 1, 3, 2};
  for (int m = 0; m < Nfp; ++m) {
    const int* b = &R.bary[R.Fmask[m] * 4];
    for (int y = 0; y < 4; ++y)
      for (int m2 = 0; m2 < Nfp; ++m2) {
        const int n2 = R.Fmask[fy[y] * Nfp + m2];
        bool same = true;
        for (int v = 0; v < 4; ++v) same = same && R.bary[n2 * 4 + v] == b[v4_image(y, v)];
        if (same) {
          tabs[4 * m + y] = (unsigned char)(fy[y] * Nfp + m2);
          tabs[4 * Nfp + 4 * m + y] = (unsigned char)n2;
        }
      }
  }
  for (int x = 0; x < 4; ++x)
    for (int m = 0; m < Nfp; ++m)
      for (int i = 0; i < B::dim(x); ++i) {
        const Signed& to = T[B::off(x) + i];
        double v = 0.0;
        for (const auto& p : to)
          for (int y = 0; y < 4; ++y)
            v += p.second * v4_sign(x, y) * R.LIFT[(size_t)p.first * NF + tabs[4 * m + y]];
        ops[L::l_off(x) + m * L::RP(x) + i] = v / (4.0 * to.size());
      }
  {  // node orbits: free, stabilised by g_1, g_2, g_3, fixed
    const NodeOrbits<N> O{};
    for (int o = 0; o < O.nful; ++o)
      for (int y = 0; y < 4; ++y) tabs.push_back((unsigned char)O.ful[o][y]);
    for (int a = 0; a < 3; ++a)
      for (int k = 0; k < 2; ++k) tabs.push_back((unsigned char)O.hal[a][k]);
    tabs.push_back((unsigned char)(O.sin < 0 ? 0 : O.sin));
    int nc = 0, best = 1 << 30;   // the node nearest the centroid
    for (int n = 0; n < Np; ++n) {
      int d = 0;
      for (int v = 0; v < 4; ++v) d += R.bary[n * 4 + v] * R.bary[n * 4 + v];
      if (d < best) {
        best = d;
        nc = n;
      }
    }
    tabs.push_back((unsigned char)nc);
    for (int n = 0; n < Np; ++n) {   // the face nodes at each node (NF: none)
      int k = 0;
      for (int fm = 0; fm < NF && k < 3; ++fm)
        if (R.Fmask[fm] == n) {
          tabs.push_back((unsigned char)fm);
          ++k;
        }
      for (; k < 3; ++k) tabs.push_back((unsigned char)NF);
    }
  }
  if (S.G == 0) return;
  const auto TR = S.G == 4 ? T : node_sums_z2<N>();
  const int G = S.G, CP = sym_cp(N, G), ng = (int)S.slots.size() / 4, per = 4 / G;
  const size_t oV = ops.size(), oP = oV + (size_t)ng * CP;
  ops.resize(oP + (size_t)ng * CP, 0.0);
  auto chr = [&](int i) -> int {   // character of adapted index i
    if (G == 4) {
      int x = 0;
      while (x < 3 && i >= B::off(x + 1)) ++x;
      return x;
    }
    return i >= Blocks<N, 2>::D0 ? 1 : 0;
  };
  auto place = [&](int o, int i) -> size_t {   // within a group's coefficients
    const int x = chr(i);
    using Z = Blocks<N, 2>;
    return G == 4 ? (size_t)(B::poff(x) + i - B::off(x))
                  : (size_t)(o * Z::PO + Z::poff(x) + i - Z::off(x));
  };
  for (int g = 0; g < ng; ++g)
    for (int o = 0; o < per; ++o) {
      const int* sl = &S.slots[4 * g + G * o];
      if (sl[0] < 0) continue;   // padding
      for (int i = 0; i < Np; ++i) {
        const int x = chr(i);
        const Signed& ti = TR[i];
        double v = 0.0, w = 0.0;
        for (int y = 0; y < G; ++y) {
          int mult = 0;
          for (int z = 0; z < G; ++z) mult += sl[z] == sl[y];
          const int sg = G == 4 ? v4_sign(x, y) : (x && y ? -1 : 1);
          for (const auto& p : ti) {
            v += sg * p.second * R.Vq[(size_t)sl[y] * Np + p.first];
            w += sg * p.second * R.Pq[(size_t)p.first * R.Nq + sl[y]] / mult;
          }
        }
        const double n = (double)G * ti.size();
        ops[oV + (size_t)g * CP + place(o, i)] = v / n;
        ops[oP + (size_t)g * CP + place(o, i)] = w / n;
      }
    }
}

}  // namespace

SymRule detect_symmetry(const RefOps& R) {
  const int n = R.Nq_rule;
  std::vector<double> lam(4 * (size_t)n);
  for (int q = 0; q < n; ++q) {
    lam[4 * q + 1] = 0.5 * (1 + R.rq[q]);
    lam[4 * q + 2] = 0.5 * (1 + R.sq[q]);
    lam[4 * q + 3] = 0.5 * (1 + R.tq[q]);
    lam[4 * q] = -0.5 * (1 + R.rq[q] + R.sq[q] + R.tq[q]);
  }
  // whether point p lies at the image of q under the vertex map `im`
  auto at_image = [&](int p, int q, const int im[4]) {
    for (int v = 0; v < 4; ++v)
      if (!(std::fabs(lam[4 * p + v] - lam[4 * q + im[v]]) <= 1e-14)) return false;
    return true;
  };
  for (int G : {4, 2}) {
    SymRule S;
    S.G = G;
    // Every point belongs to exactly one orbit.  Within an orbit a location has
    // one point (a point that an element fixes, or that two elements reach,
    // appears for each of them); a point listed twice forms orbits with the
    // other listings of its images.
    std::vector<char> seen(n, 0);
    bool ok = true;
    for (int q = 0; q < n && ok; ++q) {
      if (seen[q]) continue;
      int sl[4] = {q, q, q, q};
      seen[q] = 1;
      for (int y = 1; y < G && ok; ++y) {
        int im[4], p = -1;
        for (int v = 0; v < 4; ++v) im[v] = G == 4 ? v4_image(y, v) : (v < 2 ? 1 - v : v);
        for (int z = 0; z < y && p < 0; ++z)
          if (at_image(sl[z], q, im)) p = sl[z];
        for (int k = 0; k < n && p < 0; ++k)
          if (!seen[k] && std::fabs(R.wq[k] - R.wq[q]) <= 1e-13 * std::fabs(R.wq[q]) &&
              at_image(k, q, im))
            p = k;
        ok = p >= 0;
        if (!ok) break;
        sl[y] = p;
        seen[p] = 1;
      }
      S.slots.insert(S.slots.end(), sl, sl + G);
    }
    if (!ok) continue;
    while (S.slots.size() % 4) S.slots.push_back(-1);
    // slots are byte indices, and the kernels hold a bounded number of groups
    if ((int)S.slots.size() <= 4 * sym_groups(R.N, G)) return S;
  }
  return SymRule{};
}

namespace {
template <int N>
std::vector<float> transposed(const std::vector<double>& ops) {
  using L = SymLayout<N>;
  using B = Blocks<N, 4>;
  constexpr int Nfp = L::Nfp, RM = (Nfp + 3) & ~3;
  std::vector<float> t(L::oL + (size_t)B::Np * RM, 0.f);
  for (int y = 0; y < 4; ++y)
    for (int a = 1; a <= 3; ++a)
      for (int i = 0; i < B::dim(y ^ a); ++i)
        for (int j = 0; j < B::dim(y); ++j)
          t[L::d_off(y, a) + i * L::RP(y) + j] =
              (float)ops[L::d_off(y ^ a, a) + j * L::RP(y ^ a) + i];
  for (int x = 0; x < 4; ++x)
    for (int i = 0; i < B::dim(x); ++i)
      for (int m = 0; m < Nfp; ++m)
        t[L::oL + (size_t)(B::off(x) + i) * RM + m] = (float)ops[L::l_off(x) + m * L::RP(x) + i];
  return t;
}
}  // namespace

std::vector<float> sym_transposed(int N, const std::vector<double>& ops) {
  switch (N) {
    case 1: return transposed<1>(ops);
    case 2: return transposed<2>(ops);
    case 3: return transposed<3>(ops);
    case 4: return transposed<4>(ops);
    default: return transposed<5>(ops);
  }
}

std::vector<double> sym_adapt(int N, const std::vector<double>& f) {
  static const std::vector<Signed> sums[] = {{}, node_sums_v4<1>(), node_sums_v4<2>(),
                                             node_sums_v4<3>(), node_sums_v4<4>(),
                                             node_sums_v4<5>()};
  std::vector<double> t;
  for (const Signed& s : sums[N]) {
    double v = 0.0;
    for (const auto& p : s) v += p.second * f[p.first];
    t.push_back(v / (double)s.size());
  }
  return t;
}

void build_sym_tables(const RefOps& R, const SymRule& S, std::vector<double>& ops,
                      std::vector<unsigned char>& tabs) {
  switch (R.N) {
    case 1: tables<1>(R, S, ops, tabs); break;
    case 2: tables<2>(R, S, ops, tabs); break;
    case 3: tables<3>(R, S, ops, tabs); break;
    case 4: tables<4>(R, S, ops, tabs); break;
    case 5: tables<5>(R, S, ops, tabs); break;
    default: break;
  }
}

const std::vector<float>& sym_constants(int N) {
  static const std::vector<std::vector<float>> all = [] {
    std::vector<std::vector<float>> t(6);
    for (int n = 1; n <= 5; ++n) {
      RefOps R;
      const char* err = nullptr;
      std::vector<double> ops;
      std::vector<unsigned char> tabs;
      if (!build_ref_ops(n, R, &err)) continue;
      build_sym_tables(R, SymRule{}, ops, tabs);
      t[n].assign(ops.begin(), ops.end());
    }
    return t;
  }();
  return all[N];
}

}  // namespace wadg
