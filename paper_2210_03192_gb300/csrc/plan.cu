// Host-side class planner: builds, once per (la, lb | lc, bra_pure), the index
// tables that drive the integral kernel's stages, and chooses the launch shape.
//
// Stages and the passages they follow (arXiv:2210.03192):
//   [00|0]^(m)       Sec. 2.5.2 (Boys function times the prefactor)
//   VRR1             Eq. vrr1: [a+1_i 0|0]^(m) = PA_i [a]^(m) - rho/gamma PC_i [a]^(m+1)
//                              + a_i/(2 gamma) ([a-1_i]^(m) - rho/gamma [a-1_i]^(m+1))
//   CVRR2 prerequisites and targets  n-q form of Eq. cVRR2 (the printed closed
//                    form is garbled; the reading used is (a 0|c) = sum over
//                    u <= min(a,c) of prod_i C(a_i,u_i) C(c_i,u_i) u_i!
//                    (a-u 0)_{|u|, c-u}) with the ket transform of Sec. 2.5.1
//                    taken first: since sum_c T_Cc c!/(c-u)! X^{c-u} = d^u S_C(X)
//                    is a solid harmonic of degree lc-|u|,
//                      (a 0|C) = sum_u C(a,u) sum_m D^u_{Cm} (a-u 0)_{|u|,m},
//                      (e 0)_{k,m} = sum_prim Y^k s_{lc-k,m}(X) [e 0|0]^(lc),
//                    with 2(lc-k)+1 prerequisites per (e, k) where the monomials
//                    X^n of Eq. a0cv2 give (lc-k+1)(lc-k+2)/2;
//                    Y = rho/(2 gamma zeta_c) = 1/(2(gamma+zeta_c)), X = rho/zeta_c PC
//   HRR              Eq. hrr: (a b+1_i|C) = (a+1_i b|C) + AB_i (a b|C)
//   bra transform    optional (solid-harmonic bra)
#include <vector_types.h>

#include <algorithm>
#include <cstdio>
#include <cmath>
#include <map>
#include <mutex>
#include <set>
#include <stdexcept>
#include <string>
#include <tuple>

#include "harmonic_weights.h"
#include "lx3c_internal.h"

namespace lx3c {

int ncart(int l) { return l < 0 ? 0 : (l + 1) * (l + 2) / 2; }

int cart_index(int x, int y, int z) {
  int l = x + y + z, idx = 0;
  for (int ax = l; ax > x; --ax) idx += l - ax + 1;
  return idx + (l - x) - y;
}

namespace {

struct C3 {
  int v[3];
  int l() const { return v[0] + v[1] + v[2]; }
  bool operator<(const C3& o) const { return std::tie(v[0], v[1], v[2]) < std::tie(o.v[0], o.v[1], o.v[2]); }
  bool operator==(const C3& o) const { return v[0] == o.v[0] && v[1] == o.v[1] && v[2] == o.v[2]; }
};

std::vector<C3> cart(int l) {
  std::vector<C3> out;
  for (int x = l; x >= 0; --x)
    for (int y = l - x; y >= 0; --y) out.push_back(C3{{x, y, l - x - y}});
  return out;
}

double binom(int n, int k) {
  if (k < 0 || k > n) return 0.0;
  double r = 1.0;
  for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
  return std::round(r);
}

double fact(int n) {
  double r = 1.0;
  for (int i = 2; i <= n; ++i) r *= i;
  return r;
}

}  // namespace

// Real solid harmonics, Racah normalisation, m = -l..l, by the closed
// expansion of S_lm in Cartesian monomials (standard Schlegel-Frisch /
// Helgaker form): S_lm = N_lm sum_{t,u,v} C_tuv x^{2t+|m|-2(u+v)} y^{2(u+v)} z^{l-2t-|m|}.
std::vector<double> solid_matrix(int l) {
  int nc = ncart(l);
  std::vector<double> T((2 * l + 1) * nc, 0.0);
  for (int m = -l; m <= l; ++m) {
    int am = m < 0 ? -m : m;
    int vm2 = m < 0 ? 1 : 0;  // 2*v_m
    long double N = 1.0L / (std::pow(2.0L, am) * (long double)fact(l)) *
                    std::sqrt(2.0L * (long double)fact(l + am) * (long double)fact(l - am) / (m == 0 ? 2.0L : 1.0L));
    for (int t = 0; t <= (l - am) / 2; ++t)
      for (int u = 0; u <= t; ++u)
        for (int vv = vm2; vv <= am; vv += 2) {  // vv = 2v
          int sgn_exp = t + (vv - vm2) / 2;
          long double c = ((sgn_exp & 1) ? -1.0L : 1.0L) * std::pow(0.25L, t) * binom(l, t) * binom(l - t, am + t) *
                          binom(t, u) * binom(am, vv);
          int ex = 2 * t + am - 2 * u - vv, ey = 2 * u + vv, ez = l - 2 * t - am;
          if (ex < 0) continue;
          T[(m + l) * nc + cart_index(ex, ey, ez)] += (double)(N * c);
        }
  }
  return T;
}

namespace {

unsigned pal_id(std::vector<double>& pal, std::map<double, int>& ids, double v) {
  auto it = ids.find(v);
  if (it != ids.end()) return it->second;
  int id = (int)pal.size();
  pal.push_back(v);
  ids[v] = id;
  return id;
}

// Homogeneous polynomials of degree l as coefficients over cart(l).
typedef std::vector<long double> Poly;

Poly times_coord(const Poly& p, int l, int axis) {
  Poly r(ncart(l + 1), 0.0L);
  for (auto& c : cart(l)) {
    C3 d = c;
    d.v[axis]++;
    r[cart_index(d.v[0], d.v[1], d.v[2])] += p[cart_index(c.v[0], c.v[1], c.v[2])];
  }
  return r;
}

Poly derivative(const Poly& p, int l, int axis) {
  Poly r(ncart(l - 1), 0.0L);
  for (auto& c : cart(l))
    if (c.v[axis] > 0) {
      C3 d = c;
      d.v[axis]--;
      r[cart_index(d.v[0], d.v[1], d.v[2])] += c.v[axis] * p[cart_index(c.v[0], c.v[1], c.v[2])];
    }
  return r;
}

// The kernel's harmonic basis of degree l, m = -l..l: Q_{l,|m|}(z, r^2) times
// the real (m >= 0) or imaginary part of (x + i y)^|m|, with
// Q_{m,m} = 1, Q_{l+1,m} = z Q_{l,m} - (l^2-m^2)/(4l^2-1) r^2 Q_{l-1,m}.
const std::vector<Poly>& harmonic_basis(int l) {
  static std::map<int, std::vector<Poly>> cache;  // under class_tables_variant's lock
  auto it = cache.find(l);
  if (it != cache.end()) return it->second;
  std::vector<Poly> out(2 * l + 1);
  auto add = [](const Poly& a, const Poly& b, long double f) {
    Poly r = a;
    for (size_t i = 0; i < r.size(); ++i) r[i] += f * b[i];
    return r;
  };
  Poly A{1.0L}, B{0.0L};
  for (int m = 0; m <= l; ++m) {
    if (m > 0) {
      const Poly An = add(times_coord(A, m - 1, 0), times_coord(B, m - 1, 1), -1.0L);
      B = add(times_coord(A, m - 1, 1), times_coord(B, m - 1, 0), 1.0L);
      A = An;
    }
    for (int im = 0; im < (m > 0 ? 2 : 1); ++im) {
      Poly q0(1, 0.0L), q1 = im ? B : A;  // Q_{k-1}, Q_k times the angular factor, degrees k-1 and k
      for (int k = m; k < l; ++k) {
        Poly n = times_coord(q1, k, 2);
        if (k > m) {
          Poly r2 = times_coord(times_coord(q0, k - 1, 0), k, 0);
          for (int x = 1; x < 3; ++x) r2 = add(r2, times_coord(times_coord(q0, k - 1, x), k, x), 1.0L);
          n = add(n, r2, -(long double)(k * k - m * m) / (4.0L * k * k - 1.0L));
        }
        q0 = q1;
        q1 = n;
      }
      out[im ? l - m : l + m] = q1;
    }
  }
  return cache.emplace(l, out).first->second;
}

// D^u: rows C of the solid harmonics S_C of degree lc, d^u S_C = sum_m D[C][m]
// s_{lc-|u|,m}.  Harmonic polynomials of one degree and different m are
// orthogonal under <x^a, x^b> = a! delta_ab (rotations preserve it).
std::vector<double> harmonic_derivative(int lc, const C3& u) {
  const int k = u.l(), l = lc - k;
  const auto T = solid_matrix(lc);
  const auto& s = harmonic_basis(l);
  auto fac3 = [](const C3& c) { return (long double)(fact(c.v[0]) * fact(c.v[1]) * fact(c.v[2])); };
  std::vector<double> D((2 * lc + 1) * (2 * l + 1), 0.0);
  for (int C = 0; C < 2 * lc + 1; ++C) {
    Poly p(T.begin() + C * ncart(lc), T.begin() + (C + 1) * ncart(lc));
    int deg = lc;
    for (int x = 0; x < 3; ++x)
      for (int i = 0; i < u.v[x]; ++i) p = derivative(p, deg--, x);
    long double big = 0.0L;
    std::vector<long double> d(2 * l + 1);
    for (int m = 0; m < 2 * l + 1; ++m) {
      long double num = 0.0L, den = 0.0L;
      for (auto& c : cart(l)) {
        const int i = cart_index(c.v[0], c.v[1], c.v[2]);
        num += fac3(c) * p[i] * s[m][i];
        den += fac3(c) * s[m][i] * s[m][i];
      }
      d[m] = num / den;
      big = std::max(big, std::fabs(d[m]));
    }
    for (int m = 0; m < 2 * l + 1; ++m)
      D[C * (2 * l + 1) + m] = std::fabs(d[m]) > 1e-12L * big ? (double)d[m] : 0.0;
  }
  return D;
}

ClassTables build(int la, int lb, int lc, int bra_pure, int hrr2) {
  ClassTables ct;
  ct.la = la; ct.lb = lb; ct.lc = lc; ct.bra_pure = bra_pure;
  const int Lab = la + lb;
  ct.ncA = ncart(la); ct.ncB = ncart(lb); ct.ncc = ncart(lc);
  ct.nC = 2 * lc + 1;
  ct.nA = bra_pure ? 2 * la + 1 : ct.ncA;
  ct.nB = bra_pure ? 2 * lb + 1 : ct.ncB;
  std::map<double, int> palids;
  pal_id(ct.pal, palids, 1.0);  // id 0 is always 1.0

  // ---------------- HRR dependency analysis (Eq. hrr) ----------------
  // Rounds r = 1..R move q_r quanta from the recurrence centre to the other:
  // every q_r = 1 (1-q HRR, Eq. hrr), or with hrr2 the 2-quantum transfer of
  // Sec. 2.5.5 applied twice in one round,
  //   (a, b+1_i+1_k) = (a+1_i+1_k, b) + AB_i (a+1_k, b) + AB_k (a+1_i, b) + AB_i AB_k (a, b),
  // with one 1-q round last (topmost) when lb is odd.  Nodes (a, b) of round
  // r have |b| = the quanta moved so far; the top round holds every (a, b) of
  // the target, and each round keeps only the nodes the next one reads
  // (greedy cover: as few lower b's as possible).
  std::vector<int> step;  // q_r, r = 1..R, bottom-up
  if (hrr2) {
    for (int q = 0; q < lb / 2; ++q) step.push_back(2);
    if (lb & 1) step.push_back(1);
  } else {
    for (int q = 0; q < lb; ++q) step.push_back(1);
  }
  const int R = (int)step.size();
  std::vector<int> bl(R + 1, 0);  // |b| of round r
  for (int r = 1; r <= R; ++r) bl[r] = bl[r - 1] + step[r - 1];
  std::vector<std::vector<std::pair<C3, C3>>> lev(R + 1);
  std::vector<std::map<std::pair<C3, C3>, int>> levidx(R + 1);
  // per needed b of round r: the lower b and the axes (i, k) (k = -1 for 1-q)
  std::vector<std::map<C3, std::pair<C3, std::pair<int, int>>>> bdec(R + 1);
  for (auto& a : cart(la))
    for (auto& b : cart(lb)) {
      levidx[R][{a, b}] = (int)lev[R].size();
      lev[R].push_back({a, b});
    }
  auto add = [](C3 x, int i, int k) {
    if (i >= 0) x.v[i]++;
    if (k >= 0) x.v[k]++;
    return x;
  };
  for (int r = R; r >= 1; --r) {
    const int q = step[r - 1];
    std::set<C3> need;
    for (auto& n : lev[r]) need.insert(n.second);
    while (!need.empty()) {
      C3 best{{0, 0, 0}};
      int bestcount = -1;
      for (auto& bp : cart(bl[r - 1])) {
        int cnt = 0;
        for (int i = 0; i < 3; ++i)
          for (int k = (q == 2 ? i : -1); k < (q == 2 ? 3 : 0); ++k)
            if (need.count(add(bp, i, k))) ++cnt;
        if (cnt > bestcount) { bestcount = cnt; best = bp; }
      }
      for (int i = 0; i < 3; ++i)
        for (int k = (q == 2 ? i : -1); k < (q == 2 ? 3 : 0); ++k) {
          C3 b = add(best, i, k);
          if (need.count(b)) { bdec[r][b] = {best, {i, k}}; need.erase(b); }
        }
    }
    std::set<std::pair<C3, C3>> prev;
    for (auto& n : lev[r]) {
      const auto& dec = bdec[r][n.second];
      const C3& bp = dec.first;
      const int i = dec.second.first, k = dec.second.second;
      prev.insert({add(n.first, i, k), bp});
      prev.insert({n.first, bp});
      if (k >= 0) {
        prev.insert({add(n.first, i, -1), bp});
        prev.insert({add(n.first, k, -1), bp});
      }
    }
    // order the lower round's nodes: by |a|, then a, then b
    std::vector<std::pair<C3, C3>> pv(prev.begin(), prev.end());
    std::sort(pv.begin(), pv.end(), [](const std::pair<C3, C3>& x, const std::pair<C3, C3>& y) {
      if (x.first.l() != y.first.l()) return x.first.l() < y.first.l();
      int ix = cart_index(x.first.v[0], x.first.v[1], x.first.v[2]);
      int iy = cart_index(y.first.v[0], y.first.v[1], y.first.v[2]);
      if (ix != iy) return ix < iy;
      return cart_index(x.second.v[0], x.second.v[1], x.second.v[2]) <
             cart_index(y.second.v[0], y.second.v[1], y.second.v[2]);
    });
    lev[r - 1] = pv;
    for (size_t n = 0; n < pv.size(); ++n) levidx[r - 1][pv[n]] = (int)n;
  }
  // e0 rows (round 0): needed bra functions (a, 0)
  std::vector<C3> erows;
  for (auto& n : lev[0]) erows.push_back(n.first);
  ct.nkrow = (int)erows.size();
  for (auto& e : erows) ct.erow_xyz.push_back(int4{e.v[0], e.v[1], e.v[2], 0});
  ct.nhrr = R;
  ct.hrr2 = hrr2;
  ct.hrows.assign(R + 1, 0);
  ct.hstart.assign(R + 2, 0);
  ct.hrows[0] = ct.nkrow;
  // row = {dst | nterm << 16, src0 | src1 << 16, src2 | src3 << 16, 4-bit
  // coefficient codes}; codes index the tile's AB products: 0 one, 1..3 AB_i,
  // 4..6 2 AB_i, 7..9 AB_i^2, 10 AB_x AB_y, 11 AB_x AB_z, 12 AB_y AB_z
  auto pcode = [](int i, int k) {
    if (i == k) return 7 + i;
    const int lo = std::min(i, k), hi = std::max(i, k);
    return lo == 0 ? (hi == 1 ? 10 : 11) : 12;
  };
  for (int r = 1; r <= R; ++r) {
    ct.hstart[r] = (int)ct.htab.size();
    ct.hrows[r] = (int)lev[r].size();
    std::vector<std::pair<int, uint4>> rows;
    for (size_t n = 0; n < lev[r].size(); ++n) {
      const auto& node = lev[r][n];
      const auto& dec = bdec[r][node.second];
      const C3& bp = dec.first;
      const int i = dec.second.first, k = dec.second.second;
      const C3& a = node.first;
      unsigned src[4] = {0, 0, 0, 0}, code[4] = {0, 0, 0, 0};
      int nt;
      auto at = [&](const C3& x) { return (unsigned)levidx[r - 1].at({x, bp}); };
      if (k < 0) {
        src[0] = at(add(a, i, -1)); code[0] = 0;
        src[1] = at(a); code[1] = 1 + i;
        nt = 2;
      } else if (i == k) {
        src[0] = at(add(a, i, i)); code[0] = 0;
        src[1] = at(add(a, i, -1)); code[1] = 4 + i;
        src[2] = at(a); code[2] = pcode(i, i);
        nt = 3;
      } else {
        src[0] = at(add(a, i, k)); code[0] = 0;
        src[1] = at(add(a, k, -1)); code[1] = 1 + i;
        src[2] = at(add(a, i, -1)); code[2] = 1 + k;
        src[3] = at(a); code[3] = pcode(i, k);
        nt = 4;
      }
      rows.push_back({nt, uint4{(unsigned)n | ((unsigned)nt << 16), src[0] | (src[1] << 16), src[2] | (src[3] << 16),
                                code[0] | (code[1] << 4) | (code[2] << 8) | (code[3] << 12)}});
    }
    // rows with the same term count together, so that a warp's lanes share it
    std::stable_sort(rows.begin(), rows.end(), [](auto& x, auto& y) { return x.first < y.first; });
    for (auto& rw : rows) ct.htab.push_back(rw.second);
  }
  ct.hstart[R + 1] = (int)ct.htab.size();

  // ---------------- VRR1 buffer and items (Eq. vrr1) ----------------
  std::vector<int> voff(Lab + 2, 0);
  for (int e = 0; e <= Lab; ++e) voff[e + 1] = voff[e] + ncart(e) * (Lab - e + 1);
  ct.NV = voff[Lab + 1];
  auto vidx = [&](int e, int m, const C3& c) { return voff[e] + (m - lc) * ncart(e) + cart_index(c.v[0], c.v[1], c.v[2]); };
  ct.vlev_start.assign(Lab + 1, 0);
  for (int e = 1; e <= Lab; ++e) {
    ct.vlev_start[e - 1] = (int)ct.vtab.size();
    std::vector<uint4> simple, full;
    for (auto& t : cart(e)) {
      int ax = -1;
      for (int i = 0; i < 3; ++i)
        if (t.v[i] == 1) { ax = i; break; }
      if (ax < 0)
        for (int i = 0; i < 3; ++i)
          if (t.v[i] > 0 && (ax < 0 || t.v[i] > t.v[ax])) ax = i;
      int n = t.v[ax] - 1;
      C3 s1 = t;
      s1.v[ax]--;
      C3 s2 = s1;
      if (n > 0) s2.v[ax]--;
      for (int m = lc; m <= lc + Lab - e; ++m) {
        unsigned dst = vidx(e, m, t), a = vidx(e - 1, m, s1), an = vidx(e - 1, m + 1, s1);
        unsigned b = n > 0 ? vidx(e - 2, m, s2) : 0u, bn = n > 0 ? vidx(e - 2, m + 1, s2) : 0u;
        uint4 it{dst | (a << 16), an | (b << 16), bn | ((unsigned)ax << 16) | ((unsigned)n << 20), 0u};
        (n > 0 ? full : simple).push_back(it);
      }
    }
    ct.vtab.insert(ct.vtab.end(), simple.begin(), simple.end());
    ct.vtab.insert(ct.vtab.end(), full.begin(), full.end());
  }
  ct.vlev_start[Lab] = (int)ct.vtab.size();

  // ---------------- weights W_{k,m} = Y^k s_{lc-k,m}(X) ----------------
  // F buffer: 0..2 (rho/gamma) PC, 3 rho/gamma, 4..6 X, 7 + (k-1) Y^k
  const int kmax = std::min(Lab, lc);
  ct.kmax = kmax;
  ct.NF = 4 + (lc > 0 ? 3 + kmax : 0);
  ct.NW = (kmax + 1) * (2 * lc + 1 - kmax);
  auto woff = [&](int k) { return k * (2 * lc + 2 - k); };

  // ---------------- CVRR2 targets and prerequisites (Sec. 2.5.4) ----------------
  // prerequisites by (e, k), then m = -(lc-k)..lc-k, in the order |e|, e, k
  std::map<std::pair<C3, int>, int> accmap;
  for (int r = 0; r < ct.nkrow; ++r)
    for (int ux = 0; ux <= erows[r].v[0]; ++ux)
      for (int uy = 0; uy <= erows[r].v[1]; ++uy)
        for (int uz = 0; uz <= erows[r].v[2] && ux + uy + uz <= lc; ++uz) {
          const C3 e{{erows[r].v[0] - ux, erows[r].v[1] - uy, erows[r].v[2] - uz}};
          accmap[{e, ux + uy + uz}] = 0;
        }
  std::vector<std::pair<C3, int>> acckeys;
  for (auto& kv : accmap) acckeys.push_back(kv.first);
  std::sort(acckeys.begin(), acckeys.end(), [](auto& x, auto& y) {
    if (x.first.l() != y.first.l()) return x.first.l() < y.first.l();
    const int ix = cart_index(x.first.v[0], x.first.v[1], x.first.v[2]),
              iy = cart_index(y.first.v[0], y.first.v[1], y.first.v[2]);
    return ix != iy ? ix < iy : x.second < y.second;
  });
  ct.NACC = 0;
  for (auto& key : acckeys) {
    accmap[key] = ct.NACC;
    const unsigned v = vidx(key.first.l(), lc, key.first);
    for (int m = 0; m < 2 * (lc - key.second) + 1; ++m) ct.atab.push_back(v | ((unsigned)(woff(key.second) + m) << 16));
    ct.NACC += 2 * (lc - key.second) + 1;
  }
  // gather CSR by target id = row*nC + C, items sorted by descending term count
  int ngt = ct.nkrow * ct.nC;
  ct.gptr.assign(ngt + 1, 0);
  std::map<C3, std::vector<double>> dmap;
  for (int r = 0; r < ct.nkrow; ++r) {
    const C3& a = erows[r];
    for (int C = 0; C < ct.nC; ++C) {
      for (int ux = 0; ux <= a.v[0]; ++ux)
        for (int uy = 0; uy <= a.v[1]; ++uy)
          for (int uz = 0; uz <= a.v[2] && ux + uy + uz <= lc; ++uz) {
            const C3 u{{ux, uy, uz}};
            auto it = dmap.find(u);
            if (it == dmap.end()) it = dmap.emplace(u, harmonic_derivative(lc, u)).first;
            const int k = u.l(), nm = 2 * (lc - k) + 1;
            const double bin = binom(a.v[0], ux) * binom(a.v[1], uy) * binom(a.v[2], uz);
            const int p0 = accmap.at({C3{{a.v[0] - ux, a.v[1] - uy, a.v[2] - uz}}, k});
            for (int m = 0; m < nm; ++m) {
              const double d = it->second[C * nm + m];
              if (d != 0.0) ct.gterm.push_back((unsigned)(p0 + m) | (pal_id(ct.pal, palids, bin * d) << kGatherBits));
            }
          }
      ct.gptr[r * ct.nC + C + 1] = (int)ct.gterm.size();
    }
  }
  ct.gdst.resize(ngt);
  for (int i = 0; i < ngt; ++i) ct.gdst[i] = i;
  std::stable_sort(ct.gdst.begin(), ct.gdst.end(), [&](int x, int y) {
    return (ct.gptr[x + 1] - ct.gptr[x]) > (ct.gptr[y + 1] - ct.gptr[y]);
  });
  {
    // sliced ELL copy: padding terms read accumulator 0 with coefficient 0
    const unsigned pad = 0u | (pal_id(ct.pal, palids, 0.0) << kGatherBits);
    for (int s0 = 0; s0 < ngt; s0 += 32) {
      int mx = 0;
      for (int l = s0; l < std::min(ngt, s0 + 32); ++l) mx = std::max(mx, ct.gptr[ct.gdst[l] + 1] - ct.gptr[ct.gdst[l]]);
      ct.gslice.push_back(int2{(int)ct.gell.size(), mx});
      for (int j = 0; j < mx; ++j)
        for (int l = 0; l < 32; ++l) {
          const int r = s0 + l;
          const int id = r < ngt ? ct.gdst[r] : -1;
          const bool has = id >= 0 && j < ct.gptr[id + 1] - ct.gptr[id];
          ct.gell.push_back(has ? ct.gterm[ct.gptr[id] + j] : pad);
        }
    }
  }

  // ---------------- ket transform ----------------
  auto Tc = solid_matrix(lc);
  ct.kptr.assign(ct.nC + 1, 0);
  for (int C = 0; C < ct.nC; ++C) {
    for (int c = 0; c < ct.ncc; ++c) {
      double v = Tc[C * ct.ncc + c];
      if (v != 0.0) ct.kent.push_back(int2{c, (int)pal_id(ct.pal, palids, v)});
    }
    ct.kptr[C + 1] = (int)ct.kent.size();
  }

  // ---------------- bra transforms ----------------
  ct.nbA = ct.nbB = 0;
  if (bra_pure && la > 0) {
    auto Ta = solid_matrix(la);
    ct.baptr.assign(2 * la + 2, 0);
    for (int A = 0; A < 2 * la + 1; ++A) {
      for (int a = 0; a < ct.ncA; ++a) {
        double v = Ta[A * ct.ncA + a];
        if (v != 0.0) ct.baent.push_back(int2{a, (int)pal_id(ct.pal, palids, v)});
      }
      ct.baptr[A + 1] = (int)ct.baent.size();
    }
    ct.nbA = (2 * la + 1) * ct.ncB;
  }
  if (bra_pure && lb > 0) {
    auto Tb = solid_matrix(lb);
    ct.bbptr.assign(2 * lb + 2, 0);
    for (int B = 0; B < 2 * lb + 1; ++B) {
      for (int b = 0; b < ct.ncB; ++b) {
        double v = Tb[B * ct.ncB + b];
        if (v != 0.0) ct.bbent.push_back(int2{b, (int)pal_id(ct.pal, palids, v)});
      }
      ct.bbptr[B + 1] = (int)ct.bbent.size();
    }
    ct.nbB = ct.nA * (2 * lb + 1);
  }
  if (ct.pal.size() >= (1u << (32 - kGatherBits))) throw std::runtime_error("coefficient palette overflow");
  if (ct.NACC >= (1 << kGatherBits) || ct.NV >= 65536 || ct.NW >= 65536) throw std::runtime_error("class too large");

  // ---------------- algorithmic flop counts (FMA = 2) ----------------
  double fp = 0;
  // geometry, rsqrt, prefactor, X and powers of Y ((rho/gamma) PC only when
  // VRR1 runs)
  fp += 32 + std::max(0, kmax - 1) - (Lab == 0 ? 3.0 : 0.0);
  // Boys and [00|0]^(m): one degree-7 polynomial for F_L; the exp(-T)
  // polynomial and the downward relation only when Lab > 0 (F_L..F_lc)
  fp += Lab == 0 ? 16.0 : 32.0 + 3.0 * Lab;
  for (int e = 1; e <= Lab; ++e)
    for (int i = ct.vlev_start[e - 1]; i < ct.vlev_start[e]; ++i) fp += ((ct.vtab[i].z >> 20) & 0xF) ? 7 : 3;
  double fc;
  if (Lab == 0 || (la == 1 && lb == 0 && lc <= 4)) {
    // (s s|C) and (p s|C) run on the register-resident kernels: powers of X,
    // the monomials Y^k X^n the accumulators read, 3 ncart(lc) + ncart(lc - 1)
    // accumulators for (p s|C) or ncart(lc), a target's one or two terms, the
    // ket transform
    const int rows = Lab ? 3 : 1;
    fp += lc > 0 ? 4.0 * (lc - 1) - std::max(0, kmax - 1) : 0.0;
    for (int k = 0; k <= kmax; ++k)
      for (auto& n : cart(lc - k)) fp += std::max(0, (n.v[0] > 0) + (n.v[1] > 0) + (n.v[2] > 0) + k - 1);
    const int nmono = ct.ncc, nless = kmax ? ncart(lc - 1) : 0;
    fp += 2.0 * (rows * nmono + nless);
    fc = 2.0 * rows * (nmono + nless) + 2.0 * ct.kent.size() * rows;
  } else {
    // weights: (x + i y)^m, the Q recursion for each m, their products
    if (lc > 0) fp += 5 + 6.0 * (lc - 1);
    for (int m = 0; m <= lc; ++m) {
      fp += 4.0 * std::max(0, lc - m - 1);
      for (int k = 0; k <= kmax && k <= lc - m; ++k) fp += (k > 0) + (m > 0 ? 2 : 0);
    }
    fp += 2.0 * ct.NACC;
    fc = 2.0 * ct.gterm.size();
  }
  ct.flops_prim = fp;
  for (const uint4& h : ct.htab) fc += 2.0 * ((h.x >> 16) - 1) * ct.nC;
  auto bra = [&](const std::vector<int>& ptr, const std::vector<int2>& ent, int nother) {
    double f = 0;
    for (size_t A = 0; A + 1 < ptr.size(); ++A) {
      int n = ptr[A + 1] - ptr[A];
      bool copy = (n == 1 && ct.pal[ent[ptr[A]].y] == 1.0);
      if (!copy) f += 2.0 * n;
    }
    return f * nother * ct.nC;
  };
  if (ct.nbA) fc += bra(ct.baptr, ct.baent, ct.ncB);
  if (ct.nbB) fc += bra(ct.bbptr, ct.bbent, ct.nA);
  ct.flops_contr = fc;
  return ct;
}

}  // namespace

namespace {
std::mutex g_hrr_mu;
std::map<std::tuple<int, int, int, int>, int> g_hrr_hints;  // (la, lb, lc, pure) -> 0: 1-q, 1: 2-q HRR
}  // namespace

void set_hrr_hint(int la, int lb, int lc, int bra_pure, int variant) {
  std::lock_guard<std::mutex> lk(g_hrr_mu);
  auto key = std::make_tuple(la, lb, lc, bra_pure ? 1 : 0);
  if (variant < 0) g_hrr_hints.erase(key); else g_hrr_hints[key] = variant;
}

int hrr_variant(int la, int lb, int lc, int bra_pure) {
  std::lock_guard<std::mutex> lk(g_hrr_mu);
  auto it = g_hrr_hints.find(std::make_tuple(la, lb, lc, bra_pure ? 1 : 0));
  return it == g_hrr_hints.end() ? 0 : it->second;
}

const ClassTables& class_tables_variant(int la, int lb, int lc, int bra_pure, int hrr2) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, int, int>, ClassTables> cache;
  std::lock_guard<std::mutex> lk(mu);
  auto key = std::make_tuple(la, lb, lc, bra_pure ? 1 : 0, (hrr2 && lb >= 2) ? 1 : 0);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  return cache.emplace(key, build(la, lb, lc, bra_pure ? 1 : 0, std::get<4>(key))).first->second;
}

const ClassTables& class_tables(int la, int lb, int lc, int bra_pure) {
  return class_tables_variant(la, lb, lc, bra_pure, hrr_variant(la, lb, lc, bra_pure));
}

// Invariants of a class's host tables; empty string when they all hold.
std::string check_class_tables(const ClassTables& ct) {
  char buf[160];
  auto bad = [&](const char* what, long long i) {
    std::snprintf(buf, sizeof(buf), "%s (entry %lld)", what, i);
    return std::string(buf);
  };
  const int Lab = ct.la + ct.lb;
  const unsigned NV = (unsigned)ct.NV, NW = (unsigned)ct.NW, NACC = (unsigned)ct.NACC;
  if ((int)ct.vlev_start.size() != Lab + 1) return "VRR1 level table size";
  // VRR1: indices in range; every entry above level 0 written once; level e
  // reads only entries written before it (levels are contiguous and ordered)
  std::vector<int> written(NV, 0);
  for (int e = 1; e <= Lab; ++e) {
    unsigned lo = NV;
    for (int i = ct.vlev_start[e - 1]; i < ct.vlev_start[e]; ++i) lo = std::min(lo, ct.vtab[i].x & 0xFFFF);
    for (int i = ct.vlev_start[e - 1]; i < ct.vlev_start[e]; ++i) {
      const uint4 it = ct.vtab[i];
      const unsigned dst = it.x & 0xFFFF, a = it.x >> 16, an = it.y & 0xFFFF, b = it.y >> 16, bn = it.z & 0xFFFF;
      const unsigned axis = (it.z >> 16) & 0xF, nq = (it.z >> 20) & 0xF;
      if (dst >= NV || a >= lo || an >= lo || axis > 2 || (nq && (b >= lo || bn >= lo)))
        return bad("VRR1 item index out of range or not yet formed", i);
      ++written[dst];
    }
  }
  for (unsigned v = 0; v < NV; ++v)
    if (written[v] != (v <= (unsigned)Lab ? 0 : 1)) return bad("VRR1 entry not formed exactly once", v);
  // accumulators
  if (ct.atab.size() != NACC) return "accumulator table size";
  for (size_t i = 0; i < ct.atab.size(); ++i)
    if ((ct.atab[i] & 0xFFFF) >= NV || (ct.atab[i] >> 16) >= NW) return bad("accumulator index", (long long)i);
  // gather: CSR and its sliced-ELL copy hold the same terms
  const int ngt = ct.nkrow * ct.nC;
  if ((int)ct.gptr.size() != ngt + 1 || (int)ct.gdst.size() != ngt) return "gather table size";
  std::vector<int> seen(ngt, 0);
  for (int r = 0; r < ngt; ++r) {
    if (ct.gdst[r] < 0 || ct.gdst[r] >= ngt || seen[ct.gdst[r]]++) return bad("gather order not a permutation", r);
    if (r && ct.gptr[ct.gdst[r] + 1] - ct.gptr[ct.gdst[r]] > ct.gptr[ct.gdst[r - 1] + 1] - ct.gptr[ct.gdst[r - 1]])
      return bad("gather order not by descending term count", r);
  }
  for (int id = 0; id < ngt; ++id)
    if (ct.gptr[id + 1] < ct.gptr[id]) return bad("gather row pointers", id);
  for (size_t q = 0; q < ct.gterm.size(); ++q)
    if ((ct.gterm[q] & kGatherMask) >= NACC || (ct.gterm[q] >> kGatherBits) >= ct.pal.size()) return bad("gather term", (long long)q);
  if ((int)ct.gslice.size() != (ngt + 31) / 32) return "sliced ELL slice count";
  for (int sl = 0; sl < (int)ct.gslice.size(); ++sl)
    for (int l = 0; l < 32; ++l) {
      const int r = 32 * sl + l;
      const int id = r < ngt ? ct.gdst[r] : -1;
      const int cnt = id >= 0 ? ct.gptr[id + 1] - ct.gptr[id] : 0;
      if (cnt > ct.gslice[sl].y) return bad("sliced ELL row longer than its slice", r);
      for (int j = 0; j < ct.gslice[sl].y; ++j) {
        const size_t q = (size_t)ct.gslice[sl].x + 32 * j + l;
        if (q >= ct.gell.size()) return bad("sliced ELL entry out of range", r);
        const unsigned e = ct.gell[q];
        if (j < cnt ? e != ct.gterm[ct.gptr[id] + j]
                    : ((e >> kGatherBits) >= ct.pal.size() || ct.pal[e >> kGatherBits] != 0.0 || (e & kGatherMask) >= NACC))
          return bad("sliced ELL differs from the CSR terms", r);
      }
    }
  // ket transform
  if ((int)ct.kptr.size() != ct.nC + 1) return "ket table size";
  for (size_t q = 0; q < ct.kent.size(); ++q)
    if (ct.kent[q].x < 0 || ct.kent[q].x >= ct.ncc || ct.kent[q].y < 0 || ct.kent[q].y >= (int)ct.pal.size())
      return bad("ket entry", (long long)q);
  // HRR: round r rows built from rows of round r-1, 2..4 terms, codes < 13
  for (int r = 1; r <= ct.nhrr; ++r)
    for (int i = ct.hstart[r]; i < ct.hstart[r + 1]; ++i) {
      const uint4 h = ct.htab[i];
      const unsigned nt = h.x >> 16, src[4] = {h.y & 0xFFFF, h.y >> 16, h.z & 0xFFFF, h.z >> 16};
      if ((int)(h.x & 0xFFFF) >= ct.hrows[r] || nt < 2 || nt > 4 || (h.w & 0xF) != 0) return bad("HRR row", i);
      for (unsigned t = 0; t < nt; ++t)
        if ((int)src[t] >= ct.hrows[r - 1] || ((h.w >> (4 * t)) & 0xF) > 12) return bad("HRR term", i);
    }
  if (ct.nhrr != (ct.hrr2 ? ct.lb / 2 + (ct.lb & 1) : ct.lb)) return "HRR round count";
  // bra transforms
  if (ct.nbA)
    for (size_t q = 0; q < ct.baent.size(); ++q)
      if (ct.baent[q].x < 0 || ct.baent[q].x >= ct.ncA) return bad("bra A entry", (long long)q);
  if (ct.nbB)
    for (size_t q = 0; q < ct.bbent.size(); ++q)
      if (ct.bbent[q].x < 0 || ct.bbent[q].x >= ct.ncB) return bad("bra B entry", (long long)q);
  return "";
}

// The tables behind (a 0|C) on one primitive, as the kernel walks them: VRR1
// items from base[i] = [00|0]^(lc+i), weights, accumulators, gather.
std::vector<double> eval_targets(const ClassTables& ct, const double PA[3], const double f[3], double rg, double h,
                                 const double X[3], double Y, const double* base) {
  static const double q[36] = LX3C_QTABLE;
  const int Lab = ct.la + ct.lb, lc = ct.lc;
  std::vector<double> v(ct.NV), W(ct.NW, 1.0), P(ct.NACC), out((size_t)ct.nkrow * ct.nC);
  for (int i = 0; i <= Lab; ++i) v[i] = base[i];
  for (const uint4& it : ct.vtab) {
    const int axis = (it.z >> 16) & 0xF, nq = (it.z >> 20) & 0xF;
    double x = PA[axis] * v[it.x >> 16] - f[axis] * v[it.y & 0xFFFF];
    if (nq) x += nq * h * (v[it.y >> 16] - rg * v[it.z & 0xFFFF]);
    v[it.x & 0xFFFF] = x;
  }
  for (int m = 0; m <= lc && lc > 0; ++m)
    harmonic_weights(
        lc, ct.kmax, m, X[0], X[1], X[2], q, [&](int k) { return std::pow(Y, k); }, [&](int i, double w) { W[i] = w; });
  for (int i = 0; i < ct.NACC; ++i) P[i] = v[ct.atab[i] & 0xFFFF] * W[ct.atab[i] >> 16];
  for (size_t id = 0; id < out.size(); ++id)
    for (int t = ct.gptr[id]; t < ct.gptr[id + 1]; ++t)
      out[id] += ct.pal[ct.gterm[t] >> kGatherBits] * P[ct.gterm[t] & kGatherMask];
  return out;
}

// HRR holds exactly for moment integrals M(a, b) = int (x-A)^a (x-B)^b w(x) dx
// of any weight w, since (x-B) = (x-A) + AB.  With the moments
// mu_k = int (x-A)^k w = 1/(k+1) per axis, feed round 0 the values
// (e 0| = prod_i mu_{e_i}, run the class's HRR rows on the host and compare
// the top round with prod_i sum_j C(b_i, j) AB_i^(b_i-j) mu_{a_i+j}.
double hrr_moment_error(const ClassTables& ct, const double AB[3]) {
  auto mu = [](int k) { return 1.0 / (k + 1); };
  std::vector<double> cur(ct.nkrow);
  for (int r = 0; r < ct.nkrow; ++r)
    cur[r] = mu(ct.erow_xyz[r].x) * mu(ct.erow_xyz[r].y) * mu(ct.erow_xyz[r].z);
  const double c[13] = {1.0, AB[0], AB[1], AB[2], 2 * AB[0], 2 * AB[1], 2 * AB[2], AB[0] * AB[0], AB[1] * AB[1],
                        AB[2] * AB[2], AB[0] * AB[1], AB[0] * AB[2], AB[1] * AB[2]};
  for (int r = 1; r <= ct.nhrr; ++r) {
    std::vector<double> nxt(ct.hrows[r], 0.0);
    for (int i = ct.hstart[r]; i < ct.hstart[r + 1]; ++i) {
      const uint4 h = ct.htab[i];
      const unsigned nt = h.x >> 16, src[4] = {h.y & 0xFFFF, h.y >> 16, h.z & 0xFFFF, h.z >> 16};
      double v = 0;
      for (unsigned t = 0; t < nt; ++t) v += c[(h.w >> (4 * t)) & 0xF] * cur[src[t]];
      nxt[h.x & 0xFFFF] = v;
    }
    cur.swap(nxt);
  }
  double worst = 0;
  auto ca = cart(ct.la), cb = cart(ct.lb);
  for (size_t ia = 0; ia < ca.size(); ++ia)
    for (size_t ib = 0; ib < cb.size(); ++ib) {
      double ref = 1.0, mag = 1.0;
      for (int x = 0; x < 3; ++x) {
        double s = 0, m = 0;
        for (int j = 0; j <= cb[ib].v[x]; ++j) {
          const double t = binom(cb[ib].v[x], j) * std::pow(AB[x], cb[ib].v[x] - j) * mu(ca[ia].v[x] + j);
          s += t;
          m += std::fabs(t);
        }
        ref *= s;
        mag *= m;
      }
      worst = std::max(worst, std::fabs(cur[ia * cb.size() + ib] - ref) / mag);
    }
  return worst;
}

// ---------------------------------------------------------------------------
// Launch shape
// ---------------------------------------------------------------------------

namespace {

struct Sizes {
  long long loop, P, Y, X, pair, aux, total;
};

// per-slot sizes (in doubles) of every stage buffer for a given T, G
void buffer_sizes(const ClassTables& ct, int Kab, int Kc, int T, int G, int mode, Sizes& s,
                  ClassDesc* d) {
  int Tp = (mode == 0 && T > 1) ? (T | 1) : T;
  if (mode == 0 && T > 1 && (T % 2 == 0)) Tp = T + 1;
  auto per_t = [&](int n) -> long long { return mode == 0 ? (long long)n * Tp : (long long)T * n; };
  auto per_tg = [&](int n) -> long long { return mode == 0 ? (long long)n * G * Tp : (long long)T * G * n; };
  const long long nK = (long long)ct.nkrow * ct.nC;
  s.pair = (long long)Kab * kPairRec + 16;  // + the tile's AB products
  s.aux = (long long)T * (3 + kAuxRec * Kc);
  s.loop = per_tg(ct.NV) + per_tg(ct.NW) + per_tg(ct.NF);
  s.P = per_t(ct.NACC);
  // region assignment: Y holds P and odd HRR levels; X holds the loop
  // buffers, the gather output (level 0) and even HRR levels.
  long long Y = s.P;
  long long X = std::max(s.loop, per_t((int)nK));
  const int R = ct.nhrr;
  for (int j = 1; j <= R; ++j) {
    long long sz = per_t(ct.hrows[j] * ct.nC);
    if (j & 1) Y = std::max(Y, sz); else X = std::max(X, sz);
  }
  int cur = (R & 1) ? 0 : 1;  // 0 = Y, 1 = X
  int baR = -1, bbR = -1;
  if (ct.nbA) { cur ^= 1; baR = cur; long long sz = per_t(ct.nbA * ct.nC); if (cur) X = std::max(X, sz); else Y = std::max(Y, sz); }
  if (ct.nbB) { cur ^= 1; bbR = cur; long long sz = per_t(ct.nbB * ct.nC); if (cur) X = std::max(X, sz); else Y = std::max(Y, sz); }
  s.Y = Y;
  s.X = X;
  s.total = s.pair + s.aux + Y + X;
  if (!d) return;
  // fill descriptor layout
  d->T = T; d->Tp = Tp; d->mode = mode; d->G = G;
  d->pair_base = 0;
  d->ab_base = Kab * kPairRec;
  d->aux_base = (int)s.pair;
  int ybase = (int)(s.pair + s.aux);
  int xbase = (int)(ybase + Y);
  auto mk_t = [&](int base, int n) {
    Buf b;
    b.base = base; b.sg = 0;
    if (mode == 0) { b.si = Tp; b.st = 1; } else { b.si = 1; b.st = n; }
    return b;
  };
  auto mk_tg = [&](int base, int n) {
    Buf b;
    b.base = base;
    if (mode == 0) { b.si = G * Tp; b.sg = Tp; b.st = 1; } else { b.si = 1; b.sg = n; b.st = G * n; }
    return b;
  };
  d->V = mk_tg(xbase, ct.NV);
  d->W = mk_tg(xbase + (int)per_tg(ct.NV), ct.NW);
  d->F = mk_tg(xbase + (int)(per_tg(ct.NV) + per_tg(ct.NW)), ct.NF);
  d->P = mk_t(ybase, ct.NACC);
  d->H[0] = mk_t(xbase, (int)nK);
  for (int j = 1; j <= R; ++j) d->H[j] = mk_t((j & 1) ? ybase : xbase, ct.hrows[j] * ct.nC);
  Buf last = d->H[R];
  if (ct.nbA) { d->BA = mk_t(baR ? xbase : ybase, ct.nbA * ct.nC); last = d->BA; }
  if (ct.nbB) { d->BB = mk_t(bbR ? xbase : ybase, ct.nbB * ct.nC); last = d->BB; }
  d->OUT = last;
  d->smem_doubles = (int)s.total;
}

}  // namespace

namespace {
std::mutex g_hint_mu;
std::map<std::tuple<int, int, int, int, int, int>, int> g_hints;  // (la, lb, lc, pure, Kab, Kc) -> CTAs/SM
}  // namespace

void set_shape_hint(int la, int lb, int lc, int bra_pure, int Kab, int Kc, int ctas) {
  std::lock_guard<std::mutex> lk(g_hint_mu);
  auto key = std::make_tuple(la, lb, lc, bra_pure ? 1 : 0, Kab, Kc);
  if (ctas <= 0) g_hints.erase(key); else g_hints[key] = ctas;
}

int shape_hint(const ClassTables& ct, int Kab, int Kc) {
  std::lock_guard<std::mutex> lk(g_hint_mu);
  auto it = g_hints.find(std::make_tuple(ct.la, ct.lb, ct.lc, ct.bra_pure ? 1 : 0, Kab, Kc));
  return it == g_hints.end() ? 0 : it->second;
}

namespace {
std::map<std::tuple<int, int, int, int, int, int>, std::pair<int, int>> g_tile_hints;  // -> (T, G)
}  // namespace

void set_tile_hint(int la, int lb, int lc, int bra_pure, int Kab, int Kc, int T, int G) {
  std::lock_guard<std::mutex> lk(g_hint_mu);
  auto key = std::make_tuple(la, lb, lc, bra_pure ? 1 : 0, Kab, Kc);
  if (T <= 0) g_tile_hints.erase(key); else g_tile_hints[key] = {T, G};
}

// The hinted tile (T triples, chunks of G primitives, G balanced over the
// chunks) when one is set for the class and it fits one CTA per SM;
// smem_bytes = -1 otherwise.
LaunchShape tile_hint_shape(const ClassTables& ct, int Kab, int Kc, int smem_limit) {
  std::pair<int, int> h{0, 0};
  {
    std::lock_guard<std::mutex> lk(g_hint_mu);
    auto it = g_tile_hints.find(std::make_tuple(ct.la, ct.lb, ct.lc, ct.bra_pure ? 1 : 0, Kab, Kc));
    if (it != g_tile_hints.end()) h = it->second;
  }
  LaunchShape sh{1, 1, 1, -1};
  if (h.first <= 0) return sh;
  const int K = Kab * Kc, T = h.first;
  int G = std::max(1, std::min(h.second, K));
  const int nch = (K + G - 1) / G;
  G = (K + nch - 1) / nch;
  const int mode = T >= 32 ? 0 : 1;
  Sizes s;
  buffer_sizes(ct, Kab, Kc, T, G, mode, s, nullptr);
  if (s.total * 8 > (long long)smem_limit - 1024) return sh;
  return LaunchShape{T, G, mode, (int)(s.total * 8)};
}

namespace {

// Largest T, then largest balanced G, whose tile fits `budget` doubles with at
// least gmin(T) primitives side by side (or all of them); smem_bytes = -1 when
// none does.
template <class GMin>
LaunchShape fit_shape(const ClassTables& ct, int Kab, int Kc, long long naux, long long budget, const GMin& gmin) {
  const int K = Kab * Kc, Gmax = std::min(K, 8);
  Sizes s;
  for (int T : {512, 256, 128, 64, 32, 16, 8, 4, 2, 1}) {
    // never a tile that half its size would hold ((pp|d) with 32 kets: T = 64
    // 28.7 us a call, T = 32 26.7)
    if (T > 1 && T >= 2 * naux) continue;
    const int mode = T >= 32 ? 0 : 1;
    int G = 0;
    while (G < Gmax) {
      buffer_sizes(ct, Kab, Kc, T, G + 1, mode, s, nullptr);
      if (s.total > budget) break;
      ++G;
    }
    if (G < std::min(K, std::max(1, gmin(T)))) continue;
    // balance the primitive chunks: same number of chunks, equal sizes
    const int nch = (K + G - 1) / G;
    G = (K + nch - 1) / nch;
    buffer_sizes(ct, Kab, Kc, T, G, mode, s, nullptr);
    return LaunchShape{T, G, mode, (int)(s.total * 8)};
  }
  return LaunchShape{1, 1, 1, -1};
}

}  // namespace

// The largest tile for `ctas` CTAs per SM.
LaunchShape largest_tile(const ClassTables& ct, int Kab, int Kc, long long naux, int smem_limit, int ctas) {
  return fit_shape(ct, Kab, Kc, naux, (smem_limit / ctas - 1024) / 8, [](int) { return 1; });
}

// Shape for one or three CTAs per SM: the largest tile, or that of fewer CTAs
// when nothing fits.  For two, the default: wide tiles (T >= 64) only with three
// primitives side by side, as each chunk of primitives costs the barriers of
// its stages ((pp|p) K = 36: T, G = 128, 2 1.53 ms, 64, 6 1.35; (pp|d) K = 9:
// 128, 1 0.90, 64, 3 0.77; asking for two gives the same shapes, as a tile of
// two leaves room for the three CTAs below); and a third CTA (of 384 threads) where it takes no
// fewer triples a tile, or still a full warp of them, and two primitives: the
// barriers of three overlap better ((fd|f) K = 9 8, 5 7.64 ms, 8, 3 6.76; (ff|d)
// K = 4 8, 4 6.25, 8, 2 5.43; (gg|i) K = 36 92.4 -> 86.0), while fewer triples lose
// more than that ((dd|f) K = 9 16, 5 4.15, 8, 5 4.53), and so does one primitive at
// a time ((gs|d) K = 9 32, 3 1.56, 32, 1 1.73).
LaunchShape choose_shape_for(const ClassTables& ct, int Kab, int Kc, long long naux, int smem_limit, int ctas,
                             long long nsub, int nsm) {
  if (ctas != 2) {
    const LaunchShape sh = largest_tile(ct, Kab, Kc, naux, smem_limit, std::max(1, ctas));
    return sh.smem_bytes < 0 && ctas > 1 ? choose_shape_for(ct, Kab, Kc, naux, smem_limit, ctas - 1) : sh;
  }
  const LaunchShape two =
      fit_shape(ct, Kab, Kc, naux, (smem_limit / 2 - 1024) / 8, [](int T) { return T >= 64 ? 3 : 1; });
  if (two.smem_bytes < 0) return choose_shape_for(ct, Kab, Kc, naux, smem_limit, 1);
  const LaunchShape three =
      fit_shape(ct, Kab, Kc, naux, (smem_limit / 3 - 1024) / 8, [](int T) { return T >= 128 ? 3 : 2; });
  if (three.smem_bytes < 0 || three.T < std::min(two.T, 32)) return two;
  // nsub sub-pairs that give no third CTA of an SM a tile (nsm = 0: unknown):
  // wide tiles keep the primitives two CTAs hold side by side instead.  400 pairs
  // x 60 kets, two launches of 200 tiles, us: (pp|p) 3 x 2 x 2 primitives G = 6
  // 125, 3 149; (pp|d) 4 187, 2 210; over 40 such classes of up to 304 tiles a
  // launch 9 % on average.  With T = 32 it goes either way ((pp|f) K = 36 G = 4
  // 354, 8 538; (dd|s) 429 and 333).
  if (nsm > 0 && three.T == two.T && two.T >= 64 && nsub * ((naux + two.T - 1) / two.T) <= 2LL * nsm) return two;
  return three;
}

// The planner's shape: a tuned tile hint (T, G) for this class, contraction
// and ket contraction when one is set and fits, or a tuned number of CTAs per
// SM, or the default.
LaunchShape choose_shape(const ClassTables& ct, int Kab, int Kc, long long naux, int smem_limit, long long nsub,
                         int nsm) {
  const LaunchShape th = tile_hint_shape(ct, Kab, Kc, smem_limit);
  if (th.smem_bytes >= 0) return th;
  const int h = shape_hint(ct, Kab, Kc);
  return choose_shape_for(ct, Kab, Kc, naux, smem_limit, h > 0 ? h : 2, nsub, nsm);
}

int place_epilogue_scratch(ClassDesc& d, long long need) {
  const bool out_in_x = d.OUT.base == d.V.base;
  const long long free_base = out_in_x ? d.P.base : d.V.base;
  const long long free_size = out_in_x ? (long long)d.V.base - d.P.base : (long long)d.smem_doubles - d.V.base;
  if (need <= free_size) return (int)free_base;
  const int base = d.smem_doubles;
  d.smem_doubles += (int)need;
  return base;
}

void set_digest_scratch(ClassDesc& d) {
  d.dscr = place_epilogue_scratch(d, (long long)d.onA * d.onB + (long long)d.T * d.nC);
}

void fill_layout(ClassDesc& d, const ClassTables& ct, const LaunchShape& sh) {
  Sizes s;
  buffer_sizes(ct, d.Kab, d.Kc, sh.T, sh.G, sh.mode, s, &d);
}

}  // namespace lx3c
