// Emitter of the tile kernel's tables (see pyro_tile.cuh for the kernel and
// pyro_fixed_math.cuh for the number formats).
#include "pyro_emit_tile.h"

#include <algorithm>
#include <cmath>
#include <functional>
#include <map>
#include <sstream>
#include <vector>

#include "pyro_emit_common.h"

namespace pyro {

namespace {
using namespace emitc;

typedef long long i64;
typedef unsigned long long u64;
typedef long double ld;

const ld LOG2E = 1.442695040888963407359924681001892137L;
const ld T_HI = 5000.0L, T_T = 5000.5L;

// fixed-point conversions; `bad` is set where a value does not fit
struct Fix {
  bool bad = false;
  i64 lg(ld v) {          // f = 50, lowest bit clear
    if (!(std::fabs((double)v) < 8000.0)) { bad = true; return 0; }
    return (i64)llroundl(v * 562949953421312.0L) * 2;
  }
  i64 lg_any(ld v) {      // f = 50, all bits
    if (!(std::fabs((double)v) < 8000.0)) { bad = true; return 0; }
    return (i64)llroundl(v * 1125899906842624.0L);
  }
  i64 coef(ld v) {        // f = 51 as two signed halves
    if (!(std::fabs((double)v) < 4000.0)) { bad = true; return 0; }
    return pair((i64)llroundl(v * 2251799813685248.0L));
  }
  i64 pair(i64 x) {       // two signed halves
    const int lo = (int)(unsigned)(u64)x;
    const i64 hi = (x - lo) / 4294967296ll;
    return (i64)(((u64)hi << 32) | (unsigned)lo);
  }
};

i64 dbits(double v) {
  i64 b;
  static_assert(sizeof b == sizeof v, "");
  __builtin_memcpy(&b, &v, 8);
  return b;
}

// log2 of lambda_k = phi_k/W_k as a function of T in range r (long double)
ld lambda(const Species& s, int r, ld T) {
  const double* a = r == 0 ? s.low : s.high;
  const ld L = ((ld)a[0] - a[6] + logl(R_GAS / P_ATM) - logl((ld)s.W)) + (1.0L - a[0]) * logl(T) + a[5] / T -
               T * ((ld)a[1] / 2 + T * ((ld)a[2] / 6 + T * ((ld)a[3] / 12 + T * (ld)a[4] / 20)));
  return L * LOG2E;
}

struct Arr { ld c, b, theta; };     // log2 k = c + b log2 T - theta log2(e)/T
ld arr_at(const Arr& a, ld T) { return a.c + a.b * log2l(T) - a.theta * LOG2E / T; }

int classes(const Reaction& r) {   // tile_other's kinds; 0: plain
  switch (r.kind) {
    case RX_ARRHENIUS: return 0;
    case RX_THREEBODY: return 1;
    case RX_PLOG: return 5;
    default: return r.n_sri >= 3 ? 4 : r.n_troe >= 3 ? 3 : 2;
  }
}

template <class T>
void array(std::ostringstream& o, const char* type, const char* name, const std::vector<T>& v) {
  o << "__device__ const " << type << " " << name << "[" << std::max<size_t>(v.size(), 1) << "] = {";
  for (size_t i = 0; i < v.size(); ++i) o << (i ? "," : "") << (i % 16 == 15 ? "\n" : "") << v[i];
  if (v.empty()) o << "0";
  o << "};\n";
}

std::vector<std::string> as_ll(const std::vector<i64>& v) {
  std::vector<std::string> s;
  for (i64 x : v) s.push_back(std::to_string(x) + "ll");
  return s;
}
std::vector<std::string> as_d(const std::vector<double>& v) {
  std::vector<std::string> s;
  for (double x : v) s.push_back(lit(x));
  return s;
}

}  // namespace

TileEmit emit_tile_unit(const Mechanism& m, TileKind what) {
  const bool deriv = what != TileKind::Rates, jac = what == TileKind::Jac;
  const bool vjp = what == TileKind::Vjp || jac;   // units that look at every reaction's products
  TileEmit out;
  const int N = m.n_species(), NR = m.n_reactions();
  if (N < 1 || N > 1022 || NR < 1) { out.why = "no reactions, or more than 1022 species"; return out; }
  for (auto& r : m.reactions)
    if (side_factors(r.reactants).size() > 3 || side_factors(r.products).size() > 3 ||
        side_factors(r.reactants).empty() || (vjp && side_factors(r.products).empty()) || (r.reversible && side_factors(r.products).empty())) {
      out.why = "a reaction has more than three factors on a side";
      return out;
    }
  const double tmid = m.species[0].t_mid;      // the range switch of every species, as in the other kernels

  // ---- temperature range: the lowest T_LO from which every rate's exponent at unit
  // concentrations is below 1190 (a product with one zero, 2^-2400, then vanishes) and
  // above -8150 + 2460 per factor (a product of zeros stays in range: |lg| < 8192; with [M] 1030 higher)
  auto folded = [&](const Reaction& r, double A, double b, double theta) {
    Arr a{log2l((ld)A), (ld)b, (ld)theta};
    for (auto& p : r.reactants) a.c -= p.second * log2l((ld)m.species[p.first].W);
    return a;
  };
  std::vector<std::vector<Arr>> forms(NR);       // the Arrhenius forms of each reaction
  for (int j = 0; j < NR; ++j) {
    const Reaction& r = m.reactions[j];
    if (r.kind == RX_PLOG)
      for (auto& q : r.plog) forms[j].push_back(folded(r, q.A, q.b, q.theta));
    else
      forms[j].push_back(folded(r, r.A, r.b, r.theta));
    if (r.kind == RX_FALLOFF) {                  // the low-pressure limit bounds the falloff rate from below
      Arr a = folded(r, r.A0, r.b0, r.theta0);
      forms[j].push_back(a);
    }
  }
  auto fits_from = [&](double lo) {
    std::vector<ld> lam(N);
    for (int i = 0; i <= 200; ++i) {
      const ld T = lo * powl(T_HI / lo, i / 200.0L);
      const int rg = T >= tmid ? 1 : 0;
      for (int k = 0; k < N; ++k) {
        lam[k] = lambda(m.species[k], rg, T);
        if (deriv && !(fabsl(lam[k]) < 1000)) return false;      // exp(L_k) itself is used
      }
      for (int j = 0; j < NR; ++j) {
        ld f = 0, g = 0;
        for (auto& p : m.reactions[j].reactants) { f += p.second * lam[p.first]; g += p.second * logl((ld)m.species[p.first].W) * LOG2E; }
        ld r = 0;
        for (auto& p : m.reactions[j].products) r += p.second * lam[p.first];
        for (auto& a : forms[j]) {
          const ld K = arr_at(a, T) + g;         // log2 of the rate constant
          const ld X = arr_at(a, T) - f + r;     // reverse exponent at unit products
          const ld nf = (ld)side_factors(m.reactions[j].reactants).size(), np = (ld)side_factors(m.reactions[j].products).size();
          const int cls = classes(m.reactions[j]);
          const ld M = cls > 0 && cls < 5 ? 1030 : 0;           // [M] from the smallest normal number
          if (!(K > -8150 + 2460 * nf + M && K < 1190 && X > -8150 + 2460 * np + M && X < 1190)) return false;
        }
      }
    }
    return true;
  };
  double t_lo = 0.0;                             // (in steps of 10 K: 160 species' lies at 290 K, below room temperature)
  for (double lo = 200.0; lo <= 400.0 && t_lo == 0.0; lo += 10.0) if (fits_from(lo)) t_lo = lo;
  if (t_lo == 0.0) { out.why = "rate constants out of range above 400 K"; return out; }
  const ld T_V = (double)(0.9999L * (ld)t_lo);   // a double: the kernel divides by T what the coefficients hold

  // ---- species tables ----------------------------------------------------------
  Fix fx;
  std::vector<i64> sp((size_t)N * 16);
  std::vector<double> hc;                        // h_k/(RT) = h0 + ... + h4 T^4 + h5/T
  std::vector<double> ed((size_t)N * 12), iw(N);
  std::ostringstream ef;
  for (int k = 0; k < N; ++k) {
    const Species& s = m.species[k];
    const SpeciesCoef C = species_coef(s);
    iw[k] = 1.0 / s.W;
    for (int r = 0; r < 2; ++r) {
      const double* a = r == 0 ? s.low : s.high;
      const ld c0 = ((ld)a[0] - a[6] + logl(R_GAS / P_ATM) - logl((ld)s.W)) * LOG2E;
      const ld c[4] = {-(ld)a[1] / 2 * T_T * LOG2E, -(ld)a[2] / 6 * T_T * T_T * LOG2E,
                       -(ld)a[3] / 12 * T_T * T_T * T_T * LOG2E, -(ld)a[4] / 20 * T_T * T_T * T_T * T_T * LOG2E};
      ld sum = fabsl(c0);
      for (ld x : c) sum += fabsl(x);
      if (!(sum < 4000)) fx.bad = true;
      i64* q = &sp[((size_t)k * 2 + r) * 8];
      q[0] = fx.lg_any(c[3]); q[1] = fx.lg_any(c[2]); q[2] = fx.lg_any(c[1]); q[3] = fx.lg_any(c[0]);
      q[4] = fx.lg_any(c0);
      q[5] = fx.coef(16 * (1.0L - a[0]));
      q[6] = fx.coef((ld)a[5] * LOG2E / T_V);
      q[7] = 0;
      hc.insert(hc.end(), C.h[r], C.h[r] + 6);
      for (int i = 0; i < 6; ++i) ed[((size_t)k * 2 + r) * 6 + i] = C.d[r][i];
    }
    for (int r = 0; r < 2; ++r) for (int i = 0; i < 6; ++i) ef << (k + r + i ? "," : "") << litf(C.d[r][i]);
  }

  // ---- reactions: cost, classes --------------------------------------------------
  struct Rx { int j, cls, shape, acc; double cost; std::vector<i64> ax; };
  std::vector<std::vector<int>> groups;          // plain duplicates share a row
  {
    std::vector<bool> used(NR, false);
    for (int j = 0; j < NR; ++j) {
      if (used[j]) continue;
      std::vector<int> g{j};
      used[j] = true;
      const Reaction& r = m.reactions[j];
      if (r.duplicate && r.kind == RX_ARRHENIUS)
        for (int q = j + 1; q < NR; ++q) {
          const Reaction& o = m.reactions[q];
          if (!used[q] && o.duplicate && o.kind == RX_ARRHENIUS && o.reversible == r.reversible &&
              o.reactants == r.reactants && o.products == r.products) { g.push_back(q); used[q] = true; }
        }
      groups.push_back(g);
    }
  }
  const int rows_all = (int)groups.size();
  auto nfac = [&](int j, bool prod) { return (int)side_factors(prod ? m.reactions[j].products : m.reactions[j].reactants).size(); };
  auto n_prod = [&](int j) { return m.reactions[j].reversible ? nfac(j, true) : 0; };
  auto cost_of = [&](int j) {
    const int cls = classes(m.reactions[j]);
    const double base = 40 + 4 * nfac(j, false) + (n_prod(j) ? 25 + 2 * n_prod(j) : 0);
    return base + (cls == 0 ? 0 : cls == 1 ? 60 : cls == 2 ? 150 : cls == 5 ? 150 : 320) + 18.0 * m.reactions[j].efficiencies.size();
  };

  // ---- block shape -----------------------------------------------------------------
  // Measured (2^20 states of 53 species / 325 reactions, energy input): two blocks of 12
  // warps an SM 7.3 ms, one of 24 warps 7.6, two of 8 warps 7.9, one of 16 warps 7.8; with
  // the rows in more than one chunk two blocks lose (8.3 ms and more).  10 species / 21
  // reactions: eight blocks of 4 warps 0.81 ms, four of 8 warps 0.96 ms; 160 / 1100
  // (2^18 states): one block of 24 warps 5.6 ms, of 16 warps 6.4 ms.  Between them, 16 to 30
  // species: 60 rows, 4096 states by 4, 8 and 12 warps 38.5, 32.7, 33.0 us, 2^20 states 1.76,
  // 1.77, 1.90 ms; 80 rows 43.9, 36.6, 35.8 us, 2.33, 2.39, 2.36 ms; 110 rows 54.3, 38.8, 37.5
  // us, 3.11, 3.19, 3.02 ms: 8 warps are within 6 % of the best at every size.
  int mrows = 0;                                 // reactions with an [M] adjoint
  for (int j = 0; j < NR; ++j) if (classes(m.reactions[j])) ++mrows;
  const int fixed_bytes = jac ? 8192 + 1280 * (N + 1) + 6 * 24 * 256 + 32 * (4 * 8 + 3 * 8 + 8 + 4) + 256
                        : vjp ? 8192 + 1024 * (N + 1) + 256 * (mrows + 2) + 3 * 24 * 256 + 32 * (5 * 8 + 3 * 8 + 8 + 4) + 256
                        : deriv ? 8192 + 1024 * (N + 1) + 32 * (8 * 8 + 3 * 8 + 8 + 4) + 256 : 8192 + 512 * (N + 1) + 2064 + 256;
  int warps = rows_all < 48 ? 4 : rows_all < 120 ? 8 : 12;
  int minb = 24 / warps + (warps == 4 ? 2 : 0);
  auto red = [](int w) { return w * 256 + 6 * 256 + 14 * 128 + w * 13 * 128; };   // scratch of the temperature solve, in the rows
  while (minb > 1 && fixed_bytes + std::max(rows_all * 256, red(warps)) > kSmemPerSm / minb - kSmemPerBlock) --minb;
  if (minb == 1) warps = 24;

  // integer energy coefficients: column q scaled by 2^xs[q], the largest in [2^(hb-1), 2^hb),
  // so that a warp's sums over its species stay below 2^63 while sum |Y| < 2 (TileDot).  By
  // the number of all species, hb was 54 for 160 of them: the largest coefficients are the
  // light species', ~100 times the mixture's, and the mean error of T was 2.2e-15; now it is 1.5e-16 (FP64 sums 5.4e-16).
  std::vector<i64> ex((size_t)N * 12);
  std::vector<int> xs(6, 0);
  int hb = 57;
  while ((1 << (62 - hb)) < (N + warps - 1) / warps) --hb;
  for (int q = 0; q < 6; ++q) {
    double mx = 0.0;
    for (int i = q; i < 12 * N; i += 6) mx = std::max(mx, std::fabs(ed[i]));
    if (mx > 0.0) xs[q] = hb - 1 - std::ilogb(mx);
    for (int i = q; i < 12 * N; i += 6) ex[i] = fx.pair(llroundl(ldexpl((ld)ed[i], xs[q])));
  }

  const int lim = std::min(kSmemMaxBlock, kSmemPerSm / minb - kSmemPerBlock) - fixed_bytes;
  const int max_rows = lim / 256;
  if (lim < red(warps) || max_rows < 8) { out.why = "species arrays do not fit in shared memory"; return out; }
  const int chunks = (rows_all + max_rows - 1) / max_rows;
  if (vjp && chunks > 1) { out.why = "the reactions do not fit in shared memory at once"; return out; }
  const int rows = (rows_all + chunks - 1) / chunks;
  const int tile_rows = std::max(rows, (red(warps) + 255) / 256);

  // groups to chunks (equal rows; heaviest first so that costs even out)
  std::vector<int> order(groups.size());
  for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
  auto gcost = [&](int g) { double c = 0; for (int j : groups[g]) c += cost_of(j); return c; };
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return gcost(a) > gcost(b); });
  std::vector<std::vector<int>> in_chunk(chunks);
  {
    std::vector<double> load(chunks, 0.0);
    for (int g : order) {
      int best = -1;
      for (int c = 0; c < chunks; ++c)
        if ((int)in_chunk[c].size() < rows && (best < 0 || load[c] < load[best])) best = c;
      in_chunk[best].push_back(g);
      load[best] += gcost(g);
    }
  }
  // classes present, in code order: plain reactions by (factors, reversible), then the others
  std::map<int, int> class_id;
  auto key_of = [&](int j) {
    if (classes(m.reactions[j])) return 8;
    return (std::max(nfac(j, false), vjp ? nfac(j, true) : n_prod(j)) > 2 ? 2 : 0) + (n_prod(j) > 0 ? 1 : 0);
  };
  for (int j = 0; j < NR; ++j) class_id[key_of(j)] = 0;
  class_id[8] = 0;
  int ncls = 0;
  for (auto& kv : class_id) kv.second = ncls++;

  std::vector<i64> rx, ax;
  std::vector<double> rd, fxa;                   // b, theta of a record; FP64 companions of ax
  std::vector<int> seg;
  std::vector<int> row_of(groups.size()), mrow_of(NR, -1);
  int mrow = 0;
  for (int ch = 0; ch < chunks; ++ch) {
    std::vector<std::vector<int>> mine(warps);
    std::vector<double> load(warps, 0.0);
    int row = 0;
    for (int g : in_chunk[ch]) {
      row_of[g] = row++;
      const int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
      mine[w].push_back(g);
      load[w] += gcost(g);
    }
    for (int w = 0; w < warps; ++w) {
      for (auto& kv : class_id) {
        seg.push_back((int)(rx.size() / 8));
        for (int g : mine[w])
          for (size_t q = 0; q < groups[g].size(); ++q) {
            const int j = groups[g][q];
            if (key_of(j) != kv.first) continue;
            const Reaction& r = m.reactions[j];
            const int cls = classes(r);
            const Arr a = forms[j][0];
            i64 rec[8] = {0};
            if (cls != 5) {
              rec[0] = fx.lg(a.c);
              rec[1] = fx.coef(16 * a.b);
              rec[2] = fx.coef(-a.theta * LOG2E / T_V);
            }
            // the adjoint needs the products of an irreversible reaction too
            const std::vector<int> fr = side_factors(r.reactants),
                                   fp = r.reversible || vjp ? side_factors(r.products) : std::vector<int>();
            auto at = [](const std::vector<int>& f, size_t i) { return (u64)(i < f.size() ? f[i] : 0); };
            rd.push_back(r.b);
            rd.push_back(r.theta);
            if (cls == 0) {       // byte offsets into the species arrays and of the row
              auto off = [&](const std::vector<int>& f, size_t i) { return (u64)((i < f.size() ? f[i] : N) * 256); };
              rec[3] = (i64)(off(fr, 0) | off(fr, 1) << 32);
              rec[4] = (i64)(off(fr, 2) | off(fp, 0) << 32);
              rec[5] = (i64)(off(fp, 1) | off(fp, 2) << 32);
              rec[6] = (i64)((u64)row_of[g] * 256 | (u64)(q > 0 ? 1 : 0) << 32);
              rx.insert(rx.end(), rec, rec + 8);
              continue;
            }
            rec[3] = (i64)(at(fr, 0) | at(fr, 1) << 16 | at(fr, 2) << 32 | at(fp, 0) << 48);
            rec[4] = (i64)(at(fp, 1) | at(fp, 2) << 16 | (u64)row_of[g] << 32 | (u64)fr.size() << 48 | (u64)fp.size() << 52 | (u64)cls << 56 |
                           (u64)(r.reversible ? 1 : 0) << 60);
            rec[6] = (i64)mrow;
            mrow_of[j] = mrow++;
            rec[5] = (i64)ax.size();
            {                                    // auxiliary data
              std::vector<i64> x(16, 0);
              std::vector<double> fd(16, 0.0);
              if (cls == 5) {
                const size_t nn = r.plog.size();
                x[1] = (i64)nn;
                for (size_t i = 0; i < nn; ++i) {
                  const Arr& f = forms[j][i];
                  const ld lp = log2l((ld)r.plog[i].p);
                  x.push_back(fx.lg(lp));
                  x.push_back(dbits(i + 1 < nn ? (double)(1.0L / (log2l((ld)r.plog[i + 1].p) - lp)) : 0.0));
                  for (double v : {0.0, 0.0, 0.0, r.plog[i].b, r.plog[i].theta}) fd.push_back(v);
                  x.push_back(fx.lg(f.c)); x.push_back(fx.coef(16 * f.b)); x.push_back(fx.coef(-f.theta * LOG2E / T_V));
                }
                if (nn < 2) fx.bad = true;
              } else {
                for (auto& e : r.efficiencies) {
                  const double c = (e.second - 1.0) / m.species[e.first].W;
                  if (c == 0.0) continue;
                  x[0]++;
                  x.push_back(e.first);
                  x.push_back(dbits(c));
                }
              }
              if (cls >= 2 && cls <= 4) {
                x[2] = fx.lg(log2l((ld)r.A0) - log2l((ld)r.A));
                x[3] = fx.coef(16 * ((ld)r.b0 - r.b));
                x[4] = fx.coef(-((ld)r.theta0 - r.theta) * LOG2E / T_V);
                fd[0] = r.b0 - r.b;
                fd[1] = r.theta0 - r.theta;
              }
              // a term that is below 2^-1100 at every T of the range is left out
              auto term = [&](ld slope, ld at_lo) { return at_lo > -1100 && (fabsl(slope) < 4000 || (fx.bad = true)); };
              auto add = [&](i64 c, ld t, ld v) {      // an exponential of S: c, slopes in t and v
                fd[2 + 2 * x[1]] = (double)(t / (T_T * LOG2E));            // its logarithmic slope in T: g0 + g2/T^2
                fd[3 + 2 * x[1]] = (double)(-v * T_V / LOG2E);
                i64* e = &x[5 + 3 * x[1]++];
                e[0] = c; e[1] = fx.coef(t); e[2] = fx.coef(v);
              };
              if (cls == 3) {
                const ld A = r.troe[0], s3 = -T_T / r.troe[1] * LOG2E, s1 = -T_T / r.troe[2] * LOG2E;
                if (A != 1 && term(s3, s3 * t_lo / T_T)) add(fx.lg(log2l(fabsl(1 - A))) | (A > 1 ? 1 : 0), s3, 0);
                if (A > 0 && term(s1, s1 * t_lo / T_T)) add(fx.lg(log2l(A)), s1, 0);
                if (r.n_troe == 4) {
                  const ld s2 = -(ld)r.troe[3] / T_V * LOG2E;
                  if (term(s2, s2 * T_V / T_HI)) add(0, 0, s2);
                }
              } else if (cls == 4) {
                const ld d = r.n_sri >= 5 ? r.sri[3] : 1.0, e = r.n_sri >= 5 ? r.sri[4] : 0.0;
                const ld sb = -(ld)r.sri[1] * LOG2E / T_V, sc = -T_T / r.sri[2] * LOG2E;
                if (r.sri[0] > 0 && term(sb, sb * T_V / T_HI)) add(fx.lg(log2l((ld)r.sri[0])), 0, sb);
                if (term(sc, sc * t_lo / T_T)) add(0, sc, 0);
                x[14] = fx.lg(log2l(d));
                x[15] = fx.coef(16 * e);
                fd[8] = (double)e;
              }
              if (x.size() % 2) x.push_back(0);      // 16-byte units
              fd.resize(x.size(), 0.0);
              ax.insert(ax.end(), x.begin(), x.end());
              fxa.insert(fxa.end(), fd.begin(), fd.end());
            }
            rx.insert(rx.end(), rec, rec + 8);
          }
      }
      seg.push_back((int)(rx.size() / 8));
    }
  }
  if (fx.bad) { out.why = "a coefficient does not fit the fixed-point range"; return out; }

  // ---- species sums: owners balanced by entries, lists per chunk ------------------
  std::vector<std::vector<std::pair<int, int>>> terms(N);      // (group, nu)
  for (size_t g = 0; g < groups.size(); ++g)
    for (auto& q : net_nu(m.reactions[groups[g][0]])) if (q.second) terms[q.first].push_back({(int)g, q.second});
  const int kpw = (N + warps - 1) / warps;
  std::vector<std::vector<int>> owned(warps);
  {
    std::vector<int> idx(N);
    for (int k = 0; k < N; ++k) idx[k] = k;
    std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) { return terms[a].size() > terms[b].size(); });
    std::vector<size_t> load(warps, 0);
    for (int k : idx) {
      int best = -1;
      for (int w = 0; w < warps; ++w)
        if ((int)owned[w].size() <= kpw && (best < 0 || load[w] < load[best])) best = w;
      owned[best].push_back(k);
      load[best] += terms[k].size() + 1;
    }
  }
  int kpo = 0;
  for (auto& v : owned) kpo = std::max(kpo, (int)v.size());
  std::vector<int> chunk_of(groups.size());
  for (int ch = 0; ch < chunks; ++ch) for (int g : in_chunk[ch]) chunk_of[g] = ch;
  std::vector<int> wl, wo, we, wc;
  int hb_max = 0;
  for (int ch = 0; ch < chunks; ++ch)
    for (int w = 0; w < warps; ++w)
      for (int i = 0; i < kpo; ++i) {
        int ends[4], sum = 0, no = 0;
        ends[0] = (int)we.size();
        for (int pass = 0; pass < 3; ++pass) {
          if (i < (int)owned[w].size())
            for (auto& t : terms[owned[w][i]])
              if (chunk_of[t.first] == ch && (t.second == 1 ? 0 : t.second == -1 ? 1 : 2) == pass) {
                we.push_back(row_of[t.first] * 256);
                wc.push_back(t.second);
                sum += std::abs(t.second);
                no += pass == 2;
              }
          while (we.size() % 4) { we.push_back(tile_rows * 256); wc.push_back(0); }   // the zero row
          ends[pass + 1] = (int)we.size();
        }
        wl.insert(wl.end(), ends, ends + 4);
        int hb = 3;                              // headroom bits of the sum, more than its terms take
        while ((1 << hb) <= sum) ++hb;
        hb_max = std::max(hb_max, hb);
        wo.push_back(i < (int)owned[w].size() ? owned[w][i] : -1);
        wo.push_back(hb + 256 * no);
      }
  // spare elements (the loops read one ahead)
  for (int q = 0; q < 16; ++q) rx.push_back(0);
  for (int q = 0; q < 4; ++q) { wl.push_back(0); we.push_back(tile_rows * 256); wc.push_back(0); }
  for (int q = 0; q < 2; ++q) wo.push_back(-1);
  for (int q = 0; q < 64; ++q) ax.push_back(0);  // and the prefetches touch up to 512 bytes

  // adjoint lists: per owned species its factor occurrences (row of Db, the other factors'
  // offsets) and its efficiency terms (row of the [M] adjoint, coefficient)
  std::vector<int> vl, v1, v2, v3;
  // dense Jacobian: per species row the terms of column T and of u_k, and the stream of terms
  // per column (see pyro_tile_jac.cuh); the last row is the temperature's
  std::vector<int> jk, jl, jt, je, jx;
  std::vector<double> jc;
  if (jac) {
    for (int w = 0; w < warps; ++w) for (int i = 0; i < kpo; ++i) jk.push_back(i < (int)owned[w].size() ? owned[w][i] : -1);
    auto terms_of = [&](int g, int times, std::vector<std::vector<int>>& col) {   // times: nu of the row
      const Reaction& r = m.reactions[groups[g][0]];
      for (int side = 0; side < (r.reversible ? 2 : 1); ++side) {
        const std::vector<int> f = side_factors(side ? r.products : r.reactants);
        for (size_t q = 0; q < f.size(); ++q) {
          std::vector<int> o;
          for (size_t z = 0; z < f.size(); ++z) if (z != q) o.push_back(f[z]);
          if (o.empty()) o.push_back(N);
          const int minus = (times < 0) != (side == 1) ? 1 : 0;
          for (int t = 0; t < std::abs(times); ++t) {
            col[f[q]].push_back(row_of[g] * 256 | minus | (o.size() > 1 ? 2 : 0));
            col[f[q]].push_back(o[0] | (o.size() > 1 ? o[1] << 16 : 0));
          }
        }
      }
      const int j = groups[g][0];
      if (mrow_of[j] >= 0)
        for (auto& e : r.efficiencies) {
          if (e.second == 1.0) continue;
          col[e.first].push_back(mrow_of[j] * 256 | 4);
          col[e.first].push_back((int)jc.size());
          jc.push_back(times * (e.second - 1.0));
        }
    };
    // a stream of two-term units: the columns first, first + step, ...
    auto flush = [&](std::vector<std::vector<int>>& col, int first, int step) {
      je.push_back((int)jx.size() / 4);
      for (int c = first; c < N; c += step) {
        if (col[c].empty()) { col[c].push_back(16); col[c].push_back(0); }
        col[c][col[c].size() - 2] |= 8;
        jx.insert(jx.end(), col[c].begin(), col[c].end());
      }
      while (jx.size() % 4) { jx.push_back(16); jx.push_back(0); }
    };
    for (int k = 0; k < N; ++k) {
      std::vector<std::vector<int>> col(N);
      jl.push_back((int)jt.size());
      auto add = [&](int row, int nu) { for (int q = 0; q < std::abs(nu); ++q) jt.push_back(row * 256 | (nu < 0 ? 1 : 0)); };
      for (auto& t : terms[k]) { add(row_of[t.first], t.second); terms_of(t.first, t.second, col); }
      jl.push_back((int)jt.size());
      jl.push_back((int)jt.size());
      for (auto& t : terms[k]) if (mrow_of[groups[t.first][0]] >= 0) add(mrow_of[groups[t.first][0]], t.second);
      jl.push_back((int)jt.size());
      flush(col, 0, 1);
    }
    std::vector<std::vector<int>> col(N);
    for (size_t g = 0; g < groups.size(); ++g) terms_of((int)g, 1, col);
    for (int w = 0; w < warps; ++w) flush(col, w, warps);
    for (int q = 0; q < 16; ++q) jx.push_back(16);   // the streams are read ahead
  }
  if (vjp && !jac) {
    for (int w = 0; w < warps; ++w)
      for (int i = 0; i < kpo; ++i) {
        if (i >= (int)owned[w].size()) { for (int q = 0; q < 8; ++q) vl.push_back(q ? 0 : -1); continue; }
        const int k = owned[w][i];
        int h[8] = {k, (int)v1.size() / 2, 0, 0, (int)v2.size() / 4, 0, (int)v3.size() / 4, 0};
        for (int side = 0; side < 2; ++side) {
          for (size_t g = 0; g < groups.size(); ++g) {
            const Reaction& r = m.reactions[groups[g][0]];
            if (side && !r.reversible) continue;
            const std::vector<int> f = side_factors(side ? r.products : r.reactants);
            for (size_t q = 0; q < f.size(); ++q) {
              if (f[q] != k) continue;
              std::vector<int> o;
              for (size_t z = 0; z < f.size(); ++z) if (z != q) o.push_back(f[z] * 256);
              if (o.empty()) o.push_back(N * 256);
              if (o.size() == 1) { v1.push_back(row_of[g] * 256); v1.push_back(o[0]); }
              else for (int x : {row_of[g] * 256, o[0], o[1], side}) v2.push_back(x);
            }
          }
          h[2 + side] = (int)v1.size() / 2;
        }
        for (int j = 0; j < NR; ++j)
          for (auto& e : m.reactions[j].efficiencies) {
            const double c = (e.second - 1.0) / m.species[e.first].W;
            if (e.first != k || c == 0.0 || mrow_of[j] < 0) continue;
            const u64 b = (u64)dbits(c);
            for (int x : {mrow_of[j] * 256, 0, (int)(unsigned)b, (int)(unsigned)(b >> 32)}) v3.push_back(x);
          }
        h[5] = (int)v2.size() / 4;
        h[7] = (int)v3.size() / 4;
        vl.insert(vl.end(), h, h + 8);
      }
  }

  // ---- the unit -------------------------------------------------------------------
  std::ostringstream o;
  o << "// Tile kernel of mechanism '" << m.name << "': " << N << " species, " << NR << " reactions.\n"
    << "#define NSP " << N << "\n#define NW " << warps << "\n#define TILE_MINB " << minb << "\n#define KPW " << kpw
    << "\n#define TILE_ROUND " << (hb_max > 7 ? 1 : 0) << "\n#define KPO " << kpo << "\n#define NCH " << chunks << "\n#define NCLS " << ncls << "\n#define TILE_ROWS "
    << tile_rows << "\n#define TMID " << lit(tmid) << "\n#define TILE_OPEN " << kTileOpen << "\n#define T_LO " << lit(t_lo) << "\n#define T_HI "
    << lit((double)T_HI) << "\n#define T_V " << lit((double)T_V) << "\n#define T_T " << lit((double)T_T)
    << "\n#define T_INV_R " << lit((double)(1.0L / R_GAS)) << "\n#define T_INV_R_LO "
    << lit((double)(1.0L / R_GAS - (ld)(double)(1.0L / R_GAS))) << "\n#define T_LG_R " << fx.lg(log2l(R_GAS)) << "ll\n";
  o << "#include \"pyro_fixed_math.cuh\"\n";
  {
    std::vector<std::string> e2, l2;
    for (int j = 0; j < 1024; ++j) e2.push_back(std::to_string((u64)roundl(exp2l(j / 1024.0L) * 9223372036854775808.0L)) + "ull");
    for (int j = 0; j < 256; ++j) {
      const unsigned rc = (unsigned)roundl(2048.0L / (1.0L + (j + 0.5L) / 256));
      l2.push_back("{" + std::to_string((i64)llroundl(-log2l(rc / 2048.0L) * 4611686018427387904.0L)) + "ll," +
                   std::to_string(rc) + "u,0u}");
    }
    array(o, "unsigned long long", "t_exp2", e2);
    array(o, "pfx::Log2Entry", "t_log2", l2);
  }
  array(o, "__align__(16) long long", "t_sp", as_ll(sp));
  if (!deriv) {
    o << "__device__ const __align__(16) float t_ef[" << 12 * N << "] = {" << ef.str() << "};\n";
    array(o, "__align__(16) double", "t_ed", as_d(ed));
  }
  array(o, "double", "t_iw", as_d(iw));
  if (!deriv) {
    array(o, "__align__(16) long long", "t_ex", as_ll(ex));
    for (int& q : xs) q += 61;                   // f of the sums: the column's scale and Y's 61
    array(o, "int", "t_exs", xs);
  }
  array(o, "__align__(16) long long", "t_rx", as_ll(rx));
  array(o, "__align__(16) long long", "t_ax", as_ll(ax));
  array(o, "int", "t_seg", seg);
  array(o, "__align__(16) int", "t_wl", wl);
  array(o, "__align__(8) int", "t_wo", wo);
  array(o, "__align__(16) int", "t_we", we);
  array(o, "signed char", "t_wc", wc);
  if (deriv) {
    array(o, "__align__(16) double", "t_rd", as_d(rd));
    array(o, "double", "t_fx", as_d(fxa));
    array(o, "double", "t_h", as_d(hc));
    if (jac) {
      std::vector<double> cp;
      for (auto& sp : m.species) {
        const SpeciesCoef c = species_coef(sp);
        for (int r = 0; r < 2; ++r) { cp.insert(cp.end(), c.cp[r], c.cp[r] + 5); cp.insert(cp.end(), c.cpd[r], c.cpd[r] + 4); cp.push_back(0.0); }
      }
      o << "#define T_MROWS " << mrows << "\n#define T_NROWS " << rows << "\n#define T_R " << lit((double)R_GAS) << "\n";
      array(o, "double", "t_cp", as_d(cp));
      array(o, "int", "t_jk", jk);
      array(o, "__align__(16) int", "t_jl", jl);
      array(o, "int", "t_jt", jt);
      array(o, "int", "t_je", je);
      array(o, "__align__(16) int", "t_jx", jx);
      array(o, "double", "t_jc", as_d(jc));
    } else if (vjp) {
      o << "#define T_MROWS " << mrows << "\n";
      array(o, "__align__(16) int", "t_vl", vl);
      array(o, "__align__(8) int", "t_v1", v1);
      array(o, "__align__(16) int", "t_v2", v2);
      array(o, "__align__(16) int", "t_v3", v3);
    }
  }
  o << (deriv ? "#define TILE_PLAIN" : "#define TILE_PLAIN(SGN)");
  for (auto& kv : class_id) {
    if (kv.first == 8) continue;
    const int c = kv.second;
    o << " \\\n  { const int a = __ldg(seg + " << c << "), b = __ldg(seg + " << c + 1 << "); if (a < b) "
      << (jac ? "jac_plain<" : vjp ? "vjp_plain<" : deriv ? "jvp_plain<" : "tile_plain<") << (kv.first & 2 ? 3 : 2) << ", " << (kv.first & 1 ? "true" : "false")
      << (jac ? ">(s, a, b, u, v, invT, invT2, sum, lane); }" : vjp ? ">(s, a, b, u, v, invT, invT2, Tb, lane); }" : deriv ? ">(s, a, b, u, v, u1, u2, lane); }" : ", SGN>(s, a, b, u, v, lane); }");
  }
  o << (jac ? "\n#include \"pyro_tile_jac.cuh\"\n" : vjp ? "\n#include \"pyro_tile_vjp.cuh\"\n" : deriv ? "\n#include \"pyro_tile_jvp.cuh\"\n" : "\n#include \"pyro_tile.cuh\"\n");
  out.source = o.str();
  out.warps = warps;
  out.smem_bytes = fixed_bytes + tile_rows * 256;
  out.t_lo = t_lo;
  out.chunks = chunks;
  out.rows = rows;
  out.scratch_bytes = jac ? (2 * tile_rows + 2 * (mrows + 1)) * 256 : 0;
  return out;
}

}  // namespace pyro
