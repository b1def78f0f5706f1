// Emitter of the transport tile kernel's tables (the kernel: pyro_transport.cuh).
#include <algorithm>
#include <cmath>
#include <sstream>
#include <vector>

#include "pyro_emit_common.h"
#include "pyro_emit_tile.h"

namespace pyro {

namespace {
using namespace emitc;
typedef long long i64;
typedef unsigned long long u64;
typedef long double ld;

const ld LN2 = 0.693147180559945309417232121458176568L;

// coefficients in t = (log2 T - log2 1000)/4 of a polynomial in ln T of degree 4
void recentre(const double* a, ld* b) {
  const ld c = logl(1000.0L), h = 4 * LN2;       // ln T = c + h t
  for (int m = 0; m < 5; ++m) b[m] = 0;
  for (int m = 4; m >= 0; --m) {                 // b <- b (c + h t) + a_m
    ld nb[5];
    for (int i = 0; i < 5; ++i) nb[i] = c * b[i] + (i ? h * b[i - 1] : 0);
    nb[0] += a[m];
    for (int i = 0; i < 5; ++i) b[i] = nb[i];
  }
}

i64 halves(i64 x) {
  const int lo = (int)(unsigned)(u64)x;
  const i64 hi = (x - lo) / 4294967296ll;
  return (i64)(((u64)hi << 32) | (unsigned)lo);
}

template <class T, class F>
void array(std::ostringstream& o, const char* type, const char* name, const std::vector<T>& v, F str) {
  o << "__device__ const __align__(16) " << type << " " << name << "[" << std::max<size_t>(v.size(), 1) << "] = {";
  for (size_t i = 0; i < v.size(); ++i) o << (i ? "," : "") << (i % 16 == 15 ? "\n" : "") << str(v[i]);
  if (v.empty()) o << "0";
  o << "};\n";
}

}  // namespace

TransportTile emit_transport_tile(const Mechanism& m) {
  TransportTile out;
  const int N = m.n_species();
  if (!m.has_transport || N < 4 || N > 400) return out;
  const TransportFits& tf = m.transport;
  const double t_lo = 200.0, t_hi = 5000.0;
  const ld tl = log2l(t_lo / 1000.0L) / 4, th = log2l(t_hi / 1000.0L) / 4;

  // ---- fits in t ---------------------------------------------------------------
  std::vector<double> fit;
  ld pmin = 1e300L;
  for (int k = 0; k < N; ++k) {
    ld b[5], c[5];
    recentre(&tf.visc[(size_t)k * 5], b);
    recentre(&tf.cond[(size_t)k * 5], c);
    for (int i = 0; i <= 64; ++i) {
      const ld t = tl + (th - tl) * i / 64;
      pmin = std::min(pmin, fabsl(b[0] + t * (b[1] + t * (b[2] + t * (b[3] + t * b[4])))));
    }
    for (ld v : b) fit.push_back((double)v);
    for (ld v : c) fit.push_back((double)v);
  }
  if (!(pmin > 0) || !std::isfinite((double)pmin)) return out;
  const int sv = ilogbl(pmin), sw = 2 * sv;      // x/P 2^sv, x/P^2 2^sw below one

  // ---- Wilke's matrices, each row scaled by a power of two: the largest coefficient below 2^hb,
  // so that sums of products of halves stay below 2^63 (as in the mixture collapse).  By row:
  // the rows of heavy species are 10^-2 of the largest, and one scale for a matrix left
  // mu with a mean error of 2.0e-15 (53 species; FP64 sums 3.4e-16)
  auto W = [&](int k) { return (ld)m.species[k].W; };
  auto wil = [&](int k, int j, int q) {
    const ld c = 1.0L / sqrtl(8.0L * (1.0L + W(k) / W(j))), g = powl(W(j) / W(k), 0.25L);
    return q == 0 ? c : q == 1 ? 2 * c * g : c * g * g;
  };
  int hb = 57;
  while ((1 << (62 - hb)) < N) --hb;
  std::vector<i64> wk((size_t)N * N * 4, 0), we;   // and per row the f of the three sums
  for (int k = 0; k < N; ++k) we.insert(we.end(), 4, 0);
  for (int q = 0; q < 3; ++q) {
    ld mx = 0, mn = 1e300L;
    for (int k = 0; k < N; ++k) {
      ld row = 0;
      for (int j = 0; j < N; ++j) { row = std::max(row, wil(k, j, q)); mn = std::min(mn, wil(k, j, q)); }
      mx = std::max(mx, row);
      const int f = hb - 1 - ilogbl(row);
      for (int j = 0; j < N; ++j) wk[((size_t)k * N + j) * 4 + q] = halves(llroundl(ldexpl(wil(k, j, q), f)));
      we[(size_t)k * 4 + q] = f + 61 + (q == 0 ? 0 : q == 1 ? sv : sw);     // the row's scale, that of x, x/P or x/P^2
    }
    if (mn < mx * 1e-4L) return out;             // few bits left for the smallest: the FP64 kernel
  }

  // ---- pairs in rounds of a tournament (circle method: player 0 stays) ------------------
  const int M = N + (N & 1), rounds = M - 1, ppr = M / 2;
  const int real = N / 2;                        // pairs of a round (a bye where N is odd)
  int nw = 4;
  double best = 0;
  for (int w = 4; w <= 16; ++w) {
    const double eff = (double)real / (w * ((real + w - 1) / w));
    if (eff >= best - 1e-9) { best = eff; nw = w; }
  }
  const int per = (real + nw - 1) / nw;
  std::vector<std::vector<i64>> recs(nw);
  for (int r = 0; r < rounds; ++r) {
    std::vector<std::pair<int, int>> pairs;
    for (int i = 0; i < ppr; ++i) {
      auto player = [&](int pos) { return pos == 0 ? 0 : 1 + (pos - 1 + r) % (M - 1); };
      const int a = player(i), b = player(M - 1 - i);
      if (a < N && b < N) pairs.push_back({a, b});
    }
    for (int s = 0; s < nw * per; ++s) {
      auto& R = recs[s % nw];
      if (s >= (int)pairs.size()) {
        for (int i = 0; i < 6; ++i) R.push_back(0);
        R.push_back(-1); R.push_back(0);
        continue;
      }
      const int k = pairs[s].first, j = pairs[s].second;
      ld b[5];
      recentre(&tf.diff[((size_t)k * N + j) * 5], b);
      ld sum = 0;
      for (ld v : b) sum += fabsl(v);
      if (!(sum > 0) || !std::isfinite((double)sum)) return out;
      const int sc = 60 - ilogbl(sum);           // every partial sum below 2^61
      for (int i = 4; i >= 0; --i) R.push_back((i64)llroundl(ldexpl(b[i], sc)));
      R.push_back(sc);
      R.push_back((i64)((u64)(unsigned)(k * 256) | (u64)(unsigned)(j * 256) << 32));
      R.push_back(0);
    }
  }
  std::vector<i64> pt;
  for (auto& R : recs) pt.insert(pt.end(), R.begin(), R.end());
  for (int i = 0; i < 8; ++i) pt.push_back(0);

  const int smem = 5 * N * 256 + 4 * nw * 256 + nw * 128 + 3 * 256 + 256 + 128 + 64;
  if (smem > kSmemMaxBlock) return out;
  int minb = std::max(1, std::min({kSmemPerSm / (smem + kSmemPerBlock), 832 / (32 * nw)}));

  std::ostringstream o;
  o << "// Transport tile kernel of mechanism '" << m.name << "': " << N << " species.\n#define NSP " << N << "\n#define NW "
    << nw << "\n#define KPW " << (N + nw - 1) / nw << "\n#define TT_MINB " << minb << "\n#define TT_ROUNDS " << rounds
    << "\n#define TT_PER_WARP " << per << "\n#define TT_PAIRS_W " << rounds * per << "\n#define TT_LO " << lit(t_lo)
    << "\n#define TT_HI " << lit(t_hi) << "\n#define TT_LGC " << (i64)llroundl(log2l(1000.0L) * 576460752303423488.0L)
    << "ll\n#define TT_SV " << lit((double)ldexpl(1, sv)) << "\n#define TT_SW " << lit((double)ldexpl(1, sw)) << "\n#define TILE_OPEN " << kTileOpen << "\n#include \"pyro_fixed_math.cuh\"\n";
  auto d = [](double v) { return lit(v); };
  auto l = [](i64 v) { return std::to_string(v) + "ll"; };
  std::vector<double> iw;
  for (auto& s : m.species) iw.push_back(1.0 / s.W);
  array(o, "double", "tt_iw", iw, d);
  array(o, "double", "tt_fit", fit, d);
  array(o, "long long", "tt_wilke", wk, l);
  array(o, "int", "tt_wf", we, [](i64 v) { return std::to_string(v); });
  array(o, "long long", "tt_pair_tab", pt, l);
  std::vector<int> idx(256);
  for (int j = 0; j < 256; ++j) idx[j] = j;
  array(o, "pfx::Log2Entry", "tt_log2", idx, [](int j) {
    const unsigned rc = (unsigned)roundl(2048.0L / (1.0L + (j + 0.5L) / 256));
    return "{" + std::to_string((i64)llroundl(-log2l(rc / 2048.0L) * 4611686018427387904.0L)) + "ll," + std::to_string(rc) + "u,0u}";
  });
  o << "#include \"pyro_transport.cuh\"\n";
  out.source = o.str();
  out.warps = nw;
  out.smem_bytes = smem;
  return out;
}

}  // namespace pyro
