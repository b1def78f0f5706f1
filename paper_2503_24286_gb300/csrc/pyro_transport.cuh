// Mixture-averaged transport of a tile of 32 states per block: lane = state, the
// block's warps split the species, the rows of Wilke's rule and the species pairs.
//
// Included by the emitted unit, which defines the tables (tt_*) and sizes.  The
// per-thread kernel spent 24.5 k FP64 instructions a state on 53 species: 19 cycles of
// an SM each, 13.1 ms per 2^18 states.  This kernel takes 6.0 ms, about half of it FP64-bound
// (two FMAs a pair, the species fits), half integer work.  Here
//  * Wilke's sums (three products with constant N x N matrices) are integer dot
//    products: mole fractions and x/P, x/P^2 in fixed point, sums exact to 2^-54;
//  * the fit of a pair is a fixed-point Horner scheme in t = (log2 T - log2 1000)/4,
//    re-expanded about t = 0 by the emitter (in ln T the terms cancel by up to 1e4),
//    and its reciprocal is formed on the integer pipe from a single-precision seed;
//  * the diffusion sums keep their FP64 range: two FMAs per pair.  Pairs come in rounds
//    of a tournament: the pairs of a round share no species, so the warps update the
//    sums of both species of a pair without conflicts, with a barrier per round.
// States outside the tables' range (T outside (TT_LO, TT_HI), mole fractions or scaled
// x/P beyond 2 in magnitude, sum |x| from 2, NaN) get TILE_OPEN in the first output that is given and
// are evaluated by the FP64 kernel launched behind.
#include "pyro_device_math.cuh"
#include "pyro_fixed_math.cuh"

using pfx::Pair;
typedef pfx::i64 i64;
typedef pfx::u64 u64;

__device__ __forceinline__ Pair tt_pair(i64 v) {
  Pair p;
  p.lo = (int)v;
  p.hi = (int)((u64)v >> 32);
  return p;
}

// sum of c y: h 2^64 + l 2^32 (LOW: and the upper half of the products of the low halves;
// left out of the sums of x/P^2, whose y are the smallest, they are a mean error of 3.8e-16
// of mu, of x/P 1.2e-16, of x 1e-17, FP64 sums altogether 3.2e-16; all three 4 % of the kernel's
// time, the one 1 %).
// With |c| < 2^57 and y = x 2^61 the word h << 7 stays below 2^61 sum |x|, and l below
// 2^60 sum |x| + N 2^55.
template <bool LOW> struct TtDot {
  i64 h, l;
  __device__ __forceinline__ void add(i64 c, Pair y) {
    const int ch = (int)(c >> 32), cl = (int)c;
    h += (i64)ch * y.hi;
    l += (i64)ch * y.lo;
    l += (i64)cl * y.hi;
    if (LOW) l += (i64)pfx::mulhi_s(cl, y.lo);
  }
  __device__ __forceinline__ double value(int f) const { return pfx::scaled((h << 7) + (l >> 25), 57 - f); }
};

// a double of |y| < 2 with f = 61, rounded (truncation is a bias of the small x/P^2), as two
// signed halves: split once here, not in each of the N rows that read it
__device__ __forceinline__ i64 tt_halves(double y) {
  const u64 b = pfx::dbits(y);
  const int s = 1024 - ((int)(b >> 52) & 0x7ff);                          // from 1
  const u64 m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
  const i64 v = s > 62 ? 0ll : (i64)(m >> (s & 63)) + (i64)((m >> ((s - 1) & 63)) & 1ull);
  const Pair p = pfx::split((b >> 63) ? -v : v);
  return (i64)((u64)(unsigned)p.hi << 32 | (unsigned)p.lo);
}

// 2^s/v for a fixed-point v > 0
__device__ __forceinline__ double tt_rcp(i64 v, int s) {
  const int hi = (int)(v >> 32);
  if (hi < 4096) return 1.0 / pfx::scaled(v, -s);    // the fit is not positive, or far below its scale
  const int z = __clz(hi);
  const u64 m = (u64)v << z;                         // [1, 2), f = 63
  const unsigned mh = (unsigned)(m >> 32), ml = (unsigned)m;
  float r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(__uint_as_float(0x3f800000u | ((mh >> 8) & 0x7fffffu))));
  r0 = fminf(r0, 0.99999994f);                       // (1/2, 1)
  const unsigned R = (__float_as_uint(r0) << 8) | 0x80000000u;         // f = 32
  // e = 1 - m r0 (|e| < 2^-21), f = 63; 1/m = r0 (1 + e + e^2), the rest below 2^-63
  const i64 e = (i64)(0x8000000000000000ull - ((u64)mh * R + __umulhi(ml, R)));
  const int e2 = (int)(e >> 11);                     // f = 52
  const int t = e2 + (int)(((i64)e2 * e2) >> 52);
  const u64 r = ((u64)R << 31) + (u64)(((i64)(int)(R >> 1) * t) >> 20) +
                (((R >> 16) * ((unsigned)e & 2047u)) >> 16);               // f = 63
  // 2^s/v = r 2^(s + z - 63), r in [1/2, 1]: the leading bit adds one to the exponent field
  return __longlong_as_double((i64)(((u64)(unsigned)(s + z - 63 + 1021) << 52) + ((r + 0x200ull) >> 10)));
}

struct TtShared {
  double ys[NW * 32], mu[NW * 32], ka[NW * 32], kh[NW * 32];
  float xa[NW * 32];                           // sum |x|
  double rys[32], td[32], sqT[32];
  Pair t[32];
  int bad[32];
};

extern "C" __global__ void __launch_bounds__(32 * NW, TT_MINB)
pyro_transport_tile(i64 n, const double* __restrict__ g_T, const double* __restrict__ g_Y, double* __restrict__ g_mu,
                    double* __restrict__ g_kappa, double* __restrict__ g_Dm) {
  extern __shared__ __align__(16) char s_raw[];
  double* sx = (double*)s_raw;                 // mole fractions
  double* sP = sx + NSP * 32;                  // sqrt(mu_k/sqrt(T))
  i64* fx = (i64*)(sP + NSP * 32);             // x, x/P, x/P^2 in fixed point (two halves)
  i64* fv = fx + NSP * 32;
  i64* fw = fv + NSP * 32;
  double* S = (double*)fx;                     // diffusion sums, after Wilke's
  TtShared& sh = *(TtShared*)(fw + NSP * 32);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const i64 tiles = (n + 31) >> 5;
#pragma unroll 1
  for (i64 tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const i64 p = tile * 32 + lane, pc = p < n ? p : n - 1;
    // a tile without any state in the tables (a cold block): no work beside the FP64 kernel's
    const double T = __ldg(g_T + pc);
    if (!__any_sync(0xffffffffu, T > TT_LO && T < TT_HI)) {
      if (w == 0 && p < n) (g_mu ? g_mu : g_kappa ? g_kappa : g_Dm)[p] = __longlong_as_double(TILE_OPEN);
      continue;
    }
    const double* Yp = g_Y + pc;
    {
      double y[KPW];
      double ys = 0.0;
#pragma unroll
      for (int i = 0; i < KPW; ++i) y[i] = w + i * NW < NSP ? __ldg(Yp + (w + i * NW) * n) : 0.0;
#pragma unroll
      for (int i = 0; i < KPW; ++i)
        if (w + i * NW < NSP) {
          y[i] *= __ldg(tt_iw + w + i * NW);
          ys += y[i];
          sx[(w + i * NW) * 32 + lane] = y[i];
        }
      sh.ys[w * 32 + lane] = ys;
    }
    if (w == 0) {
      const bool in = T > TT_LO && T < TT_HI;
      const double Ts = in ? T : 1000.0;
      const u64 b = pfx::dbits(Ts);
      const i64 l = pfx::log2_mant((b & 0xfffffffffffffull) | 0x10000000000000ull, tt_log2);     // f = 62
      const i64 d = (((i64)(b >> 52) - 1023) << 59) + ((l + 4) >> 3) - TT_LGC;                    // f = 59
      sh.td[lane] = pfx::scaled(d, -61);
      sh.t[lane] = pfx::split(d << 2);
      sh.sqT[lane] = sqrt(Ts);
      sh.bad[lane] = in ? 0 : 1;
    }
    __syncthreads();
    if (w == 0) {
      double ys = 0.0;
#pragma unroll
      for (int i = 0; i < NW; ++i) ys += sh.ys[i * 32 + lane];
      sh.rys[lane] = pdm::rcp(ys);
    }
    __syncthreads();
    const double td = sh.td[lane], rys = sh.rys[lane];
    double ka = 0.0, kh = 0.0;
    float xa = 0.f;
    bool bad = false;
#pragma unroll 1
    for (int k = w; k < NSP; k += NW) {
      const double2* c = (const double2*)(tt_fit + k * 10);
      const double2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2), c3 = __ldg(c + 3), c4 = __ldg(c + 4);
      const double x = sx[k * 32 + lane] * rys;
      const double P = fabs(fma(td, fma(td, fma(td, fma(td, c2.x, c1.y), c1.x), c0.y), c0.x));
      const double K = fma(td, fma(td, fma(td, fma(td, c4.y, c4.x), c3.y), c3.x), c2.y);
      const double rP = pdm::rcp(P), v = rP * x, q = v * rP;
      const double vs = v * TT_SV, ws = q * TT_SW;
      bad |= !(fabs(vs) < 1.9 && fabs(ws) < 1.9);
      sx[k * 32 + lane] = x;
      sP[k * 32 + lane] = P;
      fx[k * 32 + lane] = tt_halves(x);
      fv[k * 32 + lane] = tt_halves(vs);
      fw[k * 32 + lane] = tt_halves(ws);
      ka = fma(x, K, ka);
      kh = fma(x, pdm::rcp(K), kh);
      xa += fabsf(pdm::to_float_trunc(x));
    }
    sh.xa[w * 32 + lane] = xa;
    sh.ka[w * 32 + lane] = ka;
    sh.kh[w * 32 + lane] = kh;
    if (bad) sh.bad[lane] = 1;
    __syncthreads();
    if (g_mu) {
      double mu = 0.0;
#pragma unroll 1
      for (int k = w; k < NSP; k += NW) {
        TtDot<false> a, b;
        TtDot<true> e;
        a.h = a.l = b.h = b.l = e.h = e.l = 0;
        const longlong2* c = (const longlong2*)(tt_wilke + k * NSP * 4);
#pragma unroll 4
        for (int j = 0; j < NSP; ++j) {
          const longlong2 c0 = __ldg(c + 2 * j), c1 = __ldg(c + 2 * j + 1);
          a.add(c0.x, tt_pair(fx[j * 32 + lane]));
          b.add(c0.y, tt_pair(fv[j * 32 + lane]));
          e.add(c1.x, tt_pair(fw[j * 32 + lane]));
        }
        const double P = sP[k * 32 + lane];
        // sum_j Phi_kj X_j; the middle table holds 2 c w, the exponents the scales of the row, v and w
        const int4 f = __ldg((const int4*)tt_wf + k);
        const double den = fma(P, fma(P, e.value(f.z), b.value(f.y)), a.value(f.x));
        mu = fma(sx[k * 32 + lane] * (P * P), pdm::rcp(den), mu);
      }
      sh.mu[w * 32 + lane] = mu;
    }
    __syncthreads();
    if (w == 0) {
      double ka = 0.0, kh = 0.0, mu = 0.0;
#pragma unroll
      for (int i = 0; i < NW; ++i) { ka += sh.ka[i * 32 + lane]; kh += sh.kh[i * 32 + lane]; }
      // Wilke's integer sums: their top word stays below 2^63 while sum |x| < 2 (TtDot)
      float xs = 0.f;
#pragma unroll
      for (int i = 0; i < NW; ++i) xs += sh.xa[i * 32 + lane];
      if (!(xs < 2.f)) sh.bad[lane] = 1;
      if (g_mu) {
#pragma unroll
        for (int i = 0; i < NW; ++i) mu += sh.mu[i * 32 + lane];
      }
      const bool open = sh.bad[lane] != 0;
      const double mark = __longlong_as_double(TILE_OPEN);
      if (p < n && g_mu) g_mu[p] = open ? mark : sh.sqT[lane] * mu;
      if (p < n && g_kappa) g_kappa[p] = open && !g_mu ? mark : 0.5 * sh.sqT[lane] * (ka + pdm::rcp(kh));
    }
    if (g_Dm) {
      for (int k = w; k < NSP; k += NW) S[k * 32 + lane] = 0.0;
      __syncthreads();
      const Pair t = sh.t[lane];
      const longlong2* c = (const longlong2*)(tt_pair_tab + (i64)w * TT_PAIRS_W * 8);
      longlong2 n0 = __ldg(c), n1 = __ldg(c + 1), n2 = __ldg(c + 2), n3 = __ldg(c + 3);
#pragma unroll 1
      for (int r = 0; r < TT_ROUNDS; ++r) {
#pragma unroll
        for (int q = 0; q < TT_PER_WARP; ++q) {
          // b4 b3 | b2 b1 | b0, scale | byte offsets of the species
          const longlong2 c0 = n0, c1 = n1, c2 = n2, c3 = n3;
          c += 4;                                  // (the table ends with a spare record)
          n0 = __ldg(c); n1 = __ldg(c + 1); n2 = __ldg(c + 2); n3 = __ldg(c + 3);
          const int ok = (int)c3.x, oj = (int)((u64)c3.x >> 32);
          if (ok < 0) continue;                    // no pair in this slot
          i64 v = pfx::horner(c0.x, t, c0.y);
          v = pfx::horner(v, t, c1.x);
          v = pfx::horner(v, t, c1.y);
          v = pfx::horner(v, t, c2.x);
          const double rc = tt_rcp(v, (int)c2.y);
          double* Sk = (double*)((char*)S + ok) + lane;
          double* Sj = (double*)((char*)S + oj) + lane;
          const double xk = ((const double*)((const char*)sx + ok))[lane], xj = ((const double*)((const char*)sx + oj))[lane];
          *Sk = fma(xj, rc, *Sk);
          *Sj = fma(xk, rc, *Sj);
        }
        __syncthreads();
      }
      const double sqT = sh.sqT[lane];
      const bool open = sh.bad[lane] != 0 && !g_mu && !g_kappa;
#pragma unroll 1
      for (int k = w; k < NSP; k += NW) {
        const double d = (1.0 - __ldg(Yp + k * n)) * sqT * pdm::rcp(S[k * 32 + lane]);
        if (p < n) g_Dm[k * n + p] = open && k == 0 ? __longlong_as_double(TILE_OPEN) : d;
      }
    }
    __syncthreads();
  }
}
