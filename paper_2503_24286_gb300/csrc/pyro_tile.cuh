// Net production rates of a tile of 32 states per block: lane = state, the block's
// warps split the species and the reactions, and all exponents are fixed point.
//
// Included by the emitted unit, which defines the mechanism's tables (t_*) and
// sizes (NSP, NW, KPW, NCH, ...).  One pass over a tile:
//   0  temperature from energy (energy input): every warp collapses the energy
//      polynomials of its species, one warp finishes the Newton iteration;
//   1  per species lambda_k = log2(phi_k/W_k) and alpha_k = log2(a_k), with
//      a_k = phi_k C_k (the activity form of Eq. equil_constants and
//      Eq. reaction_rates), in shared memory [species][lane];
//   2  per reaction the exponents of its forward and reverse rate,
//      K_j(T) - sum nu' lambda + sum nu' alpha  and  ... + sum nu'' alpha,
//      two exponentials and their difference, the rate of progress, in shared memory
//      as one 64-bit word: 52 bits of signed integer and 12 of exponent (not
//      normalised: its error is 2^-51 of the larger of the two rates);
//   3  per species the sum of its reactions' rates, aligned to the largest exponent
//      met so far, normalised once into the output.
// Bound: the integer pipes (53 species / 325 reactions: 132 k warp instructions a tile,
// issue 0.53 a cycle, ALU pipe 43 % and FP64 pipe 32 % of their limits averaged over the
// phases, which load them in turn; DRAM 2 %).  Measured against one thread per state, whose
// 7,270 FP64 instructions a state ran at the FP64 pipe's limit: 2^22 states of 53 species,
// energy input, 57.2 -> 26.4 ms; one state 332 -> 47 us; 160 species, 2^18 states (against
// one warp per state) 12.9 -> 5.4 ms.  Errors against extended precision: rates 1.5e-15 of a
// state's norm on average (FP64 kernel 1.0e-14), T 1.8e-16 (6.1e-16).  Leaving the exponential's last product and the
// difference of the two rates to FP64 was slower (7.24 against 7.11 ms per 2^20 states).
//
// All warps of a block run the same code at about the same time and the loops over
// species and reactions are rolled: a reaction is a table record, not code, so that
// the kernel stays within the instruction caches (with a loop per reaction shape and
// unrolled species loops it was 119 KB and stalled on instruction fetch).
// The FP64 pipe, which runs beside the integer work, keeps the Newton steps, the
// third-body concentrations and the blending factors of falloff reactions.
//
// States outside the tables' range (temperature outside (T_LO, T_HI), NaN or
// infinite mass fractions or ones from 2, densities beyond 2^-60..2^20, a
// falloff or PLOG reaction with [M] <= 0) get TILE_OPEN in their first output; the caller then launches the FP64
// kernel, which evaluates the states so marked.
#include "pyro_device_math.cuh"
#include "pyro_fixed_math.cuh"

using pfx::Pair;
typedef pfx::i64 i64;
typedef pfx::u64 u64;

// A rate is a 64-bit word r: read as an integer it is m 2^(e - 62 - RATE_E) with
// e = r & RATE_M, |m| < 2^63.  The exponent's bits are the last bits of the integer: they lie
// below its resolution and, near RATE_E/(RATE_M + 1) = 1/2 of one unit, are on average what
// truncation took away.  12 exponent bits, or 11 (RATE_E 1023) for words made of doubles.
#ifndef RATE_E
#define RATE_E 2048
#define RATE_M 4095
#else
#define RATE_M 2047
#endif

#ifndef TILE_DERIV
struct TileScalars {
  double T[32], ysum[32];
  Pair u[32], v[32], t[32];      // log2(T)/16, T_V/T, T/T_T
  i64 lgT[32], lgrho[32];
  float Tf[32];
  int bad[32];
  int neg;                       // the tile has negative mass fractions or densities
  int none;                      // no state of the tile is inside the tables
};

struct TileSmem {
  u64* exp2;
  i64 *lam, *alp;   // [NSP + 1][32]: the species and a unit factor; alp first holds Y
  i64* R;           // rows and one zero row; during the temperature solve its scratch (red, B, b, ys)
  i64* red;
  i64* B;
  float* b;
  double* ys;
  TileScalars* sc;
};

#endif  // TILE_DERIV

__device__ __forceinline__ Pair as_pair(i64 v) {
  Pair p;
  p.lo = (int)v;
  p.hi = (int)((u64)v >> 32);
  return p;
}

#ifndef TILE_DERIV
__device__ __forceinline__ TileSmem tile_smem(char* base) {
  TileSmem s;
  s.exp2 = (u64*)base;                     base += pfx::EXP2_TAB * 8;
  s.lam = (i64*)base;                      base += (NSP + 1) * 256;
  s.alp = (i64*)base;                      base += (NSP + 1) * 256;
  s.R = (i64*)base;
  s.ys = (double*)base;                    // NW x 32
  s.B = (i64*)(s.ys + NW * 32);            // 6 x 32
  s.b = (float*)(s.B + 6 * 32);            // 14 x 32
  s.red = (i64*)(s.b + 14 * 32);           // NW x 6 x 32 (FP32: NW x 13 x 32)
  base += (TILE_ROWS + 1) * 256;
  s.sc = (TileScalars*)base;
  return s;
}

#endif  // TILE_DERIV

// sums of products of fixed-point values c (two signed halves) and Y (f = 61): h 2^64 + l 2^32
struct TileDot {
  i64 h, l;
  __device__ __forceinline__ void add(i64 c, Pair y) {
    const int ch = (int)(c >> 32), cl = (int)c;
    h += (i64)ch * y.hi;
    l += (i64)ch * y.lo;
    l += (i64)cl * y.hi;
    l += (i64)pfx::mulhi_s(cl, y.lo);
  }
  __device__ __forceinline__ i64 sum() const { return (h << 7) + ((l + 0x1000000ll) >> 25); }   // in units of 2^57
};

// double of m 2^(e - f)
__device__ __forceinline__ double tile_to_double(i64 m, int e, int f) {
  const u64 a = m < 0 ? (u64)(-m) : (u64)m;
  const int z = pfx::clz64(a | 1ull);
  const u64 v = a << z;                               // leading one at bit 63
  u64 r = (v >> 11) + ((v >> 10) & 1ull);             // 53 bits, rounded; a carry moves to the exponent
  const int x = e - f + 63 - z + 1022;
  r += (u64)(unsigned)x << 52;
  r = (a == 0ull || x < 0) ? 0ull : r;
  r = x > 2045 ? 0x7ff0000000000000ull : r;
  return __longlong_as_double((i64)(r | ((u64)m & 0x8000000000000000ull)));
}

// arithmetic right shift; 63 where n is larger
__device__ __forceinline__ i64 tile_sar(i64 v, int n) {
  i64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
__device__ __forceinline__ u64 tile_shr(u64 v, int n) {
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}

// the rate 2^xf - 2^xr (REV false: 2^xf) with the signs in the lowest bits (SGN false: all
// are clear)
template <bool REV, bool SGN>
__device__ __forceinline__ i64 tile_rate(i64 xf, i64 xr, const u64* tab) {
  const u64 f = pfx::exp2_mant(xf, tab);
  const i64 sf = SGN ? -(xf & 1ll) : 0ll;
  const int nf = (int)(xf >> pfx::LG_F);
  i64 m;
  int e = max(nf, 50 - RATE_E);
  if (REV) {
    const u64 g = pfx::exp2_mant(xr, tab);
    const i64 sg = SGN ? -(xr & 1ll) : 0ll;
    const int ng = (int)(xr >> pfx::LG_F);
    e = max(e, ng);
    if (SGN) e += (int)(xf ^ xr) & 1;           // unlike signs: the terms add up to twice the larger
    // one's complement negation: off by one in 2^62
    m = ((i64)tile_shr(f, e + 1 - nf) ^ sf) - ((i64)tile_shr(g, e + 1 - ng) ^ sg);
  } else {
    m = (i64)tile_shr(f, e + 1 - nf) ^ sf;
  }
  return (m & ~(i64)RATE_M) | (i64)(e + RATE_E);
}

// the rate of a sum of two
__device__ __forceinline__ i64 tile_add(i64 a, i64 b) {
  const int ea = (int)a & RATE_M, eb = (int)b & RATE_M, e = max(ea, eb) + 1;
  return ((tile_sar(a, e - ea) + tile_sar(b, e - eb)) & ~(i64)RATE_M) | (i64)e;
}

// K(T) = c + beta u + tau v of a reaction, lowest bit clear
__device__ __forceinline__ i64 tile_K(i64 c, i64 beta, i64 tau, Pair u, Pair v) {
  return pfx::mul_add(as_pair(tau), v, pfx::mul_add(as_pair(beta), u, c)) & ~1ll;
}

// The temperature's factors of a state, T in (T_LO, T_HI): u = log2(T)/16, v = T_V/T and
// t = T/T_T as fracs, and its lg.  The exponents of cold states are a few hundred, so an ulp of v
// is an error of 1e-14 to 5e-14 in every rate: quotients get the remainder of the FP64
// value in units of 2^-63, and u keeps the bits of the logarithm that lg has no room for.
__device__ __forceinline__ i64 tile_quotient(double a, double b, double r) {     // a/b, r = 1/b
  const double q = a * r;
  return pfx::frac_of(q) + (i64)__double2int_rn(fma(-b, q, a) * r * 9223372036854775808.0);
}
__device__ __forceinline__ void tile_T(double T, Pair& u, Pair& v, Pair& t, i64& lgT) {
  const u64 b = pfx::dbits(T);
  const i64 e = (i64)(b >> 52) - 1023;
  const i64 l = pfx::log2_mant((b & 0xfffffffffffffull) | 0x10000000000000ull, t_log2);      // f = 62
  lgT = (e << pfx::LG_F) + (((l + 0x1000ll) >> 13) << 1);
  u = pfx::split((e << 59) + ((l + 4) >> 3));
  v = pfx::split(tile_quotient(T_V, T, pdm::rcp(T)));
  t = pfx::split(tile_quotient(T, T_T, 1.0 / T_T));
}

#ifndef TILE_DERIV
// ---------------------------------------------------------------------------
// temperature (Sec. A.3.1): FP32 Newton on the collapsed polynomials of both
// ranges, then FP64 Newton on the range found, as in the per-thread solve
// ---------------------------------------------------------------------------
__device__ __noinline__ void tile_collapse_all(const double* __restrict__ Yp, i64 n, bool hi, double* B) {
  for (int q = 0; q < 6; ++q) B[q] = 0.0;
  for (int k = 0; k < NSP; ++k) {
    const double y = __ldg(Yp + k * n);
    for (int q = 0; q < 6; ++q) B[q] = fma(y, t_ed[(k * 2 + hi) * 6 + q], B[q]);
  }
}

__device__ __forceinline__ void tile_energy(const TileSmem& s, const double* __restrict__ Yp, i64 n,
                                            double e, double T0, int max_iter, float tolf, int w, int lane,
                                            double& T, bool& ok) {
  {
    float f[13];
#pragma unroll
    for (int q = 0; q < 13; ++q) f[q] = 0.f;
    const double* y = (const double*)s.alp + lane;
#pragma unroll 2
    for (int k = w; k < NSP; k += NW) {
      const float yf = pdm::to_float_trunc(y[k * 32]);
      const float4* c = (const float4*)(t_ef + k * 12);
      const float4 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2);
      f[12] += fabsf(yf);
      f[0] = fmaf(yf, c0.x, f[0]); f[1] = fmaf(yf, c0.y, f[1]); f[2] = fmaf(yf, c0.z, f[2]); f[3] = fmaf(yf, c0.w, f[3]);
      f[4] = fmaf(yf, c1.x, f[4]); f[5] = fmaf(yf, c1.y, f[5]); f[6] = fmaf(yf, c1.z, f[6]); f[7] = fmaf(yf, c1.w, f[7]);
      f[8] = fmaf(yf, c2.x, f[8]); f[9] = fmaf(yf, c2.y, f[9]); f[10] = fmaf(yf, c2.z, f[10]); f[11] = fmaf(yf, c2.w, f[11]);
    }
    float* red = (float*)s.red;
#pragma unroll
    for (int q = 0; q < 13; ++q) red[(w * 13 + q) * 32 + lane] = f[q];
    __syncthreads();
    for (int q = w; q < 13; q += NW) {
      float a = 0.f;
#pragma unroll
      for (int i = 0; i < NW; ++i) a += red[(i * 13 + q) * 32 + lane];
      s.b[q * 32 + lane] = a;
    }
    __syncthreads();
  }
  const float* b = s.b + lane;
  if (w == 0) {
    float c[12];
#pragma unroll
    for (int q = 0; q < 12; ++q) c[q] = b[q * 32];
    float Tf = pdm::to_float_trunc(T0);
    const float eRf = pdm::to_float_trunc(e * T_INV_R);
    for (int it = 0; it < 40; ++it) {
      const bool h = Tf >= (float)TMID;
      const float c0 = h ? c[6] : c[0], c1 = h ? c[7] : c[1], c2 = h ? c[8] : c[2];
      const float c3 = h ? c[9] : c[3], c4 = h ? c[10] : c[4], c5 = h ? c[11] : c[5];
      const float ef = fmaf(Tf, fmaf(Tf, fmaf(Tf, fmaf(Tf, fmaf(Tf, c5, c4), c3), c2), c1), c0);
      const float cvf = fmaf(Tf, fmaf(Tf, fmaf(Tf, fmaf(Tf, 5.f * c5, 4.f * c4), 3.f * c3), 2.f * c2), c1);
      const float Tn = fminf(fmaxf(Tf + (eRf - ef) * __frcp_rn(cvf), 100.f), 5000.f);
      const bool conv = fabsf(Tn - Tf) <= 1e-5f * Tn;
      Tf = Tn;
      if (conv) break;
    }
    s.sc->Tf[lane] = Tf;
  }
  __syncthreads();
  const float Tf = s.sc->Tf[lane];
  bool hi = Tf >= (float)TMID;
  {
    // the collapse of one range on the integer pipe (exact up to the 2^-61 of Y)
    TileDot d[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) d[q].h = d[q].l = 0;
#pragma unroll 1
    for (int k = w; k < NSP; k += NW) {
      const Pair y = pfx::split(pfx::fix61(((const double*)s.alp)[k * 32 + lane]));
      const longlong2* c = (const longlong2*)(t_ex + (k * 2 + hi) * 6);
      const longlong2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2);
      d[0].add(c0.x, y); d[1].add(c0.y, y); d[2].add(c1.x, y);
      d[3].add(c1.y, y); d[4].add(c2.x, y); d[5].add(c2.y, y);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) s.red[(w * 6 + q) * 32 + lane] = d[q].sum();
  }
  __syncthreads();
  if (w != 0) return;
  double B[6];
  if (b[12 * 32] > 0.25f && b[12 * 32] < 2.f) {   // sum |Y| (false for NaN)
#pragma unroll 1
    for (int q = 0; q < 6; ++q) {
      i64 a = 0;
#pragma unroll
      for (int i = 0; i < NW; ++i) a += s.red[(i * 6 + q) * 32 + lane];
      s.B[q * 32 + lane] = a;
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) B[q] = pfx::scaled(s.B[q * 32 + lane], 57 - t_exs[q]);
  } else {
    tile_collapse_all(Yp, n, hi, B);
  }
  // B[0] - e/R first: the terms that cancel are large (formation energies), the rest is
  // of the size of c_v T, and the residual is rounded at that size only
  auto take_e = [&] { B[0] = fma(e, -T_INV_R_LO, fma(e, -T_INV_R, B[0])); };
  take_e();
  T = pdm::to_double(Tf);
  bool flag = false;
  ok = false;
  for (int it = 0; it < max_iter + 1; ++it) {
    const float Tc = pdm::to_float_trunc(T);
    const bool h2 = Tc >= (float)TMID;
    if (h2 != hi) { hi = h2; tile_collapse_all(Yp, n, hi, B); take_e(); }
    const double res = fma(T, fma(T, fma(T, fma(T, fma(T, B[5], B[4]), B[3]), B[2]), B[1]), B[0]);
    const float* c = b + (hi ? 6 * 32 : 0);
    const float cvf = fmaf(Tc, fmaf(Tc, fmaf(Tc, fmaf(Tc, 5.f * c[160], 4.f * c[128]), 3.f * c[96]), 2.f * c[64]), c[32]);
    const double dT = res * pdm::to_double(-__frcp_rn(cvf));
    double Tn = T + dT;
    const float Tnf = pdm::to_float_trunc(Tn);
    const bool clamped = !(Tnf >= 100.f && Tnf <= 5000.f);
    Tn = clamped ? (Tnf < 100.f ? 100.0 : 5000.0) : Tn;
    const bool conv = !clamped && fabsf(pdm::to_float_trunc(dT)) <= tolf * pdm::to_float_trunc(Tn);
    T = Tn;
    if (flag) { ok = true; break; }
    if (conv) flag = true;
    else if (it >= max_iter - 1) break;
  }
}

#endif  // TILE_DERIV

// ---------------------------------------------------------------------------
// reactions
// ---------------------------------------------------------------------------
#ifndef TILE_DERIV
// plain reactions with up to NF factors a side (missing ones: the unit factor);
// REV: reversible.  A flag marks a duplicate of a reaction before it in this warp,
// whose rate is added to the same row.
template <int NF, bool REV, bool SGN>
__device__ __forceinline__ void tile_plain(const TileSmem& s, int i0, int i1, Pair u, Pair v, int lane) {
  const char* lam = (const char*)(s.lam + lane);
  const char* alp = (const char*)(s.alp + lane);
  char* R = (char*)(s.R + lane);
  const int4* r = (const int4*)(t_rx + i0 * 8);
  int4 r0 = __ldg(r), r1 = __ldg(r + 1), r2 = __ldg(r + 2), r3 = __ldg(r + 3);
#pragma unroll 2
  for (int i = i0; i < i1; ++i) {
    const int4 c0 = r0, c1 = r1, c2 = r2, c3 = r3;
    r += 4;                                    // the next record (the table ends with a spare one)
    r0 = __ldg(r); r1 = __ldg(r + 1); r2 = __ldg(r + 2); r3 = __ldg(r + 3);
    // c0: c, beta; c1: tau, reactants 0 and 1; c2: reactant 2, products 0 to 2; c3: the row
    // (byte offsets), the flag
    Pair beta, tau;
    beta.lo = c0.z; beta.hi = c0.w;
    tau.lo = c1.x; tau.hi = c1.y;
    const i64 c = (i64)(((u64)(unsigned)c0.y << 32) | (unsigned)c0.x);
    auto at = [](const char* b, int o) { return *(const i64*)(b + o); };
    i64 X = (pfx::mul_add(tau, v, pfx::mul_add(beta, u, c)) & ~1ll) - at(lam, c1.z);
    X -= at(lam, c1.w);
    if (NF > 2) X -= at(lam, c2.x);
    i64 Xf = X + at(alp, c1.z) + at(alp, c1.w);
    if (NF > 2) Xf += at(alp, c2.x);
    i64 Xr = X;
    if (REV) {
      Xr += at(alp, c2.y) + at(alp, c2.z);
      if (NF > 2) Xr += at(alp, c2.w);
    }
    i64 rate = tile_rate<REV, SGN>(Xf, Xr, s.exp2);
    i64* o = (i64*)(R + c3.x);
    if (c3.y) rate = tile_add(*o, rate);
    *o = rate;
  }
}

#endif  // TILE_DERIV

__device__ __forceinline__ double ax_d(i64 v) { return __longlong_as_double(v); }

// sum_k eps_k Y_k/W_k of a reaction from its efficiency list.  In FP64: the integer form
// (TileDot) takes some 25 instructions a term and was slower (2^20 states 8.0 against 7.3 ms).
__device__ __forceinline__ double tile_mS(const i64* ax, int ne, double ysum, const double* __restrict__ Yp, i64 n) {
  double m = ysum;
#pragma unroll 4
  for (int q = 0; q < ne; ++q) {
    const longlong2 c = __ldg((const longlong2*)ax + q);
    m = fma(__ldg(Yp + c.x * n), ax_d(c.y), m);
  }
  return m;
}

__device__ __forceinline__ bool tile_normal_pos(double x) {
  const int h = __double2hiint(x);
  return h >= 0x00100000 && h < 0x7ff00000;
}

enum { TK_THREEBODY = 1, TK_LINDEMANN = 2, TK_TROE = 3, TK_SRI = 4, TK_PLOG = 5 };

// f l for 0 <= f <= 1 and a logarithm l
__device__ __forceinline__ i64 tile_part(double f, i64 l) {
  const bool near_one = f >= 0.9999;
  const double g = fmax(near_one ? 1.0 - f : f, 1e-300);
  const i64 p = pfx::mul_add(pfx::split(2 * l), pfx::split(pfx::frac_of(g)), 0ll);
  return near_one ? l - p : p;
}

#ifndef TILE_DERIV
// reactions of the other classes: auxiliary data ax (see the emitter for the layout)
__device__ __forceinline__ void tile_other(const TileSmem& s, int i0, int i1, int lane, double rho,
                                           const double* __restrict__ Yp, i64 n) {
  const Pair u = s.sc->u[lane], v = s.sc->v[lane], t = s.sc->t[lane];
  const double ysum = s.sc->ysum[lane];
  const i64* lam = s.lam + lane;
  const i64* alp = s.alp + lane;
  i64 an = __ldg(t_rx + i0 * 8 + 5);
#pragma unroll 1
  for (int i = i0; i < i1; ++i) {
    const i64* r = t_rx + i * 8;
    const i64 fa = __ldg(r + 3), fb = __ldg(r + 4);
    const int nr = (int)((fb >> 48) & 0xf), np = (int)((fb >> 52) & 0xf), kind = (int)((fb >> 56) & 0xf);
    const i64* ax = t_ax + an;
    an = __ldg(r + 13);                          // of the next reaction: its lines are fetched meanwhile
    if (i + 1 < i1) {
      const char* pre = (const char*)(t_ax + an) + (lane & 3) * 128;
      asm volatile("prefetch.global.L1 [%0];" ::"l"(pre));
    }
    const int ne = (int)__ldg(ax);
    // log2 [M] of the reaction (PLOG: of the total concentration).  A third body's [M] is a
    // factor of the rate and may be zero or negative (efficiencies of 0 whose sum cancels,
    // undershoots); the other classes need a positive one.
    const bool third = kind == TK_THREEBODY;
    const double M = rho * tile_mS(ax + 16, ne, ysum, Yp, n);
    const bool normal = tile_normal_pos(third ? fabs(M) : M), none = third && M == 0.0;
    if (!normal && !none) s.sc->bad[lane] = 1;
    const i64 lgM = pfx::log2_of(normal ? fabs(M) : 1.0, t_log2);
    i64 X;
    if (kind == TK_PLOG) {
      // log2 k linear in log2 p between the bracketing nodes, end nodes outside
      const int nn = (int)__ldg(ax + 1);
      const i64* nd = ax + 16;               // nodes {lg p, 1/(lg p_next - lg p), c, beta, tau}
      const i64 lgp = s.sc->lgT[lane] + lgM + T_LG_R;
      int q = 0;
      for (int j = 1; j + 1 < nn; ++j) if (lgp >= __ldg(nd + 5 * j)) q = j;
      const i64* a = nd + 5 * q;
      const i64 xa = tile_K(__ldg(a + 2), __ldg(a + 3), __ldg(a + 4), u, v);
      const i64 xb = tile_K(__ldg(a + 7), __ldg(a + 8), __ldg(a + 9), u, v);
      const double pf = fmin(fmax(pfx::to_double(lgp - __ldg(a)) * ax_d(__ldg(a + 1)), 0.0), 1.0);
      X = pf > 0.0 ? xa + tile_part(pf, xb - xa) : xa;
    } else {
      X = tile_K(__ldg(r), __ldg(r + 1), __ldg(r + 2), u, v);
    }
    if (third) X += lgM;
    if (kind >= TK_LINDEMANN && kind <= TK_SRI) {
      const i64 lgPr = tile_K(__ldg(ax + 2), __ldg(ax + 3), __ldg(ax + 4), u, v) + lgM;
      // log2(Pr/(1+Pr)) = min(lgPr, 0) - log2(1 + 2^-|lgPr|)
      const i64 am = lgPr < 0 ? lgPr : -lgPr;
      u64 q = 0x4000000000000000ull + tile_shr(pfx::exp2_mant(am, s.exp2), 1 - (int)(am >> pfx::LG_F));   // [1, 2], f = 62
      q = q > 0x7fffffffffffffffull ? 0x7fffffffffffffffull : q;
      X += (lgPr < 0 ? lgPr : 0ll) - ((pfx::log2_mant(q >> 10, t_log2) + 0x800ll) >> 12);
      if (kind != TK_LINDEMANN) {
        // the sum of up to three exponentials (Troe: F_cent, SRI: a e^(-b/T) + e^(-T/c)),
        // exponents c + beta t + gamma v
        double S = 0.0;
        const int nt = (int)__ldg(ax + 1);
#pragma unroll 1
        for (int j = 0; j < nt; ++j) {
          const i64* e = ax + 5 + 3 * j;
          const i64 x = pfx::mul_add(as_pair(__ldg(e + 1)), t, pfx::mul_add(as_pair(__ldg(e + 2)), v, 0ll)) & ~1ll;
          S += pfx::exp2_lg(x + __ldg(e), s.exp2);
        }
        const bool pos = tile_normal_pos(S);
        if (!pos) s.sc->bad[lane] = 1;
        const i64 lS = pfx::log2_of(pos ? S : 1.0, t_log2);
        // Troe: log F = log F_cent den^2/(den^2 + x^2), all logarithms to base 10;
        // SRI: F = d S^(1/(1 + log10^2 Pr)) T^e
        double x = pfx::to_double(lgPr) * 0.30102999566398119521, den2 = 1.0;
        if (kind == TK_TROE) {
          const double lf10 = pfx::to_double(lS) * 0.30102999566398119521;
          x += fma(-0.67, lf10, -0.4);
          const double den = fma(-0.14, x, fma(-1.27, lf10, 0.75));
          den2 = den * den;
        }
        X += tile_part(den2 * pdm::rcp(fma(x, x, den2)), lS);
        if (kind == TK_SRI) X += pfx::mul_add(as_pair(__ldg(ax + 15)), u, __ldg(ax + 14));
      }
    }
    X = (X & ~1ll) | (i64)(third && M < 0.0);
    // factors
    i64 Xf = 0, Xr = np ? 0ll : pfx::LG_ZERO;
    for (int q = 0; q < nr; ++q) {
      const int k = (int)((fa >> (16 * q)) & 0xffff) * 32;
      X -= lam[k];
      Xf += alp[k];
    }
    for (int q = 0; q < np; ++q) {
      const int k = (int)((q == 0 ? (fa >> 48) : (fb >> (16 * (q - 1)))) & 0xffff) * 32;
      Xr += alp[k];
    }
    const i64 rate = tile_rate<true, true>(X + Xf, X + Xr, s.exp2);
    s.R[(int)((fb >> 32) & 0xffff) * 32 + lane] = none ? 0ll : rate;
  }
}

#endif  // TILE_DERIV

// species sums of a chunk: per owned species the rows with nu = +1, with -1 (both padded to
// multiples of 4 with the zero row) and with other nu; sink(species, sum).  Every term is cut
// at the headroom hb of its list of n terms, a bias of at most n 2^(hb - 63) of the largest
// term: 2^-51 for 55 terms (160 species' longest list), but 2^-47 from 250 terms.  Units with
// such lists (TILE_ROUND: hb above 7) align four terms with 3 bits of headroom and round
// their sum to hb, 5 instructions more for four terms (3 % of the kernel's time).
struct TilePlus { static constexpr bool minus = false; };
struct TileMinus { static constexpr bool minus = true; };
template <class F>
__device__ __forceinline__ void tile_sums(const i64* rows, int ch, int w, F sink) {
  const char* R = (const char*)rows;
  // a warp's lists follow one another in the entry table: the next four entries and the
  // next species' header are loaded while the last ones are summed (both tables end
  // with a spare element)
  int4 qn = __ldg((const int4*)t_wl + (ch * NW + w) * KPO);              // first entry, ends of the three lists
  int2 on = __ldg((const int2*)t_wo + (ch * NW + w) * KPO);              // species, head-room bits + 256 others
  int4 rn = __ldg((const int4*)(t_we + qn.x));
#pragma unroll 1
  for (int i = 0; i < KPO; ++i) {
    const int4 q = qn;
    const int2 o = on;
    if (o.x < 0) break;
    qn = __ldg((const int4*)t_wl + (ch * NW + w) * KPO + i + 1);
    on = __ldg((const int2*)t_wo + (ch * NW + w) * KPO + i + 1);
#if TILE_ROUND
    const int hb = 3, up = (o.y & 0xff) - 3;    // headroom of four terms, and the rest of the list's
    const i64 half = (1ll << up) >> 1;
    auto fold = [&](i64 b) { return tile_sar(b + half, up); };
#else
    const int hb = o.y & 0xff, up = 0;
    auto fold = [&](i64 b) { return b; };
#endif
    i64 a = 0;
    int e = 0;
    auto quad = [&](int j, auto sign) {
      const int4 r = rn;
      rn = __ldg((const int4*)(t_we + j + 4));
      const i64 v0 = *(const i64*)(R + r.x), v1 = *(const i64*)(R + r.y), v2 = *(const i64*)(R + r.z),
                v3 = *(const i64*)(R + r.w);
      const int e0 = (int)v0 & RATE_M, e1 = (int)v1 & RATE_M, e2 = (int)v2 & RATE_M, e3 = (int)v3 & RATE_M;
      const int en = max(max(e, max(e0, e1)), max(e2, e3)), t = en + hb;
      a = tile_sar(a, en - e);
      e = en;
      const i64 b = fold((tile_sar(v0, t - e0) + tile_sar(v1, t - e1)) + (tile_sar(v2, t - e2) + tile_sar(v3, t - e3)));
      if (decltype(sign)::minus) a -= b; else a += b;
    };
    _Pragma("unroll 2") for (int j = q.x; j < q.y; j += 4) quad(j, TilePlus());
    _Pragma("unroll 2") for (int j = q.y; j < q.z; j += 4) quad(j, TileMinus());
    for (int j = q.z; j < q.z + (o.y >> 8); ++j) {
      const i64 x = *(const i64*)(R + __ldg(t_we + j));
      const int e0 = (int)x & RATE_M, en = max(e, e0);
      a = tile_sar(a, en - e) + fold((i64)__ldg(t_wc + j) * tile_sar(x, en + hb - e0));
      e = en;
    }
    if (q.w > q.z) rn = __ldg((const int4*)(t_we + q.w));
    sink(o.x, tile_to_double(a, e + hb + up - RATE_E, 62));
  }
}

#ifndef TILE_DERIV
extern "C" __global__ void __launch_bounds__(32 * NW, TILE_MINB)
pyro_omega_tile(i64 n, const double* __restrict__ g_rho, const double* __restrict__ g_Tin, int energy_mode,
                const double* __restrict__ g_Y, double* __restrict__ g_Tout, double* __restrict__ g_omega,
                double T_guess, int max_iter, double tol, unsigned long long* __restrict__ g_fail, int split) {
  // split: a cluster of NCH blocks per tile, one chunk of reactions each (few tiles: the
  // chunks' time is the call's; 160 species, 1024 states: 113 us by one block a tile).
  // Every block solves the temperature and prepares the species itself; the sums are added
  // in the order of the chunks, as by one block, so that both forms give the same bits.
  extern __shared__ __align__(16) char s_raw[];
  const TileSmem s = tile_smem(s_raw);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < pfx::EXP2_TAB; i += 32 * NW) s.exp2[i] = t_exp2[i];
  const i64 tiles = (n + 31) >> 5;
  if (w == 0) {                                 // the zero row that pads the lists of the species sums
    s.R[TILE_ROWS * 32 + lane] = 0;
    s.lam[NSP * 32 + lane] = 0;                 // the unit factor
    s.alp[NSP * 32 + lane] = 0;
  }
  const int rank = split ? (int)(blockIdx.x % NCH) : 0, blocks = split ? NCH : 1;
#pragma unroll 1
  for (i64 tile = blockIdx.x / blocks; tile < tiles; tile += gridDim.x / blocks) {
    const i64 p = tile * 32 + lane;
    const i64 pc = p < n ? p : n - 1;
    const double* Yp = g_Y + pc;
    const double rho = __ldg(g_rho + pc);
    // a tile without any state in the tables (a cold block): no work beside the FP64 kernel's
    const double Tin = __ldg(g_Tin + pc);
    if (!energy_mode && !__any_sync(0xffffffffu, Tin > T_LO && Tin < T_HI)) {
      if (w == 0 && p < n && rank == 0) g_omega[p] = __longlong_as_double(TILE_OPEN);
      continue;
    }
    {
      {
        double y[KPW];
        double ys = 0.0;
#pragma unroll
        for (int i = 0; i < KPW; ++i) {
          const int k = w + i * NW;
          y[i] = k < NSP ? __ldg(Yp + k * n) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < KPW; ++i) {
          const int k = w + i * NW;
          if (k < NSP) {
            ys = fma(y[i], __ldg(t_iw + k), ys);
            s.alp[k * 32 + lane] = __double_as_longlong(y[i]);
          }
        }
        s.ys[w * 32 + lane] = ys;
      }
      bool bad = false;
      double T;
      bool ok = true;
      if (energy_mode) {
        tile_energy(s, Yp, n, Tin, T_guess, max_iter, (float)tol, w, lane, T, ok);
      } else {
        T = Tin;
        __syncthreads();
      }
      if (w == 0) {
        if (energy_mode && p < n && rank == 0) {
          if (!ok) atomicAdd(g_fail, 1ull);
          g_Tout[p] = T;
        }
        // state scalars; states outside the tables' range are left to the FP64 kernel
        const unsigned re = ((unsigned)__double2hiint(rho) >> 20) & 0x7ff;
        const bool in = T > T_LO && T < T_HI && re >= 1023 - 60 && re <= 1023 + 20;
        const double Ts = in ? T : 1000.0;
        s.sc->T[lane] = Ts;
        tile_T(Ts, s.sc->u[lane], s.sc->v[lane], s.sc->t[lane], s.sc->lgT[lane]);
        s.sc->lgrho[lane] = pfx::log2_of(in ? fabs(rho) : 1.0, t_log2) | (i64)((u64)__double_as_longlong(rho) >> 63);
        s.sc->bad[lane] = in ? 0 : 1;
        const bool none = !__any_sync(0xffffffffu, in);
        if (lane == 0) { s.sc->neg = 0; s.sc->none = none; }
        __syncwarp();
        if (__double_as_longlong(rho) < 0) s.sc->neg = 1;
      }
      if (w == NW - 1) {
        double a = 0.0;
#pragma unroll
        for (int i = 0; i < NW; ++i) a += s.ys[i * 32 + lane];
        s.sc->ysum[lane] = a;
      }
      __syncthreads();
      if (s.sc->none) {                          // the same, its temperatures solved
        if (w == 0 && p < n && rank == 0) g_omega[p] = __longlong_as_double(TILE_OPEN);
        __syncthreads();
        continue;
      }
      // species: lambda_k and alpha_k
      const Pair u = s.sc->u[lane], v = s.sc->v[lane], t = s.sc->t[lane];
      const i64 lgrho = s.sc->lgrho[lane];
      const int hi = pdm::to_float_trunc(s.sc->T[lane]) >= (float)TMID ? 1 : 0;
#pragma unroll 1
      for (int k = w; k < NSP; k += NW) {
        const longlong2* c = (const longlong2*)(t_sp + (k * 2 + hi) * 8);
        const longlong2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2), c3 = __ldg(c + 3);   // c4 c3 | c2 c1 | c0 cl | ci -
        i64 q = pfx::horner(c0.x, t, c0.y);
        q = pfx::horner(q, t, c1.x);
        q = pfx::horner(q, t, c1.y);
        q = pfx::horner(q, t, c2.x);
        q = tile_K(q, c2.y, c3.x, u, v);
        const u64 yb = (u64)s.alp[k * 32 + lane];
        int ye = (int)(yb >> 52) & 0x7ff;
        const bool zero = (yb << 1) == 0ull;
        bad |= ye > 1023;
        u64 ym = (yb & 0xfffffffffffffull) | 0x10000000000000ull;
        if (ye == 0) {                           // subnormal
          const int sh = pfx::clz64(ym ^ 0x10000000000000ull) - 11;
          ym = (ym ^ 0x10000000000000ull) << sh;
          ye = 1 - sh;
        }
        i64 ly = ((i64)(ye - 1023) << pfx::LG_F) + (((pfx::log2_mant(ym, t_log2) + 0x1000ll) >> 13) << 1);
        ly = zero ? pfx::LG_ZERO : (ly | (i64)(yb >> 63));
        if ((i64)yb < 0 && !zero) s.sc->neg = 1;
        s.lam[k * 32 + lane] = q;
        s.alp[k * 32 + lane] = q + ly + lgrho;
      }
      if (bad) s.sc->bad[lane] = 1;
      __syncthreads();
    }
    const Pair u = s.sc->u[lane], v = s.sc->v[lane];
    const bool signs = s.sc->neg != 0;
#pragma unroll 1
    for (int ch = rank; ch < (split ? rank + 1 : NCH); ++ch) {
      const int* seg = t_seg + (ch * NW + w) * (NCLS + 1);
      // every other warp takes the plain reactions last: they load the integer pipes, the
      // others the FP64 pipe
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        if ((w & 1) == half) {
          if (signs) {
            TILE_PLAIN(true)
          } else {
            TILE_PLAIN(false)
          }
        } else {
          const int a = __ldg(seg + NCLS - 1), b = __ldg(seg + NCLS);
          if (a < b) tile_other(s, a, b, lane, rho, Yp, n);
        }
      }
      __syncthreads();
      const bool open = s.sc->bad[lane] != 0;         // behind the barrier: reactions set it too
      tile_sums(s.R + lane, ch, w, [&](int k, double v) {
        if (split) {
          ((double*)s.lam)[k * 32 + lane] = v;       // the species arrays are free after the only chunk
        } else if (p < n) {
          double* out = g_omega + k * n + p;
          if (ch > 0) v += *out;
          if (open && k == 0) v = __longlong_as_double(TILE_OPEN);
          *out = v;
        }
      });
      __syncthreads();
    }
#if NCH > 1
    if (split) {
      auto barrier = [] {
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      };
      auto remote = [](const void* a, int r) {
        unsigned b, l = (unsigned)__cvta_generic_to_shared(a);
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(l), "r"(r));
        return b;
      };
      barrier();
#pragma unroll 1
      for (int k = rank + w * NCH; k < NSP; k += NW * NCH) {
        double v = 0.0;
        int any = 0;
#pragma unroll
        for (int r = 0; r < NCH; ++r) {
          double x;
          int b;
          asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(remote(s.lam + k * 32 + lane, r)) : "memory");
          asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(b) : "r"(remote(s.sc->bad + lane, r)) : "memory");
          v = r ? x + v : x;
          any |= b;
        }
        if (any && k == 0) v = __longlong_as_double(TILE_OPEN);
        if (p < n) g_omega[k * n + p] = v;
      }
      barrier();                                 // the other blocks read this one's arrays
    }
#endif
  }
}
#endif  // TILE_DERIV
