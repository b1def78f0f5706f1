// Jacobian-vector product of the net production rates for a tile of 32 states per block
// (lane = state, warps split species and reactions), over the tables of pyro_tile.cuh.
//
// The per-thread kernel needed some 13 k FP64 instructions a state on 53 species (19
// cycles of an SM each) in 500 KB of straight-line code.  Here the exponents, the
// exponentials and the sums of the tangents are integer work; the FP64 pipe keeps the
// activities a_k = exp(L_k) rho Y_k with their tangents and, per reaction,
//   dR = kk (dx D + dP' - dP''),  dx = (b/T + theta/T^2) dT - sum nu' dL,
// 12 instructions for two factors a side (262,139 states: 7.73 -> 4.48 ms; FP64 pipe 81 of its
// 84 %).  A reaction's dR is kept as a rate word.
// States outside the tables' range, and states with a tangent that overflows or is not
// finite, get TILE_OPEN in their first output and are evaluated by the FP64 kernel.
#define TILE_DERIV
#define RATE_E 1023
#include "pyro_tile.cuh"

struct JvpScalars {
  double T[32], invT[32], rho[32], drho[32], drr[32], dT[32], ysum[32], dysum[32];
  Pair u[32], v[32], t[32];
  i64 lgT[32];
  int bad[32];
};

struct JvpSmem {
  u64* exp2;
  i64* lam;             // [NSP + 1][32], as the next three: the species and a unit factor
  double *a, *da, *dL;
  i64* R;               // rows and one zero row; first the partial sums of Y/W and dY/W
  JvpScalars* sc;
};

// a double as a rate word (0 below the normal range); e = 2047 marks overflow or NaN.  Its 53
// bits fill the word but for one: the last one is rounded off by the exponent's bits (RATE_M).
__device__ __forceinline__ i64 jvp_word(double x) {
  const int h = __double2hiint(x), e = (h >> 20) & 0x7ff;
  const u64 m = ((u64)__double_as_longlong(x) & 0xfffffffffffffull) << 10 | 0x4000000000000000ull;   // 1.f 2^62
  const i64 w = (((i64)m ^ (i64)(h >> 31)) & ~(i64)RATE_M) | (i64)e;
  return e == 0 ? 0ll : w;
}
__device__ __forceinline__ bool jvp_finite(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }

template <int NF, bool REV>
__device__ __forceinline__ void jvp_plain(const JvpSmem& s, int i0, int i1, Pair u, Pair v, double u1, double u2, int lane) {
  const char* lam = (const char*)(s.lam + lane);
  const char *a = (const char*)(s.a + lane), *da = (const char*)(s.da + lane), *dL = (const char*)(s.dL + lane);
  char* R = (char*)(s.R + lane);
  const int4* r = (const int4*)(t_rx + i0 * 8);
  int4 r0 = __ldg(r), r1 = __ldg(r + 1), r2 = __ldg(r + 2), r3 = __ldg(r + 3);
#pragma unroll 1
  for (int i = i0; i < i1; ++i) {
    const int4 c0 = r0, c1 = r1, c2 = r2, c3 = r3;
    const double2 bt = __ldg((const double2*)t_rd + i);    // b, theta
    r += 4;
    r0 = __ldg(r); r1 = __ldg(r + 1); r2 = __ldg(r + 2); r3 = __ldg(r + 3);
    Pair beta, tau;
    beta.lo = c0.z; beta.hi = c0.w;
    tau.lo = c1.x; tau.hi = c1.y;
    const i64 c = (i64)(((u64)(unsigned)c0.y << 32) | (unsigned)c0.x);
    auto lg = [&](int o) { return *(const i64*)(lam + o); };
    auto d = [](const char* b, int o) { return *(const double*)(b + o); };
    i64 X = (pfx::mul_add(tau, v, pfx::mul_add(beta, u, c)) & ~1ll) - lg(c1.z) - lg(c1.w);
    if (NF > 2) X -= lg(c2.x);
    const double kk = pfx::exp2_lg(X, s.exp2);
    double dx = fma(bt.x, u1, bt.y * u2) - d(dL, c1.z) - d(dL, c1.w);
    if (NF > 2) dx -= d(dL, c2.x);
    const double a0 = d(a, c1.z), a1 = d(a, c1.w);
    double P = a0 * a1, dP = fma(d(da, c1.z), a1, a0 * d(da, c1.w));
    if (NF > 2) {
      const double a2 = d(a, c2.x);
      dP = fma(dP, a2, P * d(da, c2.x));
      P *= a2;
    }
    if (REV) {
      const double b0 = d(a, c2.y), b1 = d(a, c2.z), e0 = d(da, c2.y), e1 = d(da, c2.z);
      if (NF > 2) {
        const double b2 = d(a, c2.w), q = b0 * b1, dq = fma(e0, b1, b0 * e1);
        P = fma(-q, b2, P);
        dP -= fma(dq, b2, q * d(da, c2.w));
      } else {
        P = fma(-b0, b1, P);
        dP = fma(-e0, b1, fma(-b0, e1, dP));
      }
    }
    const double dR = kk * fma(dx, P, dP);
    if (!jvp_finite(dR)) s.sc->bad[lane] = 1;
    i64 w = jvp_word(dR);
    i64* o = (i64*)(R + c3.x);
    if (c3.y) w = tile_add(*o, w);
    *o = w;
  }
}

__device__ __forceinline__ void jvp_other(const JvpSmem& s, int i0, int i1, int lane, const double* __restrict__ Yp,
                                          const double* __restrict__ dYp, i64 n) {
  const JvpScalars& z = *s.sc;
  const Pair u = z.u[lane], v = z.v[lane], t = z.t[lane];
  const double invT = z.invT[lane], invT2 = invT * invT, rho = z.rho[lane], dT = z.dT[lane];
  const double LOG10_2 = 0.30102999566398119521, LN_2 = 0.69314718055994530942, LN10_INV = 0.43429448190325182765;
#pragma unroll 1
  for (int i = i0; i < i1; ++i) {
    const i64* r = t_rx + i * 8;
    const i64 fa = __ldg(r + 3), fb = __ldg(r + 4);
    const int nr = (int)((fb >> 48) & 0xf), np = (int)((fb >> 52) & 0xf), kind = (int)((fb >> 56) & 0xf);
    const i64* ax = t_ax + __ldg(r + 5);
    const double* fx = t_fx + __ldg(r + 5);
    const int ne = (int)__ldg(ax);
    double mS = z.ysum[lane], dmS = z.dysum[lane];
#pragma unroll 4
    for (int q = 0; q < ne; ++q) {
      const longlong2 c = __ldg((const longlong2*)(ax + 16) + q);
      mS = fma(__ldg(Yp + c.x * n), ax_d(c.y), mS);
      dmS = fma(__ldg(dYp + c.x * n), ax_d(c.y), dmS);
    }
    const double M = rho * mS, dM = fma(z.drho[lane], mS, rho * dmS);
    // (a third body's [M] is a factor: zero or negative as it may be)
    if (!(kind == TK_THREEBODY ? jvp_finite(M) : tile_normal_pos(M)) || !jvp_finite(dM)) s.sc->bad[lane] = 1;
    const i64 lgM = pfx::log2_of(M, t_log2);
    i64 X;
    double tau, sM = 0.0;          // d ln kk/dT, d ln kk/d ln M
    if (kind == TK_PLOG) {
      const int nn = (int)__ldg(ax + 1);
      const i64* nd = ax + 16;
      const double* fd = fx + 16;
      const i64 lgp = z.lgT[lane] + lgM + T_LG_R;
      int q = 0;
      for (int j = 1; j + 1 < nn; ++j) if (lgp >= __ldg(nd + 5 * j)) q = j;
      const i64* a = nd + 5 * q;
      const i64 xa = tile_K(__ldg(a + 2), __ldg(a + 3), __ldg(a + 4), u, v);
      const i64 xb = tile_K(__ldg(a + 7), __ldg(a + 8), __ldg(a + 9), u, v);
      const double inv = ax_d(__ldg(a + 1)), pu = pfx::to_double(lgp - __ldg(a)) * inv;
      const double pf = fmin(fmax(pu, 0.0), 1.0);
      X = pf > 0.0 ? xa + tile_part(pf, xb - xa) : xa;
      sM = pu > 0.0 && pu < 1.0 ? pfx::to_double(xb - xa) * inv : 0.0;
      const double ta = fma(__ldg(fd + 5 * q + 3), invT, __ldg(fd + 5 * q + 4) * invT2);
      const double tb = fma(__ldg(fd + 5 * q + 8), invT, __ldg(fd + 5 * q + 9) * invT2);
      tau = fma(sM, invT, fma(pf, tb - ta, ta));
    } else {
      X = tile_K(__ldg(r), __ldg(r + 1), __ldg(r + 2), u, v);
      const double2 bt = __ldg((const double2*)t_rd + i);
      tau = fma(bt.x, invT, bt.y * invT2);
    }
    double scale = 1.0;
    if (kind == TK_THREEBODY) {
      scale = M;
      sM = 1.0;
    }
    if (kind >= TK_LINDEMANN && kind <= TK_SRI) {
      const i64 lgPr = tile_K(__ldg(ax + 2), __ldg(ax + 3), __ldg(ax + 4), u, v) + lgM;
      const double pT = fma(__ldg(fx), invT, __ldg(fx + 1) * invT2);      // d ln Pr/dT at fixed [M]
      // 1 - Pr/(1+Pr) = q Pr/(1+Pr), q = 1/Pr, formed as a product (the difference cancels)
      const double q = pfx::exp2_lg((-lgPr) & ~1ll, s.exp2);
      scale = pdm::rcp(1.0 + q);
      sM = q * scale;
      double extra = 0.0;
      if (kind != TK_LINDEMANN) {
        double S = 0.0, dS = 0.0;
        const int nt = (int)__ldg(ax + 1);
#pragma unroll 1
        for (int j = 0; j < nt; ++j) {
          const i64* e = ax + 5 + 3 * j;
          const i64 x = pfx::mul_add(as_pair(__ldg(e + 1)), t, pfx::mul_add(as_pair(__ldg(e + 2)), v, 0ll)) & ~1ll;
          const double y = pfx::exp2_lg(x + __ldg(e), s.exp2);
          S += y;
          dS = fma(y, fma(__ldg(fx + 3 + 2 * j), invT2, __ldg(fx + 2 + 2 * j)), dS);
        }
        if (!tile_normal_pos(S)) s.sc->bad[lane] = 1;
        const i64 lS = pfx::log2_of(S, t_log2);
        const double lp10 = pfx::to_double(lgPr) * LOG10_2, ls = pfx::to_double(lS), rS = pdm::rcp(S);
        if (kind == TK_TROE) {
          const double lf = ls * LOG10_2, x = lp10 + fma(-0.67, lf, -0.4), den = fma(-0.14, x, fma(-1.27, lf, 0.75));
          const double den2 = den * den, rD = pdm::rcp(fma(x, x, den2)), f = den2 * rD, w = 2.0 * lf * rD * rD;
          const double Ax = -w * den2 * x, Ad = w * den * x * x;
          X += tile_part(f, lS);
          sM += fma(-0.14, Ad, Ax);
          extra = fma(-0.67, Ax, fma(-1.1762, Ad, f)) * dS * rS;
        } else {
          const double f = pdm::rcp(fma(lp10, lp10, 1.0));
          X += tile_part(f, lS) + pfx::mul_add(as_pair(__ldg(ax + 15)), u, __ldg(ax + 14));
          sM = fma(ls * LN_2, -2.0 * lp10 * f * f * LN10_INV, sM);
          extra = fma(f * dS, rS, __ldg(fx + 8) * invT);
        }
      }
      tau += fma(sM, pT, extra);
    }
    double dx = tau * dT;
    const i64* lam = s.lam + lane;
    const double *a = s.a + lane, *da = s.da + lane, *dL = s.dL + lane;
    double Pf = 1.0, dPf = 0.0, Pr = np ? 1.0 : 0.0, dPr = 0.0;
    for (int q = 0; q < nr; ++q) {
      const int k = (int)((fa >> (16 * q)) & 0xffff) * 32;
      X -= lam[k];
      dx -= dL[k];
      dPf = fma(dPf, a[k], Pf * da[k]);
      Pf *= a[k];
    }
    for (int q = 0; q < np; ++q) {
      const int k = (int)((q == 0 ? (fa >> 48) : (fb >> (16 * (q - 1)))) & 0xffff) * 32;
      dPr = fma(dPr, a[k], Pr * da[k]);
      Pr *= a[k];
    }
    const double kt = pfx::exp2_lg(X & ~1ll, s.exp2);
    const double D = Pf - Pr, kk = kt * scale;
    // d kk = kk (dx + sM dM/M); a third body's kk/M is kt
    const double dkk = kind == TK_THREEBODY ? fma(kk, dx, kt * dM) : kk * fma(sM * dM, pdm::rcp(M), dx);
    const double dR = fma(dkk, D, kk * (dPf - dPr));
    if (!jvp_finite(dR)) s.sc->bad[lane] = 1;
    s.R[(int)((fb >> 32) & 0xffff) * 32 + lane] = jvp_word(dR);
  }
}

extern "C" __global__ void __launch_bounds__(32 * NW, TILE_MINB)
pyro_jvp_tile(i64 n, const double* __restrict__ g_rho, const double* __restrict__ g_T, const double* __restrict__ g_Y,
              const double* __restrict__ g_drho, const double* __restrict__ g_dT, const double* __restrict__ g_dY,
              double* __restrict__ g_dw) {
  extern __shared__ __align__(16) char s_raw[];
  JvpSmem s;
  s.exp2 = (u64*)s_raw;
  s.lam = (i64*)(s_raw + pfx::EXP2_TAB * 8);
  s.a = (double*)(s.lam + (NSP + 1) * 32);
  s.da = s.a + (NSP + 1) * 32;
  s.dL = s.da + (NSP + 1) * 32;
  s.R = (i64*)(s.dL + (NSP + 1) * 32);
  s.sc = (JvpScalars*)(s.R + (TILE_ROWS + 1) * 32);
  double* part = (double*)s.R;                   // NW x 2 x 32
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < pfx::EXP2_TAB; i += 32 * NW) s.exp2[i] = t_exp2[i];
  if (w == 0) {
    s.R[TILE_ROWS * 32 + lane] = 0;
    s.lam[NSP * 32 + lane] = 0;                  // the unit factor
    s.a[NSP * 32 + lane] = 1.0;
    s.da[NSP * 32 + lane] = 0.0;
    s.dL[NSP * 32 + lane] = 0.0;
  }
  const i64 tiles = (n + 31) >> 5;
#pragma unroll 1
  for (i64 tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const i64 p = tile * 32 + lane, pc = p < n ? p : n - 1;
    // a tile without any state in the tables (a cold block): no work beside the FP64 kernel's
    const double T_in = __ldg(g_T + pc);
    if (!__any_sync(0xffffffffu, T_in > T_LO && T_in < T_HI)) {
      if (w == 0 && p < n) g_dw[p] = __longlong_as_double(TILE_OPEN);
      continue;
    }
    const double *Yp = g_Y + pc, *dYp = g_dY + pc;
    {
      double y[KPW], dy[KPW], ys = 0.0, dys = 0.0;
#pragma unroll
      for (int i = 0; i < KPW; ++i) {
        const int k = w + i * NW;
        y[i] = k < NSP ? __ldg(Yp + k * n) : 0.0;
        dy[i] = k < NSP ? __ldg(dYp + k * n) : 0.0;
      }
#pragma unroll
      for (int i = 0; i < KPW; ++i) {
        const int k = w + i * NW;
        if (k < NSP) {
          const double c = __ldg(t_iw + k);
          ys = fma(y[i], c, ys);
          dys = fma(dy[i], c, dys);
          s.a[k * 32 + lane] = y[i];             // until the species phase
          s.da[k * 32 + lane] = dy[i];
        }
      }
      part[(w * 2) * 32 + lane] = ys;
      part[(w * 2 + 1) * 32 + lane] = dys;
    }
    if (w == 0) {
      const double T = T_in, rho = __ldg(g_rho + pc), drho = __ldg(g_drho + pc), dT = __ldg(g_dT + pc);
      const unsigned re = ((unsigned)__double2hiint(rho) >> 20) & 0x7ff;
      const bool in = T > T_LO && T < T_HI && re >= 1023 - 60 && re <= 1023 + 20 && rho > 0.0 && jvp_finite(drho) &&
                      jvp_finite(dT);
      const double Ts = in ? T : 1000.0, rs = in ? rho : 1.0;
      JvpScalars& z = *s.sc;
      z.T[lane] = Ts;
      z.invT[lane] = pdm::rcp(Ts);
      z.rho[lane] = rs;
      z.drho[lane] = in ? drho : 0.0;
      z.drr[lane] = in ? drho * pdm::rcp(rs) : 0.0;
      z.dT[lane] = in ? dT : 0.0;
      tile_T(Ts, z.u[lane], z.v[lane], z.t[lane], z.lgT[lane]);
      z.bad[lane] = in ? 0 : 1;
    }
    __syncthreads();
    if (w == NW - 1) {
      double a = 0.0, b = 0.0;
#pragma unroll
      for (int i = 0; i < NW; ++i) { a += part[i * 64 + lane]; b += part[i * 64 + 32 + lane]; }
      s.sc->ysum[lane] = a;
      s.sc->dysum[lane] = b;
    }
    const Pair u = s.sc->u[lane], v = s.sc->v[lane];
    const double T = s.sc->T[lane], invT = s.sc->invT[lane], dT = s.sc->dT[lane];
    {
      const Pair t = s.sc->t[lane];
      const double rho = s.sc->rho[lane], drr = s.sc->drr[lane];
      const int hi = pdm::to_float_trunc(T) >= (float)TMID ? 1 : 0;
      bool bad = false;
#pragma unroll 1
      for (int k = w; k < NSP; k += NW) {
        const longlong2* c = (const longlong2*)(t_sp + (k * 2 + hi) * 8);
        const longlong2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2), c3 = __ldg(c + 3);
        i64 q = pfx::horner(c0.x, t, c0.y);
        q = pfx::horner(q, t, c1.x);
        q = pfx::horner(q, t, c1.y);
        q = pfx::horner(q, t, c2.x);
        q = tile_K(q, c2.y, c3.x, u, v);
        const double* h = t_h + (k * 2 + hi) * 6;
        double hr = fma(T, fma(T, fma(T, fma(T, __ldg(h + 4), __ldg(h + 3)), __ldg(h + 2)), __ldg(h + 1)), __ldg(h));
        hr = fma(__ldg(h + 5), invT, hr);
        const double Lp = fma(-hr, invT, invT), E = pfx::exp2_lg(q, s.exp2);
        const double y = s.a[k * 32 + lane], dy = s.da[k * 32 + lane];
        bad |= !jvp_finite(y) || !jvp_finite(dy);
        const double a = E * (rho * y);
        s.lam[k * 32 + lane] = q;
        s.a[k * 32 + lane] = a;
        s.da[k * 32 + lane] = fma(a, fma(Lp, dT, drr), E * (rho * dy));
        s.dL[k * 32 + lane] = Lp * dT;
      }
      if (bad) s.sc->bad[lane] = 1;
    }
    __syncthreads();
    const double u1 = dT * invT, u2 = u1 * invT;
#pragma unroll 1
    for (int ch = 0; ch < NCH; ++ch) {
      const int* seg = t_seg + (ch * NW + w) * (NCLS + 1);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        if ((w & 1) == half) {
          TILE_PLAIN
        } else {
          const int a = __ldg(seg + NCLS - 1), b = __ldg(seg + NCLS);
          if (a < b) jvp_other(s, a, b, lane, Yp, dYp, n);
        }
      }
      __syncthreads();
      const bool open = s.sc->bad[lane] != 0;
      tile_sums(s.R + lane, ch, w, [&](int k, double x) {
        if (p < n) {
          double* out = g_dw + k * n + p;
          if (ch > 0) x += *out;
          if (open && k == 0) x = __longlong_as_double(TILE_OPEN);
          *out = x;
        }
      });
      __syncthreads();
    }
  }
}
