// Vector-Jacobian product of the net production rates for a tile of 32 states per block
// (lane = state, warps split species and reactions), over the tables of pyro_tile.cuh.
//
// Exponents and exponentials are integer work.  Per reaction the FP64 pipe forms
//   Rbar = sum nu wbar,  Db = Rbar kk,  xb = Db (P' - P''),  Tbar += xb (tau - sum nu' L'),
// and stores Db; the adjoints of the activities are then gathered per species,
//   abar_i = sum_j +-Db_j (product of the side's other factors),
// in a fixed order, with no conflicts between warps: 17 FP64 instructions a reaction of two
// factors a side in all, against some 40 of the per-thread kernel (2^18 states 8.6 -> 5.3 ms,
// FP64 pipe 81 of its 84 %).  [M] adjoints likewise.
// States outside the tables' range, with non-finite inputs or results, get TILE_OPEN in
// rho_bar and are evaluated by the FP64 kernel.
#define TILE_DERIV
#define RATE_E 1023
#include "pyro_tile.cuh"

struct VjpScalars {
  double T[32], invT[32], rho[32], ysum[32], Mtot[32];
  Pair u[32], v[32], t[32];
  i64 lgT[32];
  int bad[32];
};

struct VjpSmem {
  u64* exp2;
  i64* lam;             // [NSP + 1][32], as the next three: the species and a unit factor
  double *a, *Lp, *wb;
  double* Db;           // rows; first the partial sums of Y/W
  double* Mb;           // rows of the reactions with [M]
  double *pT, *pM, *pR; // NW x 32 partial sums
  VjpScalars* sc;
};

__device__ __forceinline__ bool vjp_finite(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }

template <int NF, bool REV>
__device__ __forceinline__ void vjp_plain(const VjpSmem& s, int i0, int i1, Pair u, Pair v, double invT, double invT2,
                                          double& Tb, int lane) {
  const char* lam = (const char*)(s.lam + lane);
  const char *a = (const char*)(s.a + lane), *Lp = (const char*)(s.Lp + lane), *wb = (const char*)(s.wb + lane);
  char* R = (char*)(s.Db + lane);
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
    double sT = fma(bt.x, invT, bt.y * invT2) - d(Lp, c1.z) - d(Lp, c1.w);
    double Rb = (d(wb, c2.y) + d(wb, c2.z)) - (d(wb, c1.z) + d(wb, c1.w));
    double P = d(a, c1.z) * d(a, c1.w);
    if (NF > 2) {
      X -= lg(c2.x);
      sT -= d(Lp, c2.x);
      Rb += d(wb, c2.w) - d(wb, c2.x);
      P *= d(a, c2.x);
    }
    if (REV) P = fma(-d(a, c2.y), NF > 2 ? d(a, c2.z) * d(a, c2.w) : d(a, c2.z), P);
    const double Db = Rb * pfx::exp2_lg(X, s.exp2);
    Tb = fma(Db * P, sT, Tb);
    double* o = (double*)(R + c3.x);
    *o = c3.y ? *o + Db : Db;
  }
}

__device__ __forceinline__ void vjp_other(const VjpSmem& s, int i0, int i1, int lane, const double* __restrict__ Yp, i64 n,
                                          double& Tb, double& Mtot, double& rhobM) {
  const VjpScalars& z = *s.sc;
  const Pair u = z.u[lane], v = z.v[lane], t = z.t[lane];
  const double invT = z.invT[lane], invT2 = invT * invT, rho = z.rho[lane];
  const double LOG10_2 = 0.30102999566398119521, LN_2 = 0.69314718055994530942, LN10_INV = 0.43429448190325182765;
#pragma unroll 1
  for (int i = i0; i < i1; ++i) {
    const i64* r = t_rx + i * 8;
    const i64 fa = __ldg(r + 3), fb = __ldg(r + 4);
    const int nr = (int)((fb >> 48) & 0xf), np = (int)((fb >> 52) & 0xf), kind = (int)((fb >> 56) & 0xf);
    const bool rev = ((fb >> 60) & 1) != 0;
    const i64* ax = t_ax + __ldg(r + 5);
    const double* fx = t_fx + __ldg(r + 5);
    const double mS = tile_mS(ax + 16, (int)__ldg(ax), z.ysum[lane], Yp, n), M = rho * mS;
    // (a third body's [M] is a factor: zero or negative as it may be)
    if (!(kind == TK_THREEBODY ? vjp_finite(M) : tile_normal_pos(M))) s.sc->bad[lane] = 1;
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
    if (kind == TK_THREEBODY) scale = M;
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
    const i64* lam = s.lam + lane;
    const double *a = s.a + lane, *Lp = s.Lp + lane, *wb = s.wb + lane;
    double Pf = 1.0, Pr = rev ? 1.0 : 0.0, Rb = 0.0;
    for (int q = 0; q < nr; ++q) {
      const int k = (int)((fa >> (16 * q)) & 0xffff) * 32;
      X -= lam[k];
      tau -= Lp[k];
      Rb -= wb[k];
      Pf *= a[k];
    }
    for (int q = 0; q < np; ++q) {
      const int k = (int)((q == 0 ? (fa >> 48) : (fb >> (16 * (q - 1)))) & 0xffff) * 32;
      Rb += wb[k];
      Pr *= a[k];
    }
    const double kt = pfx::exp2_lg(X & ~1ll, s.exp2), kk = kt * scale, D = Pf - Pr;
    const double Db = Rb * kk;
    Tb = fma(Db * D, tau, Tb);
    // [M] adjoint: Rbar D dkk/dM (a third body's dkk/dM is kt)
    const double m = kind == TK_THREEBODY ? Rb * kt * D : Db * D * sM * pdm::rcp(M);
    Mtot += m;
    rhobM = fma(m, mS, rhobM);
    s.Db[(int)((fb >> 32) & 0xffff) * 32 + lane] = Db;
    s.Mb[(int)__ldg(r + 6) * 32 + lane] = m;
  }
}

extern "C" __global__ void __launch_bounds__(32 * NW, TILE_MINB)
pyro_vjp_tile(i64 n, const double* __restrict__ g_rho, const double* __restrict__ g_T, const double* __restrict__ g_Y,
              const double* __restrict__ g_wb, double* __restrict__ g_rhob, double* __restrict__ g_Tb,
              double* __restrict__ g_Yb) {
  extern __shared__ __align__(16) char s_raw[];
  VjpSmem s;
  s.exp2 = (u64*)s_raw;
  s.lam = (i64*)(s_raw + pfx::EXP2_TAB * 8);
  s.a = (double*)(s.lam + (NSP + 1) * 32);
  s.Lp = s.a + (NSP + 1) * 32;
  s.wb = s.Lp + (NSP + 1) * 32;
  s.Db = s.wb + (NSP + 1) * 32;
  s.Mb = s.Db + (TILE_ROWS + 1) * 32;
  s.pT = s.Mb + (T_MROWS + 1) * 32;
  s.pM = s.pT + NW * 32;
  s.pR = s.pM + NW * 32;
  s.sc = (VjpScalars*)(s.pR + NW * 32);
  double* part = s.Db;                           // NW x 32
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < pfx::EXP2_TAB; i += 32 * NW) s.exp2[i] = t_exp2[i];
  if (w == 0) {
    s.lam[NSP * 32 + lane] = 0;                  // the unit factor
    s.a[NSP * 32 + lane] = 1.0;
    s.Lp[NSP * 32 + lane] = 0.0;
    s.wb[NSP * 32 + lane] = 0.0;
  }
  const i64 tiles = (n + 31) >> 5;
#pragma unroll 1
  for (i64 tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const i64 p = tile * 32 + lane, pc = p < n ? p : n - 1;
    // a tile without any state in the tables (a cold block): no work beside the FP64 kernel's
    const double T_in = __ldg(g_T + pc);
    if (!__any_sync(0xffffffffu, T_in > T_LO && T_in < T_HI)) {
      if (w == 0 && p < n) g_rhob[p] = __longlong_as_double(TILE_OPEN);
      continue;
    }
    const double* Yp = g_Y + pc;
    bool bad = false;
    {
      double y[KPW], b[KPW], ys = 0.0;
#pragma unroll
      for (int i = 0; i < KPW; ++i) {
        const int k = w + i * NW;
        y[i] = k < NSP ? __ldg(Yp + k * n) : 0.0;
        b[i] = k < NSP ? __ldg(g_wb + k * n + pc) : 0.0;
      }
#pragma unroll
      for (int i = 0; i < KPW; ++i) {
        const int k = w + i * NW;
        if (k < NSP) {
          ys = fma(y[i], __ldg(t_iw + k), ys);
          s.a[k * 32 + lane] = y[i];             // until the species phase
          s.wb[k * 32 + lane] = b[i];
          bad |= !vjp_finite(y[i]) || !vjp_finite(b[i]);
        }
      }
      part[w * 32 + lane] = ys;
    }
    if (w == 0) {
      const double T = T_in, rho = __ldg(g_rho + pc);
      const unsigned re = ((unsigned)__double2hiint(rho) >> 20) & 0x7ff;
      const bool in = T > T_LO && T < T_HI && re >= 1023 - 60 && re <= 1023 + 20 && rho > 0.0;
      const double Ts = in ? T : 1000.0;
      VjpScalars& z = *s.sc;
      z.T[lane] = Ts;
      z.invT[lane] = pdm::rcp(Ts);
      z.rho[lane] = in ? rho : 1.0;
      tile_T(Ts, z.u[lane], z.v[lane], z.t[lane], z.lgT[lane]);
      z.bad[lane] = in ? 0 : 1;
    }
    __syncthreads();
    if (w == NW - 1) {
      double a = 0.0;
#pragma unroll
      for (int i = 0; i < NW; ++i) a += part[i * 32 + lane];
      s.sc->ysum[lane] = a;
    }
    const Pair u = s.sc->u[lane], v = s.sc->v[lane];
    const double T = s.sc->T[lane], invT = s.sc->invT[lane], rho = s.sc->rho[lane];
    {
      const Pair t = s.sc->t[lane];
      const int hi = pdm::to_float_trunc(T) >= (float)TMID ? 1 : 0;
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
        s.lam[k * 32 + lane] = q;
        s.a[k * 32 + lane] = pfx::exp2_lg(q, s.exp2) * (rho * s.a[k * 32 + lane]);
        s.Lp[k * 32 + lane] = fma(-hr, invT, invT);
      }
      if (bad) s.sc->bad[lane] = 1;
    }
    __syncthreads();
    {
      const double invT2 = invT * invT;
      double Tb = 0.0, Mtot = 0.0, rhobM = 0.0;
      const int* seg = t_seg + w * (NCLS + 1);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        if ((w & 1) == half) {
          TILE_PLAIN
        } else {
          const int a = __ldg(seg + NCLS - 1), b = __ldg(seg + NCLS);
          if (a < b) vjp_other(s, a, b, lane, Yp, n, Tb, Mtot, rhobM);
        }
      }
      s.pT[w * 32 + lane] = Tb;
      s.pM[w * 32 + lane] = Mtot;
      s.pR[w * 32 + lane] = rhobM;
    }
    __syncthreads();
    double Tsum = 0.0, Rsum = 0.0;               // warp 0: the reactions' parts of T_bar and rho_bar
    if (w == 0) {
      double m = 0.0;
#pragma unroll 4
      for (int i = 0; i < NW; ++i) {
        m += s.pM[i * 32 + lane];
        Tsum += s.pT[i * 32 + lane];
        Rsum += s.pR[i * 32 + lane];
      }
      s.sc->Mtot[lane] = m;
    }
    __syncthreads();
    // adjoints of the activities and of [M], per owned species
    double Tb = 0.0, rb = 0.0;
    {
      const char *Db = (const char*)(s.Db + lane), *a = (const char*)(s.a + lane), *Mb = (const char*)(s.Mb + lane);
      auto at = [](const char* b, int o) { return *(const double*)(b + o); };
      const double Mt = s.sc->Mtot[lane];
      bad = false;
#pragma unroll 1
      for (int i = 0; i < KPO; ++i) {
        // species; ends of the lists: reactant and product factors with one other factor,
        // with two others, efficiencies
        const int4 h0 = __ldg((const int4*)t_vl + (w * KPO + i) * 2), h1 = __ldg((const int4*)t_vl + (w * KPO + i) * 2 + 1);
        const int k = h0.x;
        if (k < 0) break;
        double ab = 0.0, sc = 0.0;
        int j = h0.y;
#pragma unroll 4
        for (; j < h0.z; ++j) {
          const int2 e = __ldg((const int2*)t_v1 + j);
          ab = fma(at(Db, e.x), at(a, e.y), ab);
        }
#pragma unroll 4
        for (; j < h0.w; ++j) {
          const int2 e = __ldg((const int2*)t_v1 + j);
          ab = fma(-at(Db, e.x), at(a, e.y), ab);
        }
        for (j = h1.x; j < h1.y; ++j) {
          const int4 e = __ldg((const int4*)t_v2 + j);       // w: 0 reactant, 1 product
          const double q = at(Db, e.x) * at(a, e.y);
          ab = fma(e.w ? -q : q, at(a, e.z), ab);
        }
#pragma unroll 2
        for (j = h1.z; j < h1.w; ++j) {
          const int4 e = __ldg((const int4*)t_v3 + j);
          sc = fma(at(Mb, e.x), __hiloint2double(e.w, e.z), sc);
        }
        const double ta = ab * at(a, k * 256);
        Tb = fma(ta, s.Lp[k * 32 + lane], Tb);
        rb += ta;
        const double E = pfx::exp2_lg(s.lam[k * 32 + lane], s.exp2);
        const double y = fma(ab, E * rho, rho * fma(Mt, __ldg(t_iw + k), sc));
        bad |= !vjp_finite(y);
        if (p < n) g_Yb[k * n + p] = y;
      }
      if (bad) s.sc->bad[lane] = 1;
    }
    s.pT[w * 32 + lane] = Tb;
    s.pR[w * 32 + lane] = rb;
    __syncthreads();
    if (w == 0) {
      double r = 0.0;
#pragma unroll 4
      for (int i = 0; i < NW; ++i) {
        Tsum += s.pT[i * 32 + lane];
        r += s.pR[i * 32 + lane];
      }
      const double rhob = fma(r, pdm::rcp(rho), Rsum);
      const bool open = s.sc->bad[lane] != 0 || !vjp_finite(Tsum) || !vjp_finite(rhob);
      if (p < n) {
        g_Tb[p] = Tsum;
        g_rhob[p] = open ? __longlong_as_double(TILE_OPEN) : rhob;
      }
    }
    __syncthreads();
  }
}
