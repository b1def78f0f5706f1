// Dense Jacobian d(Tdot, omega)/d(T, Y) at fixed density for a tile of 32 states per block
// (lane = state, warps split species, reactions and rows), over the tables of pyro_tile.cuh.
//
// The per-thread kernel stored some 2,000 partial derivatives a state in global memory and
// spent 30 k FP64 instructions a state on 53 species.  Here a reaction leaves its rate
// constant kk (in shared memory), dR/dT, rho dR/d[M] and S' - S'' = sum (nu' - nu'') L' (in a
// per-block scratch that stays in L2); an entry is gathered where it is written,
//   J_ki = E_i rho sum_j +-kk_j (product of the other factors) + (u_k + ...)/W_i,
// one FP64 instruction a term, from an emitted stream of (row of kk, other factor) pairs per
// matrix row, and the temperature row from the same gather with kk_j scaled by the
// reaction's energy change -R T^2 (S'' - S').  Bound by the FP64 pipe (82 of its 84 %): 65,536
// states 5.44 -> 4.25 ms, up to 4,864 states (one tile an SM) 1.5-2.0 -> 0.39 ms.
// States outside the tables' range or with a non-finite entry get TILE_OPEN in their first
// output and are evaluated by the FP64 kernel.
#define TILE_DERIV
#define RATE_E 1023
#include "pyro_tile.cuh"

struct JacScalars {
  double T[32], invT[32], rho[32], ysum[32];
  Pair u[32], v[32], t[32];
  i64 lgT[32];
  int bad[32];
};

struct JacSmem {
  u64* exp2;
  i64* lam;             // [NSP + 1][32], as the next four: the species and a unit factor
  double *a, *E, *Lp, *c;        // activity, its derivative E rho, L', R(c_p/R - 1)
  double* kk;           // rows; first the partial sums of Y/W
  double* part;         // 6 x NW x 32 partial sums
  double *Rt, *Q, *M, *Mq;       // per block in global memory
  JacScalars* sc;
};

struct JacSums { double a, b, c, u; };

__device__ __forceinline__ bool jac_finite(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff; }

template <int NF, bool REV>
__device__ __forceinline__ void jac_plain(const JacSmem& s, int i0, int i1, Pair u, Pair v, double invT, double invT2,
                                          JacSums& sum, int lane) {
  const char* lam = (const char*)(s.lam + lane);
  const char *a = (const char*)(s.a + lane), *Lp = (const char*)(s.Lp + lane), *cp = (const char*)(s.c + lane);
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
    double q = (d(Lp, c1.z) + d(Lp, c1.w)) - (d(Lp, c2.y) + d(Lp, c2.z));
    double dc = (d(cp, c2.y) + d(cp, c2.z)) - (d(cp, c1.z) + d(cp, c1.w));
    double P = d(a, c1.z) * d(a, c1.w), Pr = 0.0;
    if (REV) Pr = d(a, c2.y) * d(a, c2.z);
    if (NF > 2) {
      X -= lg(c2.x);
      q += d(Lp, c2.x) - d(Lp, c2.w);
      dc += d(cp, c2.w) - d(cp, c2.x);
      P *= d(a, c2.x);
      if (REV) Pr *= d(a, c2.w);
    }
    const double kk = pfx::exp2_lg(X, s.exp2), D = P - Pr, R = kk * D;
    const double Rt = kk * fma(D, fma(bt.x, invT, bt.y * invT2), Pr * q);
    sum.a = fma(q, R, sum.a);
    sum.b = fma(q, Rt, sum.b);
    sum.c = fma(dc, R, sum.c);
    const int o = (c3.x >> 3) + lane;
    if (c3.y) {                                  // a duplicate of the row's reaction
      s.kk[o] += kk;
      s.Rt[o] += Rt;
    } else {
      s.kk[o] = kk;
      s.Rt[o] = Rt;
      s.Q[o] = q;
    }
  }
}

__device__ __forceinline__ void jac_other(const JacSmem& s, int i0, int i1, int lane, const double* __restrict__ Yp, i64 n,
                                          JacSums& sum) {
  const JacScalars& z = *s.sc;
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
    if (!(kind == TK_THREEBODY ? jac_finite(M) : tile_normal_pos(M))) s.sc->bad[lane] = 1;
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
    const double *a = s.a + lane, *Lp = s.Lp + lane, *cp = s.c + lane;
    double Pf = 1.0, Pr = rev ? 1.0 : 0.0, q = 0.0, dc = 0.0;
    for (int f = 0; f < nr; ++f) {
      const int k = (int)((fa >> (16 * f)) & 0xffff) * 32;
      X -= lam[k];
      q += Lp[k];
      dc -= cp[k];
      Pf *= a[k];
    }
    for (int f = 0; f < np; ++f) {
      const int k = (int)((f == 0 ? (fa >> 48) : (fb >> (16 * (f - 1)))) & 0xffff) * 32;
      q -= Lp[k];
      dc += cp[k];
      Pr *= a[k];
    }
    const double kt = pfx::exp2_lg(X & ~1ll, s.exp2), kk = kt * scale, D = Pf - Pr;
    // rho dR/d[M] (a third body's dkk/dM is kt)
    const double uj = rho * (kind == TK_THREEBODY ? kt * D : kk * D * sM * pdm::rcp(M));
    const double R = kk * D, Rt = kk * fma(D, tau, Pr * q);
    sum.a = fma(q, R, sum.a);
    sum.b = fma(q, Rt, sum.b);
    sum.c = fma(dc, R, sum.c);
    sum.u = fma(q, uj, sum.u);
    const int row = (int)((fb >> 32) & 0xffff) * 32 + lane, mr = (int)__ldg(r + 6) * 32 + lane;
    s.kk[row] = kk;
    s.Rt[row] = Rt;
    s.Q[row] = q;
    s.M[mr] = uj;
    s.Mq[mr] = uj * q;
  }
}

extern "C" __global__ void __launch_bounds__(32 * NW, TILE_MINB)
pyro_jacobian_tile(i64 n, const double* __restrict__ g_rho, const double* __restrict__ g_T, const double* __restrict__ g_Y,
                   double* __restrict__ g_J, double* __restrict__ g_scratch) {
  extern __shared__ __align__(16) char s_raw[];
  JacSmem s;
  s.exp2 = (u64*)s_raw;
  s.lam = (i64*)(s_raw + pfx::EXP2_TAB * 8);
  s.a = (double*)(s.lam + (NSP + 1) * 32);
  s.E = s.a + (NSP + 1) * 32;
  s.Lp = s.E + (NSP + 1) * 32;
  s.c = s.Lp + (NSP + 1) * 32;
  s.kk = s.c + (NSP + 1) * 32;
  s.part = s.kk + (TILE_ROWS + 1) * 32;
  s.sc = (JacScalars*)(s.part + 6 * NW * 32);
  s.Rt = g_scratch + (i64)blockIdx.x * (2 * TILE_ROWS + 2 * (T_MROWS + 1)) * 32;
  s.Q = s.Rt + TILE_ROWS * 32;
  s.M = s.Q + TILE_ROWS * 32;
  s.Mq = s.M + (T_MROWS + 1) * 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < pfx::EXP2_TAB; i += 32 * NW) s.exp2[i] = t_exp2[i];
  if (w == 0) {
    s.lam[NSP * 32 + lane] = 0;                  // the unit factor
    s.a[NSP * 32 + lane] = 1.0;
    s.Lp[NSP * 32 + lane] = 0.0;
    s.c[NSP * 32 + lane] = 0.0;
  }
  const i64 tiles = (n + 31) >> 5;
#pragma unroll 1
  for (i64 tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const i64 p = tile * 32 + lane, pc = p < n ? p : n - 1;
    // a tile without any state in the tables (a cold block): no work beside the FP64 kernel's
    const double T_in = __ldg(g_T + pc);
    if (!__any_sync(0xffffffffu, T_in > T_LO && T_in < T_HI)) {
      if (w == 0 && p < n) g_J[p] = __longlong_as_double(TILE_OPEN);
      continue;
    }
    const double* Yp = g_Y + pc;
    bool bad = false;
    {
      double y[KPW], ys = 0.0;
#pragma unroll
      for (int i = 0; i < KPW; ++i) y[i] = w + i * NW < NSP ? __ldg(Yp + (w + i * NW) * n) : 0.0;
#pragma unroll
      for (int i = 0; i < KPW; ++i) {
        const int k = w + i * NW;
        if (k < NSP) {
          ys = fma(y[i], __ldg(t_iw + k), ys);
          s.a[k * 32 + lane] = y[i];             // until the species phase
          bad |= !jac_finite(y[i]);
        }
      }
      s.part[w * 32 + lane] = ys;
    }
    if (w == 0) {
      const double T = T_in, rho = __ldg(g_rho + pc);
      const unsigned re = ((unsigned)__double2hiint(rho) >> 20) & 0x7ff;
      const bool in = T > T_LO && T < T_HI && re >= 1023 - 60 && re <= 1023 + 20 && rho > 0.0;
      const double Ts = in ? T : 1000.0;
      JacScalars& z = *s.sc;
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
      for (int i = 0; i < NW; ++i) a += s.part[i * 32 + lane];
      s.sc->ysum[lane] = a;
    }
    const Pair u = s.sc->u[lane], v = s.sc->v[lane];
    const double T = s.sc->T[lane], invT = s.sc->invT[lane], rho = s.sc->rho[lane];
    double cv = 0.0, dcv = 0.0;                  // c_v and dc_v/dT, this warp's species
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
        // h/(RT) = h0 + h1 T + ... + h5/T; c_p/R = h0 + 2 h1 T + 3 h2 T^2 + ...
        const double h0 = __ldg(h), h1 = __ldg(h + 1), h2 = __ldg(h + 2), h3 = __ldg(h + 3), h4 = __ldg(h + 4);
        double hr = fma(T, fma(T, fma(T, fma(T, h4, h3), h2), h1), h0);
        hr = fma(__ldg(h + 5), invT, hr);
        const double* g = t_cp + (k * 2 + hi) * 10;
        const double cp = fma(T, fma(T, fma(T, fma(T, __ldg(g + 4), __ldg(g + 3)), __ldg(g + 2)), __ldg(g + 1)), __ldg(g));
        const double dcp = fma(T, fma(T, fma(T, __ldg(g + 8), __ldg(g + 7)), __ldg(g + 6)), __ldg(g + 5));
        const double y = s.a[k * 32 + lane], E = pfx::exp2_lg(q, s.exp2) * rho;
        const double ci = fma(cp, T_R, -T_R), yw = y * __ldg(t_iw + k);
        cv = fma(yw, ci, cv);
        dcv = fma(yw * T_R, dcp, dcv);
        s.lam[k * 32 + lane] = q;
        s.E[k * 32 + lane] = E;
        s.a[k * 32 + lane] = E * y;
        s.Lp[k * 32 + lane] = fma(-hr, invT, invT);
        s.c[k * 32 + lane] = ci;
      }
      if (bad) s.sc->bad[lane] = 1;
    }
    __syncthreads();
    {
      const double invT2 = invT * invT;
      JacSums sum;
      sum.a = sum.b = sum.c = sum.u = 0.0;
      const int* seg = t_seg + w * (NCLS + 1);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        if ((w & 1) == half) {
          TILE_PLAIN
        } else {
          const int a = __ldg(seg + NCLS - 1), b = __ldg(seg + NCLS);
          if (a < b) jac_other(s, a, b, lane, Yp, n, sum);
        }
      }
      double* o = s.part + w * 32 + lane;
      o[0] = sum.a;
      o[NW * 32] = sum.b;
      o[2 * NW * 32] = sum.c;
      o[3 * NW * 32] = sum.u;
      o[4 * NW * 32] = cv;
      o[5 * NW * 32] = dcv;
    }
    __syncthreads();
    // rows of the species: column T, then the columns of the mass fractions
    const char *kk = (const char*)(s.kk + lane), *a = (const char*)(s.a + lane), *Mr = (const char*)(s.M + lane);
    auto at = [](const char* b, int o) { return *(const double*)(b + o); };
    // sign by the lowest bit of x, on the integer pipe
    auto flip = [](double q, int x) { return __hiloint2double(__double2hiint(q) ^ (x << 31), __double2loint(q)); };
    // A row's stream of terms, column after column: x is a row offset with flags in its low
    // bits (1: minus, 2: two other factors, 4: an [M] term with the coefficient of index y, 8:
    // the column's last term, 16: none, a column without terms), y the other factors.  Two
    // terms a load, the next two loads in flight: read term by term the stream's latency
    // from L2 bounds the kernel (6.0 ms per
    // 65,536 states).  sink(column, sum, [M] sum)
    auto row = [&](int b0, int cols, int step, const char* M, double u0, auto sink) {
      const int4* e = (const int4*)t_jx + b0;
      int4 x0 = __ldg(e), x1 = __ldg(e + 1), x2 = __ldg(e + 2);
      double acc = 0.0, cr = u0;
      int c = 0;
      auto term = [&](int x, int y) {
        if (!(x & 20)) {
          double q = at(kk, x & ~255);
          if (x & 2) q *= at(a, (y >> 16) << 8);
          q = flip(q, x);
          acc = fma(q, at(a, (y & 0xffff) << 8), acc);
        } else if (x & 4) {
          cr = fma(at(M, x & ~255), __ldg(t_jc + y), cr);
        }
        if (x & 8) {
          sink(c, acc, cr, !(x & 16));           // (uniform: the column has terms)
          c += step;
          acc = 0.0;
          cr = u0;
        }
      };
#pragma unroll 1
      while (c < cols) {
        const int4 x = x0;
        x0 = x1;
        x1 = x2;
        x2 = __ldg(e + 3);
        ++e;
        term(x.x, x.y);
        term(x.z, x.w);
      }
    };
    bad = false;
    const i64 stride = n;
#pragma unroll 1
    for (int i = 0; i < KPO; ++i) {
      const int k = __ldg(t_jk + w * KPO + i);
      if (k < 0) break;
      double jt = 0.0, uk = 0.0;
      const int4 l = __ldg((const int4*)t_jl + k);           // terms of column T and of u_k: row offset, 1: minus (|nu| times)
#pragma unroll 4
      for (int j = l.x; j < l.y; ++j) {
        const int e = __ldg(t_jt + j);
        jt += flip(at((const char*)(s.Rt + lane), e & ~255), e);
      }
      for (int j = l.z; j < l.w; ++j) {
        const int e = __ldg(t_jt + j);
        uk += flip(at(Mr, e & ~255), e);
      }
      double* Jr = g_J + (i64)(k + 1) * (NSP + 1) * stride + p;
      bad |= !jac_finite(jt);
      if (p < n) *Jr = jt;
      row(__ldg(t_je + k), NSP, 1, Mr, uk, [&](int c, double acc, double cr, bool some) {
        Jr += stride;
        double x = cr * __ldg(t_iw + c);
        if (some) x = fma(acc, at((const char*)(s.E + lane), c << 8), x);
        bad |= !jac_finite(x);
        if (p < n) *Jr = x;
      });
    }
    if (bad) s.sc->bad[lane] = 1;
    __syncthreads();
    // temperature row: kk_j q_j in place of kk_j, and the sums over the warps
    for (int j = w; j < T_NROWS; j += NW) s.kk[j * 32 + lane] *= s.Q[j * 32 + lane];
    for (int q = w; q < 6; q += NW) {
      double x = 0.0;
      for (int i = 0; i < NW; ++i) x += s.part[(q * NW + i) * 32 + lane];
      s.part[(q * NW) * 32 + lane] = x;
    }
    __syncthreads();
    const double e = T_R * T * T, A = s.part[lane], B = s.part[NW * 32 + lane], Cs = s.part[2 * NW * 32 + lane];
    const double U = s.part[3 * NW * 32 + lane], cvs = s.part[4 * NW * 32 + lane], dcvs = s.part[5 * NW * 32 + lane];
    const double rcv = pdm::rcp(cvs), f = -rcv * pdm::rcp(rho), Td = f * (e * A);
    bad = false;
    // columns w, w + NW, ... (each warp's stream holds its columns)
    row(__ldg(t_je + NSP + w), w < NSP ? (NSP - w + NW - 1) / NW * NW : 0, NW, (const char*)(s.Mq + lane), U,
        [&](int c0, double acc, double cr, bool) {
          const int c = c0 + w;
          const double iw = __ldg(t_iw + c);
          const double x = f * (e * fma(acc, s.E[c * 32 + lane], cr * iw)) - Td * (rcv * (s.c[c * 32 + lane] * iw));
          bad |= !jac_finite(x);
          if (p < n) g_J[(i64)(c + 1) * stride + p] = x;
        });
    if (bad) s.sc->bad[lane] = 1;
    __syncthreads();
    if (w == 0) {
      const double x = f * fma(e, B, Cs) - Td * (dcvs * rcv);
      const bool open = s.sc->bad[lane] != 0 || !jac_finite(x);
      if (p < n) g_J[p] = open ? __longlong_as_double(TILE_OPEN) : x;
    }
    __syncthreads();
  }
}
