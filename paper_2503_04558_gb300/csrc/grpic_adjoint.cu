// grpic_adjoint.cu -- the differentiable form: a hand-written adjoint of the
// FP64 time step (push + deposit + field update, arXiv:2503.04558 Sec. 2) for
// the time-averaged radial Poynting flux through the horizon ring,
//   L = (1/N) sum_n sum_j (E_th H_ph - E_ph H_th)(i_H, j+1/2) dtheta,
// with respect to the initial particle state and the initial fields.
//
// Reverse sweep per step n (state S_n = particles, F_n = D, B):
//   * seed   lambda_F^{n+1} += dL/dF^{n+1}  (through the auxiliary fields);
//   * fields the field update is linear in (F^n, J): its transpose runs the
//            predictor-corrector stages backwards with the transposed circulation
//            and auxiliary-field stencils, each point gathering what its readers
//            hand back (two launches a stage, no atomics), the boundary copies
//            transposed into their source cells;
//   * particles for every particle: the transpose of the deposit (derivatives of
//            the piecewise-linear CIC weights), the axis reflection, the geodesic
//            step (the predictor and correctors as run, transposed one by one,
//            or the implicit-function theorem at the converged trapezoid,
//            (I - dt/2 dF/dy)^T w = lambda, a 5x5 solve), the Boris step and the
//            interpolation (scatter of lambda_E into lambda_F).  Vector-Jacobian
//            products of the right-hand side and of the Boris step are reverse
//            passes written out through the push's point quantities; the window's
//            transpose interpolates the adjoint currents.  Forward-mode dual
//            numbers through the metric code give the full Jacobian that the
//            implicit-function form needs.
//            Bound by the FP64 pipe (88 % busy; 1120 of its instructions a
//            particle; 4.24 ms for 2e6 particles, 9.5 ms with dual numbers and
//            row-by-row window contractions; the early correctors' transposes in
//            double-FP32 pairs: slower, 8 warps per SM do not hide their chains).
// Recompute checkpoints every `checkpoint_every` steps bound the memory; the
// segment's recompute runs the FP64 push in its recording form, so the
// particle adjoint reads the Boris output and the corrector iterates (with
// sin, cos of theta) instead of running the push again.
#include "grpic_geo.cuh"

#include <cstring>
#include <new>
#include <vector>

namespace grpic {

// ---- forward-mode dual numbers ---------------------------------------------
template <int N>
struct DN {
    double v;
    double d[N];
    __device__ DN() {}
    __device__ DN(double x) : v(x)
    {
#pragma unroll
        for (int k = 0; k < N; ++k) d[k] = 0.0;
    }
};
template <int N>
__device__ __forceinline__ DN<N> operator+(const DN<N> &a, const DN<N> &b)
{
    DN<N> r;
    r.v = a.v + b.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k] + b.d[k];
    return r;
}
template <int N>
__device__ __forceinline__ DN<N> operator-(const DN<N> &a, const DN<N> &b)
{
    DN<N> r;
    r.v = a.v - b.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k] - b.d[k];
    return r;
}
template <int N>
__device__ __forceinline__ DN<N> operator-(const DN<N> &a)
{
    DN<N> r;
    r.v = -a.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = -a.d[k];
    return r;
}
template <int N>
__device__ __forceinline__ DN<N> operator*(const DN<N> &a, const DN<N> &b)
{
    DN<N> r;
    r.v = a.v * b.v;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k] * b.v + a.v * b.d[k];
    return r;
}
template <int N>
__device__ __forceinline__ DN<N> operator/(const DN<N> &a, const DN<N> &b)
{
    DN<N> r;
    double ib = rcp_t(b.v);
    r.v = a.v * ib;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = (a.d[k] - r.v * b.d[k]) * ib;
    return r;
}
template <int N>
__device__ __forceinline__ DN<N> rcp_t(const DN<N> &a)
{
    DN<N> r;
    r.v = rcp_t(a.v);
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = -a.d[k] * r.v * r.v;
    return r;
}
template <int N>
__device__ __forceinline__ DN<N> sqrt_t(const DN<N> &a)
{
    DN<N> r;
    r.v = sqrt_t(a.v);
    double h = a.v > 0.0 ? 0.5 * rcp_t(r.v) : 0.0;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = a.d[k] * h;
    return r;
}
template <int N>
__device__ __forceinline__ void sincos_t(const DN<N> &a, DN<N> *s, DN<N> *c)
{
    double sv, cv;
    sincos(a.v, &sv, &cv);
    s->v = sv;
    c->v = cv;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        s->d[k] = cv * a.d[k];
        c->d[k] = -sv * a.d[k];
    }
}

namespace {

// ---- the particle's local maps ---------------------------------------------
// right-hand side of Eq. particle-eom (no Lorentz force) at y = (r, th, ur, ut, up)
template <typename T>
__device__ __forceinline__ void rhs_y(double a, double eps, const T y[5], T f[6])
{
    T s, c;
    sincos_t(y[1], &s, &c);
    KSGeo<T> m;
    ks_geo_sc<T>(T(a), y[0], s, c, m);
    RhsT<T> o;
    geo_rhs_m<T, T>(m, T(eps), y[2], y[3], y[4], o);
    f[0] = o.xr;
    f[1] = o.xt;
    f[2] = o.xp;
    f[3] = o.ur;
    f[4] = o.ut;
    f[5] = T(0.0);
}

// F = (X^r, X^th, U_r, U_th, U_ph) and X^ph at y, with dF/dy and dX^ph/dy
__device__ void rhs_jac(double a, double eps, const double y[5], double F[5], double J[5][5], double &Fp,
                        double dFp[5])
{
    DN<5> yd[5], f[6];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        yd[k] = DN<5>(y[k]);
        yd[k].d[k] = 1.0;
    }
    rhs_y<DN<5>>(a, eps, yd, f);
    const int map[5] = {0, 1, 3, 4, 5};
    for (int r = 0; r < 5; ++r) {
        F[r] = f[map[r]].v;
        for (int k = 0; k < 5; ++k) J[r][k] = f[map[r]].d[k];
    }
    Fp = f[2].v;
    for (int k = 0; k < 5; ++k) dFp[k] = f[2].d[k];
}

// Adjoints of the point quantities of pointT (rho^2's inverse, z, 1 + z, its
// inverse, beta, 1 / sin^2, a^2 + r^2, sin cos, E), collected by the reverse
// passes below, and their transpose into r, theta (and a through a^2).
struct PtAdj {
    double ir, z, o, io, be, is2, A, cs, E;
};
__device__ __forceinline__ void point_vjp(const PtT<double> &m, double a2, double m2a2, double r, double c2, PtAdj L,
                                          double Lrho2, double &Lr, double &Lth, double &La2)
{
    // E = -2 a^2 sin cos / rho^2
    const double e = m2a2 * L.E;
    L.cs = fma(e, m.ir, L.cs);
    L.ir = fma(e, m.cs, L.ir);
    // beta = z / (1 + z), 1 / (1 + z), z = 2 r / rho^2
    L.z = fma(L.be, m.iopz, L.z);
    L.io = fma(L.be, m.z, L.io);
    L.z += fma(-L.io, m.iopz * m.iopz, L.o);
    L.ir = fma(L.z, r + r, L.ir);
    // 1 / rho^2, rho^2 = r^2 + a^2 cos^2, a^2 + r^2
    const double R = fma(-L.ir, m.ir * m.ir, Lrho2);
    Lr = fma(r + r, R + L.A, (L.z + L.z) * m.ir);
    // d cos^2 = -2 sin cos, d (sin cos) = cos^2 - sin^2, d sin^-2 = -2 sin cos / sin^4
    const double k = m.cs * m.is2;
    Lth = fma(L.cs, c2 - m.s2, fma(m2a2 * m.cs, R, -(L.is2 + L.is2) * (k * m.is2)));
    La2 = fma(R, c2, fma(-2.0 * m.cs * m.ir, L.E, L.A));
}

// w^T dF/dy + wp dX^ph/dy at y = (r, th, u_r, u_th, u_ph) for F = (X^r, X^th,
// U_r, U_th, 0): the reverse pass through the right-hand side exactly as the push
// evaluates it (pointT and rhsT), about 165 FP64 operations.  (Through dual
// numbers in r and theta for thirteen metric quantities: about 350.)  out_a
// (ND = 3) receives the part through the spin.  sv, cv = sin, cos y[1].
template <int ND>
__device__ __forceinline__ void rhs_vjp_p(double a, double eps, const double y[5], double sv, double cv,
                                          const double w[5], double wp, double out[5], double *out_a = nullptr)
{
    double a2 = a * a, m2a2 = -2.0 * a2, r = y[0], ur = y[2], ut = y[3], up = y[4], aup = a * up;
    const PtT<double> m = pointT<double>(a2, m2a2, r, sv, cv);
    // forward (rhsT)
    double ur2 = ur * ur, p = m.is2 * up, p2 = p * up;
    double W = fma(m.ar2, ur, aup), P = fma(ur, W + aup, fma(ut, ut, p2));
    double I = m.ir * P, Q = fma(-m.beta, ur2, I + eps);
    double iu = rsqrt_fast(m.opz * Q), h = 0.5 * iu, ii = m.ir * iu;
    double T1 = m.iopz * ur, T2 = fma(h, ur, 1.0), T = fma(T1, T2, h * Q), K = m.iopz * T;
    double B2 = I - ur2, B4 = m.cs * m.is2;
    // reverse: U_r = K (2 / rho^2 - z^2) + h z B2, U_th = E (h I - K z) + ii B4 p2,
    // X^r = iu (ir W - beta u_r) - beta, X^th = ii u_th, X^ph = ii (a u_r + p)
    double Lr = w[2], Lt = w[3];
    double rK = Lr * K, tE = Lt * m.E, rh = Lr * h;
    PtAdj L;
    double LK = fma(Lr, fma(-m.z, m.z, m.ir + m.ir), -tE * m.z);
    L.z = fma(rh, B2, fma(-(m.z + m.z), rK, -tE * K));
    double Lh = fma(Lr * m.z, B2, tE * I);
    double rhz = rh * m.z;
    double LI = fma(tE, h, rhz);
    L.E = Lt * fma(h, I, -K * m.z);
    double tp2 = Lt * p2;
    double Lii = fma(tp2, B4, fma(w[1], ut, wp * fma(a, ur, p)));
    double b4 = tp2 * ii;
    L.cs = b4 * m.is2;
    L.is2 = b4 * m.cs;
    double Lp2 = Lt * ii * B4;
    double Lut = w[1] * ii;
    double pii = wp * ii;
    double V = w[0] * iu;
    double Liu = w[0] * fma(m.ir, W, -m.beta * ur);
    double Lw = V * m.ir;
    L.be = -fma(V, ur, w[0]);
    double Lur = fma(pii, a, fma(-V, m.beta, -2.0 * rhz * ur));
    // K = T / (1 + z), T = T1 T2 + h Q
    double LT = LK * m.iopz;
    L.io = fma(LK, T, LT * ur * T2);
    Lur = fma(LT, fma(T1, h, m.iopz * T2), Lur);
    Lh = fma(LT, fma(T1, ur, Q), Lh);
    double LQ = LT * h;
    // ii = ir iu, h = iu / 2, iu = ((1 + z) Q)^-1/2
    L.ir = fma(Lii, iu, fma(V, W, rK + rK));
    Liu = fma(Lii, m.ir, fma(0.5, Lh, Liu));
    double G = -h * iu * iu * Liu;
    L.o = G * Q;
    LQ = fma(G, m.opz, LQ);
    // Q = I - beta u_r^2 + eps, I = P / rho^2, P = u_r (W + a u_ph) + u_th^2 + p2
    LI += LQ;
    L.be = fma(-LQ, ur2, L.be);
    L.ir = fma(LI, P, L.ir);
    double LP = LI * m.ir;
    Lw = fma(LP, ur, Lw);
    Lur = fma(-2.0 * LQ * m.beta, ur, fma(LP, W + aup, Lur));
    Lur = fma(Lw, m.ar2, Lur);
    Lut = fma(LP + LP, ut, Lut);
    Lp2 += LP;
    L.A = Lw * ur;
    // p2 = p u_ph, p = u_ph / sin^2
    double Lp = fma(Lp2, up, pii);
    L.is2 = fma(Lp, up, L.is2);
    out[2] = Lur;
    out[3] = Lut;
    out[4] = fma(Lp2, p, fma(Lp, m.is2, a * fma(LP, ur, Lw)));
    double La2;
    point_vjp(m, a2, m2a2, r, cv * cv, L, 0.0, out[0], out[1], La2);
    if constexpr (ND > 2) *out_a += fma(2.0 * a, La2, fma(pii, ur, up * fma(LP, ur, Lw)));
}

// lo^T d(u')/dz for the generalized Boris step (Eqs. boris-plus-minus, u0bar,
// boris-scheme) u' = u'(z), z = (r, th, u_r, u_th, u_ph, D^r, D^th, D^ph, B^r,
// B^th, B^ph): its reverse pass written out by hand, the metric's through the
// point quantities; sn, cs = sin, cos of theta
template <int ND>
__device__ __forceinline__ void boris_vjp(double a, double qm, double dt, const double z[11], double sn, double cs,
                                          const double lo[3], double out[11], double *out_a = nullptr)
{
    // (not const: the host compiler front end folds chains of const doubles in
    // time exponential in their length)
    double a2 = a * a, m2a2 = -2.0 * a2, r = z[0];
    const PtT<double> m = pointT<double>(a2, m2a2, r, sn, cs);
    double alpha = lapse(m);
    double gz = fma(m.z * a2, m.s2, m.ar2);  // g_pp = sin^2 (a^2 + r^2 + z a^2 sin^2)
    double as2 = a * m.s2, sgo = m.rho2 * sn;
    double grr = m.opz, grp = -as2 * m.opz, gtt = m.rho2, gpp = m.s2 * gz;
    double irr = fma(m.ar2, m.ir, -m.beta), irp = a * m.ir, itt = m.ir, ipp = m.ir * m.is2;
    double oa = m.opz * alpha;               // sqrt(1 + z)
    double sg = sgo * oa;
    double u[3] = {z[2], z[3], z[4]}, D[3] = {z[5], z[6], z[7]}, B[3] = {z[8], z[9], z[10]};
    double c1 = 0.5 * qm * dt;
    // forward values
    double Dl[3] = {grr * D[0] + grp * D[2], gtt * D[1], grp * D[0] + gpp * D[2]};
    double h = c1 * alpha;
    double um[3] = {u[0] + h * Dl[0], u[1] + h * Dl[1], u[2] + h * Dl[2]};
    double v[3] = {irr * um[0] + irp * um[2], itt * um[1], irp * um[0] + ipp * um[2]};
    double S = 1.0 + um[0] * v[0] + um[1] * v[1] + um[2] * v[2];
    double irS = rsqrt_fast(S);
    double iu0b = alpha * irS;               // 1 / u0bar
    double kt = c1 * iu0b;
    double t[3] = {kt * B[0], kt * B[1], kt * B[2]};
    double Gt[3] = {grr * t[0] + grp * t[2], gtt * t[1], grp * t[0] + gpp * t[2]};
    double tt = t[0] * Gt[0] + t[1] * Gt[1] + t[2] * Gt[2];
    double i1tt = rcp_t(1.0 + tt);
    double ks = 2.0 * i1tt;
    double sv[3] = {ks * t[0], ks * t[1], ks * t[2]};
    double vt[3] = {v[1] * t[2] - v[2] * t[1], v[2] * t[0] - v[0] * t[2], v[0] * t[1] - v[1] * t[0]};
    double w[3] = {um[0] + sg * vt[0], um[1] + sg * vt[1], um[2] + sg * vt[2]};
    double x[3] = {irr * w[0] + irp * w[2], itt * w[1], irp * w[0] + ipp * w[2]};
    double C[3] = {x[1] * sv[2] - x[2] * sv[1], x[2] * sv[0] - x[0] * sv[2], x[0] * sv[1] - x[1] * sv[0]};
    // reverse: out_i = um_i + sg C_i + h Dl_i; the metric's adjoints
    double Lgrr, Lgrp, Lgtt, Lgpp, Lirr, Lirp, Litt, Lipp, Lsg, Lal;
    double Lum[3] = {lo[0], lo[1], lo[2]};
    double Lh = lo[0] * Dl[0] + lo[1] * Dl[1] + lo[2] * Dl[2];
    double LDl[3] = {lo[0] * h, lo[1] * h, lo[2] * h};
    Lsg = lo[0] * C[0] + lo[1] * C[1] + lo[2] * C[2];
    double LC[3] = {lo[0] * sg, lo[1] * sg, lo[2] * sg};
    // C = x cross s
    double Lx[3] = {sv[1] * LC[2] - sv[2] * LC[1], sv[2] * LC[0] - sv[0] * LC[2], sv[0] * LC[1] - sv[1] * LC[0]};
    double Ls[3] = {LC[1] * x[2] - LC[2] * x[1], LC[2] * x[0] - LC[0] * x[2], LC[0] * x[1] - LC[1] * x[0]};
    // x = Ginv w
    double Lw[3] = {irr * Lx[0] + irp * Lx[2], itt * Lx[1], irp * Lx[0] + ipp * Lx[2]};
    Lirr = Lx[0] * w[0];
    Lirp = Lx[0] * w[2] + Lx[2] * w[0];
    Litt = Lx[1] * w[1];
    Lipp = Lx[2] * w[2];
    // w = um + sg (v cross t)
    for (int i = 0; i < 3; ++i) Lum[i] += Lw[i];
    Lsg += Lw[0] * vt[0] + Lw[1] * vt[1] + Lw[2] * vt[2];
    double LD_[3] = {Lw[0] * sg, Lw[1] * sg, Lw[2] * sg};
    double Lv[3] = {t[1] * LD_[2] - t[2] * LD_[1], t[2] * LD_[0] - t[0] * LD_[2], t[0] * LD_[1] - t[1] * LD_[0]};
    double Lt[3] = {LD_[1] * v[2] - LD_[2] * v[1], LD_[2] * v[0] - LD_[0] * v[2], LD_[0] * v[1] - LD_[1] * v[0]};
    // s = ks t, ks = 2 / (1 + tt), tt = t^T G t
    double Lks = Ls[0] * t[0] + Ls[1] * t[1] + Ls[2] * t[2];
    for (int i = 0; i < 3; ++i) Lt[i] += ks * Ls[i];
    double Ltt = -Lks * 2.0 * i1tt * i1tt;
    for (int i = 0; i < 3; ++i) Lt[i] += 2.0 * Ltt * Gt[i];
    Lgrr = Ltt * t[0] * t[0];
    Lgrp = Ltt * 2.0 * t[0] * t[2];
    Lgtt = Ltt * t[1] * t[1];
    Lgpp = Ltt * t[2] * t[2];
    // t = kt B, kt = c1 alpha / sqrt(S)
    double Lkt = Lt[0] * B[0] + Lt[1] * B[1] + Lt[2] * B[2];
    double LB[3] = {kt * Lt[0], kt * Lt[1], kt * Lt[2]};
    Lal = Lkt * c1 * irS;
    double LS = -0.5 * Lkt * kt * irS * irS;
    // S = 1 + um . v, v = Ginv um
    for (int i = 0; i < 3; ++i) {
        Lum[i] += LS * v[i];
        Lv[i] += LS * um[i];
    }
    Lum[0] += irr * Lv[0] + irp * Lv[2];
    Lum[1] += itt * Lv[1];
    Lum[2] += irp * Lv[0] + ipp * Lv[2];
    Lirr += Lv[0] * um[0];
    Lirp += Lv[0] * um[2] + Lv[2] * um[0];
    Litt += Lv[1] * um[1];
    Lipp += Lv[2] * um[2];
    // um = u + h Dl, h = c1 alpha, Dl = G D
    for (int i = 0; i < 3; ++i) {
        Lh += Lum[i] * Dl[i];
        LDl[i] += h * Lum[i];
    }
    Lal += c1 * Lh;
    double LDv[3] = {grr * LDl[0] + grp * LDl[2], gtt * LDl[1], grp * LDl[0] + gpp * LDl[2]};
    Lgrr += LDl[0] * D[0];
    Lgrp += LDl[0] * D[2] + LDl[2] * D[0];
    Lgtt += LDl[1] * D[1];
    Lgpp += LDl[2] * D[2];
    // the metric from the point quantities: sqrt(gamma) = rho^2 sin sqrt(1 + z), alpha =
    // (1 + z)^-1/2, gamma_rph = -a sin^2 (1 + z), gamma_phph = sin^2 gz and the upper one
    PtAdj L;
    L.o = Lgrr - as2 * Lgrp + 0.5 * (Lsg * sgo * alpha - Lal * alpha * m.iopz);
    double Lgz = Lgpp * m.s2;
    L.A = Lgz + Lirr * m.ir;
    L.z = Lgz * a2 * m.s2;
    L.be = -Lirr;
    L.ir = Lirr * m.ar2 + Lirp * a + Litt + Lipp * m.is2;
    L.is2 = Lipp * m.ir;
    L.io = L.cs = L.E = 0.0;
    double Lrho2 = Lgtt + Lsg * sn * oa;
    double Ls2 = Lgpp * gz + Lgz * m.z * a2 - Lgrp * a * m.opz;  // through sin^2
    double La2;
    point_vjp(m, a2, m2a2, r, cs * cs, L, Lrho2, out[0], out[1], La2);
    out[1] += 2.0 * m.cs * Ls2 + Lsg * m.rho2 * oa * cs;
    if constexpr (ND > 2) *out_a += 2.0 * a * (La2 + Lgz * m.z * m.s2) + Lirp * m.ir - Lgrp * m.s2 * m.opz;
    for (int i = 0; i < 3; ++i) {
        out[2 + i] = Lum[i];
        out[5 + i] = LDv[i];
        out[8 + i] = LB[i];
    }
}

// small dense solve M x = b (n = 5), Gaussian elimination with partial pivoting
__device__ void solve5(double M[5][5], double b[5])
{
    for (int c = 0; c < 5; ++c) {
        int p = c;
        for (int r = c + 1; r < 5; ++r)
            if (fabs(M[r][c]) > fabs(M[p][c])) p = r;
        if (p != c) {
            for (int k = 0; k < 5; ++k) {
                double t = M[c][k];
                M[c][k] = M[p][k];
                M[p][k] = t;
            }
            double t = b[c];
            b[c] = b[p];
            b[p] = t;
        }
        double iv = 1.0 / M[c][c];
        for (int r = c + 1; r < 5; ++r) {
            double f = M[r][c] * iv;
            for (int k = c; k < 5; ++k) M[r][k] -= f * M[c][k];
            b[r] -= f * b[c];
        }
    }
    for (int c = 4; c >= 0; --c) {
        double s = b[c];
        for (int k = c + 1; k < 5; ++k) s -= M[c][k] * b[k];
        b[c] = s / M[c][c];
    }
}

// a component's bilinear stencil (as the push's gather): column and rows of the
// corners, offsets, mirror rows of an odd component
struct St {
    int c0, r0, r1;
    double f, gg;
    bool flip0, flip1;
};
// value and d/dx1, d/dx2 (logical) of the interpolant
__device__ __forceinline__ void gather_d(const double *F, int64_t ld, const St &S, double &v, double &d1, double &d2)
{
    const double *a = F + (size_t)S.r0 * ld + S.c0, *b = F + (size_t)S.r1 * ld + S.c0;
    double a0 = flip_sign(__ldg(a), S.flip0), b0 = flip_sign(__ldg(b), S.flip1);
    double da = flip_sign(__ldg(a + 1), S.flip0) - a0, db = flip_sign(__ldg(b + 1), S.flip1) - b0;
    double x = fma(S.f, da, a0);
    d2 = fma(S.f, db, b0) - x;
    v = fma(S.gg, d2, x);
    d1 = fma(S.gg, db - da, da);
}
__device__ __forceinline__ void scatter_w(double *L, int64_t ld, const St &S, double lam)
{
    double *a = L + (size_t)S.r0 * ld + S.c0, *b = L + (size_t)S.r1 * ld + S.c0;
    double hi = S.gg * lam, lo = lam - hi, fl = S.f * lo, fh = S.f * hi;
    atomicAdd(a, flip_sign(lo - fl, S.flip0));
    atomicAdd(a + 1, flip_sign(fl, S.flip0));
    atomicAdd(b, flip_sign(hi - fh, S.flip1));
    atomicAdd(b + 1, flip_sign(fh, S.flip1));
}

// two neighbouring values along one dimension: their interpolant and difference
struct Pair2 {
    double v, d;
};
__device__ __forceinline__ Pair2 pair_at(double a, double b, double f) { return {fma(f, b - a, a), b - a}; }

constexpr int MAX_ITER = 16;  // correctors the adjoint accepts

struct PAdjArgs {
    GridDev g;
    double dt;
    int n_iter;
    int ift;                  // 1: implicit-function theorem at the converged trapezoid
    double qm[4], qw[4];
    int massive[4];
    int64_t n;
    const double *x[5];       // state n: r, th, ur, ut, up
    const uint32_t *tag0;     // tags at n
    const uint32_t *tag1;     // tags at n+1
    const double *F[6];       // fields at n
    const double *tape;       // the forward push's record of step n (layout in grpic_internal.cuh)
    int64_t tape_ld;
    const double *lamJ[3];    // adjoint of J A
    const double *lam1[5];    // adjoint of state n+1
    double *lam0[5];          // adjoint of state n (output)
    double *lamF[6];          // adjoint of fields at n (accumulated)
    double *La;               // per particle: its part of dL/da (may be null)
    int64_t ld;
};

template <bool SPIN>
__global__ void __launch_bounds__(128) particle_adjoint(PAdjArgs A)
{
    constexpr int ND = SPIN ? 3 : 2;
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= A.n) return;
    const GridDev &g = A.g;
    double out[5] = {0, 0, 0, 0, 0};
    uint32_t t0 = A.tag0[p];
    if (SPIN) A.La[p] = 0.0;
    if (t0 & DEAD) {
        for (int k = 0; k < 5; ++k) A.lam0[k][p] = 0.0;
        return;
    }
    const int sp = t0 & 3u;
    const bool massive = A.massive[sp] != 0, charged = massive && A.qm[sp] != 0.0;
    double r = A.x[0][p], th = A.x[1][p];
    double u[3] = {A.x[2][p], A.x[3][p], A.x[4][p]};
    // a state the push refused (outside the domain, non-finite) moved nothing
    bool inside = finite64(r) && finite64(th) && finite64(u[0]) && finite64(u[1]) && finite64(u[2]) && r >= g.r_in &&
                  r < g.r_out && th >= 0.0 && th <= M_PI;
    if (!inside) {
        for (int k = 0; k < 5; ++k) A.lam0[k][p] = 0.0;
        return;
    }
    const ColPos ca = r_column_in(g, r);  // as in the push
    const double x2a = theta_cells(g, th);
    const double dt = A.dt, eps = massive ? 1.0 : 0.0;
    // the forward push's record: u' after the Boris step, the corrector
    // iterates, x^{n+1} before the reflection
    const double *T = A.tape + p;
    const int64_t tl = A.tape_ld;
    const int N = A.n_iter, te = tape_end(N);
    const double y0[5] = {r, th, T[(TAPE_U + 0) * tl], T[(TAPE_U + 1) * tl], T[(TAPE_U + 2) * tl]};
    const double s0 = T[TAPE_SC0 * tl], c0 = T[(TAPE_SC0 + 1) * tl];
    const double y1[5] = {T[te * tl], T[(te + 1) * tl], T[(te + 2) * tl], T[(te + 3) * tl], y0[4]};
    const double dphi = T[(te + 4) * tl];
    double refl = 1.0;
    double th1 = y1[1];
    if (th1 < 0.0) { th1 = -th1; refl = -1.0; }
    else if (th1 > M_PI) { th1 = 2.0 * M_PI - th1; refl = -1.0; }
    const ColPos cb = r_column(g, y1[0]);
    const double x2b = theta_cells(g, th1);
    const int i0 = ca.i, j0 = row_of(g, x2a), j1 = row_of(g, x2b);
    const int di = cb.i - i0, dj = j1 - j0;
    // offsets of the start and end points in their cells
    const double fa1 = ca.f, fa2 = x2a - j0, fb1 = cb.f, fb2 = x2b - j1;
    // the push's own checks: a finite end point, at most one cell away
    bool moved_ok = di >= -1 && di <= 1 && dj >= -1 && dj <= 1 && y1[0] > 0.0 && finite64(y1[0]) && finite64(x2b) &&
                    finite64(y1[2]) && finite64(y1[3]) && finite64(dphi);
    if (!moved_ok) {
        for (int k = 0; k < 5; ++k) A.lam0[k][p] = 0.0;
        return;
    }

    // ---- adjoint -------------------------------------------------------
    double l1[5] = {0, 0, 0, 0, 0};
    if (!(A.tag1[p] & DEAD))
        for (int k = 0; k < 5; ++k) l1[k] = A.lam1[k][p];
    double ldphi = 0.0, lx1a = 0.0, lx2a = 0.0, lx1b = 0.0, lx2b = 0.0;
    double qw = A.qw[sp];
    if (qw != 0.0) {
        // Transpose of the Esirkepov window.  The start's weights are (1 - f, f) at the
        // nodes of its cell (columns / rows 1, 2 of the window), the end's at those of
        // its own (di, dj cells on), so a current's window contracted with its adjoint L
        // is interpolation of L:
        //   J^r A_r at face k: cr P_r(k) (L interpolated in theta at the start + at the
        //   end), P_r nonzero at face 1 and, for a move in r, at the extra face, and
        //   P_r's derivatives -1 at the start's and the end's own face;
        //   J^theta A_theta likewise; J^phi dV: cp (I_11 / 3 + (I_10 + I_01) / 6 + I_00 / 3),
        //   I_pq bilinear with the end's (1) or start's (0) weights in r (p) and theta (q).
        // At a node itself (offset 0) the weights' derivative is taken as 0.
        double cr = -0.5 * qw / dt, cq = qw / dt, cp = cq * dphi;
        const size_t w0 = (size_t)j0 * A.ld + (i0 + NG);  // the start cell's node
        const size_t w1 = (size_t)j1 * A.ld + (i0 + di + NG);
        const int64_t ld = A.ld;
        {   // J^r: rows j0, j0 + 1 (start) and j1, j1 + 1 (end) at a face's column
            const double *L = A.lamJ[0];
            auto face = [&](int c, Pair2 &a, Pair2 &b) {
                const double *s0 = L + (w0 + c), *s1 = L + (w0 + (int64_t)dj * ld + c);
                a = pair_at(__ldg(s0), __ldg(s0 + ld), fa2);
                b = pair_at(__ldg(s1), __ldg(s1 + ld), fb2);
            };
            Pair2 a, b;
            face(0, a, b);
            double P = cr * (fa1 - (di == 0 ? fb1 : (di > 0 ? 1.0 : 0.0))), U = cr * (a.v + b.v);
            lx1a += U;
            lx2a += P * a.d;
            lx2b += P * b.d;
            if (di != 0) {
                face(di, a, b);
                P = cr * (di > 0 ? -fb1 : 1.0 - fb1);
                U = cr * (a.v + b.v);
                lx2a += P * a.d;
                lx2b += P * b.d;
            }
            lx1b -= U;
        }
        {   // J^theta: columns of the start and of the end at a theta face's row
            const double *L = A.lamJ[1];
            auto face = [&](int l, Pair2 &a, Pair2 &b) {
                const double *s0 = L + (w0 + (int64_t)l * ld), *s1 = s0 + di;
                a = pair_at(__ldg(s0), __ldg(s0 + 1), fa1);
                b = pair_at(__ldg(s1), __ldg(s1 + 1), fb1);
            };
            Pair2 a, b;
            face(0, a, b);
            double P = cr * (fa2 - (dj == 0 ? fb2 : (dj > 0 ? 1.0 : 0.0))), U = cr * (a.v + b.v);
            lx2a += U;
            lx1a += P * a.d;
            lx1b += P * b.d;
            if (dj != 0) {  // (the end's row j1: the extra face lies in the grid)
                face(dj, a, b);
                P = cr * (dj > 0 ? -fb2 : 1.0 - fb2);
                U = cr * (a.v + b.v);
                lx1a += P * a.d;
                lx1b += P * b.d;
            }
            lx2b -= U;
        }
        {   // J^phi: the four corner sets
            const double *L = A.lamJ[2];
            auto corners = [&](const double *q, double f1, double f2, double &I, double &I1, double &I2) {
                Pair2 a = pair_at(__ldg(q), __ldg(q + 1), f1), b = pair_at(__ldg(q + ld), __ldg(q + ld + 1), f1);
                I2 = b.v - a.v;
                I = fma(f2, I2, a.v);
                I1 = fma(f2, b.d - a.d, a.d);
            };
            double I00, R00, T00, I01, R01, T01, I10, R10, T10, I11, R11, T11;
            corners(L + w0, fa1, fa2, I00, R00, T00);
            corners(L + (w0 + (int64_t)dj * ld), fa1, fb2, I01, R01, T01);
            corners(L + (w0 + di), fb1, fa2, I10, R10, T10);
            corners(L + w1, fb1, fb2, I11, R11, T11);
            const double c3 = 1.0 / 3.0, c6 = 1.0 / 6.0;
            double p3 = cp * c3, p6 = cp * c6;
            ldphi += cq * fma(c3, I11 + I00, c6 * (I10 + I01));
            lx1a = fma(p3, R00, fma(p6, R01, lx1a));
            lx1b = fma(p3, R11, fma(p6, R10, lx1b));
            lx2a = fma(p3, T00, fma(p6, T10, lx2a));
            lx2b = fma(p3, T11, fma(p6, T01, lx2b));
        }
        if (zero64(fa1)) lx1a = 0.0;
        if (zero64(fa2)) lx2a = 0.0;
        if (zero64(fb1)) lx1b = 0.0;
        if (zero64(fb2)) lx2b = 0.0;
    }
    // end point: logical -> (r, theta) after reflection, then the reflection
    l1[0] = fma(lx1b, rcp_t(y1[0]) * g.idx1, l1[0]);
    l1[1] = fma(lx2b, g.idth, l1[1]);
    l1[1] *= refl;
    l1[3] *= refl;
    const double hh = 0.5 * dt;
    double l0[5];
    double la = 0.0;                       // dL/da through the metric of this push
    double *pla = &la;
    if (A.ift) {
        // the converged trapezoid y1 = y0 + dt/2 (F(y1) + F(y0)), dphi = dt/2
        // (X^ph(y1) + X^ph(y0)), by the implicit-function theorem:
        // (I - dt/2 dF/dy(y1))^T w = lambda_1, lambda_0 = (I + dt/2 dF/dy(y0))^T w
        double F1[5], J1[5][5], Fp1, dFp1[5];
        rhs_jac(g.a, eps, y1, F1, J1, Fp1, dFp1);
        for (int k = 0; k < 5; ++k) l1[k] += hh * ldphi * dFp1[k];
        double M[5][5];
        for (int a = 0; a < 5; ++a)
            for (int b = 0; b < 5; ++b) M[a][b] = (a == b ? 1.0 : 0.0) - hh * J1[b][a];  // transposed
        double w[5] = {l1[0], l1[1], l1[2], l1[3], l1[4]};
        solve5(M, w);
        double hw[5], v0[5];
        for (int k = 0; k < 5; ++k) hw[k] = hh * w[k];
        if constexpr (SPIN) {
            // the a-dependence of F(y1): w . dt/2 dF/da(y1) + dt/2 ldphi dX^ph/da(y1)
            double unused[5], s1, c1;
            sincos(y1[1], &s1, &c1);
            rhs_vjp_p<ND>(g.a, eps, y1, s1, c1, hw, hh * ldphi, unused, pla);
        }
        rhs_vjp_p<ND>(g.a, eps, y0, s0, c0, hw, hh * ldphi, v0, pla);
        for (int k = 0; k < 5; ++k) l0[k] = w[k] + v0[k];
    } else {
        // transpose of the iteration the push runs: y~_0 = y0 + dt F(y0),
        // y~_{k+1} = y0 + dt/2 (F(y~_k) + F(y0)), dphi = dt/2 (X^ph(y~_{N-1}) + X^ph(y0))
        double gk[5] = {l1[0], l1[1], l1[2], l1[3], l1[4]};
        double lF0[5] = {0, 0, 0, 0, 0}, ly0[5] = {0, 0, 0, 0, 0}, lFp0 = 0.0;
        if (N == 0) {
            lFp0 += dt * ldphi;
        } else {
            for (int it = N - 1; it >= 0; --it) {
                for (int k = 0; k < 5; ++k) {
                    ly0[k] += gk[k];
                    lF0[k] += hh * gk[k];
                }
                double ap = (it == N - 1) ? hh * ldphi : 0.0;
                lFp0 += ap;
                double hg[5], gn[5];
                for (int k = 0; k < 5; ++k) hg[k] = hh * gk[k];
                const double *q = T + (int64_t)(TAPE_IT + 6 * it) * tl;
                const double yi[5] = {q[0], q[tl], q[2 * tl], q[3 * tl], y0[4]};
                rhs_vjp_p<ND>(g.a, eps, yi, q[4 * tl], q[5 * tl], hg, ap, gn, pla);
                for (int k = 0; k < 5; ++k) gk[k] = gn[k];
            }
        }
        for (int k = 0; k < 5; ++k) {
            ly0[k] += gk[k];
            lF0[k] += dt * gk[k];
        }
        double v0[5];
        rhs_vjp_p<ND>(g.a, eps, y0, s0, c0, lF0, lFp0, v0, pla);
        for (int k = 0; k < 5; ++k) l0[k] = ly0[k] + v0[k];
    }
    // start point: deposit's start-weight derivatives
    const double ir1 = rcp_t(r) * g.idx1;  // d x1 / d r
    l0[0] = fma(lx1a, ir1, l0[0]);
    l0[1] = fma(lx2a, g.idth, l0[1]);
    // Boris: y0 = (r, th, u'(r, th, u, E))
    out[0] = l0[0];
    out[1] = l0[1];
    if (charged) {
        // fields at x^n and their logical derivatives
        St S[6];
        double E[6], dE1[6], dE2[6];
        int ih, jh;
        double fh, gh;
        half_node(i0, fa1, ih, fh);
        half_node(j0, fa2, jh, gh);
        const bool m0 = jh < 0, m1 = jh + 1 > g.nth - 1;  // rows mirrored at the axis
        const int h0 = m0 ? 0 : jh, h1 = m1 ? g.nth - 1 : jh + 1;
        S[0] = {ih + NG, j0, j0 + 1, fh, fa2, false, false};  // D^r
        S[1] = {i0 + NG, h0, h1, fa1, gh, m0, m1};            // D^th (odd across the axis)
        S[2] = {i0 + NG, j0, j0 + 1, fa1, fa2, false, false};  // D^ph
        S[3] = {i0 + NG, h0, h1, fa1, gh, false, false};      // B^r
        S[4] = S[0];                                          // B^th
        S[5] = {ih + NG, h0, h1, fh, gh, false, false};       // B^ph
        for (int c = 0; c < 6; ++c) gather_d(A.F[c], A.ld, S[c], E[c], dE1[c], dE2[c]);
        double zv[11] = {r, th, u[0], u[1], u[2], E[0], E[1], E[2], E[3], E[4], E[5]};
        double lb[11];
        boris_vjp<ND>(g.a, A.qm[sp], dt, zv, s0, c0, l0 + 2, lb, pla);
        out[0] += lb[0];
        out[1] += lb[1];
        for (int k = 0; k < 3; ++k) out[2 + k] = lb[2 + k];
        double lE[6];
        for (int c = 0; c < 6; ++c) lE[c] = lb[5 + c];
        double lx1 = 0.0, lx2 = 0.0;
        for (int c = 0; c < 6; ++c) {
            scatter_w(A.lamF[c], A.ld, S[c], lE[c]);
            lx1 += lE[c] * dE1[c];
            lx2 += lE[c] * dE2[c];
        }
        out[0] = fma(lx1, ir1, out[0]);
        out[1] = fma(lx2, g.idth, out[1]);
    } else {
        for (int k = 0; k < 3; ++k) out[2 + k] = l0[2 + k];
    }
    for (int k = 0; k < 5; ++k) A.lam0[k][p] = out[k];
    if (SPIN) A.La[p] = la;
}

// ---- field update transpose -------------------------------------------------
struct FAdj {
    int nr, nth;
    int64_t ld, ldt;
    size_t slab;
    const double *tab, *col1d;
};

__device__ __forceinline__ double tb(const FAdj &A, int slot, int i, int j)
{
    return A.tab[slot * A.slab + (size_t)j * A.ldt + (i + NG)];
}

// device pointers of up to six arrays, passed by value
struct P6 {
    double *p[6];
    __host__ __device__ double *operator[](int k) const { return p[k]; }
};

__device__ __forceinline__ bool phys(int comp, int i, int j, int nr, int nth)
{
    bool half_r = (comp == 0 || comp == 4 || comp == 5), half_t = (comp == 1 || comp == 3 || comp == 5);
    if (i < 0 || i > (half_r ? nr - 1 : nr)) return false;
    if (j > (half_t ? nth - 1 : nth)) return false;
    return true;
}

// The field update's transpose works on mu_k, the adjoint of stage k's value before
// its boundary copies.  A stage's mu gives the adjoints h of the auxiliary
// fields (transpose of the circulations), these the previous iterate's adjoint
// (transpose of the auxiliary fields), and the guard copies' transpose the
// previous mu: two launches a stage, every entry gathered by its own thread (the
// scatter with atomics took 8 launches and 12 clears).  The sums over the stages
// that the rest needs follow from M = sum_k mu_k and mu_0.

// mu (zero where a component is not updated) -> scale * h: H_r, H_th, H_ph, E_r,
// E_th, E_ph (transpose of Eqs. D-update, B-update), every column and row
__global__ void __launch_bounds__(256) stage_h(FAdj A, P6 mu, P6 h, double scale, double dth)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (c >= (int)A.ldt || j > A.nth) return;
    const int i = c - NG;
    const int inv[6] = {T_INV_ADR, T_INV_ADT, T_INV_ADP, T_INV_ABR, T_INV_ABT, T_INV_ABP};
    auto g = [&](int k, int ii, int jj) {
        if (ii < 0 || ii > A.nr || jj < 0 || jj > A.nth) return 0.0;
        return __ldg(mu[k] + (size_t)jj * A.ld + (ii + NG)) * tb(A, inv[k], ii, jj);
    };
    const double drp = A.col1d[c], drd = A.col1d[A.ldt + c];
    const size_t q = (size_t)j * A.ld + c;
    const double g1 = g(1, i, j), g2 = g(2, i, j), g5 = g(5, i, j);
    h[0][q] = scale * (g(2, i, j + 1) - g2) * drd;
    h[1][q] = scale * (g2 - g(2, i + 1, j)) * dth;
    h[2][q] = scale * ((j < A.nth ? g(0, i, j) : 0.0) - g(0, i, j + 1) + g(1, i + 1, j) - g1);
    h[3][q] = scale * (g(5, i, j - 1) - g5) * drp;
    h[4][q] = scale * (g5 - g(5, i - 1, j)) * dth;
    h[5][q] = scale * (g(3, i, j) - g(3, i, j - 1) + g(4, i - 1, j) - g(4, i, j));
}

// component k of the iterate's adjoint at (column c, row j) from h (transpose of
// Eqs. auxH, auxE); zero beyond the columns
__device__ __forceinline__ double from_h(const FAdj &A, const P6 &h, int k, int c, int j)
{
    if (c < 0 || c >= (int)A.ldt) return 0.0;
    const int i = c - NG;
    const size_t q = (size_t)j * A.ld + c;
    const bool l = c > 0, r = c + 1 < (int)A.ldt;
    auto pair = [&](int n, bool right) {
        const double *x = h[n] + q;
        return __ldg(x) + (right ? (r ? __ldg(x + 1) : 0.0) : (l ? __ldg(x - 1) : 0.0));
    };
    switch (k) {
    case 0: return tb(A, T_AGRR_DR, i, j) * __ldg(h[3] + q) + 0.5 * tb(A, T_AGRP_DR, i, j) * pair(5, true);
    case 1: return tb(A, T_AGTT_DT, i, j) * __ldg(h[4] + q) - 0.5 * tb(A, T_SGB_DT, i, j) * pair(2, false);
    case 2:
        return tb(A, T_AGPP_DP, i, j) * __ldg(h[5] + q) + 0.5 * (tb(A, T_SGB_DP, i, j) * pair(1, false) +
                                                                  tb(A, T_AGRP_DP, i, j) * pair(3, false));
    case 3: return tb(A, T_AGRR_BR, i, j) * __ldg(h[0] + q) + 0.5 * tb(A, T_AGRP_BR, i, j) * pair(2, false);
    case 4: return tb(A, T_AGTT_BT, i, j) * __ldg(h[1] + q) + 0.5 * tb(A, T_SGB_BT, i, j) * pair(5, true);
    default:
        return tb(A, T_AGPP_BP, i, j) * __ldg(h[2] + q) + 0.5 * (tb(A, T_AGRP_BP, i, j) * pair(0, true) -
                                                                  tb(A, T_SGB_BP, i, j) * pair(4, true));
    }
}

// the boundary copies' transpose of X(column): the physical columns' values plus
// those of their guard copies, zero in the guards and on the axis (D^ph, B^th)
template <typename XF>
__device__ __forceinline__ void put_mu(const FAdj &A, int k, int i, int j, const XF &X, double damp, P6 mu, P6 M,
                                       bool add)
{
    const bool hr = (k == 0 || k == 4 || k == 5);
    const size_t row = (size_t)j * A.ld;
    double v = 0.0;
    if (phys(k, i, j, A.nr, A.nth) && !((k == 2 || k == 4) && (j == 0 || j == A.nth))) {
        const int last = hr ? A.nr - 1 : A.nr;
        v = X(i + NG);
        if (i == 0) v += X(0) + X(1);
        if (i == last)
            for (int c = last + 1 + NG; c < A.nr + 2 * NG; ++c) v += X(c);
        v *= damp;
    }
    const size_t q = row + i + NG;
    mu[k][q] = v;
    M[k][q] = add ? M[k][q] + v : v;
    for (int c = 0; c < NG && i == 0; ++c) mu[k][row + c] = M[k][row + c] = 0.0;
    for (int c = A.nr + 1 + NG; c < A.nr + 2 * NG && i == A.nr; ++c) mu[k][row + c] = M[k][row + c] = 0.0;
}

// mu, M <- the projection's transpose of lam (the last stage's, damped)
__global__ void __launch_bounds__(256) stage_first(FAdj A, P6 lam, P6 mu, P6 M, int damp)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i > A.nr || j > A.nth) return;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double *L = lam[k] + (size_t)j * A.ld;
        const double f = damp ? A.col1d[((k == 0 || k == 4 || k == 5) ? 3 : 2) * A.ldt + i + NG] : 1.0;
        put_mu(A, k, i, j, [&](int c) { return __ldg(L + c); }, f, mu, M, false);
    }
}

// mu <- the previous stage's from h; M += mu
__global__ void __launch_bounds__(256) stage_mu(FAdj A, P6 h, P6 mu, P6 M)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i > A.nr || j > A.nth) return;
#pragma unroll
    for (int k = 0; k < 6; ++k)
        put_mu(A, k, i, j, [&](int c) { return from_h(A, h, k, c, j); }, 1.0, mu, M, true);
}

// after the stages: lam_out <- M (the identity for entries that an update never
// writes: rows past the last half-theta row, columns past the last guard),
// lam_J <- -dt M / A, mu <- dt (alpha_s (M - mu_0) + mu_0) = the adjoint of C(X^n)
__global__ void __launch_bounds__(256) stages_close(FAdj A, P6 lam, P6 mu, P6 M, P6 out, P6 lamJ, double dt, double as)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (c >= A.ld || j > A.nth) return;
    const int i = c - NG, inv[3] = {T_INV_ADR, T_INV_ADT, T_INV_ADP};
    const size_t q = (size_t)j * A.ld + c;
    const bool in = c < (int)A.ldt;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const bool ht = (k == 1 || k == 3 || k == 5);
        const bool written = in && j <= (ht ? A.nth - 1 : A.nth);
        const double m = in ? M[k][q] : 0.0;
        out[k][q] = written ? m : lam[k][q];
        if (in) {
            const double m0 = mu[k][q];
            mu[k][q] = dt * (as * (m - m0) + m0);
        }
        if (k < 3) lamJ[k][q] = in && i >= 0 && i <= A.nr ? -dt * m * tb(A, inv[k], i, j) : 0.0;
    }
}

// out += the iterate's adjoint from h, entry by entry
__global__ void __launch_bounds__(256) add_from_h(FAdj A, P6 h, P6 out)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    if (c >= (int)A.ldt || j > A.nth) return;
#pragma unroll
    for (int k = 0; k < 6; ++k) out[k][(size_t)j * A.ld + c] += from_h(A, h, k, c, j);
}

// ---- objective ------------------------------------------------------------
__device__ __forceinline__ double fx(const double *F, int64_t ld, int i, int j) { return F[(size_t)j * ld + i + NG]; }

// auxiliary fields needed at the ring (same formulas as the field update)
struct Ring {
    double Eth, Hph, Eph, Hth;
};
__device__ Ring ring_vals(FAdj A, P6 F, int iH, int j)
{
    auto Hph = [&](int i, int jj) {
        return tb(A, T_AGPP_BP, i, jj) * fx(F[5], A.ld, i, jj) +
               0.5 * (tb(A, T_AGRP_BR, i, jj) * fx(F[3], A.ld, i, jj) + tb(A, T_AGRP_BR, i + 1, jj) * fx(F[3], A.ld, i + 1, jj)) -
               0.5 * (tb(A, T_SGB_DT, i, jj) * fx(F[1], A.ld, i, jj) + tb(A, T_SGB_DT, i + 1, jj) * fx(F[1], A.ld, i + 1, jj));
    };
    auto Hth = [&](int i, int jj) {
        return tb(A, T_AGTT_BT, i, jj) * fx(F[4], A.ld, i, jj) +
               0.5 * (tb(A, T_SGB_DP, i, jj) * fx(F[2], A.ld, i, jj) + tb(A, T_SGB_DP, i + 1, jj) * fx(F[2], A.ld, i + 1, jj));
    };
    auto Eth = [&](int i, int jj) {
        return tb(A, T_AGTT_DT, i, jj) * fx(F[1], A.ld, i, jj) -
               0.5 * (tb(A, T_SGB_BP, i, jj) * fx(F[5], A.ld, i, jj) + tb(A, T_SGB_BP, i - 1, jj) * fx(F[5], A.ld, i - 1, jj));
    };
    auto Eph = [&](int i, int jj) {
        return tb(A, T_AGPP_DP, i, jj) * fx(F[2], A.ld, i, jj) +
               0.5 * (tb(A, T_AGRP_DR, i, jj) * fx(F[0], A.ld, i, jj) + tb(A, T_AGRP_DR, i - 1, jj) * fx(F[0], A.ld, i - 1, jj)) +
               0.5 * (tb(A, T_SGB_BT, i, jj) * fx(F[4], A.ld, i, jj) + tb(A, T_SGB_BT, i - 1, jj) * fx(F[4], A.ld, i - 1, jj));
    };
    Ring R;
    R.Eth = Eth(iH, j);
    R.Hph = 0.5 * (Hph(iH - 1, j) + Hph(iH, j));
    R.Eph = 0.5 * (Eph(iH, j) + Eph(iH, j + 1));
    R.Hth = 0.25 * (Hth(iH - 1, j) + Hth(iH, j) + Hth(iH - 1, j + 1) + Hth(iH, j + 1));
    return R;
}

// flux at the ring (one block reduction) accumulated into *out with weight w
__global__ void flux_kernel(FAdj A, P6 F, int iH, double dth, double w, double *out)
{
    __shared__ double red[256];
    double s = 0.0;
    for (int j = threadIdx.x; j < A.nth; j += blockDim.x) {
        Ring R = ring_vals(A, F, iH, j);
        s += (R.Eth * R.Hph - R.Eph * R.Hth) * dth;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out += w * red[0];
}

// seed: aux adjoints of w * flux (then aux_T maps them to the fields)
__global__ void flux_seed(FAdj A, P6 F, int iH, double dth, double w, P6 lamA)
{
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= A.nth) return;
    Ring R = ring_vals(A, F, iH, j);
    double c = w * dth;
    auto at = [&](int comp, int i, int jj, double v) { atomicAdd(lamA[comp] + (size_t)jj * A.ld + i + NG, v); };
    // aux order: 0 H_r, 1 H_th, 2 H_ph, 3 E_r, 4 E_th, 5 E_ph
    at(4, iH, j, c * R.Hph);
    at(2, iH - 1, j, 0.5 * c * R.Eth);
    at(2, iH, j, 0.5 * c * R.Eth);
    at(5, iH, j, -0.5 * c * R.Hth);
    at(5, iH, j + 1, -0.5 * c * R.Hth);
    for (int di = -1; di <= 0; ++di)
        for (int dj = 0; dj <= 1; ++dj) at(1, iH + di, j + dj, -0.25 * c * R.Eph);
}

// ---- spin derivative of the field update and of the objective -------------
// At fixed fields the update and the flux depend on the spin only through
// the static tables (face-area inverses, metric products of the auxiliary
// fields); dtab holds their a-derivatives.  A value and its a-derivative:
struct VD {
    double v, d;
};
__device__ __forceinline__ VD operator+(VD x, VD y) { return {x.v + y.v, x.d + y.d}; }
__device__ __forceinline__ VD operator-(VD x, VD y) { return {x.v - y.v, x.d - y.d}; }
__device__ __forceinline__ VD operator*(double c, VD x) { return {c * x.v, c * x.d}; }

// auxiliary fields of App. B (the field update's formulas) with their
// a-derivatives at fixed X
struct DAux {
    FAdj A;
    const double *dtab;
    P6 X;
    __device__ VD p(int slot, int comp, int i, int j) const
    {
        size_t q = slot * A.slab + (size_t)j * A.ldt + (i + NG);
        double x = X[comp][(size_t)j * A.ld + (i + NG)];
        return {A.tab[q] * x, dtab[q] * x};
    }
    __device__ VD t(int slot, int i, int j) const
    {
        size_t q = slot * A.slab + (size_t)j * A.ldt + (i + NG);
        return {A.tab[q], dtab[q]};
    }
    __device__ VD Hr(int i, int j) const
    {
        return p(T_AGRR_BR, 3, i, j) + 0.5 * (p(T_AGRP_BP, 5, i, j) + p(T_AGRP_BP, 5, i - 1, j));
    }
    __device__ VD Hth(int i, int j) const
    {
        return p(T_AGTT_BT, 4, i, j) + 0.5 * (p(T_SGB_DP, 2, i, j) + p(T_SGB_DP, 2, i + 1, j));
    }
    __device__ VD Hph(int i, int j) const
    {
        return p(T_AGPP_BP, 5, i, j) + 0.5 * (p(T_AGRP_BR, 3, i, j) + p(T_AGRP_BR, 3, i + 1, j)) -
               0.5 * (p(T_SGB_DT, 1, i, j) + p(T_SGB_DT, 1, i + 1, j));
    }
    __device__ VD Er(int i, int j) const
    {
        return p(T_AGRR_DR, 0, i, j) + 0.5 * (p(T_AGRP_DP, 2, i, j) + p(T_AGRP_DP, 2, i + 1, j));
    }
    __device__ VD Eth(int i, int j) const
    {
        return p(T_AGTT_DT, 1, i, j) - 0.5 * (p(T_SGB_BP, 5, i, j) + p(T_SGB_BP, 5, i - 1, j));
    }
    __device__ VD Eph(int i, int j) const
    {
        return p(T_AGPP_DP, 2, i, j) + 0.5 * (p(T_AGRP_DR, 0, i, j) + p(T_AGRP_DR, 0, i - 1, j)) +
               0.5 * (p(T_SGB_BT, 4, i, j) + p(T_SGB_BT, 4, i - 1, j));
    }
};

// block sum of v added to *out (blockDim.x * blockDim.y = 256)
__device__ __forceinline__ void block_add(double v, double *out)
{
    __shared__ double red[256];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    red[t] = v;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (t < o) red[t] += red[t + o];
        __syncthreads();
    }
    if (t == 0 && red[0] != 0.0) atomicAdd(out, red[0]);
}

// *out += sum over points of w . dC/da (X): C the circulation of one stage
// (Eqs. D-update, B-update divided by the face areas), w adjoint-shaped
__global__ void __launch_bounds__(256) dcirc_dot(FAdj A, const double *dtab, P6 X, P6 w, double scale, double dth,
                                                 double *out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    double acc = 0.0;
    if (i <= A.nr && j <= A.nth) {
        DAux X_{A, dtab, X};
        const int nr = A.nr, nth = A.nth;
        const size_t q = (size_t)j * A.ld + (i + NG);
        const double drd = A.col1d[1 * A.ldt + i + NG], drp = A.col1d[0 * A.ldt + i + NG];
        auto term = [&](int comp, int inv_slot, VD circ) {
            VD inv = X_.t(inv_slot, i, j);
            return w[comp][q] * (circ.d * inv.v + circ.v * inv.d);
        };
        if (i <= nr - 1) {
            VD hp = (j < nth) ? X_.Hph(i, j) : VD{0.0, 0.0};
            VD hm = (j > 0) ? X_.Hph(i, j - 1) : VD{0.0, 0.0};
            acc += term(0, T_INV_ADR, hp - hm);
        }
        if (j < nth) {
            acc += term(1, T_INV_ADT, X_.Hph(i - 1, j) - X_.Hph(i, j));
            acc += term(3, T_INV_ABR, -1.0 * (X_.Eph(i, j + 1) - X_.Eph(i, j)));
        }
        if (j > 0 && j < nth) {
            acc += term(2, T_INV_ADP, dth * (X_.Hth(i, j) - X_.Hth(i - 1, j)) + drd * (X_.Hr(i, j - 1) - X_.Hr(i, j)));
            if (i <= nr - 1) acc += term(4, T_INV_ABT, -1.0 * (X_.Eph(i, j) - X_.Eph(i + 1, j)));
        }
        if (i <= nr - 1 && j < nth)
            acc += term(5, T_INV_ABP,
                        -1.0 * (dth * (X_.Eth(i + 1, j) - X_.Eth(i, j)) + drp * (X_.Er(i, j) - X_.Er(i, j + 1))));
    }
    block_add(scale * acc, out);
}

// *out += sj * sum over the D points a stage writes of w . d(invA)/da J A
// (the current term of Eq. fld-predictor / fld-corrector)
__global__ void __launch_bounds__(256) jinv_dot(FAdj A, const double *dtab, P6 w,
                                                P6 J, double sj, double *out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = blockIdx.y * blockDim.y + threadIdx.y;
    double acc = 0.0;
    if (i <= A.nr && j <= A.nth) {
        const size_t q = (size_t)j * A.ld + (i + NG), qt = (size_t)j * A.ldt + (i + NG);
        if (i <= A.nr - 1) acc += w[0][q] * dtab[T_INV_ADR * A.slab + qt] * J[0][q];
        if (j < A.nth) acc += w[1][q] * dtab[T_INV_ADT * A.slab + qt] * J[1][q];
        if (j > 0 && j < A.nth) acc += w[2][q] * dtab[T_INV_ADP * A.slab + qt] * J[2][q];
    }
    block_add(sj * acc, out);
}

// *out += w * d(flux)/da at fixed fields F (the ring values of the objective)
__global__ void __launch_bounds__(256) flux_da(FAdj A, const double *dtab, P6 F, int iH, double dth,
                                               double w, double *out)
{
    double acc = 0.0;
    int j = blockIdx.x * 256 + threadIdx.x;
    if (j < A.nth) {
        DAux X_{A, dtab, F};
        VD Eth = X_.Eth(iH, j);
        VD Hph = 0.5 * (X_.Hph(iH - 1, j) + X_.Hph(iH, j));
        VD Eph = 0.5 * (X_.Eph(iH, j) + X_.Eph(iH, j + 1));
        VD Hth = 0.25 * (X_.Hth(iH - 1, j) + X_.Hth(iH, j) + X_.Hth(iH - 1, j + 1) + X_.Hth(iH, j + 1));
        acc = w * dth * (Eth.d * Hph.v + Eth.v * Hph.d - Eph.d * Hth.v - Eph.v * Hth.d);
    }
    block_add(acc, out);
}

// dtab = (tab(a + h) - tab(a - h)) / (2h)
__global__ void central_diff(const double *tp, const double *tm, double inv2h, size_t n, double *d)
{
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) d[e] = (tp[e] - tm[e]) * inv2h;
}

// *out += sum of x[0..n)
__global__ void __launch_bounds__(256) sum_into(const double *x, int64_t n, double *out)
{
    double acc = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < n; e += (int64_t)gridDim.x * 256) acc += x[e];
    block_add(acc, out);
}

}  // namespace
}  // namespace grpic

using namespace grpic;

namespace {

P6 six(double *const *h, int n = 6)
{
    P6 q;
    for (int k = 0; k < 6; ++k) q.p[k] = k < n ? h[k] : nullptr;
    return q;
}

}  // namespace

extern "C" grpic_status grpic_horizon_flux(grpic_ctx *ctx, const grpic_fields *f, int i_horizon, double *out,
                                           void *stream)
{
    if (!ctx || !f || !out || ctx->prm.precision != 64 || f->ld < ctx->g.nr + 2 * NG || i_horizon < 1 ||
        i_horizon > ctx->g.nr - 1)
        return GRPIC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    double *hp[6];
    for (int k = 0; k < 3; ++k) {
        hp[k] = (double *)f->D[k];
        hp[3 + k] = (double *)f->B[k];
    }
    FAdj A{ctx->g.nr, ctx->g.nth, f->ld, ctx->g.ld_tab, ctx->slab, ctx->tab, ctx->col1d};
    // the call's own word: calls on one context from several streams or threads
    // do not meet
    double *dev = nullptr;
    if (cudaMalloc(&dev, sizeof(double)) != cudaSuccess) return GRPIC_ENOMEM;
    cudaMemsetAsync(dev, 0, sizeof(double), s);
    flux_kernel<<<1, 256, 0, s>>>(A, six(hp), i_horizon, ctx->g.dth, 1.0, dev);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, dev, sizeof(double), cudaMemcpyDeviceToHost, s);
    const cudaError_t es = cudaStreamSynchronize(s);
    cudaFree(dev);
    return e == cudaSuccess && es == cudaSuccess ? GRPIC_OK : GRPIC_ECUDA;
}

// What the spin derivative of one field update needs: the derivative
// tables, the update's input fields Xn, its currents J and every stage's
// output Y[6 k ..], and the scalar it accumulates into.
struct SpinField {
    const double *dtab;
    P6 Xn, J;
    double *const *Y;
    double *La;
};

// Transpose of one field update: lam (adjoint of F^{n+1}) -> out, the adjoint of
// F^n, and lamJ, of the integrated currents J A.  work: mu[6], M[6], h[6].
// With sp, also adds the update's a-derivative contracted with the stage
// adjoints to sp->La: every stage's pre-projection value
//   dt (c_k C(Xn) + beta_s C(Y_{k-1})) - dt invA J   (c_0 = 1, c_k = alpha_s)
// depends on a through the tables of C and invA.
static grpic_status field_adjoint(grpic_ctx *ctx, P6 lam, P6 out, P6 lamJ, double *const *work, int64_t ld,
                                  cudaStream_t s, const SpinField *sp = nullptr)
{
    const int N = ctx->prm.n_field_iter;
    const double dt = ctx->prm.dt, bs = ctx->prm.beta_field, as = 1.0 - bs, dth = ctx->g.dth;
    FAdj A{ctx->g.nr, ctx->g.nth, ld, ctx->g.ld_tab, ctx->slab, ctx->tab, ctx->col1d};
    const dim3 blk(64, 4), rows((ctx->g.nth + 1 + 3) / 4);
    const dim3 gphys((ctx->g.nr + 1 + 63) / 64, rows.x), gcol((ctx->g.ld_tab + 63) / 64, rows.x),
        gld((unsigned)((ld + 63) / 64), rows.x);
    const P6 mu = six(work), M = six(work + 6), h = six(work + 12);
    stage_first<<<gphys, blk, 0, s>>>(A, lam, mu, M, 1);
    for (int k = N; k > 0; --k) {
        if (sp)  // dt beta_s mu_k . dC/da (Y_{k-1})
            dcirc_dot<<<gphys, blk, 0, s>>>(A, sp->dtab, six(sp->Y + (k - 1) * 6), mu, dt * bs, dth, sp->La);
        stage_h<<<gcol, blk, 0, s>>>(A, mu, h, dt * bs, dth);
        stage_mu<<<gphys, blk, 0, s>>>(A, h, mu, M);
    }
    if (sp)  // the currents' term: -dt M . d(invA)/da J
        jinv_dot<<<gphys, blk, 0, s>>>(A, sp->dtab, M, sp->J, -dt, sp->La);
    stages_close<<<gld, blk, 0, s>>>(A, lam, mu, M, out, lamJ, dt, as);
    if (sp)  // (sum_k dt c_k mu_k) . dC/da (X^n)
        dcirc_dot<<<gphys, blk, 0, s>>>(A, sp->dtab, sp->Xn, mu, 1.0, dth, sp->La);
    // lam X^n += C^T lam C(X^n)
    stage_h<<<gcol, blk, 0, s>>>(A, mu, h, 1.0, dth);
    add_from_h<<<gcol, blk, 0, s>>>(A, h, out);
    return cudaGetLastError() == cudaSuccess ? GRPIC_OK : GRPIC_ECUDA;
}

extern "C" grpic_status grpic_adjoint_field_step(grpic_ctx *ctx, const grpic_fields *lam_in, grpic_fields *lam_out,
                                                 void *stream)
{
    if (!ctx || !lam_in || !lam_out || ctx->prm.precision != 64 || lam_in->ld != lam_out->ld ||
        lam_in->ld < ctx->g.nr + 2 * NG || ctx->prm.n_field_iter < 1)
        return GRPIC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    int64_t ld = lam_in->ld;
    size_t fn = (size_t)(ctx->g.nth + 1) * ld;
    double *base = nullptr;
    if (ctx_malloc(ctx, &base, 18 * fn * sizeof(double)) != cudaSuccess) return GRPIC_ENOMEM;
    double *work[18], *in[6], *out[6], *J[3];
    for (int k = 0; k < 18; ++k) work[k] = base + k * fn;
    for (int k = 0; k < 3; ++k) {
        in[k] = (double *)lam_in->D[k];
        in[3 + k] = (double *)lam_in->B[k];
        out[k] = (double *)lam_out->D[k];
        out[3 + k] = (double *)lam_out->B[k];
        J[k] = (double *)lam_out->J[k];
    }
    grpic_status st = field_adjoint(ctx, six(in), six(out), six(J, 3), work, ld, s);
    cudaStreamSynchronize(s);
    cudaFree(base);
    return st;
}

// ---------------------------------------------------------------------------
// full gradient: forward with checkpoints, reverse sweep
// ---------------------------------------------------------------------------
extern "C" grpic_status grpic_adjoint_grad(grpic_ctx *ctx, const grpic_particles *p0, const grpic_fields *f0,
                                           int nsteps, int checkpoint_every, int i_horizon, int trapezoid_ift,
                                           double *L_out, double *const grad_p[5], double *const grad_f[6],
                                           double *dL_da, void *stream)
{
    if (!ctx || !p0 || !f0 || !L_out || ctx->prm.precision != 64 || nsteps < 1 || checkpoint_every < 1 ||
        i_horizon < 1 || i_horizon > ctx->g.nr - 1 || ctx->prm.n_field_iter < 1 || f0->ld < ctx->g.nr + 2 * NG ||
        p0->n < 0 || p0->n > INT32_MAX || (!grad_p && (grad_f || dL_da)) || ctx->prm.n_push_iter > MAX_ITER ||
        ctx->prm.pusher != 0 || ctx->prm.shape_order != 1 || ctx->prm.radiation != 0 || ctx->prm.injection != 0)
        return GRPIC_EINVAL;
    const bool want = grad_p != nullptr;  // NULL: the objective alone
    if (want)
        for (int k = 0; k < 5; ++k)
            if (!grad_p[k]) return GRPIC_EINVAL;
    if (p0->n > 0 && (!p0->x1 || !p0->x2 || !p0->u1 || !p0->u2 || !p0->u3 || !p0->tag)) return GRPIC_EINVAL;
    for (int k = 0; k < 3; ++k)
        if (!f0->D[k] || !f0->B[k]) return GRPIC_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t ld = f0->ld, np = p0->n;
    const size_t fn = (size_t)(ctx->g.nth + 1) * ld;
    const int ck = checkpoint_every;
    const int nseg = (nsteps + ck - 1) / ck;
    const int sl = std::min(ck, nsteps);  // steps of the longest segment
    const int last0 = (nseg - 1) * ck;    // first step of the last segment
    const bool spin = dL_da != nullptr;
    const int NF = ctx->prm.n_field_iter, TW = tape_width(ctx->prm.n_push_iter);
    const size_t ntab = ctx->slab * T_COUNT;
    // states: checkpoints of every segment but the last (which is recorded during
    // the forward pass), the current segment's states
    struct State {
        double *F[6];
        double *x[5];
        uint32_t *tag;
    };
    std::vector<State> cks(want ? nseg - 1 : 0), seg(want ? sl + 1 : 0);
    State W;  // working particles / fields of the forward runs
    double *Jw[3], *Ldev, *lamFa[6], *lamFb[6], *lamJ[3], *lamP[5], *lamP2[5], *aux[6], *tape = nullptr;
    std::vector<double *> work(want ? 18 : 0, nullptr);
    // spin derivative: derivative tables (and those of a +- h), per-particle parts,
    // the segment's currents and one update's stage outputs
    double *dtab = nullptr, *tp = nullptr, *tm = nullptr, *c1 = nullptr, *Ladev = nullptr, *Lap = nullptr;
    std::vector<double *> segJ(spin ? 3 * sl : 0, nullptr), Ystage(spin ? 6 * (NF + 1) : 0, nullptr);
    // one block holds all of it: the first pass measures, the second places
    char *base = nullptr;
    size_t need = 0;
    auto place = [&](size_t bytes) -> double * {
        double *q = base ? (double *)(base + need) : nullptr;
        need += (bytes + 255) & ~(size_t)255;
        return q;
    };
    auto layout = [&]() {
        need = 0;
        auto state = [&](State &S) {
            for (int k = 0; k < 6; ++k) S.F[k] = place(fn * sizeof(double));
            for (int k = 0; k < 5; ++k) S.x[k] = place(np * sizeof(double));
            S.tag = (uint32_t *)place(np * sizeof(uint32_t));
        };
        for (auto &S : cks) state(S);
        for (auto &S : seg) state(S);
        state(W);
        for (int k = 0; k < 3; ++k) Jw[k] = place(fn * sizeof(double));
        Ldev = place(sizeof(double));
        if (!want) return;
        for (int k = 0; k < 6; ++k) lamFa[k] = place(fn * sizeof(double));
        for (int k = 0; k < 6; ++k) lamFb[k] = place(fn * sizeof(double));
        double *a6 = place(6 * fn * sizeof(double));
        for (int k = 0; k < 6; ++k) aux[k] = a6 + (base ? k * fn : 0);
        for (int k = 0; k < 3; ++k) lamJ[k] = place(fn * sizeof(double));
        for (int k = 0; k < 5; ++k) lamP[k] = place(np * sizeof(double));
        for (int k = 0; k < 5; ++k) lamP2[k] = place(np * sizeof(double));
        tape = place((size_t)sl * TW * (size_t)np * sizeof(double));  // the push's record of a segment
        for (auto &w : work) w = place(fn * sizeof(double));
        if (!spin) return;
        dtab = place(ntab * sizeof(double));
        tp = place(ntab * sizeof(double));
        tm = place(ntab * sizeof(double));
        c1 = place(4 * ctx->g.ld_tab * sizeof(double));
        Ladev = place(sizeof(double));
        Lap = place(np * sizeof(double));
        for (auto &q : segJ) q = place(fn * sizeof(double));
        for (auto &q : Ystage) q = place(fn * sizeof(double));
    };
    layout();
    // (the context's own scratch first: it may take the kept block's memory)
    if (ensure_field_scratch_ext(ctx, ld) != GRPIC_OK || ensure_particle_scratch_ext(ctx, np) != GRPIC_OK)
        return GRPIC_ENOMEM;
    // The block stays with the context for the next gradient while it is at most a
    // sixteenth of the device's memory (mapping 5.5 GB and unmapping it took 27 of
    // 98 ms); a larger one is given back at once, the kept one by grpic_destroy, when
    // a gradient needs more, or when another call of the context finds no memory.
    if (ctx->adj_bytes < need) {
        cudaFree(ctx->adj_block);
        ctx->adj_block = nullptr;
        ctx->adj_bytes = 0;
        if (cudaMalloc(&ctx->adj_block, need) != cudaSuccess) {
            cudaGetLastError();
            ctx->adj_block = nullptr;
            return GRPIC_ENOMEM;
        }
        ctx->adj_bytes = need;
    }
    base = (char *)ctx->adj_block;
    layout();
    auto cleanup = [&]() {
        cudaStreamSynchronize(s);
        size_t free_b = 0, total = 0;
        cudaMemGetInfo(&free_b, &total);
        if (ctx->adj_bytes > total / 16) {
            cudaFree(ctx->adj_block);
            ctx->adj_block = nullptr;
            ctx->adj_bytes = 0;
        }
    };
    if (spin) {
        // a-derivatives of the tables by central differences, h = 1e-5 (the
        // quadratures are smooth in a: truncation ~h^2, rounding ~1e-16/h)
        const double h = 1e-5;
        if (launch_tables_at(ctx, ctx->g.a + h, tp, c1, s) != cudaSuccess ||
            launch_tables_at(ctx, ctx->g.a - h, tm, c1, s) != cudaSuccess) {
            cleanup();
            return GRPIC_ECUDA;
        }
        central_diff<<<(unsigned)((ntab + 255) / 256), 256, 0, s>>>(tp, tm, 0.5 / h, ntab, dtab);
        cudaMemsetAsync(Ladev, 0, sizeof(double), s);
    }
    auto copy_state = [&](State &dst, const State &src) {
        for (int k = 0; k < 6; ++k) cudaMemcpyAsync(dst.F[k], src.F[k], fn * sizeof(double), cudaMemcpyDeviceToDevice, s);
        for (int k = 0; k < 5; ++k) cudaMemcpyAsync(dst.x[k], src.x[k], np * sizeof(double), cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(dst.tag, src.tag, np * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
    };
    // initial state -> W
    for (int k = 0; k < 3; ++k) {
        cudaMemcpyAsync(W.F[k], f0->D[k], fn * sizeof(double), cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(W.F[3 + k], f0->B[k], fn * sizeof(double), cudaMemcpyDeviceToDevice, s);
    }
    void *px[5] = {p0->x1, p0->x2, p0->u1, p0->u2, p0->u3};
    for (int k = 0; k < 5; ++k) cudaMemcpyAsync(W.x[k], px[k], np * sizeof(double), cudaMemcpyDeviceToDevice, s);
    cudaMemcpyAsync(W.tag, p0->tag, np * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
    cudaMemsetAsync(Ldev, 0, sizeof(double), s);

    grpic_fields FW;
    for (int k = 0; k < 3; ++k) {
        FW.D[k] = W.F[k];
        FW.B[k] = W.F[3 + k];
        FW.J[k] = Jw[k];
    }
    FW.ld = ld;
    grpic_particles PW;
    memset(&PW, 0, sizeof PW);
    PW.n = np;
    PW.capacity = np;
    PW.d_count = nullptr;
    PW.x1 = W.x[0];
    PW.x2 = W.x[1];
    PW.u1 = W.x[2];
    PW.u2 = W.x[3];
    PW.u3 = W.x[4];
    PW.tag = W.tag;
    FAdj A{ctx->g.nr, ctx->g.nth, ld, ctx->g.ld_tab, ctx->slab, ctx->tab, ctx->col1d};
    const double wL = 1.0 / nsteps, dth = ctx->g.dth;
    grpic_status st = GRPIC_OK;
    // one forward step; with a tape slice, the push also records itself there
    auto fwd_step = [&](double *tp) -> grpic_status {
        for (int k = 0; k < 3; ++k) cudaMemsetAsync(Jw[k], 0, fn * sizeof(double), s);
        cudaError_t e = tp ? launch_push64_tape(ctx, &PW, &FW, tp, np, s)
                           : launch_push64(ctx, &PW, &PW, nullptr, nullptr, nullptr, &FW, false, s);
        if (e != cudaSuccess) return GRPIC_ECUDA;
        grpic_status r = GRPIC_OK;
        if (launch_field64(ctx, &FW, s) != cudaSuccess) r = GRPIC_ECUDA;
        return r;
    };
    // ---- forward with checkpoints --------------------------------------
    // the last segment, the first the reverse sweep needs, is recorded here
    // (its states, the push's record and, for the spin derivative, its
    // currents) instead of being recomputed from a checkpoint
    for (int n = 0; n < nsteps && st == GRPIC_OK; ++n) {
        if (want && n % ck == 0 && n < last0) copy_state(cks[n / ck], W);
        const bool rec = want && n >= last0;
        const int m = n - last0;
        if (rec && m == 0) copy_state(seg[0], W);
        st = fwd_step(rec ? tape + (size_t)m * TW * (size_t)np : nullptr);
        if (rec) {
            copy_state(seg[m + 1], W);
            if (spin)
                for (int k = 0; k < 3; ++k)
                    cudaMemcpyAsync(segJ[3 * m + k], Jw[k], fn * sizeof(double), cudaMemcpyDeviceToDevice, s);
        }
        flux_kernel<<<1, 256, 0, s>>>(A, six(W.F), i_horizon, dth, wL, Ldev);
        if (spin)  // the objective's own tables at F^{n+1}
            flux_da<<<(ctx->g.nth + 255) / 256, 256, 0, s>>>(A, dtab, six(W.F), i_horizon, dth, wL, Ladev);
    }
    cudaMemcpyAsync(L_out, Ldev, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (!want) {
        int hst = 0;
        cudaMemcpyAsync(&hst, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, s);
        cudaMemsetAsync(ctx->d_status, 0, sizeof(int), s);
        ctx->keys_valid = 0;
        ctx->hist_valid = 0;
        cleanup();
        if (cudaGetLastError() != cudaSuccess && st == GRPIC_OK) st = GRPIC_ECUDA;
        if (st == GRPIC_OK && hst != 0) st = (grpic_status)hst;
        return st;
    }
    // ---- reverse sweep -----------------------------------------------------
    for (int k = 0; k < 6; ++k) cudaMemsetAsync(lamFa[k], 0, fn * sizeof(double), s);
    for (int k = 0; k < 5; ++k) cudaMemsetAsync(lamP[k], 0, np * sizeof(double), s);
    P6 lamF = six(lamFa), lamF2 = six(lamFb);  // the fields' adjoint and the previous step's
    SpinField spf{dtab, P6(), P6(), Ystage.data(), Ladev};
    dim3 gfull((ctx->g.ld_tab + 63) / 64, (ctx->g.nth + 1 + 3) / 4), blk(64, 4);
    for (int sgi = nseg - 1; sgi >= 0 && st == GRPIC_OK; --sgi) {
        int n0 = sgi * ck, len = std::min(ck, nsteps - n0);
        // recompute the segment's states (the last one was recorded in the forward pass)
        if (sgi != nseg - 1) {
            copy_state(W, cks[sgi]);
            copy_state(seg[0], W);
        }
        for (int m = 0; m < len && st == GRPIC_OK && sgi != nseg - 1; ++m) {
            st = fwd_step(tape + (size_t)m * TW * (size_t)np);
            copy_state(seg[m + 1], W);
            if (spin)
                for (int k = 0; k < 3; ++k)
                    cudaMemcpyAsync(segJ[3 * m + k], Jw[k], fn * sizeof(double), cudaMemcpyDeviceToDevice, s);
        }
        for (int m = len - 1; m >= 0 && st == GRPIC_OK; --m) {
            // seed: lamF (adjoint of F^{n+1}) += wL dflux/dF^{n+1}
            cudaMemsetAsync(aux[0], 0, 6 * fn * sizeof(double), s);
            flux_seed<<<(ctx->g.nth + 127) / 128, 128, 0, s>>>(A, six(seg[m + 1].F), i_horizon, dth, wL, six(aux));
            add_from_h<<<gfull, blk, 0, s>>>(A, six(aux), lamF);
            // fields: lamF -> lamF2 (adjoint of F^n through the field update), lamJ
            if (spin) {
                // the update of step m again, every stage kept
                if (launch_field64_stages(ctx, seg[m].F, &segJ[3 * m], Ystage.data(), ld, s) != cudaSuccess) {
                    st = GRPIC_ECUDA;
                    break;
                }
                spf.Xn = six(seg[m].F);
                spf.J = six(&segJ[3 * m], 3);
            }
            st = field_adjoint(ctx, lamF, lamF2, six(lamJ, 3), work.data(), ld, s, spin ? &spf : nullptr);
            if (st != GRPIC_OK) break;
            // particles
            PAdjArgs P;
            P.g = ctx->g;
            P.dt = ctx->prm.dt;
            P.n_iter = ctx->prm.n_push_iter;
            P.ift = trapezoid_ift ? 1 : 0;
            for (int k = 0; k < 4; ++k) {
                P.qm[k] = ctx->prm.q_over_m[k];
                P.qw[k] = ctx->prm.q_weight[k];
                P.massive[k] = ctx->prm.massive[k];
            }
            P.n = np;
            for (int k = 0; k < 5; ++k) {
                P.x[k] = seg[m].x[k];
                P.lam1[k] = lamP[k];
                P.lam0[k] = lamP2[k];
            }
            P.tape = tape + (size_t)m * TW * (size_t)np;
            P.tape_ld = np;
            P.tag0 = seg[m].tag;
            P.tag1 = seg[m + 1].tag;
            for (int k = 0; k < 6; ++k) {
                P.F[k] = seg[m].F[k];
                P.lamF[k] = lamF2[k];
            }
            for (int k = 0; k < 3; ++k) P.lamJ[k] = lamJ[k];
            P.ld = ld;
            P.La = spin ? Lap : nullptr;
            if (np > 0 && spin) particle_adjoint<true><<<(unsigned)((np + 127) / 128), 128, 0, s>>>(P);
            if (np > 0 && !spin) particle_adjoint<false><<<(unsigned)((np + 127) / 128), 128, 0, s>>>(P);
            if (spin && np > 0) {
                unsigned nb = (unsigned)std::min<int64_t>((np + 255) / 256, 4 * 152);
                sum_into<<<nb, 256, 0, s>>>(Lap, np, Ladev);
            }
            if (cudaGetLastError() != cudaSuccess) st = GRPIC_ECUDA;
            for (int k = 0; k < 5; ++k) std::swap(lamP[k], lamP2[k]);
            std::swap(lamF, lamF2);
        }
    }
    for (int k = 0; k < 5; ++k) cudaMemcpyAsync(grad_p[k], lamP[k], np * sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (grad_f)
        for (int k = 0; k < 6; ++k)
            if (grad_f[k]) cudaMemcpyAsync(grad_f[k], lamF[k], fn * sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (spin) cudaMemcpyAsync(dL_da, Ladev, sizeof(double), cudaMemcpyDeviceToHost, s);
    // a particle the forward refused (range, non-finite) is reported like the step does
    int hst = 0;
    cudaMemcpyAsync(&hst, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaMemsetAsync(ctx->d_status, 0, sizeof(int), s);
    ctx->keys_valid = 0;
    ctx->hist_valid = 0;
    cleanup();
    if (cudaGetLastError() != cudaSuccess && st == GRPIC_OK) st = GRPIC_ECUDA;
    if (st == GRPIC_OK && hst != 0) st = (grpic_status)hst;
    return st;
}
