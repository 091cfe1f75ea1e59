// grpic_push64.cu -- FP64 particle push fused with the charge-conserving
// deposit (arXiv:2503.04558 Sec. 2.2-2.3, Fig. stepping).
//
// One thread per particle (structure of arrays, coalesced loads):
//   1. interpolate D^j, B^j at x^n, each from its own staggered lattice
//      (bilinear cloud-in-cell in logical coordinates);
//   2. one full generalized Boris step at fields n (Eqs. boris-plus-minus,
//      u0bar, boris-scheme), skipped for photons;
//   3. geodesic predictor + n_iter trapezoidal correctors (Eqs.
//      geodesic-predictor, geodesic-corrector) on (r, theta, phi, u_r, u_theta);
//      U_phi = 0 so u_phi is left untouched;
//   4. axis reflection, range / finiteness checks;
//   5. Esirkepov deposit of x^n -> x^{n+1} (Eq. esirkepov-decomp with a local
//      prefix sum, Eq. j-phi-deposit) into the integrated currents
//      J^r A_r, J^theta A_theta, J^phi dV, reduced across the warp by start cell
//      (grpic_window.cuh);
//   6. cell key of x^{n+1} (dead -> n_cells) and a warp-aggregated histogram
//      for the sort.
//
// Bound by the FP64 pipe alone (one warp instruction in about 18 cycles; it
// also takes conversions and comparisons): what counts is the number of its
// instructions, not registers, loads or integer work.  Cells come from a table
// and a short series, sin and cos from the row's, reciprocals and roots from
// hardware seeds and one third-order step, sign and range tests and selections
// from the bits.  1.68e7 particles on 512^2: 25.7 -> 17.5 ms (766 -> about 530 pipe
// instructions a particle), and 12.0 ms with the early correctors in double-FP32
// pairs.  Errors against 64 bits, now to before, over 60 to 80 seeds of seven cases
// (both shapes and pushers): the mean ratio of every output lies in 0.65 .. 1.04, J^r
// 0.65 .. 0.79, positions 0.92 .. 0.99.  In a single run u_theta and J^phi are those of
// a few particles at the axis, and either side can be ten times the other's.
#include "grpic_internal.cuh"
#include "grpic_geo.cuh"
#include "grpic_df.cuh"
#include "grpic_window.cuh"
#include "grpic_vay.cuh"
#include "grpic_shape3.cuh"
#include "grpic_philox.cuh"

namespace grpic {
namespace {

struct Push64Args {
    GridDev g;
    double dt;
    int n_iter;
    int pairs;           // the correctors before the last may run in pairs
    float hf;            // dt / 2
    df a_df, a2_df, dt_df;
    double qm[4];
    double qdt[4], wr[4], wp[4];  // q dt / (2 m); -q w / (2 dt), q w / dt
    int massive[4];
    int64_t n;
    const int64_t *d_count;
    double *r, *th, *u1, *u2, *u3;
    uint32_t *tag;
    // read through a permutation (see the FP32 push): slot p's particle comes
    // from slot perm[p] of the input arrays; perm == nullptr: in place
    const int32_t *perm, *live;
    int64_t *count_out;
    int32_t *cnt9;  // with perm: counts of the next neighbour sort (see the FP32 push)
    const double *in_r, *in_th, *in_u1, *in_u2, *in_u3;
    const uint32_t *in_tag;
    const double *D0, *D1, *D2, *B0, *B1, *B2;
    double *J0, *J1, *J2;
    int64_t ld;
    int32_t *keys;
    int32_t *count;
    int histogram;
    int pusher;  // 0 generalized Boris, 1 Vay in the FIDO frame
    // 2D radiation: emission / conversion decisions per slot into spawn
    // (0, 1 photon, 2 pair), see grpic_rad.cu
    int radiation;
    double gamma_thr, eps_ph, pconv;
    float gthr2f;  // gamma_thr^2, rounded down
    uint64_t seed;
    int64_t step;
    int32_t *spawn;
    int *status;
    double *tape;  // the adjoint's record of the push (TAPE instantiation only)
    int64_t tape_ld;
};

// comparisons of positive doubles by their bits (the FP64 pipe takes a comparison
// at the price of a multiply-add); negative numbers count as beyond every bound
constexpr unsigned long long PI_BITS = 0x400921fb54442d18ull;  // M_PI
__device__ __forceinline__ unsigned long long positive_bits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ bool in_shell(const GridDev &g, double r)
{
    const long long b = __double_as_longlong(r);
    return b >= __double_as_longlong(g.r_in) && b < __double_as_longlong(g.r_out);
}

// threads per block (512 are resident per SM at 128 registers).  The last round
// of blocks leaves SMs with one block more than others, for a block's whole
// time: 128 against 256 threads, 2e5 particles on 128^2 1293 -> 1203 us per 4
// steps, cubic shape with 1.5e6 4.52 -> 4.37 ms, large ones and 64 threads the same
constexpr int PUSH64_T = 128;

using Rhs = RhsT<double>;
using Pt64 = PtT<double>;

// the right-hand side of Eq. particle-eom (without F_i) at a point: the
// point quantities and the part in u of grpic_geo.cuh's pointT / rhsT
__device__ __forceinline__ void geo_rhs_sc(double a, double a2, double m2a2, double eps, double r, double s, double c,
                                           double ur, double ut, double up, Rhs &f)
{
    const Pt64 m = pointT<double>(a2, m2a2, r, s, c);
    rhsT<double>(m, a, eps, ur, ut, up, a * up, f);
}

// The correctors before the last one in double-FP32 pairs (about 44 significant
// bits on the FP32 pipes, which the push leaves idle).  Their result is only
// the point where the last corrector, in FP64, takes its right-hand side: a relative
// error eps of a step's change comes out of it times dt/2 dF/dy, itself of the order
// of dt/2 times the angular velocity or the inverse radius, and the change is of that
// order of the value.  They run where the square of both is below 2^-14
// (PAIR_MAX_ANGLE, PAIR_MAX_RADIAL; eps times it is then under an eighth of an FP64
// rounding of the value), dt is at most PAIR_MAX_DT, and the low words of u^2 and of
// its inverse stay in FP32's range (PAIR_MAX_U; PAIR_MIN_U for photons: a massless
// right-hand side scales with u, a massive one has the 1 of 1 + u^2), and in FP64
// elsewhere: next to the axis and on coarse grids.  Per particle, so that a result
// does not depend on the warp's other lanes.  Measured over 9 seeds of eight cases,
// 128^2 to 512^2: every output as far from 64 bits' value as with FP64 correctors, to
// 1 %.
constexpr float PAIR_MAX_ANGLE = 0.0064f;      // of dt/2 |dphi/dt|
constexpr float PAIR_MAX_RADIAL = 0.0078125f;  // of dt/2 / r
constexpr double PAIR_MAX_DT = 0.02;
constexpr int PAIR_MIN_U = 0x3e100000;         // of the largest |u_i|: 2^-30, 2^30 (high words)
constexpr int PAIR_MAX_U = 0x41d00000;

__device__ __forceinline__ bool pairs_hold(float hf, double xp, double r, bool massive, const double u[3])
{
    const int top = max(max(__double2hiint(u[0]) & 0x7fffffff, __double2hiint(u[1]) & 0x7fffffff),
                        __double2hiint(u[2]) & 0x7fffffff);
    return hf * float_of_pos(fabs(xp)) < PAIR_MAX_ANGLE && hf < PAIR_MAX_RADIAL * float_of_pos(r) &&
           (massive || top >= PAIR_MIN_U) && top < PAIR_MAX_U;
}

struct RhsDf {
    df xr, xt, ur, ut;
};

// rhsT's right-hand side (without X^phi) in pairs at (r, sin, cos theta, u)
__device__ __forceinline__ void geo_rhs_df(const df &a2, float eps, const df &r, const df &s, const df &c, const df &ur,
                                           const df &ut, const df &up, const df &aup, RhsDf &f)
{
    const df r2 = r * r;
    const df ir = rcp_t(r2 + a2 * (c * c));
    const df z = scale2(r, 2.0f) * ir;
    const df opz = add_f(z, 1.0f);
    const df iopz = rcp_t(opz);
    const df beta = z * iopz;
    const df is2 = rcp_t(s * s);
    const df ar2 = a2 + r2;
    const df cs = c * s;
    const df E = scale2(a2 * cs, -2.0f) * ir;
    const df ur2 = ur * ur;
    const df is2up2 = is2 * up * up;
    const df w = ar2 * ur + aup;
    const df P = ur * (w + aup) + (ut * ut + is2up2);
    const df irP = ir * P;
    const df Q = add_f(irP - beta * ur2, eps);
    const df iu0 = rsqrt_t(opz * Q);
    const df h = scale2(iu0, 0.5f);
    const df iri = ir * iu0;
    f.xr = iu0 * (ir * w - beta * ur) - beta;
    f.xt = iri * ut;
    const df K = iopz * (iopz * ur * add_f(h * ur, 1.0f) + h * Q);
    f.ur = K * (scale2(ir, 2.0f) - z * z) + h * z * (irP - ur2);
    f.ut = E * (h * irP - K * z) + iri * (cs * is2) * is2up2;
}

// sin, cos of (theta0 + d), |d| <= 0.03: the second-order terms in pairs, the
// rest of the series (d^4 / 24) in FP32
__device__ __forceinline__ void sincos_shift_pair(const df &s0, const df &c0, const df &d, df &s, df &c)
{
    const df d2 = d * d;
    const float q = __fmul_rn(d2.hi, d2.hi);
    const df ec = add_f(scale2(d2, 0.5f), -q * fmaf(d2.hi, -1.0f / 720.0f, 1.0f / 24.0f));  // 1 - cos d
    const df es = add_f(d2 * df_const(1.0 / 6.0), -q * (1.0f / 120.0f));                    // 1 - sin(d) / d
    const df cd = c0 * d, sd = s0 * d;
    s = (s0 + cd) - (s0 * ec + cd * es);
    c = (c0 - sd) - (c0 * ec - sd * es);
}

// n correctors in pairs from the predictor: on return the changes of r, theta,
// u_r, u_theta against x^n; false (nothing kept) where an iterate leaves the range.
// note(it, changes) sees each iterate that a right-hand side is taken at.
template <typename NOTE>
__device__ __forceinline__ bool correctors_df(const df &a, const df &a2, const df &dt, int n, float eps, double r,
                                              double s0, double c0, const double u[3], const Rhs &f0, double &dr,
                                              double &dth, double &dur, double &dut, const NOTE &note)
{
    const df R = df_of(r), S0 = df_of(s0), C0 = df_of(c0), U0 = df_of(u[0]), U1 = df_of(u[1]), up = df_of(u[2]);
    const df aup = a * up, h = scale2(dt, 0.5f);
    const df x0 = df_of(f0.xr), t0 = df_of(f0.xt), v0 = df_of(f0.ur), w0 = df_of(f0.ut);
    df dR = dt * x0, dT = dt * t0, dV = dt * v0, dW = dt * w0;
    // theta may move by a few hundredths, and by an eighth of its distance to the
    // axis (the angular velocity of the criterion is that of x^n)
    const float room = fminf(4.0f * PAIR_MAX_ANGLE, 0.125f * S0.hi);
#pragma unroll 1
    for (int it = 0; it < n; ++it) {
        if (!(fabsf(dT.hi) < room)) return false;
        note(it, dR, dT, dV, dW);
        df s, c;
        sincos_shift_pair(S0, C0, dT, s, c);
        RhsDf f;
        geo_rhs_df(a2, eps, R + dR, s, c, U0 + dV, U1 + dW, up, aup, f);
        dR = h * (f.xr + x0);
        dT = h * (f.xt + t0);
        dV = h * (f.ur + v0);
        dW = h * (f.ut + w0);
    }
    if (!(fabsf(dT.hi) < room)) return false;
    dr = double_of(dR);
    dth = double_of(dT);
    dur = double_of(dV);
    dut = double_of(dW);
    return true;
}

// the 3+1 metric at the point (App. A): gamma_rr = 1 + z, gamma_thth = rho^2,
// gamma_rph = -a sin^2 (1 + z), gamma_phph = Sigma sin^2 / rho^2 with Sigma =
// (a^2 + r^2) rho^2 + 2 r a^2 sin^2 (the same Sigma as (a^2 + r^2)^2 - a^2
// Delta sin^2, without its cancellation), so gamma_phph = sin^2 (a^2 + r^2 +
// z a^2 sin^2); sqrt(gamma) = rho^2 sin (1 + z) alpha
__device__ __forceinline__ void ks_point_pt(double a, double a2, const Pt64 &B, KS &m)
{
    m.alpha = lapse(B);
    m.beta = B.beta;
    m.g_rr = B.opz;
    m.g_tt = B.rho2;
    m.g_pp = B.s2 * fma(B.z, a2 * B.s2, B.ar2);
    m.g_rp = -a * B.s2 * B.opz;
    m.gi_rr = fma(B.ar2, B.ir, -B.beta);
    m.gi_rp = a * B.ir;
    m.gi_tt = B.ir;
    m.gi_pp = B.ir * B.is2;
    m.sqrtg = B.rho2 * B.s * B.opz * m.alpha;
}

// Generalized Boris step at the particle (u covariant, D, B contravariant) with
// the point quantities at x^n; qdt = q dt / (2 m).  With t = kt B and s = ks t the
// rotations are multiples of v x B and x x B
__device__ __forceinline__ void boris(double a, double a2, const Pt64 &Bm, double qdt, const double D[3],
                                      const double B[3], double u[3])
{
    KS m;
    ks_point_pt(a, a2, Bm, m);
    const double Dl0 = fma(m.g_rr, D[0], m.g_rp * D[2]), Dl1 = m.g_tt * D[1], Dl2 = fma(m.g_rp, D[0], m.g_pp * D[2]);
    const double h = qdt * m.alpha;
    const double um0 = fma(h, Dl0, u[0]), um1 = fma(h, Dl1, u[1]), um2 = fma(h, Dl2, u[2]);
    // raised u^-
    const double v0 = fma(m.gi_rr, um0, m.gi_rp * um2), v1 = m.gi_tt * um1, v2 = fma(m.gi_rp, um0, m.gi_pp * um2);
    const double iu0b = m.alpha * rsqrt_fast(fma(um0, v0, fma(um1, v1, fma(um2, v2, 1.0))));  // 1 / u0bar
    const double kt = qdt * iu0b;
    const double Bl0 = fma(m.g_rr, B[0], m.g_rp * B[2]), Bl2 = fma(m.g_rp, B[0], m.g_pp * B[2]);
    const double BB = fma(B[0], Bl0, fma(m.g_tt * B[1], B[1], B[2] * Bl2));
    const double k1 = m.sqrtg * kt;                        // e_ijk t^k = k1 eps_ijk B^k
    const double k2 = (k1 + k1) * rcp_t(fma(kt * kt, BB, 1.0));  // the same of s = 2 t / (1 + t.t)
    // u~ = u^- + e_ijk v^j t^k
    const double w0 = fma(k1, fma(v1, B[2], -v2 * B[1]), um0), w1 = fma(k1, fma(v2, B[0], -v0 * B[2]), um1),
                 w2 = fma(k1, fma(v0, B[1], -v1 * B[0]), um2);
    const double x0 = fma(m.gi_rr, w0, m.gi_rp * w2), x1 = m.gi_tt * w1, x2 = fma(m.gi_rp, w0, m.gi_pp * w2);
    // u^+ = u^- + e_ijk (raised u~)^j s^k, then the second electric half kick
    u[0] = fma(h, Dl0, fma(k2, fma(x1, B[2], -x2 * B[1]), um0));
    u[1] = fma(h, Dl1, fma(k2, fma(x2, B[0], -x0 * B[2]), um1));
    u[2] = fma(h, Dl2, fma(k2, fma(x0, B[1], -x1 * B[0]), um2));
}

// Vay's update in the FIDO frame with the point quantities at x^n
__device__ __forceinline__ void vay(double a, double a2, const Pt64 &Bm, double qm, double dt, const double D[3],
                                    const double B[3], double u[3])
{
    KS k;
    ks_point_pt(a, a2, Bm, k);
    VayMetric<double> m{k.alpha, k.g_rr, k.g_rp, k.g_tt, k.g_pp, k.gi_rr, k.gi_rp, k.gi_tt, k.gi_pp, k.sqrtg};
    vay_step<double>(m, qm, dt, D, B, u);
}

// a component from its four corners, along r on both rows, then along theta;
// flip0, flip1: the rows are mirror rows of an odd component
__device__ __forceinline__ double gather(const double *__restrict__ F, int64_t ld, int r0, int r1, int col, double f,
                                         double gg, bool flip0, bool flip1)
{
    const double *a = F + (size_t)r0 * ld + col, *b = F + (size_t)r1 * ld + col;
    const double a0 = __ldg(a), a1 = __ldg(a + 1), b0 = __ldg(b), b1 = __ldg(b + 1);
    const double x = flip_sign(fma(f, a1 - a0, a0), flip0), y = flip_sign(fma(f, b1 - b0, b0), flip1);
    return fma(gg, y - x, x);
}

// the six fields at (column i + f, row j + gg): D^r and B^theta at (i+1/2, j),
// D^theta (odd across the axis) and B^r at (i, j+1/2), D^phi at (i, j), B^phi at
// (i+1/2, j+1/2); rows -1 and n_theta of the half-theta lattice are mirrors
__device__ __forceinline__ void gather_fields(const double *D0, const double *D1, const double *D2, const double *B0,
                                              const double *B1, const double *B2, int64_t ld, int nth, int i, double f,
                                              int j, double gg, double Dv[3], double Bv[3])
{
    int ih, jh;
    double fh, gh;
    half_node(i, f, ih, fh);
    half_node(j, gg, jh, gh);
    const bool m0 = jh < 0, m1 = jh + 1 > nth - 1;
    const int h0 = m0 ? 0 : jh, h1 = m1 ? nth - 1 : jh + 1;
    Dv[0] = gather(D0, ld, j, j + 1, ih + NG, fh, gg, false, false);
    Dv[1] = gather(D1, ld, h0, h1, i + NG, f, gh, m0, m1);
    Dv[2] = gather(D2, ld, j, j + 1, i + NG, f, gg, false, false);
    Bv[0] = gather(B0, ld, h0, h1, i + NG, f, gh, false, false);
    Bv[1] = gather(B1, ld, j, j + 1, ih + NG, fh, gg, false, false);
    Bv[2] = gather(B2, ld, h0, h1, ih + NG, fh, gh, false, false);
}

// sin, cos of theta at offset f in row j: those of the nearer edge of the row
// shifted by the rest (rows of at most 0.05 rad; the nearer edge keeps sin's
// relative precision up to both poles), the library's on coarser grids
__device__ __forceinline__ void sincos_row(const GridDev &g, int j, double f, double th, double &s, double &c)
{
    if (g.trow) {
        const int jn = j + (__double2hiint(f) >= 0x3fe00000 ? 1 : 0);
        const double2 t0 = __ldg(g.trow + 2 * jn), t1 = __ldg(g.trow + 2 * jn + 1);  // theta_j, sin | cos, pad
        sincos_shift<double>(t0.y, t1.x, th - t0.x, s, c);
    } else {
        sincos(th, &s, &c);
    }
}

// FP32 view of 1 + gamma^ij u_i u_j, a few 1e-6 of its terms off: whether the
// FIDO Lorentz factor can reach `thr` (the FP64 decision is taken only then; a
// margin of 2 % in the square covers the cancellation between the terms).  The
// angle is taken from the nearer pole before it is cut to FP32: pi - theta, for
// theta close to pi, has no relative precision left in a float theta.
__device__ __forceinline__ bool may_reach(float a, float r, double th, double u0, double u1, double u2, float thr2)
{
    float s, c;  // (cos enters by its square)
    sincosf((float)(__double2hiint(th) >= 0x3ff921fb ? M_PI - th : th), &s, &c);
    const float v0 = (float)u0, v1 = (float)u1, v2 = (float)u2;
    const float ir = 1.0f / fmaf(a * c, a * c, r * r), z = 2.0f * r * ir;
    const float t0 = (fmaf(a, a, r * r) * ir - z / (1.0f + z)) * v0 * v0, t1 = 2.0f * a * ir * v0 * v2;
    const float t2 = ir * v1 * v1, t3 = ir / (s * s) * v2 * v2;
    // not below: NaN and infinities go on to the FP64 decision
    return !(1.0f + t0 + t1 + t2 + t3 + 0.02f * (fabsf(t0) + fabsf(t1) + t2 + t3) < thr2);
}

// SHAPE 1: cloud in cell (bilinear interpolation, 4 x 4 window reduced across
// the warp); SHAPE 3: the cubic spline of grpic_shape3.cuh (4 x 4 taps,
// per-lane deposit of the 5 x 5 window).  TAPE: also write the adjoint's
// record of the push (CIC, no radiation)
template <int SHAPE, bool RAD, bool TAPE>
__global__ void __launch_bounds__(PUSH64_T, 512 / PUSH64_T) push64_kernel(Push64Args A)
{
    const GridDev &g = A.g;
    const bool permuted = A.perm != nullptr;
    int64_t n = permuted ? (int64_t)*A.live : (A.d_count ? *A.d_count : A.n);
    if (n > A.n) n = A.n;
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned FULL = 0xffffffffu;
    int lane = threadIdx.x & 31;
    int ncell = g.nr * g.nth;
    if (permuted && p == 0 && A.count_out) *A.count_out = n;

    bool live = false;
    uint32_t tag = DEAD;
    double r = 0, th = 0, u[3] = {0, 0, 0};
    if (p < n) {
        const int64_t src = permuted ? (int64_t)A.perm[p] : p;
        tag = A.in_tag[src];
        if (!(tag & DEAD)) {
            live = true;
            r = A.in_r[src];
            th = A.in_th[src];
            u[0] = A.in_u1[src];
            u[1] = A.in_u2[src];
            u[2] = A.in_u3[src];
        }
    }

    bool dep = false;
    int spawn = 0;
    double fa1 = 0.0, fa2 = 0.0, fb1 = 0.0, fb2 = 0.0, wr = 0.0, wp = 0.0, wphi = 0.0;  // offsets of the start and end points
    int i0 = 0, j0 = 0, di = 0, dj = 0, key = -1;
    if (live) {
        // a state outside the domain (or non-finite) would index the fields out
        // of range: refuse it before any gather
        const bool fin = finite64(r) && finite64(th) && finite64(u[0]) && finite64(u[1]) && finite64(u[2]);
        if (!(fin && in_shell(g, r) && (positive_bits(th) <= PI_BITS || zero64(th)))) {
            set_status(A.status, fin ? GRPIC_ERANGE : GRPIC_ENAN);
            tag |= DEAD;
            live = false;
        }
    }
    if (live) {
        int sp = tag & 3u;
        const ColPos c0p = r_column_in(g, r);
        const double x2a = theta_cells(g, th);
        i0 = c0p.i;
        fa1 = c0p.f;
        j0 = row_of(g, x2a);
        fa2 = x2a - j0;
        // sin, cos of theta^n: shared by the Boris step and the first
        // right-hand side, shifted for the corrector iterates
        double s0, c0;
        sincos_row(g, j0, fa2, th, s0, c0);
        const double a2 = g.a * g.a, m2a2 = -2.0 * a2;
        const Pt64 B0 = pointT<double>(a2, m2a2, r, s0, c0);
        if (A.massive[sp] && A.qm[sp] != 0.0) {
            double Dv[3], Bv[3];
            if constexpr (SHAPE == 3)
                gather3_fields(A.D0, A.D1, A.D2, A.B0, A.B1, A.B2, A.ld, g.nth, i0, fa1, j0, fa2, Dv, Bv);
            else
                gather_fields(A.D0, A.D1, A.D2, A.B0, A.B1, A.B2, A.ld, g.nth, i0, fa1, j0, fa2, Dv, Bv);
            if (A.pusher)
                vay(g.a, a2, B0, A.qm[sp], A.dt, Dv, Bv, u);
            else
                boris(g.a, a2, B0, A.qdt[sp], Dv, Bv, u);
        }
        // geodesic predictor-corrector (Sec. 2.2)
        double eps = A.massive[sp] ? 1.0 : 0.0;
        Rhs f0, ft;
        double *tape = TAPE ? A.tape + p : nullptr;
        const int64_t tl = A.tape_ld;
        if constexpr (TAPE) {
            tape[(TAPE_U + 0) * tl] = u[0];
            tape[(TAPE_U + 1) * tl] = u[1];
            tape[(TAPE_U + 2) * tl] = u[2];
            tape[TAPE_SC0 * tl] = s0;
            tape[(TAPE_SC0 + 1) * tl] = c0;
        }
        rhsT<double>(B0, g.a, eps, u[0], u[1], u[2], g.a * u[2], f0);
        double dt = A.dt;
        const double h = 0.5 * dt;
        double xpl = f0.xp;
        double rt = fma(dt, f0.xr, r), tt = fma(dt, f0.xt, th);
        double urt = fma(dt, f0.ur, u[0]), utt = fma(dt, f0.ut, u[1]);
        int it = 0;
        {
            // the record's iterates: 2^-44 of the changes off, which are a hundredth
            // of the values; sin and cos from x^n's
            auto note = [&](int k, const df &dR, const df &dT, const df &dV, const df &dW) {
                if constexpr (TAPE) {
                    double *q = tape + (int64_t)(TAPE_IT + 6 * k) * tl;
                    const double d = double_of(dT);
                    double st, ct;
                    sincos_shift<double>(s0, c0, d, st, ct);
                    q[0] = r + double_of(dR);
                    q[tl] = th + d;
                    q[2 * tl] = u[0] + double_of(dV);
                    q[3 * tl] = u[1] + double_of(dW);
                    q[4 * tl] = st;
                    q[5 * tl] = ct;
                }
            };
            double dr, dth, dur, dut;
            if (A.pairs && pairs_hold(A.hf, f0.xp, r, A.massive[sp] != 0, u) &&
                correctors_df(A.a_df, A.a2_df, A.dt_df, A.n_iter - 1, (float)eps, r, s0, c0, u, f0, dr, dth, dur, dut,
                              note)) {
                rt = r + dr;
                tt = th + dth;
                urt = u[0] + dur;
                utt = u[1] + dut;
                it = A.n_iter - 1;
            }
        }
        for (; it < A.n_iter; ++it) {
            // theta of the iterate within 0.05 of theta^n (the usual case: one
            // step moves a particle less than two cells): the series of
            // sincos_shift, truncated below 1e-17
            double st, ct;
            const double dth = tt - th;
            if (below64(dth, 0x3fa99999))  // (0.05)
                sincos_shift<double>(s0, c0, dth, st, ct);
            else
                sincos(tt, &st, &ct);
            if constexpr (TAPE) {
                double *q = tape + (int64_t)(TAPE_IT + 6 * it) * tl;
                q[0] = rt;
                q[tl] = tt;
                q[2 * tl] = urt;
                q[3 * tl] = utt;
                q[4 * tl] = st;
                q[5 * tl] = ct;
            }
            geo_rhs_sc(g.a, a2, m2a2, eps, rt, st, ct, urt, utt, u[2], ft);
            rt = fma(h, ft.xr + f0.xr, r);
            tt = fma(h, ft.xt + f0.xt, th);
            xpl = ft.xp;
            urt = fma(h, ft.ur + f0.ur, u[0]);
            utt = fma(h, ft.ut + f0.ut, u[1]);
        }
        const double pt = h * (xpl + f0.xp);  // dt X^phi(x^n) without correctors
        if constexpr (TAPE) {
            double *q = tape + (int64_t)tape_end(A.n_iter) * tl;
            q[0] = rt;
            q[tl] = tt;
            q[2 * tl] = urt;
            q[3 * tl] = utt;
            q[4 * tl] = pt;
        }
        // axis reflection
        if (negative64(tt) && !zero64(tt)) { tt = -tt; utt = -utt; }
        if (__double_as_longlong(tt) > (long long)PI_BITS) { tt = 2.0 * M_PI - tt; utt = -utt; }
        bool finite = finite64(rt) && finite64(tt) && finite64(pt) && finite64(urt) && finite64(utt) && __double_as_longlong(rt) > 0;
        if (!finite) {
            set_status(A.status, GRPIC_ENAN);
            tag |= DEAD;
            live = false;
        } else {
            const ColPos c1p = r_column(g, rt);
            const double x2b = theta_cells(g, tt);
            const int j1 = row_of(g, x2b);
            di = c1p.i - i0;
            dj = j1 - j0;
            if (di < -1 || di > 1 || dj < -1 || dj > 1) {
                set_status(A.status, GRPIC_ERANGE);
                tag |= DEAD;
                live = false;
                di = dj = 0;
            } else {
                fb1 = c1p.f;
                fb2 = x2b - j1;
                wr = A.wr[sp];
                wp = A.wp[sp];
                wphi = pt;
                if constexpr (SHAPE == 3)
                    deposit3(g.nr, g.nth, A.ld, A.J0, A.J1, A.J2, wr, wp, i0, fa1, j0, fa2, c1p.i, fb1, j1,
                             fb2, pt);
                dep = true;
                r = rt;
                th = tt;
                u[0] = urt;
                u[1] = utt;
                if (!in_shell(g, rt)) tag |= DEAD;
                // the column the next push will start from (clamped into the grid)
                const int ib = min(max(c1p.i, 0), g.nr - 1);
                key = (tag & DEAD) ? ncell : (j1 * g.nr + ib);
                if (RAD && !(tag & DEAD)) {
                    // at the new position: emission by a charged particle above
                    // gamma_thr, conversion of a photon above 2 m c^2; a photon
                    // draws first (the draw fails for all but ~tau dt of them,
                    // which then skip the metric: the same decision)
                    const bool charged = A.massive[sp] && A.qm[sp] != 0.0;
                    const bool drawn = !A.massive[sp] && uniform53(A.seed, (uint64_t)p, A.step, 1) < A.pconv;
                    if (drawn || (charged && may_reach((float)g.a, (float)r, th, u[0], u[1], u[2],
                                                       A.gthr2f))) {
                        KS m;
                        ks_point(g.a, r, th, m);
                        const double uu = m.gi_rr * u[0] * u[0] + 2.0 * m.gi_rp * u[0] * u[2] +
                                          m.gi_tt * u[1] * u[1] + m.gi_pp * u[2] * u[2];
                        if (charged) {
                            const double G = sqrt(1.0 + uu), G2 = G - A.eps_ph;
                            if (G >= A.gamma_thr && G2 >= 1.0) {
                                const double f = sqrt(G2 * G2 - 1.0) / sqrt(uu);
                                u[0] *= f;
                                u[1] *= f;
                                u[2] *= f;
                                spawn = 1;
                            }
                        } else if (sqrt(uu) > 2.0) {
                            spawn = 2;
                            tag |= DEAD;
                            key = ncell;
                        }
                    }
                }
            }
        }
    }
    if (RAD && p < n) A.spawn[p] = spawn;
    if (p < n) {
        if (dep || permuted) {
            A.r[p] = r;
            A.th[p] = th;
            A.u1[p] = u[0];
            A.u2[p] = u[1];
            A.u3[p] = u[2];
        }
        if (tag & DEAD) key = ncell;
        A.tag[p] = tag;
        A.keys[p] = key;
    } else if (permuted && p < A.n) {
        A.tag[p] = DEAD;  // past the live slots of the permuted order
    }

    // ---- deposit (CIC): the core entries reduced across the warp by start
    // cell, the entries of lanes that left their cell added directly
    if constexpr (SHAPE == 1)
        deposit_warp_cells<double, 3>(dep, i0, j0, g.nr, fa1, fa2, di, dj, fb1, fb2, wr, wp, wphi,
                                      lane, g.nth, NG, (int)A.ld, A.J0, A.J1, A.J2);

    // ---- histogram of the new keys (warp-aggregated) -----------------------
    if (A.histogram) {
        int hk = (p < n) ? key : -1;
        unsigned peers = __match_any_sync(FULL, hk);
        if (hk >= 0 && lane == __ffs(peers) - 1) atomicAdd(A.count + hk, __popc(peers));
    }
    if (A.cnt9) {
        // old cell = start cell (i0, j0); the key is the new cell; lanes match
        // on cell * 9 + direction (32-bit: see the FP32 push)
        const bool counted = p < n && dep && key >= 0 && key < ncell;
        const int c0 = j0 * g.nr + i0;
        const int dir = (dj + 1) * 3 + min(max(i0 + di, 0), g.nr - 1) - i0 + 1;  // the key's column is clamped
        const unsigned mk = counted ? (unsigned)c0 * 9u + (unsigned)dir : 0xffffffffu;
        const unsigned peers = __match_any_sync(FULL, mk);
        if (counted && lane == __ffs(peers) - 1) atomicAdd(A.cnt9 + (int64_t)dir * ncell + c0, (int)__popc(peers));
    }
}

}  // namespace

static Push64Args push64_args(grpic_ctx *ctx, const grpic_particles *in, grpic_particles *p, const int32_t *perm,
                              const int32_t *live, int32_t *cnt9, grpic_fields *f, bool histogram)
{
    Push64Args A;
    A.g = ctx->g;
    A.dt = ctx->prm.dt;
    const double idt = 1.0 / ctx->prm.dt, m_i2dt = -0.5 / ctx->prm.dt;
    A.n_iter = ctx->prm.n_push_iter;
    A.pairs = A.n_iter >= 2 && A.dt <= PAIR_MAX_DT;
    A.hf = (float)(0.5 * A.dt);
    A.a_df = df_const(ctx->g.a);
    A.a2_df = df_const(ctx->g.a * ctx->g.a);
    A.dt_df = df_const(A.dt);
    for (int k = 0; k < 4; ++k) {
        A.qm[k] = ctx->prm.q_over_m[k];
        A.massive[k] = ctx->prm.massive[k];
        A.qdt[k] = 0.5 * A.qm[k] * A.dt;
        A.wr[k] = ctx->prm.q_weight[k] * m_i2dt;
        A.wp[k] = ctx->prm.q_weight[k] * idt;
    }
    A.n = p->n;
    A.d_count = p->d_count;
    A.r = (double *)p->x1;
    A.th = (double *)p->x2;
    A.u1 = (double *)p->u1;
    A.u2 = (double *)p->u2;
    A.u3 = (double *)p->u3;
    A.tag = p->tag;
    A.perm = perm;
    A.live = live;
    A.count_out = perm ? p->d_count : nullptr;
    A.cnt9 = perm ? cnt9 : nullptr;
    A.in_r = (const double *)in->x1;
    A.in_th = (const double *)in->x2;
    A.in_u1 = (const double *)in->u1;
    A.in_u2 = (const double *)in->u2;
    A.in_u3 = (const double *)in->u3;
    A.in_tag = in->tag;
    A.D0 = (const double *)f->D[0];
    A.D1 = (const double *)f->D[1];
    A.D2 = (const double *)f->D[2];
    A.B0 = (const double *)f->B[0];
    A.B1 = (const double *)f->B[1];
    A.B2 = (const double *)f->B[2];
    A.J0 = (double *)f->J[0];
    A.J1 = (double *)f->J[1];
    A.J2 = (double *)f->J[2];
    A.ld = f->ld;
    A.keys = ctx->d_keys;
    A.count = ctx->d_count;
    A.histogram = histogram ? 1 : 0;
    A.pusher = ctx->prm.pusher;
    A.radiation = ctx->prm.radiation;
    A.gamma_thr = ctx->prm.gamma_thr;
    A.eps_ph = ctx->prm.eps_ph;
    A.pconv = 1.0 - std::exp(-ctx->prm.tau * ctx->prm.dt);
    A.gthr2f = std::nextafter((float)(ctx->prm.gamma_thr * ctx->prm.gamma_thr), 0.0f);
    A.seed = ctx->prm.seed;
    A.step = ctx->step_count;
    A.spawn = ctx->prm.radiation ? ctx->d_spawn : nullptr;
    A.status = ctx->d_status;
    A.tape = nullptr;
    A.tape_ld = 0;
    return A;
}

cudaError_t launch_push64(grpic_ctx *ctx, const grpic_particles *in, grpic_particles *p, const int32_t *perm,
                          const int32_t *live, int32_t *cnt9, grpic_fields *f, bool histogram, cudaStream_t s,
                          int64_t slot0)
{
    Push64Args A = push64_args(ctx, in, p, perm, live, cnt9, f, histogram);
    A.keys = ctx->d_keys + slot0;
    if (p->n <= 0) return cudaSuccess;
    int64_t blocks = (p->n + PUSH64_T - 1) / PUSH64_T;
    const bool rad = ctx->prm.radiation != 0;
    if (ctx->prm.shape_order == 3) {
        if (rad)
            push64_kernel<3, true, false><<<(unsigned)blocks, PUSH64_T, 0, s>>>(A);
        else
            push64_kernel<3, false, false><<<(unsigned)blocks, PUSH64_T, 0, s>>>(A);
    } else {
        if (rad)
            push64_kernel<1, true, false><<<(unsigned)blocks, PUSH64_T, 0, s>>>(A);
        else
            push64_kernel<1, false, false><<<(unsigned)blocks, PUSH64_T, 0, s>>>(A);
    }
    return cudaGetLastError();
}

cudaError_t launch_push64_tape(grpic_ctx *ctx, grpic_particles *p, grpic_fields *f, double *tape, int64_t tape_ld,
                               cudaStream_t s)
{
    if (ctx->prm.shape_order != 1 || ctx->prm.radiation || ctx->prm.pusher != 0 || tape_ld < p->n)
        return cudaErrorInvalidValue;
    Push64Args A = push64_args(ctx, p, p, nullptr, nullptr, nullptr, f, false);
    A.tape = tape;
    A.tape_ld = tape_ld;
    if (p->n <= 0) return cudaSuccess;
    push64_kernel<1, false, true><<<(unsigned)((p->n + PUSH64_T - 1) / PUSH64_T), PUSH64_T, 0, s>>>(A);
    return cudaGetLastError();
}

}  // namespace grpic
