// grpic_field.cu -- semi-implicit D/B field update (arXiv:2503.04558 Sec. 2.1,
// Eqs. fld-predictor and fld-corrector; discrete forms of App. B).
//
// A stage (the predictor, then n_field_iter correctors) evaluates the auxiliary
// fields E_i, H_i from the current iterate (Eqs. auxE, auxH: metric products
// formed first, then the two-point averages), the circulations C_H, C_E (Eqs.
// D-update, B-update) and the new iterate:
//   predictor:  X~ = X^n + dt (C(X^n) - J),  C(X^n) kept for the correctors
//   corrector:  X  = X^n + dt (alpha_s C(X^n) + beta_s C(X~)) - dt J
// The boundary conditions are applied inside the stage: the guard columns are
// zero-derivative copies of the first and last physical columns, D^phi and
// B^theta are zero on the axis, D^r on the axis uses only the interior H_phi
// edge over the half-width face (Eq. Dr-axis); the last stage multiplies by the
// outer damping factor before the copy.  J holds the integrated currents J A
// (the deposit output) and is divided by the face areas here.
#include "grpic_internal.cuh"
#include "grpic_geo.cuh"

#include <algorithm>

namespace grpic {
namespace {

// ---------------------------------------------------------------------------
// Both kernels below form every quantity once per point and stage and pass it
// to the neighbours through shared memory: first the products whose column
// neighbours the auxiliary fields average (products()), then the auxiliary
// fields E_i, H_i themselves (auxiliary()), then the circulations (circulation()),
// so no table value of a neighbour is read.
//
// FP64: the predictor leaves the part of a corrector's circulation that does not
// change, alpha_s circ(X^n) - J, and a corrector is
//   X^n + (dt / A) (beta_s circ(X) + that),
// one rounding of X's size per stage.  56 operations per point and stage (122 when
// each point evaluated its neighbours' auxiliary fields and combined X^n, C^n and J
// in every stage; 52 with X^n folded in too, whose second rounding left B^r 1.4
// times further from 64 bits' value at 128^2).
//
// FP32: the order of the roundings is fixed, operation by operation:
//   products t x of a pair: fma(own t, own x, round(neighbour's t x)), halved;
//   auxiliary fields: fma(t, x, half pair), then -+ the second half pair;
//   C = round(circ / A), Jd = round(J / A);
//   predictor: fma(dt, C - Jd, X^n);
//   corrector: fma(-Jd, dt, fma(dt, m, X^n)), m = alpha_s C^n + beta_s C with one of
//   the products inside the fused multiply-add (FieldArgs::lead).
// A step's currents amplify the last bit of the fields: next to the axis J^phi is
// decided by a few particles, and a field off by one rounding moves them by up to
// 1e-3 of their size.  With the order fixed a run's fields are the same bits on
// every launch shape, and the same as before the shapes were changed.  (Folding
// alpha_s, J and dt / A into a base as in FP64: 0.63 ms an update at 2048^2, but two
// steps at that size then ended with J^phi 2.4e-4 off.)
// One update (8 stages): FP32 2048^2 1.29 -> 0.81 ms, FP64 1024^2 2.44 -> 1.21
// ms; FP64 128^2 0.128 -> 0.066 ms.
template <typename T>
struct FieldArgs {
    int nr, nth, ldt, ld;
    size_t slab;
    T dt, as, bs, dth;
    const T *tab;
    const T *col1d;  // dr_prim, dr_dual, damp_int, damp_half
    const T *Xi[6];  // the iterate at the launch's first stage
    T *Xo[6];        // the iterate after its last one
    T *Bs[6];        // FP64: alpha_s circ(X^n) - J; FP32: C^n, times alpha_s if `lead`
                     // (written by the first launch, read by the others)
    const T *Xn[6];  // X^n for the launches after the first
    T *Xs[6];        // FP32 tiles: a copy of X^n, written by the first launch
    const T *J[3];
    int lead;        // FP32: fma(beta_s, C, alpha_s C^n), else fma(alpha_s, C^n, beta_s C)
    int j_lo, j_hi;  // the rows updated
    int rows;        // strip kernel: rows per CTA
    int ns;          // tile kernel: stages of this launch
    int ahead;       // tile kernel: CTAs running at a time
    int last;        // the last stage is damped
    int carry;       // strip kernel: copy the rows next to the range to the next iterate
};

__host__ __device__ constexpr bool half_r(int k) { return k == 0 || k == 4 || k == 5; }
__host__ __device__ constexpr bool half_t(int k) { return k == 1 || k == 3 || k == 5; }

// own-point coefficients of the products (0..7) and auxiliary fields (8..13),
// and the inverse areas
__host__ __device__ constexpr int coef(int k)
{
    constexpr int t[14] = {T_AGRP_BP, T_SGB_DP,  T_AGRP_BR, T_SGB_DT,  T_AGRP_DP, T_SGB_BP,  T_AGRP_DR,
                           T_SGB_BT,  T_AGRR_BR, T_AGTT_BT, T_AGPP_BP, T_AGRR_DR, T_AGTT_DT, T_AGPP_DP};
    return t[k];
}
__host__ __device__ constexpr int inv_area(int k)
{
    constexpr int t[6] = {T_INV_ADR, T_INV_ADT, T_INV_ADP, T_INV_ABR, T_INV_ABT, T_INV_ABP};
    return t[k];
}

// alpha gamma_rph B^ph, sqrt(gamma) beta D^ph, alpha gamma_rph B^r - sqrt(gamma) beta D^th,
// alpha gamma_rph D^ph, sqrt(gamma) beta B^ph, alpha gamma_rph D^r + sqrt(gamma) beta B^th,
// each at its own location, into S[q * n + e]
template <typename T>
__device__ __forceinline__ void products(const T *K, const T *X, T *S, int n, int e)
{
    S[e] = K[0] * X[5];
    S[n + e] = K[1] * X[2];
    S[2 * n + e] = fmat(K[2], X[3], -K[3] * X[1]);
    S[3 * n + e] = K[4] * X[2];
    S[4 * n + e] = K[5] * X[5];
    S[5 * n + e] = fmat(K[6], X[0], K[7] * X[4]);
}

// H_r, H_th, H_ph, E_r, E_th, E_ph (App. B) into E[q * m + o]; el, er: the
// column neighbours' places in S
template <typename T>
__device__ __forceinline__ void auxiliary(const T *K, const T *X, const T *S, int n, int el, int er, T *E, int m, int o)
{
    const T h = T(0.5);
    E[o] = fmat(h, fmat(K[0], X[5], S[el]), K[8] * X[3]);
    E[m + o] = fmat(h, fmat(K[1], X[2], S[n + er]), K[9] * X[4]);
    E[2 * m + o] = fmat(h, fmat(K[2], X[3], fmat(-K[3], X[1], S[2 * n + er])), K[10] * X[5]);
    E[3 * m + o] = fmat(h, fmat(K[4], X[2], S[3 * n + er]), K[11] * X[0]);
    E[4 * m + o] = fmat(-h, fmat(K[5], X[5], S[4 * n + el]), K[12] * X[1]);
    E[5 * m + o] = fmat(h, fmat(K[6], X[0], fmat(K[7], X[4], S[5 * n + el])), K[13] * X[2]);
}

// FP32: the same with every pair's products apart, K[0..7] halved
__device__ __forceinline__ void products(const float *K, const float *X, float *S, int n, int e)
{
    S[e] = K[0] * X[5];
    S[n + e] = K[1] * X[2];
    S[2 * n + e] = K[2] * X[3];
    S[3 * n + e] = K[3] * X[1];
    S[4 * n + e] = K[4] * X[2];
    S[5 * n + e] = K[5] * X[5];
    S[6 * n + e] = K[6] * X[0];
    S[7 * n + e] = K[7] * X[4];
}
__device__ __forceinline__ void auxiliary(const float *K, const float *X, const float *S, int n, int el, int er, float *E,
                                          int m, int o)
{
    E[o] = fmaf(K[8], X[3], fmaf(K[0], X[5], S[el]));
    E[m + o] = fmaf(K[9], X[4], fmaf(K[1], X[2], S[n + er]));
    E[2 * m + o] = __fsub_rn(fmaf(K[10], X[5], fmaf(K[2], X[3], S[2 * n + er])), fmaf(K[3], X[1], S[3 * n + er]));
    E[3 * m + o] = fmaf(K[11], X[0], fmaf(K[4], X[2], S[4 * n + er]));
    E[4 * m + o] = fmaf(K[12], X[1], -fmaf(K[5], X[5], S[5 * n + el]));
    E[5 * m + o] = __fadd_rn(fmaf(K[13], X[2], fmaf(K[6], X[0], S[6 * n + el])), fmaf(K[7], X[4], S[7 * n + el]));
}
template <typename T>
constexpr int N_PROD = sizeof(T) == 4 ? 8 : 6;
// a coefficient as the products take it
template <typename T>
__device__ __forceinline__ T coef_value(int k, T v)
{
    return sizeof(T) == 4 && k < 8 ? T(0.5) * v : v;
}

// the circulations of Eqs. D-update, B-update (not yet divided by the areas)
// from the auxiliary fields at the point o, its column neighbours l, r and its
// row neighbours d (below), u (above).  Beyond the axis rows H_phi is zero (its
// tables are), which leaves D^r there the one edge of Eq. Dr-axis.
template <typename T>
__device__ __forceinline__ void circulation(const T *E, int m, int o, int l, int r, int d, int u, T dth, T drp, T drd,
                                            T *C)
{
    const T hp = E[2 * m + o], ep = E[5 * m + o];
    C[0] = hp - E[2 * m + d];
    C[1] = E[2 * m + l] - hp;
    C[2] = fmat(E[m + o] - E[m + l], dth, (E[d] - E[o]) * drd);
    C[3] = ep - E[5 * m + u];
    C[4] = E[5 * m + r] - ep;
    C[5] = fmat(E[4 * m + o] - E[4 * m + r], dth, (E[3 * m + u] - E[3 * m + o]) * drp);
}

// FP32: the predictor at one component (J: its current, 0 for B), X^n -> X~; Q: C^n
// as the correctors take it, Jd: J / A
__device__ __forceinline__ void predict(float C, float W, float J, const FieldArgs<float> &A, float &X, float &Q, float &Jd)
{
    const float Cn = __fmul_rn(C, W);
    Jd = __fmul_rn(J, W);
    Q = A.lead ? __fmul_rn(A.as, Cn) : Cn;
    X = fmaf(A.dt, __fsub_rn(Cn, Jd), X);
}
// ... and a corrector
__device__ __forceinline__ float correct(float C, float W, float Q, float Xn, float Jd, const FieldArgs<float> &A)
{
    const float c = __fmul_rn(C, W);
    const float m = A.lead ? fmaf(A.bs, c, Q) : fmaf(A.as, Q, __fmul_rn(A.bs, c));
    return fmaf(-Jd, A.dt, fmaf(A.dt, m, Xn));
}

// FP64: the predictor at one component, X^n -> X~; Q: alpha_s circ^n - J, what the
// correctors add to beta_s circ
__device__ __forceinline__ void predict(double C, double W, double J, const FieldArgs<double> &A, double &X, double &Q)
{
    Q = fma(A.as, C, -J);
    X = fma(C - J, A.dt * W, X);
}
// ... and beta_s circ + Q of a corrector (bd, bp, br: beta_s times dth, drp, drd)
__device__ __forceinline__ void circulation_on(const double *E, int m, int o, int l, int r, int d, int u, double bs,
                                               double bd, double bp, double br, const double *Q, double *C)
{
    const double hp = E[2 * m + o], ep = E[5 * m + o];
    C[0] = fma(bs, hp - E[2 * m + d], Q[0]);
    C[1] = fma(bs, E[2 * m + l] - hp, Q[1]);
    C[2] = fma(E[m + o] - E[m + l], bd, fma(E[d] - E[o], br, Q[2]));
    C[3] = fma(bs, ep - E[5 * m + u], Q[3]);
    C[4] = fma(bs, E[5 * m + r] - ep, Q[4]);
    C[5] = fma(E[4 * m + o] - E[4 * m + r], bd, fma(E[3 * m + u] - E[3 * m + o], bp, Q[5]));
}

// one component's new value at (i, j) with the guard copies of the first and
// last physical columns
template <typename T>
__device__ __forceinline__ void put_value(T *row, int c, int i, int last, int ldt, T v)
{
    row[c] = v;
    if (i == 0) row[0] = row[1] = v;
    if (i == last)
        for (int g = c + 1; g < ldt; ++g) row[g] = v;
}

// NS consecutive stages per launch on a BW x BH tile of points, P of them per
// thread (a fixed column, rows RS apart): the points' iterate, inverse areas and
// coefficients stay in registers over the launch, X^n, C^n and J / A in shared
// memory (each thread reads its own).  A stage reads one point beyond the one it
// writes, so the outer NS points of the tile are a halo that neighbouring CTAs
// compute too.  The first launch leaves a copy of X^n for the later ones, so that
// the last one can write the caller's arrays.  Points that a component does not
// update (rows beyond the axis) carry W = 0 and X^n = 0; guard columns are set from
// the physical ones after each stage.  FP32 only: issue and the loads at a tile's
// start bound it (the next tile's lines are asked for ahead); FP64 is bound by its
// pipe, which the halo's second computation would load.
template <int BW, int BH, int P, int NS, int MINB, bool FIRST>
__global__ void __launch_bounds__(BW *BH / P, MINB) field_tile_kernel(const __grid_constant__ FieldArgs<float> A)
{
    constexpr int NT = BW * BH / P, RS = NT / BW, OW = BW - 2 * NS, OH = BH - 2 * NS, BOX = BW * BH;
    static_assert(NT % BW == 0 && NT % 32 == 0, "a thread's points share their column");
    extern __shared__ __align__(16) unsigned char field_smem[];
    float *const S = reinterpret_cast<float *>(field_smem);
    float *const E = S + N_PROD<float> * BOX;
    float *const Q = E + 6 * BOX;    // C^n as the correctors take it
    float *const XN = Q + 6 * BOX;   // X^n
    float *const JD = XN + 6 * BOX;  // J / A
    float *const Gd = JD + 3 * BOX;  // guard copies, 12 x BH
    const int nr = A.nr, nth = A.nth;
    const int bc = threadIdx.x % BW, br0 = threadIdx.x / BW;
    const int c0 = (int)blockIdx.x * OW - NS, r0 = A.j_lo + (int)blockIdx.y * OH - NS;
    const int c = c0 + bc, i = c - NG;
    const bool col_in = c >= 0 && c < A.ldt;
    const bool ph_i = i >= 0 && i <= nr, ph_h = i >= 0 && i <= nr - 1;  // integer, half-r components
    float drp = 0.0f, drd = 0.0f, dmi = 1.0f, dmh = 1.0f;
    if (col_in) {
        drp = __ldg(A.col1d + c);
        drd = __ldg(A.col1d + A.ldt + c);
        dmi = __ldg(A.col1d + 2 * A.ldt + c);
        dmh = __ldg(A.col1d + 3 * A.ldt + c);
    }
    // the lines of the tile that this SM is likely to take next, into L2
    for (int t = threadIdx.x; t < (FIRST ? 26 : 41) * BH; t += NT) {
        const int next = (int)(blockIdx.y * gridDim.x + blockIdx.x) + A.ahead, q = t / BH;
        const int j = next / (int)gridDim.x * OH - NS + t % BH, col = max(next % (int)gridDim.x * OW - NS, 0);
        if (j < 0 || j > nth) continue;
        const float *row = q < 20   ? A.tab + (q < 6 ? q : q + 6) * A.slab + (unsigned)(j * A.ldt)
                           : q < 26 ? A.Xi[q - 20] + (unsigned)(j * A.ld)
                           : q < 32 ? A.Bs[q - 26] + (unsigned)(j * A.ld)
                           : q < 38 ? A.Xn[q - 32] + (unsigned)(j * A.ld)
                                    : A.J[q - 38] + (unsigned)(j * A.ld);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(col, A.ldt - 1)));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(col + 32, A.ldt - 1)));
    }
    float X[P][6], W[P][6], K[P][14];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int j = r0 + br0 + p * RS, e = threadIdx.x + p * NT;
        const bool in = col_in && j >= 0 && j <= nth, axis = j == 0 || j == nth;
        const unsigned q = (unsigned)(j * A.ld + c), qt = (unsigned)(j * A.ldt + c);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const bool row = in && !(half_t(k) && j == nth);
            const bool upd = row && (half_r(k) ? ph_h : ph_i) && !((k == 2 || k == 4) && axis);
            X[p][k] = row ? __ldg(A.Xi[k] + q) : 0.0f;
            W[p][k] = upd ? __ldg(A.tab + inv_area(k) * A.slab + qt) : 0.0f;
            XN[k * BOX + e] = !upd ? 0.0f : (FIRST ? X[p][k] : __ldg(A.Xn[k] + q));
            if (!FIRST) {
                Q[k * BOX + e] = upd ? __ldg(A.Bs[k] + q) : 0.0f;
                if (k < 3) JD[k * BOX + e] = upd ? __fmul_rn(__ldg(A.J[k < 3 ? k : 0] + q), W[p][k]) : 0.0f;
            }
        }
#pragma unroll
        for (int k = 0; k < 14; ++k) K[p][k] = in ? coef_value(k, __ldg(A.tab + coef(k) * A.slab + qt)) : 0.0f;
    }
    const int dl = bc > 0 ? 1 : 0, dr = bc < BW - 1 ? 1 : 0;
    const int dd = br0 > 0 ? BW : 0, du = br0 < RS - 1 ? BW : 0;  // of a thread's first and last point
    auto fields = [&]() {
#pragma unroll
        for (int p = 0; p < P; ++p) products(K[p], X[p], S, BOX, (int)threadIdx.x + p * NT);
        __syncthreads();
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int e = threadIdx.x + p * NT;
            auxiliary(K[p], X[p], S, BOX, e - dl, e + dr, E, BOX, e);
        }
        __syncthreads();
    };
    auto circ_of = [&](int p, float(&C)[6]) {
        const int e = threadIdx.x + p * NT;
        circulation(E, BOX, e, e - dl, e + dr, e - (p == 0 ? dd : BW), e + (p == P - 1 ? du : BW), A.dth, drp, drd, C);
    };
    // guard columns i = -1, n_r (half-r components) and n_r + 1: zero-derivative
    // copies of the first / last physical column
    const bool edge = c0 <= NG || c0 + BW > nr + NG;  // the tile holds some
    auto guards = [&]() {
        if (!edge) return;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int br = br0 + p * RS;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                if (i == 0) Gd[k * BH + br] = X[p][k];
                if (i == (half_r(k) ? nr - 1 : nr)) Gd[(6 + k) * BH + br] = X[p][k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int br = br0 + p * RS;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                if (i == -1) X[p][k] = Gd[k * BH + br];
                if (i == nr + 1 || (i == nr && half_r(k))) X[p][k] = Gd[(6 + k) * BH + br];
            }
        }
    };
    int st = 0;
    if constexpr (FIRST) {
        fields();
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int j = r0 + br0 + p * RS, e = threadIdx.x + p * NT;
            float C[6];
            circ_of(p, C);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                float J = 0.0f, q, jd;
                if (k < 3 && W[p][k] != 0.0f) J = __ldg(A.J[k < 3 ? k : 0] + (unsigned)(j * A.ld + c));
                predict(C[k], W[p][k], J, A, X[p][k], q, jd);
                if ((k == 2 || k == 4) && (j == 0 || j == nth)) X[p][k] = 0.0f;  // D^ph, B^th on the axis
                Q[k * BOX + e] = q;
                if (k < 3) JD[k * BOX + e] = jd;
            }
        }
        if (++st < A.ns) guards();
    }
    while (st < A.ns) {
        fields();
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int e = threadIdx.x + p * NT;
            float C[6];
            circ_of(p, C);
#pragma unroll
            for (int k = 0; k < 6; ++k)
                X[p][k] = correct(C[k], W[p][k], Q[k * BOX + e], XN[k * BOX + e], k < 3 ? JD[(k < 3 ? k : 0) * BOX + e] : 0.0f, A);
        }
        if (++st < A.ns) guards();
    }
    if (A.last)
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int k = 0; k < 6; ++k) X[p][k] *= half_r(k) ? dmh : dmi;
    // the tile without its halo to global memory
    if (bc < NS || bc >= NS + OW || !ph_i) return;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int br = br0 + p * RS, j = r0 + br, e = threadIdx.x + p * NT;
        if (br < NS || br >= NS + OH || j > nth) continue;
        const size_t row = (size_t)j * A.ld;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            if ((half_r(k) && !ph_h) || (half_t(k) && j == nth)) continue;
            put_value(A.Xo[k] + row, c, i, half_r(k) ? nr - 1 : nr, A.ldt, X[p][k]);
            if (FIRST && A.Xs[k]) {
                A.Bs[k][row + c] = Q[k * BOX + e];
                A.Xs[k][row + c] = XN[k * BOX + e];
            }
        }
    }
}

// One stage per launch on strips of BW - 2 columns: a CTA of BW x RT threads
// walks down A.rows rows, RT at a time, the auxiliary fields of the last rows
// kept in a ring in shared memory, so that only one row at each end and two
// columns are computed twice.  The next rows' loads and the update's are issued
// ahead of the arithmetic that hides them (FP64 1024^2: 1.49 -> 1.25 ms).  For
// FP64 (bound by the FP64 pipe), for row ranges and, in FP32, on request.
template <typename T, int BW, int RT, int RES, bool FIRST>
__global__ void __launch_bounds__(BW *RT, RES) field_strip_kernel(const __grid_constant__ FieldArgs<T> A)
{
    constexpr int RING = RT <= 2 ? 4 : (RT <= 6 ? 8 : 16), NE = BW * RING, NP = BW * RT;
    static_assert(RING >= RT + 2, "the update reads two rows above the new ones");
    __shared__ T S[N_PROD<T> * NP], E[6 * NE];
    const int nr = A.nr, nth = A.nth;
    const int bc = threadIdx.x % BW, rt = threadIdx.x / BW;
    const int c = (int)blockIdx.x * (BW - 2) - 1 + bc, i = c - NG;
    const int ja = A.j_lo + (int)blockIdx.y * A.rows, jb = min(ja + A.rows, A.j_hi);  // rows [ja, jb)
    const bool col_in = c >= 0 && c < A.ldt;
    const bool ph_i = i >= 0 && i <= nr, ph_h = i >= 0 && i <= nr - 1;
    const bool mine = bc >= 1 && bc <= BW - 2 && ph_i;
    T drp = T(0), drd = T(0), dmi = T(1), dmh = T(1);
    if (col_in) {
        drp = __ldg(A.col1d + c);
        drd = __ldg(A.col1d + A.ldt + c);
        if (A.last) {
            dmi = __ldg(A.col1d + 2 * A.ldt + c);
            dmh = __ldg(A.col1d + 3 * A.ldt + c);
        }
    }
    const int el = threadIdx.x - (bc > 0 ? 1 : 0), er = threadIdx.x + (bc < BW - 1 ? 1 : 0);
    T X[6], K[14];
    auto load = [&](int j) {
        const bool in = col_in && j >= 0 && j <= nth && j <= jb;
        const unsigned q = (unsigned)(j * A.ld + c), qt = (unsigned)(j * A.ldt + c);
#pragma unroll
        for (int k = 0; k < 6; ++k) X[k] = in && !(half_t(k) && j == nth) ? __ldg(A.Xi[k] + q) : T(0);
#pragma unroll
        for (int k = 0; k < 14; ++k) K[k] = in ? coef_value(k, __ldg(A.tab + coef(k) * A.slab + qt)) : T(0);
    };
    load(ja - 1 + rt);
    for (int jt = ja - 1; jt <= jb; jt += RT) {
        const int j = jt + rt;
        // the row this thread updates: the one below, whose neighbours'
        // auxiliary fields are complete after this round
        const int ju = j - 1;
        const bool upd = mine && ju >= ja && ju < jb, axis = ju == 0 || ju == nth;
        const unsigned q = (unsigned)(ju * A.ld + c);
        T W[6], B[6], XN[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const bool on = upd && !(half_r(k) && !ph_h) && !(half_t(k) && ju == nth) && !((k == 2 || k == 4) && axis);
            W[k] = on ? __ldg(A.tab + inv_area(k) * A.slab + (unsigned)(ju * A.ldt + c)) : T(0);
            B[k] = on ? __ldg((FIRST ? A.Xi[k] : A.Bs[k]) + q) : T(0);  // X^n or what the predictor left
        }
        if (A.carry && (j == A.j_lo - 1 || j == A.j_hi) && j <= jb && j >= 0 && j <= nth && col_in && bc >= 1 &&
            bc <= BW - 2) {
#pragma unroll
            for (int k = 0; k < 6; ++k)
                if (!(half_t(k) && j == nth)) A.Xo[k][(size_t)j * A.ld + c] = X[k];
        }
        products(K, X, S, NP, (int)threadIdx.x);
        __syncthreads();
        auxiliary(K, X, S, NP, el, er, E, NE, ((j + 1) & (RING - 1)) * BW + bc);
        load(j + RT);
        // (X^n here, where the coefficients' registers are free, not with W and B: FP64
        // 512^2 0.46 -> 0.40 ms)
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const bool on = upd && !(half_r(k) && !ph_h) && !(half_t(k) && ju == nth) && !((k == 2 || k == 4) && axis);
            if (!FIRST) XN[k] = on ? __ldg(A.Xn[k] + q) : T(0);
        }
        __syncthreads();
        if (upd) {
            const int o = (j & (RING - 1)) * BW + bc;
            const int d = (ju & (RING - 1)) * BW + bc, u = ((j + 1) & (RING - 1)) * BW + bc;
            T C[6];
            if constexpr (FIRST || sizeof(T) == 4)
                circulation(E, NE, o, o - 1, o + 1, d, u, A.dth, drp, drd, C);
            else
                circulation_on(E, NE, o, o - 1, o + 1, d, u, A.bs, A.bs * A.dth, A.bs * drp, A.bs * drd, B, C);
            const size_t row = (size_t)ju * A.ld;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                if ((half_r(k) && !ph_h) || (half_t(k) && ju == nth)) continue;
                T v, b = T(0);
                T J = T(0);
                if ((FIRST || sizeof(T) == 4) && k < 3) J = __ldg(A.J[k < 3 ? k : 0] + q);
                if constexpr (FIRST) {
                    v = B[k];
                    if constexpr (sizeof(T) == 4) {
                        float jd;
                        predict(C[k], W[k], J, A, v, b, jd);
                    } else {
                        predict(C[k], W[k], J, A, v, b);
                    }
                    if ((k == 2 || k == 4) && axis) v = b = T(0);
                } else {
                    if constexpr (sizeof(T) == 4)
                        v = correct(C[k], W[k], B[k], XN[k], __fmul_rn(J, W[k]), A);
                    else
                        v = fma(C[k], A.dt * W[k], XN[k]);
                    if ((k == 2 || k == 4) && axis) v = T(0);
                }
                if (A.last) v *= half_r(k) ? dmh : dmi;
                put_value(A.Xo[k] + row, c, i, half_r(k) ? nr - 1 : nr, A.ldt, v);
                if (FIRST && !A.last) A.Bs[k][row + c] = b;
            }
        }
    }
}

template <typename T>
T *fslot(grpic_ctx *ctx, int k, int64_t ld)
{
    size_t n = (size_t)(ctx->g.nth + 1) * ld;
    return (T *)ctx->fscratch + (size_t)k * n;
}

// a launch shape of the tile kernel
template <int BW, int BH, int P, int NS, int MINB>
struct Tiles {
    static constexpr int OW = BW - 2 * NS, OH = BH - 2 * NS, threads = BW * BH / P, stages = NS;
    static constexpr int smem = ((N_PROD<float> + 6 + 15) * BW * BH + 12 * BH) * (int)sizeof(float);
    static dim3 grid(const FieldArgs<float> &A) { return dim3((A.ldt + OW - 1) / OW, (A.j_hi - A.j_lo + OH - 1) / OH); }
    static cudaError_t setup(FieldArgs<float> &A, int sms)
    {
        A.ahead = sms * MINB;
        cudaError_t e = cudaFuncSetAttribute(field_tile_kernel<BW, BH, P, NS, MINB, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return e ? e : cudaFuncSetAttribute(field_tile_kernel<BW, BH, P, NS, MINB, false>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    }
    static void launch(const FieldArgs<float> &A, bool first, cudaStream_t s)
    {
        if (first)
            field_tile_kernel<BW, BH, P, NS, MINB, true><<<grid(A), threads, smem, s>>>(A);
        else
            field_tile_kernel<BW, BH, P, NS, MINB, false><<<grid(A), threads, smem, s>>>(A);
    }
};

// A launch shape of the strip kernel.  The rows per CTA are those for which the
// fullest SM has the least to do: each of its CTAs forms the auxiliary fields of
// rows + 2 rows (28 operations a point) and updates `rows` of them (28; the rule
// takes 24, which measured the same or better), in
// (rows + 2) / RT rounds whose latency (about ROUND operations' time) CTAs
// resident together hide from each other.  So long strips on large grids (few
// halo rows) and one short round, spread over all SMs, on small ones.
template <typename T, int BW, int RT, int RES>
struct Strips {
    static constexpr int stages = 1, ROUND = 3000;
    static dim3 grid(const FieldArgs<T> &A)
    {
        return dim3((A.ldt + BW - 3) / (BW - 2), (A.j_hi - A.j_lo + A.rows - 1) / A.rows);
    }
    static int64_t cost(int ldt, int rows, int sms, int &best)
    {
        const int64_t nx = (ldt + BW - 3) / (BW - 2);
        int64_t least = INT64_MAX;
        for (int r = std::max(RT - 2, 1); r < 96; r += RT) {
            const int64_t per_sm = (nx * ((rows + r - 1) / r) + sms - 1) / sms;
            const int64_t c = per_sm * BW * (28 * (r + 2) + 24 * r) + (per_sm + RES - 1) / RES * ((r + 2) / RT) * ROUND;
            if (c < least) {
                least = c;
                best = r;
            }
        }
        return least;
    }
    static cudaError_t setup(FieldArgs<T> &A, int sms)
    {
        cost(A.ldt, A.j_hi - A.j_lo, sms, A.rows);
        return cudaSuccess;
    }
    static void launch(const FieldArgs<T> &A, bool first, cudaStream_t s)
    {
        if (first)
            field_strip_kernel<T, BW, RT, RES, true><<<grid(A), BW * RT, 0, s>>>(A);
        else
            field_strip_kernel<T, BW, RT, RES, false><<<grid(A), BW * RT, 0, s>>>(A);
    }
};

// The update of rows [j_lo, j_hi) of X (D, then B; in place) with currents J
// by launches of the shape SH: the rows outside are left as they are and feed
// the range's edge rows in every stage (their two neighbours go along with the
// iterates).  Y: nullptr, or every stage's own output arrays
// (SH::stages == 1; X is then not written).  Without correctors the step is
// the forward-Euler predictor alone, undamped.  lead: FieldArgs.
template <typename T, typename SH>
cudaError_t run_field(grpic_ctx *ctx, T *const X[6], T *const J[3], int64_t ld, const T *tab, const T *col1d,
                      cudaStream_t s, int j_lo, int j_hi, T *const *Y = nullptr, bool lead = false)
{
    const int N = ctx->prm.n_field_iter;
    FieldArgs<T> A;
    A.nr = ctx->g.nr;
    A.nth = ctx->g.nth;
    A.ldt = ctx->g.ld_tab;
    A.ld = (int)ld;
    A.slab = ctx->slab;
    A.dt = (T)ctx->prm.dt;
    A.as = (T)(1.0 - ctx->prm.beta_field);
    A.bs = (T)ctx->prm.beta_field;
    A.lead = lead;
    A.dth = (T)ctx->g.dth;
    A.tab = tab;
    A.col1d = col1d;
    A.j_lo = j_lo;
    A.j_hi = j_hi;
    A.rows = 0;
    const bool whole = j_lo == 0 && j_hi == ctx->g.nth + 1;
    for (int k = 0; k < 3; ++k) A.J[k] = J[k];
    const int launches = (N + SH::stages) / SH::stages;
    // A launch's halo reads the iterate at other CTAs' points, so it writes other
    // arrays.  Tiles: the iterate alternates between a buffer and, X^n being copied
    // by the first launch, the caller's arrays; strips: between two buffers, the
    // last stage writing the caller's (of X^n each thread reads its own point).
    constexpr bool tiles = SH::stages > 1;
    const bool in_buffer = !Y && (tiles ? launches % 2 == 1 : launches == 1);  // the result
    cudaError_t e = SH::setup(A, sm_count(ctx->device));
    for (int l = 0; l < launches && e == cudaSuccess; ++l) {
        const bool last = l == launches - 1;
        A.last = last && N > 0;
        A.carry = !tiles && !whole && !last;
        A.ns = std::min(SH::stages, N + 1 - l * SH::stages);
        for (int k = 0; k < 6; ++k) {
            T *const buf[2] = {fslot<T>(ctx, 6 + k, ld), fslot<T>(ctx, 12 + k, ld)};
            A.Bs[k] = fslot<T>(ctx, k, ld);
            if (tiles) {
                A.Xi[k] = l % 2 ? buf[0] : X[k];
                A.Xo[k] = l % 2 ? X[k] : buf[0];
                A.Xn[k] = buf[1];
                A.Xs[k] = launches > 1 ? buf[1] : nullptr;
            } else {
                A.Xi[k] = l == 0 ? X[k] : (Y ? Y[6 * (l - 1) + k] : buf[(l - 1) & 1]);
                A.Xo[k] = Y ? Y[6 * l + k] : (last && l > 0 ? X[k] : buf[l & 1]);
                A.Xn[k] = X[k];
            }
        }
        SH::launch(A, l == 0, s);
        e = cudaGetLastError();
    }
    if (in_buffer)
        for (int k = 0; k < 6 && e == cudaSuccess; ++k) {
            const int hi = std::min(j_hi, ctx->g.nth + (half_t(k) ? 0 : 1));
            if (hi > j_lo)
                e = cudaMemcpy2DAsync(X[k] + (size_t)j_lo * ld, ld * sizeof(T),
                                      fslot<T>(ctx, 6 + k, ld) + (size_t)j_lo * ld, ld * sizeof(T),
                                      ctx->g.ld_tab * sizeof(T), hi - j_lo, cudaMemcpyDeviceToDevice, s);
        }
    return e;
}

using Strips64 = Strips<double, 64, 4, 2>;
using Narrow64 = Strips<double, 32, 8, 2>;
using Strips32 = Strips<float, 64, 4, 3>;
using Wide32 = Tiles<64, 24, 3, 4, 1>;
using Small32 = Tiles<32, 16, 1, 4, 2>;

cudaError_t run_field64(grpic_ctx *ctx, double *const X[6], double *const J[3], int64_t ld, cudaStream_t s, int j_lo,
                        int j_hi, double *const *Y = nullptr)
{
    const int sms = sm_count(ctx->device), ldt = ctx->g.ld_tab, rows = j_hi - j_lo;
    int r;
    return Strips64::cost(ldt, rows, sms, r) <= Narrow64::cost(ldt, rows, sms, r)
               ? run_field<double, Strips64>(ctx, X, J, ld, ctx->tab, ctx->col1d, s, j_lo, j_hi, Y)
               : run_field<double, Narrow64>(ctx, X, J, ld, ctx->tab, ctx->col1d, s, j_lo, j_hi, Y);
}

template <typename T>
struct FieldPtrs {
    T *X[6], *J[3];
    explicit FieldPtrs(const grpic_fields *f)
    {
        for (int k = 0; k < 3; ++k) {
            X[k] = (T *)f->D[k];
            X[3 + k] = (T *)f->B[k];
            J[k] = (T *)f->J[k];
        }
    }
};

}  // namespace

// The FP64 field update from Xn with currents J, every stage's output kept:
// Y[k][0..5] for k = 0 (predictor) .. N (the last corrector, damped) -- the
// iterates the adjoint needs to differentiate the update w.r.t. its tables.
// Xn is not modified; Y buffers are (nth+1) x ld each.
cudaError_t launch_field64_stages(grpic_ctx *ctx, double *const Xn[6], double *const J[3], double *const *Y,
                                  int64_t ld, cudaStream_t s)
{
    return run_field64(ctx, Xn, J, ld, s, 0, ctx->g.nth + 1, Y);
}

cudaError_t launch_field64(grpic_ctx *ctx, grpic_fields *f, cudaStream_t s, int j_lo, int j_hi)
{
    if (j_hi < 0) j_hi = ctx->g.nth + 1;
    const FieldPtrs<double> P(f);
    return run_field64(ctx, P.X, P.J, f->ld, s, j_lo, j_hi);
}

// Launches of four stages over the whole grid, of one stage over a row range
// (whose rows outside must not move between stages) or on request
// (grpic_set_field_path); the same operations per point either way.  Of the
// two tiles the wide one has the smaller halo; the small one is taken while
// the wide one's CTAs do not fill the SMs.
// Which product of the corrector's sum is inside the fused multiply-add
// (FieldArgs::lead) goes by the arrays: beta_s C on the whole grid with 16-byte
// rows and bases, alpha_s C^n elsewhere.  Both are equally good; these are the
// orders that runs on such arrays have always had, so a run that is continued or
// repeated keeps its bits.
cudaError_t launch_field32(grpic_ctx *ctx, grpic_fields *f, cudaStream_t s, int j_lo, int j_hi)
{
    const int rows = ctx->g.nth + 1, sms = sm_count(ctx->device);
    if (j_hi < 0) j_hi = rows;
    const FieldPtrs<float> P(f);
    const bool whole = j_lo == 0 && j_hi == rows;
    bool lead = whole && f->ld % 4 == 0;
    for (int k = 0; k < 6; ++k) lead = lead && (uintptr_t)P.X[k] % 16 == 0;
    if (!(ctx->field_fused && whole))
        return run_field<float, Strips32>(ctx, P.X, P.J, f->ld, ctx->tab32, ctx->col1d32, s, j_lo, j_hi, nullptr, lead);
    const int64_t wide = (int64_t)((ctx->g.ld_tab + Wide32::OW - 1) / Wide32::OW) * ((rows + Wide32::OH - 1) / Wide32::OH);
    return wide <= sms ? run_field<float, Small32>(ctx, P.X, P.J, f->ld, ctx->tab32, ctx->col1d32, s, j_lo, j_hi, nullptr,
                                                   lead)
                       : run_field<float, Wide32>(ctx, P.X, P.J, f->ld, ctx->tab32, ctx->col1d32, s, j_lo, j_hi, nullptr,
                                                  lead);
}

}  // namespace grpic
