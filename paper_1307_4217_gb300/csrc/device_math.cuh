// Device arithmetic of the formal solver (Sec. 3.2-3.3 of Stepan & Trujillo
// Bueno 2013): BESSER control points, the exponential-integral coefficients
// of the Bezier/DELO step, and the Hanle statistical-equilibrium solve (Eq. 2).
#pragma once
#include <cuda_runtime.h>

namespace porta {

// ---------------------------------------------------------------------------
// Coefficients of Eq. 7 for an upwind optical path t = tau_MO:
//   e = exp(-t),
//   psi'_M = (1 - e (1 + t)) / t,          psi'_O = (e + t - 1) / t,
//   w_M = (2 - e (t^2 + 2t + 2)) / t^2,    w_O = 1 - 2 (e + t - 1) / t^2,
//   w_C = 2 (t - 2 + e (t + 2)) / t^2      (Eqs. 9-13).
// Near t = 0 the closed forms lose digits to cancellation; polynomials in t take their place.
// ---------------------------------------------------------------------------
template <typename Real>
struct Coef {
    Real e, pm, po, wm, wo, wc;
};

// The linear-interpolation coefficients follow from the quadratic ones: a
// linear source on MO is the Bezier curve whose control point is the midpoint
// c_M = (y_M + y_O)/2, so psi'_M = w_M + w_C/2 and psi'_O = w_O + w_C/2 (all
// terms positive: no cancellation). Only the three w series are evaluated.

// reciprocal. In FP64, whose operations run at 2 lanes per cycle and SM here (1/64 of the FP32
// rate): the hardware's 20-bit approximation and two Newton steps, 4 of them, within an ulp
// for normal x. In FP32 the hardware approximation rcp.approx.ftz (max 1 ulp; the operands
// here are normal numbers below 2^126), since the FP32 form's error budget is 1e-5. The bare
// instruction saves the scaling steps of a general approximate division (4% of the J^K_Q
// sweep's time).
__device__ __forceinline__ double rcp(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}
__device__ __forceinline__ float rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Double precision. With q = w_O, h = t (1 - q) / 2 gives e0 = 1 - e = t (1 - h) and
// w_C = e0 - w_M - w_O. Below t = 1, w_M and w_O over t are polynomials minimax in relative
// error (Remez exchange on the Taylor series, 5e-17); above, the closed forms in e0. Every
// coefficient is within 2e-15 of its value. (26 operations, 34 and an exponential above,
// where Taylor series below 0.14 and 0.18 and the closed forms above took up to 60 and left
// 1e-13 at the crossover: 6% of the FP64 J^K_Q sweep's time.) e0 out: 1 - e.
__device__ __forceinline__ Coef<double> coefficients(double t, double &e0)
{
    Coef<double> c;
    if (t < 1.0) {
        double m = fma(t, -1.1202256902396886e-09, 1.9558584056821613e-08), o = fma(t, 2.1752747810916859e-10, -3.9450135294101958e-09);
        m = fma(t, m, -2.2723481708323534e-07);
        o = fma(t, o, 4.9804374537587804e-08);
        m = fma(t, m, 2.2524008032884722e-06);
        o = fma(t, o, -5.5090033985190619e-07);
        m = fma(t, m, -1.9839818101854985e-05);
        o = fma(t, o, 5.5113331078707397e-06);
        m = fma(t, m, 0.00015432036885733235);
        o = fma(t, o, -4.9603129765952493e-05);
        m = fma(t, m, -0.0010416664919878616);
        o = fma(t, o, 0.00039682538720382121);
        m = fma(t, m, 0.0059523809209458198);
        o = fma(t, o, -0.0027777777765696106);
        m = fma(t, m, -0.027777777774420587);
        o = fma(t, o, 0.016666666666588639);
        m = fma(t, m, 0.099999999999813557);
        o = fma(t, o, -0.083333333333331358);
        m = fma(t, m, -0.24999999999999592);
        o = fma(t, o, 0.33333333333333331);
        m = fma(t, m, 0.33333333333333331);
        c.wm = t * m;
        c.wo = t * o;
        const double ht = 0.5 * t;
        e0 = fma(-t, fma(-ht, c.wo, ht), t);
        c.e = 1.0 - e0;
        c.wc = (e0 - c.wm) - c.wo;
    } else {
        const double it = rcp(t);
        c.e = exp(-t);
        e0 = 1.0 - c.e;
        const double h2 = fma(-2.0 * e0, it, 2.0);
        c.wo = fma(-h2, it, 1.0);
        c.wc = 2.0 * it * (h2 - e0);
        c.wm = fma(-c.e, fma(t, t + 2.0, 2.0), 2.0) * (it * it);
    }
    c.pm = c.wm + 0.5 * c.wc;
    c.po = c.wo + 0.5 * c.wc;
    return c;
}
__device__ __forceinline__ Coef<double> coefficients(double t)
{
    double e0;
    return coefficients(t, e0);
}

// Single precision: two regimes. Below t = 1.5, w / t as a polynomial whose relative
// error on [0, 1.5] is minimax (Remez exchange on the Taylor series, coefficients
// rounded to FP32: 5e-9 for w_M, 3e-9 for w_O, 1e-9 for w_C before rounding); above,
// the closed forms, where their cancellation costs at most a factor ~3. Every
// coefficient stays within 4e-7 relative of its exact value (rms 6e-8 to 8e-8). One
// polynomial range of degree 6 or 7 takes the place of Taylor series of degree 6
// below 0.25 and 12 below 1.5 (23 multiply-adds instead of 18 or 36, and lanes of a
// warp no longer diverge between the two).
__device__ __forceinline__ void wpoly(float t, float &wm, float &wo, float &wc)
{
    float m = fmaf(t, -9.985858924e-06f, 1.324526238e-04f);
    float c = fmaf(t, -2.395259799e-06f, 3.410954741e-05f);
    float o = fmaf(t, 3.294269391e-06f, -4.541862290e-05f);
    m = fmaf(t, m, -1.014578040e-03f);
    c = fmaf(t, c, -2.921269333e-04f);
    o = fmaf(t, o, 3.927011858e-04f);
    m = fmaf(t, m, 5.933146924e-03f);
    c = fmaf(t, c, 1.980281435e-03f);
    o = fmaf(t, o, -2.775641857e-03f);
    m = fmaf(t, m, -2.777018584e-02f);
    c = fmaf(t, c, -1.110962220e-02f);
    o = fmaf(t, o, 1.666613296e-02f);
    m = fmaf(t, m, 9.999849647e-02f);
    c = fmaf(t, c, 4.999971390e-02f);
    o = fmaf(t, o, -8.333328366e-02f);
    m = fmaf(t, m, -2.499998808e-01f);
    c = fmaf(t, c, -1.666666418e-01f);
    o = fmaf(t, o, 3.333333433e-01f);
    wm = t * fmaf(t, m, 3.333333433e-01f);
    wc = t * fmaf(t, c, 3.333333433e-01f);
    wo = t * o;
}
// w_M, w_O, w_C of one optical path t given e = exp(-t)
__device__ __forceinline__ void wcoef(float t, float e, float &wm, float &wo, float &wc)
{
    if (t < 1.5f) {
        wpoly(t, wm, wo, wc);
    } else {
        const float it = rcp(t), it2 = it * it;
        wm = (2.0f - e * (t * t + 2.0f * t + 2.0f)) * it2;
        wo = 1.0f - 2.0f * (e + t - 1.0f) * it2;
        wc = 2.0f * (t - 2.0f + e * (t + 2.0f)) * it2;
    }
}

__device__ __forceinline__ Coef<float> coefficients(float t)
{
    Coef<float> c;
    c.e = expf(-t);
    wcoef(t, c.e, c.wm, c.wo, c.wc);
    c.pm = c.wm + 0.5f * c.wc;
    c.po = c.wo + 0.5f * c.wc;
    return c;
}

// Profile shape exp(-(x - s)^2). In FP32 it is evaluated as a power of two by
// the hardware approximation ex2.approx.ftz (max 2 ulp; the rounding of the FP32
// argument x - s already bounds its accuracy to ~1e-7 (x-s)^2 relative), and the
// exponent is capped at 60 so that eta_I and its reciprocal stay normal numbers
// far in the wings (the flush-to-zero form then never sees a subnormal result);
// the capped terms are below 1e-26 relative to line centre, where the optical
// paths vanish.
__device__ __forceinline__ float profile_shape(float xs)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fminf(xs * xs, 60.0f) * -1.4426950408889634f));
    return r;
}
// (FP64: capped at 1e-282 of the line centre, so that eta_I stays a normal number)
__device__ __forceinline__ double profile_shape(double xs)
{
    const double x = xs * xs;
    return exp(-(__double2hiint(x) > __double2hiint(650.0) ? 650.0 : x));
}

// exp(-x^2) in FP64 by a table of 2^(j/64) at the shared-memory address tab (Tang, ACM TOMS 15,
// 1989): -x^2 = (64 m + j) ln 2 / 64 + r with |r| < 0.0055, e^r by its Taylor polynomial of
// degree 5 (4e-17), 10 operations of the FP64 pipe and 2^m by the exponent; within an ulp.
// Capped as profile_shape is. (J^K_Q sweep, one per node and frequency: 16 x 16 x 32,
// unpolarized, 48 rays, 11 frequencies, ten iterations 14.3 -> 13.4 ms; adjoint, ten per
// point and frequency: 16 x 16 x 24, 32 rays, 7 frequencies 2.28 -> 2.14 ms.)
__device__ __forceinline__ double profile_shape(double xs, unsigned tab)
{
    double y = -xs * xs;
    y = __double2hiint(y) > __double2hiint(-650.0) ? -650.0 : y;      // (both negative: the larger magnitude)
    double k = fma(y, 92.33248261689366, 6755399441055744.0);
    const int n = __double2loint(k);
    k -= 6755399441055744.0;
    const double r = fma(k, -3.623510646634843e-19, fma(k, -0.010830424696249145, y));
    const double q = fma(r, fma(r, fma(r, 1.0 / 120, 1.0 / 24), 1.0 / 6), 0.5);
    double t;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(t) : "r"(tab + 8 * (n & 63)));
    t = fma(t, fma(r * r, q, r), t);
    return __hiloint2double(__double2hiint(t) + ((n >> 6) << 20), __double2loint(t));
}
__device__ __forceinline__ float profile_shape(float xs, unsigned) { return profile_shape(xs); }
// the table, by the first 64 threads of a block (FP64; a barrier follows)
template <typename Real> __device__ __forceinline__ void profile_table(double *tab)
{
    if (sizeof(Real) == 8 && threadIdx.x < 64) tab[threadIdx.x] = exp2(threadIdx.x / 64.0);
}

// ---------------------------------------------------------------------------
// BESSER upwind control point c_M of the quadratic Bezier spline on MO
// (Sec. 3.2, steps 1-9); ihM = 1/h_M, ihP = 1/h_P, ihMP = 1/(h_M + h_P).
// ---------------------------------------------------------------------------
// Per-update constants shared by the four Stokes parameters:
//   g.a = h_M/(h_P (h_M + h_P)), g.b = h_P/(h_M (h_M + h_P)), so that the derivative
//   of Eq. 6 is y'_O = g.a (y_P - y_O) + g.b (y_O - y_M);
//   g.hm2 = h_M/2, g.hp2 = h_P/2, g.r = h_M/h_P.
template <typename Real>
struct BesserGeom {
    Real a, b, hm2, hp2, r;
};

template <typename Real>
__device__ __forceinline__ BesserGeom<Real> besser_geom(Real hM, Real hP)
{
    BesserGeom<Real> g;
    const Real is = rcp(hM + hP);
    const Real ihM = rcp(hM), ihP = rcp(hP);
    g.a = hM * ihP * is;
    g.b = hP * ihM * is;
    g.hm2 = Real(0.5) * hM;
    g.hp2 = Real(0.5) * hP;
    g.r = hM * ihP;
    return g;
}

// Branch-free form: every step is evaluated and the outcome selected, so lanes
// of a warp that take different branches do not diverge. Interval tests use
// the sign of products ((c - y1)(c - y2) > 0 <=> c outside [min, max]).
// `branch` reports the outcome: 0 extremum at O (step 2), 1 c_M clipped to y_M
// (steps 5-6), 2 c_P clipped to y_P (steps 7-9), 3 the parabola (step 4).
template <typename Real>
__device__ __forceinline__ Real control_point_branch(Real yM, Real yO, Real yP, const BesserGeom<Real> &g, int &branch)
{
    const Real dm = yO - yM, dp = yP - yO;           // step 1 (h_M d_M, h_P d_P)
    const Real yp = g.a * dp + g.b * dm;             // step 3 (Eq. 6)
    const Real w = g.hm2 * yp;                       // step 4: c_M = y_O - w
    Real u = g.hp2 * yp;                             //         c_P = y_O + u
    const bool clip = u * (u - dp) > Real(0);        // step 7: c_P outside [y_O, y_P] -> y_P
    u = clip ? dp : u;
    const Real cM9 = yO - g.r * u;                   // steps 8-9: y'_O = 2 (c_P - y_O)/h_P
    const bool over = (dm - w) * w < Real(0);        // steps 5-6: c_M outside [y_M, y_O] -> y_M
    const Real r = over ? yM : cM9;
    const bool ext = dm * dp <= Real(0);             // step 2: extremum at O
    branch = ext ? 0 : (over ? 1 : (clip ? 2 : 3));
    return ext ? yO : r;
}

// The same in FP64 with the signs of the products taken from their factors' bits, in the
// integer pipe (6 of 16 FP64 operations less).
__device__ __forceinline__ bool nonzero(double a) { return ((unsigned)__double2hiint(a) << 1 | (unsigned)__double2loint(a)) != 0u; }
// a b > 0, a b < 0
__device__ __forceinline__ bool same_sign(double a, double b) { return (__double2hiint(a) ^ __double2hiint(b)) >= 0 && nonzero(a) && nonzero(b); }
__device__ __forceinline__ bool opposite_sign(double a, double b) { return (__double2hiint(a) ^ __double2hiint(b)) < 0 && nonzero(a) && nonzero(b); }
__device__ __forceinline__ double control_point_branch(double yM, double yO, double yP, const BesserGeom<double> &g, int &branch)
{
    const double dm = yO - yM, dp = yP - yO;
    const double yp = g.a * dp + g.b * dm;
    const double w = g.hm2 * yp;
    double u = g.hp2 * yp;
    const bool clip = same_sign(u, u - dp);
    u = clip ? dp : u;
    const double cM9 = yO - g.r * u;
    const bool over = opposite_sign(dm - w, w);
    const double r = over ? yM : cM9;
    const bool ext = !same_sign(dm, dp);
    branch = ext ? 0 : (over ? 1 : (clip ? 2 : 3));
    return ext ? yO : r;
}

template <typename Real>
__device__ __forceinline__ Real control_point(Real yM, Real yO, Real yP, const BesserGeom<Real> &g)
{
    int branch;
    return control_point_branch(yM, yO, yP, g, branch);
}

// ---------------------------------------------------------------------------
// The BESSER-DELO step (Eq. 7) with a general propagation matrix: the seven
// elements (eta_I, eta_Q, eta_U, eta_V, rho_Q, rho_U, rho_V) at M and at O,
// K' = K/eta_I - 1 with the off-diagonal pattern of the Unno-Rachkovsky
// matrix, kappa^-1 = 1 + psi'_O K'_O (Eq. 8) solved by Gaussian elimination
// with partial pivoting. The two-level sweeps use its specializations (an I-V
// block, or the arrow of dichroism); this form is the general one.
// ---------------------------------------------------------------------------
template <typename Real>
__device__ __forceinline__ void kprime4(const Real *eta, Real K[4][4])
{
    const Real a = Real(1) / eta[0];
    const Real q = eta[1] * a, u = eta[2] * a, v = eta[3] * a, rq = eta[4] * a, ru = eta[5] * a, rv = eta[6] * a;
    K[0][0] = 0;  K[0][1] = q;   K[0][2] = u;   K[0][3] = v;
    K[1][0] = q;  K[1][1] = 0;   K[1][2] = rv;  K[1][3] = -ru;
    K[2][0] = u;  K[2][1] = -rv; K[2][2] = 0;   K[2][3] = rq;
    K[3][0] = v;  K[3][1] = ru;  K[3][2] = -rq; K[3][3] = 0;
}

template <typename Real>
__device__ __forceinline__ void delo_step_general(const Real IM[4], const Real etaM[7], const Real epsM[4],
                                                  const Real etaO[7], const Real epsO[4], Real etaP_I,
                                                  const Real epsP[4], Real dsM, Real dsP, bool has_p, Real IO[4],
                                                  Real &lstar)
{
    Real SM[4], SO[4], SP[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        SM[s] = epsM[s] / etaM[0];
        SO[s] = epsO[s] / etaO[0];
        SP[s] = has_p ? epsP[s] / etaP_I : Real(0);
    }
    const Real tMO = Real(0.5) * (etaM[0] + etaO[0]) * dsM;
    const Real tOP = has_p ? Real(0.5) * (etaO[0] + etaP_I) * dsP : Real(1);
    const Coef<Real> co = coefficients(tMO);
    Real cM[4];
    if (has_p) {
        const BesserGeom<Real> bg = besser_geom(tMO, tOP);
#pragma unroll
        for (int s = 0; s < 4; ++s) cM[s] = control_point(SM[s], SO[s], SP[s], bg);
    } else {
#pragma unroll
        for (int s = 0; s < 4; ++s) cM[s] = Real(0.5) * (SM[s] + SO[s]);
    }
    Real kM[4][4], kO[4][4], A[4][5];
    kprime4(etaM, kM);
    kprime4(etaO, kO);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        Real acc = co.e * IM[r];
#pragma unroll
        for (int s = 0; s < 4; ++s) acc -= co.pm * kM[r][s] * IM[s];
        A[r][4] = acc + co.wm * SM[r] + co.wo * SO[r] + co.wc * cM[r];
#pragma unroll
        for (int s = 0; s < 4; ++s) A[r][s] = (r == s ? Real(1) : Real(0)) + co.po * kO[r][s];
    }
    // elimination with partial pivoting (the diagonal is 1 + 0, off-diagonals psi'_O K'_O)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        int piv = c;
#pragma unroll
        for (int r = c + 1; r < 4; ++r)
            if (fabs(A[r][c]) > fabs(A[piv][c])) piv = r;
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            const Real x = A[c][s];
            A[c][s] = A[piv][s];
            A[piv][s] = x;
        }
        const Real inv = Real(1) / A[c][c];
#pragma unroll
        for (int r = c + 1; r < 4; ++r) {
            const Real f = A[r][c] * inv;
#pragma unroll
            for (int s = c; s < 5; ++s) A[r][s] -= f * A[c][s];
        }
    }
#pragma unroll
    for (int r = 3; r >= 0; --r) {
        Real s = A[r][4];
#pragma unroll
        for (int q = r + 1; q < 4; ++q) s -= A[r][q] * IO[q];
        IO[r] = s / A[r][r];
    }
    lstar = co.wo + (has_p ? co.wc : Real(0.5) * co.wc);
}

// ---------------------------------------------------------------------------
// Hanle statistical equilibrium for K = 2 of the upper level (Eq. 2):
//   S_Q + i Gamma sum_Q' K_QQ'(B) S_Q' = R_Q,
// written for the real unknowns x = (S^2_0, Re S^2_1, Im S^2_1, Re S^2_2, Im S^2_2)
// using S_{-Q} = (-1)^Q conj(S_Q). With g = Gamma * B / |B| the real matrix is
//   [ 1          sqrt6 gy  -sqrt6 gx  0      0     ]
//   [-sqrt6/2 gy  1         -gz        gy    -gx    ]
//   [ sqrt6/2 gx  gz         1         gx     gy    ]
//   [ 0          -gy        -gx        1     -2 gz  ]
//   [ 0           gx        -gy        2 gz   1     ]
// Scaling the Q != 0 unknowns and equations by sqrt(2) makes the matrix the
// identity plus an antisymmetric matrix, whose symmetric part is positive
// definite; Gaussian elimination without pivoting is then stable (FP64).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void hanle_solve5(double gx, double gy, double gz, const double r[5], double x[5])
{
    const double s6 = 2.449489742783178098197284;  // sqrt(6)
    double A[5][6] = {
        {1.0, s6 * gy, -s6 * gx, 0.0, 0.0, r[0]},
        {-0.5 * s6 * gy, 1.0, -gz, gy, -gx, r[1]},
        {0.5 * s6 * gx, gz, 1.0, gx, gy, r[2]},
        {0.0, -gy, -gx, 1.0, -2.0 * gz, r[3]},
        {0.0, gx, -gy, 2.0 * gz, 1.0, r[4]},
    };
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        double inv = 1.0 / A[c][c];
#pragma unroll
        for (int q = c + 1; q < 5; ++q) {
            double f = A[q][c] * inv;
#pragma unroll
            for (int s = c; s < 6; ++s) A[q][s] -= f * A[c][s];
        }
    }
#pragma unroll
    for (int q = 4; q >= 0; --q) {
        double s = A[q][5];
#pragma unroll
        for (int t = q + 1; t < 5; ++t) s -= A[q][t] * x[t];
        x[q] = s / A[q][q];
    }
}

// y = M x with M the real matrix of hanle_solve5 (same unknowns and equations)
__device__ __forceinline__ void hanle_apply5(double gx, double gy, double gz, const double x[5], double y[5])
{
    const double s6 = 2.449489742783178098197284;  // sqrt(6)
    y[0] = x[0] + s6 * gy * x[1] - s6 * gx * x[2];
    y[1] = -0.5 * s6 * gy * x[0] + x[1] - gz * x[2] + gy * x[3] - gx * x[4];
    y[2] = 0.5 * s6 * gx * x[0] + gz * x[1] + x[2] + gx * x[3] + gy * x[4];
    y[3] = -gy * x[1] - gx * x[2] + x[3] - 2.0 * gz * x[4];
    y[4] = gx * x[1] - gy * x[2] + 2.0 * gz * x[3] + x[4];
}

}  // namespace porta
