// Formal solution for the radiation-field tensors (Sec. 3 of Stepan & Trujillo
// Bueno 2013): the short-characteristics BESSER sweep of every ray direction
// and frequency, fused with the frequency integration of the Stokes parameters
// and Lambda* that feeds J^K_Q (Eq. 1, Eq. 14) and the Jacobi update; and the same
// sweep for emergent Stokes profiles, with the Stokes vectors of every node for the
// reverse mode where asked.
//
// The decomposition is that of the general sweep (sweep.cu): one thread-block
// cluster per ray and frequency group at a time, the plane split into strips of
// sheared rows, one per CTA; the stencils of the bilinear interpolation at the
// upwind point M and downwind point P are fixed nearest-neighbour accesses in the
// frame sheared along the characteristics.
//
// The transfer coefficients of a node depend on the frequency only through the
// profile, eta_I = chi phi(x - s) and eta_V = b (x - s) eta_I, while its source
// vector S(Omega) does not (CRD). When a plane enters the 4-slot ring, a thread per
// node writes the node's source vector once and its (eta_I, eta_V) at every
// frequency of the pass. A point update then interpolates eps = sum_k w_k eta_k S_k
// and eta = sum_k w_k eta_k from its 4 upwind and 4 downwind corners without
// evaluating a profile.
//
// An update thread owns a point and takes the frequencies of the pass one unit after
// the other: two adjacent frequencies in FP32, whose operations are packed (FFMA2,
// FMUL2, FADD2) wherever no factor is common to both, one frequency in FP64.
//
// Strips exchange only their first row: the CTA that computed it writes it into the
// halo row of the strip before with st.async, which counts the bytes on that CTA's
// mbarrier, so no CTA waits for another one except for the halo row itself, and
// nothing waits for a fence of the fixed-point sums in flight. The inputs of the next
// planes' nodes travel by cp.async during the updates.
//
// What bounds it: instruction issue and the length of a plane's chain of operations, not
// memory (the inputs are re-read from L2). A plane and pass takes about 2660 cycles of fixed
// chain, 1106 per unit of its points' rounds and 1190 + 151 per unit for the nodes (NS = 4,
// FP32; jsweep_plane_cost), whatever the strip, so a pass has few units over as many points
// as the threads hold. Against the kernel of sweep_jw.cu, which this one replaces where it
// fits (one frequency of one point per thread and step, one cluster barrier per plane), ms
// per formal solution: 64 x 64 x 64 x 160 rays x 21 frequencies 20.1 -> 17.9, 33 x 27 x 41 x
// 80 x 21 1.91 -> 1.20, 24 x 24 x 32 x 48 x 11 in FP64 10.6 -> 6.1, 64 x 64 x 48 x 160 x 31
// x 4 lines, unpolarized, 46.4 -> 31.4 (with the rate equations).
//
// FP32 errors against 64 bits, that kernel's and this one's: J^K_Q of 33 x 27 x 41 9.0e-8 and
// 3.6e-8, Lambda-bar* 4.1e-8 and 2.3e-8; iterates of 64 x 64 x 64 6.2e-6 and 4.5e-6. What kept them
// above were roundings that are the same for all rays or planes and do not average out (those
// of the geometry, of the weights and of the reciprocal in kappa^-1; each is explained at its place).
//
// Shared memory per CTA (X: 8 bytes, a frequency unit):
//   ring[4][nodes]        source vectors, Real
//   coef[4][FX][nodes]    (eta_I, eta_V) (NS = 4) or eta_I (NS = 1), X
//   ibuf[2][FX][points + a halo row]   Stokes vectors of planes q - 1 and q, X
//   tot, stage, ...       point totals, inputs in flight, geometry
// with nodes = (rows + 2) nx (one halo row on each side, recomputed locally).
#include <cooperative_groups.h>

#include <type_traits>

#include "device_math.cuh"
#include "porta_internal.cuh"
#include "sweep_common.cuh"

namespace cg = cooperative_groups;

namespace porta {

namespace {

template <typename Real, int NS>
struct JW {
    static constexpr int per = 16 / (int)sizeof(Real);        // Reals per 16-byte chunk
    static constexpr int s_words = NS == 1 ? 1 : 4;            // source words per node
    static constexpr int s_chunks = NS == 1 ? 0 : 4 / per;     // 16-byte chunks per node (NS = 4)
    static constexpr int staged = NS == 1 ? 4 : 12;            // words of a voxel's packed inputs
    static constexpr int cw = NS == 1 ? 1 : 2;                 // coefficients (X) per node and unit
    static constexpr int na = NS == 1 ? 2 : 4;                 // accumulated quantities per point
    static constexpr int nacc = NS == 1 ? 2 : 7;               // fixed-point accumulators per voxel
};

constexpr int kJFrac = 46;   // fixed-point fraction bits below a voxel's reference value

// one term of the fixed-point sum: the integer nearest to y (an FP32 value times a power of
// two) added to *p. Integer additions are exact and commute, so the sums do not depend on
// the order in which rays, frequency passes and concurrent launches add their terms.
// Returns whether the term is beyond 2^62 (or not finite); its sum is then void and the
// caller reports it.
// y = h 2^40 + m 2^18 + l by adding 1.5 2^23, whose sum's low bits are the integer nearest
// to the addend: every step is exact but the last, which rounds y to an integer. (The
// conversion instruction, float to 64-bit integer, runs in the FP64 pipe at two lanes a
// cycle and SM: 16 cycles each, 7 per point, 12% of the time of a 64 x 64 plane.)
__device__ __forceinline__ bool jadd(unsigned long long *p, float y)
{
    constexpr float M = 12582912.0f;
    constexpr unsigned B = 0x4b400000u;                        // bits of M
    const float h = fmaf(y, 0x1p-40f, M), r = fmaf(M - h, 0x1p40f, y);
    const float m = fmaf(r, 0x1p-18f, M), l = fmaf(M - m, 0x1p18f, r) + M;
    const unsigned long long k = (unsigned long long)__float_as_uint(m) * (1u << 18) +
                                 (((unsigned long long)(__float_as_uint(h) - B) << 40) - (unsigned long long)B * ((1u << 18) + 1u));
    atomicAdd(p, k + __float_as_uint(l));
    return !(fabsf(y) < 4.6116860e18f);
}
// the same for |y| <= 2^45 (terms up to half the voxel's reference value) in two parts, 5
// instructions less for each of a point's 7 terms
__device__ __forceinline__ void jadd_small(unsigned long long *p, float y)
{
    constexpr float M = 12582912.0f;
    constexpr unsigned B = 0x4b400000u;
    const float h = fmaf(y, 0x1p-23f, M), l = fmaf(M - h, 0x1p23f, y) + M;
    const unsigned long long k = (unsigned long long)__float_as_uint(h) * (1u << 23) - (unsigned long long)B * ((1u << 23) + 1u);
    atomicAdd(p, k + __float_as_uint(l));
}

// byte offsets of the dynamic shared memory (the ring of source vectors comes first) and
// strides of its coefficient and Stokes planes (one frequency unit each)
struct JSmem { unsigned coef, ibuf, tot, stage, geo, freq, wgt, vox, stw, ste, stv, end, cplane, iplane; };
template <typename Real, int NS>
__host__ __device__ inline JSmem jsmem(int nodes, int pts, int tots, int FX)
{
    using W = JW<Real, NS>;
    const unsigned rb = (unsigned)sizeof(Real);
    auto up16 = [](unsigned x) { return (x + 15u) / 16u * 16u; };
    JSmem s;
    s.cplane = up16(nodes * W::cw * 8);
    s.iplane = up16(pts * NS * 8);
    s.coef = up16(4 * nodes * W::s_words * rb);
    s.ibuf = s.coef + 4 * FX * s.cplane;
    s.tot = s.ibuf + 2 * FX * s.iplane;
    s.stage = s.tot + up16(2 * tots * W::na * rb);
    s.geo = s.stage + W::staged * nodes * rb;
    s.freq = s.geo + 8 * (unsigned)sizeof(PlaneGeom<Real>);
    s.wgt = s.freq + 2 * FX * 8;
    s.stw = s.wgt + 4 * nodes * rb;
    s.vox = s.stw + nodes * rb;
    s.ste = s.vox + 4 * nodes * 4;
    s.stv = s.ste + nodes * 4;
    s.end = s.stv + nodes * 4;
    return s;
}

}  // namespace

template <typename Real, int NS>
int jsweep_smem_bytes(int nodes, int ipts, int tots, int F)
{
    constexpr int W = jsweep_lanes<Real>();
    return (int)jsmem<Real, NS>(nodes, ipts, tots, (F + W - 1) / W).end;
}

// ---- frequency units: a pair of floats (every operation packed; each lane rounds as the
// scalar operation) or one double -----------------------------------------------------
template <typename Real> struct XOf;
template <> struct XOf<float> { using X = float2; };
template <> struct XOf<double> { using X = double; };

__device__ __forceinline__ float2 xset(float a) { return make_float2(a, a); }
__device__ __forceinline__ double xset(double a) { return a; }
__device__ __forceinline__ float2 xmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 xfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 xadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double xmul(double a, double b) { return a * b; }
__device__ __forceinline__ double xfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double xadd(double a, double b) { return a + b; }
__device__ __forceinline__ float2 xneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ double xneg(double a) { return -a; }
__device__ __forceinline__ float2 xrcp(float2 a) { return make_float2(rcp(a.x), rcp(a.y)); }
__device__ __forceinline__ double xrcp(double a) { return rcp(a); }
// -1 / a
__device__ __forceinline__ float2 xnrcp(float2 a) { return make_float2(rcp(-a.x), rcp(-a.y)); }
__device__ __forceinline__ double xnrcp(double a) { return rcp(-a); }
// the same Real times both lanes (scalar operations: a pair made of one value costs a move)
__device__ __forceinline__ float2 xms(float s, float2 a) { return make_float2(s * a.x, s * a.y); }
__device__ __forceinline__ double xms(double s, double a) { return s * a; }
__device__ __forceinline__ float2 xfs(float s, float2 a, float2 c) { return make_float2(fmaf(s, a.x, c.x), fmaf(s, a.y, c.y)); }
__device__ __forceinline__ double xfs(double s, double a, double c) { return fma(s, a, c); }
// s + sum over the lanes of a b
__device__ __forceinline__ float xdot(float2 a, float2 b, float s) { return fmaf(a.y, b.y, fmaf(a.x, b.x, s)); }
__device__ __forceinline__ double xdot(double a, double b, double s) { return fma(a, b, s); }
__device__ __forceinline__ float2 xprofile(float2 xs, unsigned) { return make_float2(profile_shape(xs.x), profile_shape(xs.y)); }
__device__ __forceinline__ double xprofile(double xs, unsigned tab) { return profile_shape(xs, tab); }
__device__ __forceinline__ float xlane(float2 a, int i) { return i ? a.y : a.x; }
__device__ __forceinline__ double xlane(double a, int) { return a; }

// Coefficients of the step (Eqs. 9-13) of a unit: e = e^-t, their sum e0 = 1 - e, and the
// three w. With q = w_O, h = t (1 - q) / 2 gives e0 = t (1 - h), w_O + w_C = e0 - w_M (or
// 2 h - q): below t = 1.5 two polynomials (w_M and w_O over t, minimax in relative error:
// 5e-9 and 3e-9) yield all five, above it closed forms whose cancellation costs a factor of
// about 3. Measured over t from 1e-7 to 1e3 (porta_eval_unit): e0 within 7.3e-8 of its value
// and e + e0 = 1 to rounding, so a constant source function is kept; w_O within 1.6e-7, w_M
// within 5.4e-7 (just above 1.5) and w_C, which multiplies differences of source functions,
// 5.6e-7. The polynomials are evaluated for both lanes always; the closed forms replace them
// where some lane needs them. (Three polynomials, an exponential per lane and the sums: 26
// instructions more per unit, 3% of the sweep's time, and the same errors of J.)
template <typename X> struct XCoef { X e, e0, wm, wo, wc; };
__device__ __forceinline__ XCoef<double> xcoef(double t)
{
    double e0;
    const Coef<double> c = coefficients(t, e0);
    return {c.e, e0, c.wm, c.wo, c.wc};
}
__device__ __forceinline__ XCoef<float2> xcoef(float2 t)
{
    XCoef<float2> c;
    const float2 one = xset(1.0f), nt = xneg(t);
    float2 m = xset(-9.985858924e-06f), o = xset(3.294269391e-06f);
    m = xfma(t, m, xset(1.324526238e-04f));
    m = xfma(t, m, xset(-1.014578040e-03f));
    o = xfma(t, o, xset(-4.541862290e-05f));
    m = xfma(t, m, xset(5.933146924e-03f));
    o = xfma(t, o, xset(3.927011858e-04f));
    m = xfma(t, m, xset(-2.777018584e-02f));
    o = xfma(t, o, xset(-2.775641857e-03f));
    m = xfma(t, m, xset(9.999849647e-02f));
    o = xfma(t, o, xset(1.666613296e-02f));
    m = xfma(t, m, xset(-2.499998808e-01f));
    o = xfma(t, o, xset(-8.333328366e-02f));
    m = xfma(t, m, xset(3.333333433e-01f));
    o = xfma(t, o, xset(3.333333433e-01f));
    c.wm = xmul(t, m);
    c.wo = xmul(t, o);
    const float2 ht = xms(0.5f, t);
    c.e0 = xfma(nt, xfma(xneg(ht), c.wo, ht), t);
    c.e = xadd(one, xneg(c.e0));
    c.wc = xadd(xadd(c.e0, xneg(c.wm)), xneg(c.wo));
    if (fmaxf(t.x, t.y) >= 1.5f) {
        const float2 two = xset(2.0f), u = xms(-1.4426950408889634f, t), it = xrcp(t);
        float2 e;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(u.x));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(u.y));
        const float2 e0 = xadd(one, xneg(e)), h = xfma(xneg(e0), it, one), h2 = xadd(h, h);
        const float2 wm = xmul(xfma(xneg(e), xfma(t, xadd(t, two), two), two), xmul(it, it));
        const float2 wo = xfma(xneg(h2), it, one), hd = xadd(h2, xneg(e0)), wc = xmul(xadd(hd, hd), it);
        if (t.x >= 1.5f) { c.e.x = e.x; c.e0.x = e0.x; c.wm.x = wm.x; c.wo.x = wo.x; c.wc.x = wc.x; }
        if (t.y >= 1.5f) { c.e.y = e.y; c.e0.y = e0.y; c.wm.y = wm.y; c.wo.y = wo.y; c.wc.y = wc.y; }
    }
    return c;
}

// y_O - c_M of the BESSER control point (Sec. 3.2, steps 1-9) from d_M = y_O - y_M and
// -d_P = y_O - y_P. The parabola's c_M = y_O - w has w = a d_P + b d_M, and the step clipped
// at c_P = y_P has w = r d_P (Eq. 6 times h_M / 2). Past step 2 (d_M d_P <= 0: c_M = y_O)
// both differences and w have one sign, so the interval tests compare magnitudes: |w| >
// |d_M| is c_M outside [y_M, y_O] (steps 5-6, c_M = y_M), |w| > |r d_P| is c_P outside
// [y_O, y_P] (steps 7-9). na = -a, nr = -r.
__device__ __forceinline__ float cp_select(float dm, float w, float rdp, float te)
{
    float c = fabsf(w) > fabsf(rdp) ? rdp : w;
    c = fabsf(w) > fabsf(dm) ? dm : c;
    return te < 0.0f ? c : 0.0f;
}
__device__ __forceinline__ float2 xoffset(float2 dm, float2 ndp, float2 na, float2 b, float2 nr)
{
    const float2 w = xfma(na, ndp, xmul(b, dm)), rdp = xmul(nr, ndp), te = xmul(dm, ndp);
    return make_float2(cp_select(dm.x, w.x, rdp.x, te.x), cp_select(dm.y, w.y, rdp.y, te.y));
}
// (the comparisons on the bits, in the integer pipe; where a difference is 0, so is the
// selected value, and step 2 needs the signs alone)
__device__ __forceinline__ double xoffset(double dm, double ndp, double na, double b, double nr)
{
    const double w = fma(na, ndp, b * dm), rdp = nr * ndp;
    auto mag = [](double x) { return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull; };
    double c = mag(w) > mag(rdp) ? rdp : w;
    c = mag(w) > mag(dm) ? dm : c;
    return (__double2hiint(dm) ^ __double2hiint(ndp)) < 0 ? c : 0.0;
}

// ---- shared memory by 32-bit address -------------------------------------------------
// (a generic pointer to the dynamic array costs an addition of the CTA's window per
// access). volatile keeps the accesses' order against barriers; stores clobber memory.
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void lds(unsigned a, int &x) { asm volatile("ld.shared.s32 %0, [%1];" : "=r"(x) : "r"(a)); }
__device__ __forceinline__ void lds4i(unsigned a, int *x)
{
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(a));
}
__device__ __forceinline__ int wrap(int x, int n) { return (int)min((unsigned)x, (unsigned)(x - n)); }
__device__ __forceinline__ void lds(unsigned a, float &x) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(a)); }
__device__ __forceinline__ void lds(unsigned a, double &x) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(x) : "r"(a)); }
__device__ __forceinline__ void lds(unsigned a, float2 &x)
{
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x.x), "=f"(x.y) : "r"(a));
}
// two units (16 bytes)
__device__ __forceinline__ void lds2(unsigned a, float2 &x, float2 &y)
{
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(y.x), "=f"(y.y) : "r"(a));
}
__device__ __forceinline__ void lds2(unsigned a, double &x, double &y)
{
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(x), "=d"(y) : "r"(a));
}
// four Reals: one 16-byte chunk in FP32, two in FP64, `ch` bytes apart
__device__ __forceinline__ void lds4(unsigned a, unsigned, float *w)
{
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3]) : "r"(a));
}
__device__ __forceinline__ void lds4(unsigned a, unsigned ch, double *w)
{
    lds2(a, w[0], w[1]);
    lds2(a + ch, w[2], w[3]);
}
__device__ __forceinline__ void sts(unsigned a, int x) { asm volatile("st.shared.s32 [%0], %1;" ::"r"(a), "r"(x) : "memory"); }
__device__ __forceinline__ void sts(unsigned a, float x) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory"); }
__device__ __forceinline__ void sts(unsigned a, double x) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(x) : "memory"); }
__device__ __forceinline__ void sts(unsigned a, float2 x)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x.x), "f"(x.y) : "memory");
}
__device__ __forceinline__ void sts2(unsigned a, float2 x, float2 y)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x.x), "f"(x.y), "f"(y.x), "f"(y.y) : "memory");
}
__device__ __forceinline__ void sts2(unsigned a, double x, double y)
{
    asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(x), "d"(y) : "memory");
}
__device__ __forceinline__ void sts4(unsigned a, unsigned, const float *w)
{
    sts2(a, make_float2(w[0], w[1]), make_float2(w[2], w[3]));
}
__device__ __forceinline__ void sts4(unsigned a, unsigned ch, const double *w)
{
    sts2(a, w[0], w[1]);
    sts2(a + ch, w[2], w[3]);
}
// copies from global to shared memory that pass through no register (completed by
// copies_wait of the same thread)
template <typename T> __device__ __forceinline__ void copy_async(unsigned dst, const T *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"((int)sizeof(T)) : "memory");
}
__device__ __forceinline__ void copy_async16(unsigned dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// a w / b rounded up or down: to the nearest of the exact value plus `shift` (-1/2 to 1/2) of
// its last place. The rounding of a node's weight w_m / (chi N) would be the same for all rays
// of one w_m, N being nearly so, and go into J and Lambda* undiminished (2e-8, which Lambda*
// near 1 multiplies in the update: 64 x 64 x 48, Lambda-bar* 3.5e-8 from its value in place of
// 2.5e-8, populations 1.3 times as far); with a shift of its own for every ray it averages out.
__device__ __forceinline__ float quotient(float a, float w, float b, float shift)
{
    const float aw = __fmul_rn(a, w), r = rcp(b), q = __fmul_rn(aw, r);
    const float place = __uint_as_float(__float_as_uint(q) & 0x7f800000u) * 0x1p-23f;
    return __fadd_rn(q, fmaf(fmaf(-q, b, aw) + fmaf(a, w, -aw), r, shift * place));
}

// the shift of ray m: multiples of the golden ratio, modulo 1, fill the interval evenly (formed
// anew for every node: kept through the updates it is one register too many)
__device__ __forceinline__ float ray_shift(unsigned m)
{
    asm volatile("" : "+r"(m));
    return (float)(m * 2654435769u >> 8) * 0x1p-24f - 0.5f;
}

// keeps the compiler from rebuilding a corner's address from its parts at every use
__device__ __forceinline__ unsigned opaque(unsigned x)
{
    asm("" : "+r"(x));
    return x;
}

// ---- the halo exchange -----------------------------------------------------------------
__device__ __forceinline__ unsigned map_rank(unsigned addr, int rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// stores to another CTA's shared memory that count their bytes on its mbarrier
__device__ __forceinline__ void push(unsigned dst, unsigned bar, float2 x)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(dst),
                 "f"(x.x), "f"(x.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void push(unsigned dst, unsigned bar, double x)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(dst), "d"(x),
                 "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void push2(unsigned dst, unsigned bar, float2 x, float2 y)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                     dst), "f"(x.x), "f"(x.y), "f"(y.x), "f"(y.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void push2(unsigned dst, unsigned bar, double x, double y)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(dst),
                 "d"(x), "d"(y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bar_init(unsigned bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive_remote(unsigned bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ unsigned bar_try(unsigned bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok;
}
// Bounded wait for the phase of the given parity. A wait that runs out (the neighbouring
// CTA stopped) marks the CTA, which from then on waits for and signals nothing (its
// neighbours' waits run out in turn), and sets the error flag; the kernel then ends with
// wrong sums and the next call that synchronizes reports the flag. The limit is a time, a
// hundred thousand times a plane's: the tries themselves may sleep. It is read after the
// waits of ordinary length only (read at once it cost 1 to 2% of every sweep).
constexpr unsigned long long kHaloWaitNs = 2000000000ull;
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __noinline__ void bar_wait_long(unsigned bar, unsigned parity, volatile int *dead, int *err)
{
    for (int i = 0; i < 1024; ++i)
        if (bar_try(bar, parity) || *dead) return;
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < kHaloWaitNs)
        if (bar_try(bar, parity) || *dead) return;
    *dead = 1;
    atomicOr(err, 4);
}
__device__ __forceinline__ void bar_wait(unsigned bar, unsigned parity, volatile int *dead, int *err)
{
    if (!*dead && !bar_try(bar, parity)) bar_wait_long(bar, parity, dead, err);
}

// Shared control words of a CTA: full (word b) counts the bytes of the halo row of the
// planes of parity b that the next strip's CTA writes here; freed (word b) receives the
// arrival of the CTA before once it has read the halo row that this CTA wrote there.
// JPhase counts the completed phases of each.
struct JBars { unsigned full, freed; volatile int *dead; };   // [2] words of 8 bytes each
struct JPhase { unsigned full0, full1, freed0, freed1; };

// what a sweep leaves: the J^K_Q and Lambda* sums (SUMS; with one ray's Stokes vectors and
// Lambda*, PROBE), or the emergent Stokes profiles and, for the reverse mode, the Stokes
// vectors of every node (EMERGENT: no sums, no profile normalization)
enum JMode { SUMS = 0, PROBE_RAY = 1, EMERGENT = 2 };
// PACKED: the voxels' inputs lie side by side in a.pack. (A form of its own: the test of
// a.pack in one kernel cost 1.2% of a 64 x 64 x 64 formal solution, 17.89 -> 18.11 ms.)
template <typename Real, int NS, int MODE, bool PACKED>
__device__ __forceinline__ void jsweep_item(const SweepArgs<Real> &a, const unsigned sbase, const JSmem &sm,
                                            const JBars &bars, JPhase &ph, const unsigned sray, const unsigned stab, int box, int m, int g,
                                            int rank, int C)
{
    using X = typename XOf<Real>::X;
    using W = JW<Real, NS>;
    constexpr bool PROBE = MODE == PROBE_RAY, EMG = MODE == EMERGENT;
    constexpr int XW = jsweep_lanes<Real>();
    constexpr int NA = W::na;
    constexpr unsigned SZ = sizeof(Real);
    constexpr unsigned CB = W::cw * 8;               // bytes of a node's coefficients and of a Stokes element
                                                     // (NS = 4: of each of its two chunks)
    constexpr int SCH = W::staged * (int)SZ / 16;    // 16-byte chunks of a voxel's packed inputs
    const BoxDev B = a.boxes[box];
    const int nx = B.nx, ny = B.ny, nz = B.nz, FX = (a.F + XW - 1) / XW;
    const int row0 = (int)(((long long)rank * ny) / C);
    const int R = (int)(((long long)(rank + 1) * ny) / C) - row0;
    // the CTAs that own the sheared rows before and after this strip
    const int prev_row = row0 == 0 ? ny - 1 : row0 - 1, next_row = (row0 + R) % ny;
    const int prev_owner = (int)(((long long)(prev_row + 1) * C + ny - 1) / ny) - 1;
    const int prev_R = prev_row + 1 - (int)(((long long)prev_owner * ny) / C);
    const int next_owner = (int)(((long long)(next_row + 1) * C + ny - 1) / ny) - 1;
    // the pass's frequencies: the units of the grid split evenly over the groups
    const int nunit = (a.nnu + XW - 1) / XW;
    const int nper = nunit / a.ngroups, nextra = nunit - nper * a.ngroups;
    const int j0 = XW * (g * nper + min(g, nextra));
    const int nf = nper + (g < nextra ? 1 : 0);      // units
    const PlaneGeom<Real> *G = a.geom + B.geom0 + (long long)m * nz;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int nodes = a.ring_plane;                  // node capacity of a ring slot
    const int nn = (R + 2) * nx;                     // nodes of this strip's slot
    const int ipts = a.ipts_max;
    const int npts = R * nx;
    // voxel indices fit in 32 bits (porta_create limits nvox to 2^31)
    const int nvox = (int)a.nvox, vox0 = (int)B.vox0;
    const Real *__restrict__ invn = a.invn + (long long)m * a.nvox;
    const unsigned geo = sbase + sm.geo;             // plane q's PlaneGeom at q % 8
    constexpr unsigned GB = sizeof(PlaneGeom<Real>);
    // four words of the ray's constants (mu, ox, oy, oz | T[18], w, pad)
    auto ray4 = [&](int i, Real *w) { lds4(sray + i * 4 * SZ, 16, w); };
    constexpr int GW = (int)sizeof(PlaneGeom<Real>) / 4;

    // the pass's frequency nodes and weights (a last half-empty unit repeats its frequency
    // with weight 0) and the first planes' geometry; later planes follow five ahead. (The
    // previous item ended at a CTA barrier: no reader is left.)
    for (int f = tid; f < nf * XW; f += nt) {
        const bool in = j0 + f < a.nnu;
        sts(sbase + sm.freq + f * SZ, a.xf[in ? j0 + f : a.nnu - 1]);
        sts(sbase + sm.freq + (FX * XW + f) * SZ, in ? a.wf[j0 + f] : Real(0));
    }
    for (int i = tid; i < GW * min(6, nz); i += nt) sts(geo + 4 * i, reinterpret_cast<const int *>(G)[i]);
    __syncthreads();

    // Update threads: a point (or several in rounds) and every Lg-th unit of the pass from fg
    // on; the threads of a group are whole warps. (The warp's index comes from a warp
    // reduction so that the compiler knows that what follows from it is the same for all
    // lanes and keeps it in uniform registers.)
    const int pw = min(nt, (npts + 31) / 32 * 32);
    const int wid = (int)__reduce_max_sync(0xffffffffu, (unsigned)tid >> 5);
    const int Lg = npts > 0 ? min(nf, nt / pw) : 1;
    const int fg = npts > 0 ? wid * 32 / pw : 0, ptid = tid - fg * pw;
    const int p_own = min(ptid, max(npts - 1, 0)), l_own = p_own / nx, c_own = p_own - l_own * nx;
    // the work beside the updates goes to the last threads first (where the units do not
    // divide evenly, the last groups have one less)
    const int rtid = nt - 1 - tid, rowt = rtid / nx, colt = rtid - rowt * nx;
    const int dl = nt / nx, dc = nt - dl * nx;

    // voxel of point (l, c) of the strip in a plane (l = -1: the row before the strip)
    auto point_voxel = [&](int q, int l, int c) {
        const unsigned o = geo + (q & 7) * GB;
        int ax, ay, kz;
        lds(o, ax);
        lds(o + 4, ay);
        lds(o + 8, kz);
        int pi = c + ax;
        pi -= pi >= nx ? nx : 0;
        int pj = row0 + l + ay;
        pj += pj < 0 ? ny : 0;
        pj -= pj >= ny ? ny : 0;
        pj -= pj >= ny ? ny : 0;
        return vox0 + (kz * ny + pj) * nx + pi;
    };

    // Inputs of plane q's nodes on their way to shared memory; the thread that asked for a
    // node's values is the one that fills the node a phase later. (Wrapped by an unsigned
    // minimum: x - n is huge below n.)
    // (no room for the packed inputs: a node's words one by one from where they are, into the
    // places of the packed ones)
    auto fetch_words = [&](unsigned d, int v) {
        auto put = [&](int w, const Real *src) {
            copy_async(d + w / W::per * nodes * 16 + w % W::per * SZ, src + v);
        };
        put(0, a.chi);
        put(1, a.vel);
#pragma unroll 1
        for (int k = 0; k < (NS == 1 ? 1 : 6); ++k) put(2 + k, a.rho + (size_t)k * a.nvox);
        if constexpr (NS == 4) {
            put(8, a.bx);
            put(9, a.by);
            put(10, a.bz);
        }
    };
    const int jown = row0 + rowt - 1 + (row0 + rowt == 0 ? ny : 0) - (row0 + rowt > ny ? ny : 0);
    auto fetch = [&](int q) {
        if (rtid >= nn) return;
        int g4[4];
        lds4i(geo + (q & 7) * GB, g4);
        const int base = vox0 + g4[2] * ny * nx;
        int j = jown, c = colt;
        for (int idx = rtid; idx < nn; idx += nt) {
            const int pi = wrap(c + g4[0], nx), pj = wrap(j + g4[1], ny);
            const int v = base + pj * nx + pi;
            const unsigned d = sbase + sm.stage + idx * 16;
            sts(sbase + sm.stv + idx * 4, v);
            if (!EMG) copy_async(sbase + sm.stw + idx * SZ, invn + v);
            if (!EMG && a.jacc) copy_async(sbase + sm.ste + idx * 4, a.jexp + v);
            if constexpr (PACKED) {
                const Real *src = a.pack + (size_t)(unsigned)v * W::staged;
#pragma unroll
                for (int h = 0; h < SCH; ++h) copy_async16(d + h * nodes * 16, src + h * W::per);
            } else {
                fetch_words(d, v);
            }
            c += dc;
            j += dl;
            if (c >= nx) { c -= nx; ++j; }
            j = wrap(wrap(j, ny), ny);      // (from the row before the strip to the one after: up to 2 ny)
        }
    };

    // Plane q into ring slot q % 4: a thread takes a node, writes its source vector and its
    // (eta_I, eta_V) at every unit of the pass.
    auto fill = [&](int q) {
        const unsigned s = q & 3;
        copies_wait();
        if (rtid >= nn) return;
        Real o[4];
        ray4(0, o);
        for (int idx = rtid; idx < nn; idx += nt) {
            Real d[W::staged];
            const unsigned src = sbase + sm.stage + idx * 16;
#pragma unroll
            for (int h = 0; h < SCH; ++h) {
                if constexpr (SZ == 4) lds4(src + h * nodes * 16, 0, d + 4 * h);
                else lds2(src + h * nodes * 16, d[2 * h], d[2 * h + 1]);
            }
            const X chi_n = xset(d[0]), ns_n = xset(-d[1] * o[0]);
            // weight of the node's frequency sums, 1 / (chi N) and, for the fixed-point sums
            // (FP32), the ray's weight and the voxel's power of two
            Real t[20];
#pragma unroll
            for (int i = 0; i < 5; ++i)
                if (NS == 4 || (i == 4 && !EMG)) ray4(1 + i, t + 4 * i);
            if constexpr (!EMG) {
                Real wn;
                lds(sbase + sm.stw + idx * SZ, wn);
                if constexpr (SZ == 4) {
                    int ex;
                    lds(sbase + sm.ste + idx * 4, ex);
                    wn = quotient(wn, t[18], d[0], ray_shift(m)) * pow2(ex);
                } else {
                    wn *= rcp(d[0]);
                }
                sts(sbase + sm.wgt + (s * nodes + idx) * SZ, wn);
            }
            int v;
            lds(sbase + sm.stv + idx * 4, v);
            sts(sbase + sm.vox + (s * nodes + idx) * 4, v);
            unsigned oc = opaque(sbase + sm.coef + s * FX * sm.cplane + idx * CB), of = sbase + sm.freq;
            if constexpr (NS == 1) {
                sts(sbase + (s * nodes + idx) * SZ, d[2]);
                for (int f = 0; f < nf; ++f, oc += sm.cplane, of += 8) {
                    X x;
                    lds(of, x);
                    sts(oc, xmul(chi_n, xprofile(xadd(x, ns_n), stab)));
                }
            } else {
                const X b_n = xset(a.bfac * (d[8] * o[1] + d[9] * o[2] + d[10] * o[3]));
                Real w[4];
                // S_i(Omega) = sum_KQ (-1)^Q T^K_Q(i, Omega) S^K_-Q (Eq. 1 tensors, two-level emissivity)
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    w[i] = t[6 * i] * d[2] + t[6 * i + 1] * d[3] + Real(2) * (t[6 * i + 2] * d[4] + t[6 * i + 3] * d[5] +
                                                                              t[6 * i + 4] * d[6] + t[6 * i + 5] * d[7]);
                w[3] = d[2];
                sts4(sbase + (s * W::s_chunks * nodes + idx) * 16, nodes * 16, w);
#pragma unroll 2
                for (int f = 0; f < nf; ++f, oc += sm.cplane, of += 8) {
                    X x;
                    lds(of, x);
                    const X xs = xadd(x, ns_n), eta = xmul(chi_n, xprofile(xs, stab));
                    sts2(oc, eta, xmul(xmul(b_n, xs), eta));
                }
            }
        }
    };

    // A point's sums over the pass, times its node's weight: the fixed-point terms J^K_Q +=
    // w_m sum_p T^K_Q(p, m) I_p, Lambda-bar* += w_m L, or the per-ray partials (FP64).
    auto add_point = [&](unsigned n, const Real *sum) {
        Real wn, t[4] = {0, 0, 0, 0};
        int v;
        lds(sbase + sm.wgt + n * SZ, wn);
        lds(sbase + sm.vox + n * 4, v);
#pragma unroll
        for (int s = 0; s < NA; ++s) t[s] = sum[s] * wn;
        if (!a.jacc) {
            store_partial<Real, NS>(a, m, v, g, t);
            return;
        }
        if constexpr (SZ == 4) {
            Real y[W::nacc], sum_abs = 0;
            if constexpr (NS == 1) {
                y[0] = t[0];
                y[1] = t[1];
            } else {
                Real T[20];
#pragma unroll
                for (int i = 0; i < 5; ++i) ray4(1 + i, T + 4 * i);
#pragma unroll
                for (int k = 0; k < 6; ++k) y[k] = T[k] * t[0] + T[6 + k] * t[1] + T[12 + k] * t[2];
                y[6] = t[3];
            }
#pragma unroll
            for (int k = 0; k < W::nacc; ++k) sum_abs += fabsf(y[k]);
            unsigned long long *acc = a.jacc + v;
            if (sum_abs <= 0x1p45f) {
#pragma unroll
                for (int k = 0; k < W::nacc; ++k, acc += nvox) jadd_small(acc, y[k]);
            } else {
                // large terms, one after the other; or the weight is beyond FP32, as it is where chi
                // times the voxel's reference value is below 1e-27 or so: the sums are then as far
                // below, and 2^64 goes from one to the other
                if (!(wn < __int_as_float(0x7f800000))) {
                    Real w[4];
                    ray4(5, w);
                    wn = quotient(invn[v], w[2], a.chi[v], ray_shift(m)) * pow2(a.jexp[v] - 64);
#pragma unroll
                    for (int s = 0; s < NA; ++s) t[s] = sum[s] * Real(0x1p64) * wn;
                }
                bool bad = false;
#pragma unroll 1
                for (int k = 0; k < W::nacc; ++k, acc += nvox) {
                    Real x = k + 1 < W::nacc ? t[0] : t[NA - 1];
                    if (NS == 4 && k < 6) {
                        Real T[3];
#pragma unroll
                        for (int i = 0; i < 3; ++i) lds(sray + (4 + 6 * i + k) * SZ, T[i]);
                        x = T[0] * t[0] + T[1] * t[1] + T[2] * t[2];
                    }
                    bad |= jadd(acc, x);
                }
                if (bad) atomicOr(a.jerr, 1);
            }
        }
    };
    // the same from the totals of several groups of threads (written a phase before)
    auto add_totals = [&](int q) {
        for (int p = rtid; p < npts; p += nt) {
            Real t[4] = {0, 0, 0, 0};
            for (int h = 0; h < Lg; ++h) {
                Real w[4] = {0, 0, 0, 0};
                const unsigned o = sbase + sm.tot + ((q & 1) * a.tots + h * pw + p) * NA * SZ;
                if constexpr (NS == 1) {
                    lds(o, w[0]);
                    lds(o + SZ, w[1]);
                } else {
                    lds4(o, 16, w);
                }
#pragma unroll
                for (int s = 0; s < NA; ++s) t[s] += w[s];
            }
            add_point((q & 3) * nodes + p + nx, t);
        }
    };

    // A point's frequency integral over the thread's units
    auto totals = [&](int q, int p, const Real *acc) {
        if (Lg == 1) {
            add_point((q & 3) * nodes + p + nx, acc);
            return;
        }
        const unsigned o = sbase + sm.tot + ((q & 1) * a.tots + fg * pw + p) * NA * SZ;
        if constexpr (NS == 1) {
            sts(o, acc[0]);
            sts(o + SZ, acc[1]);
        } else {
            sts4(o, 16, acc);
        }
    };

    // The work of phase q beside the update of plane q: the nodes of plane q + 2, the sums
    // of plane q - 1, and the inputs of later planes.
    auto aside = [&](int q) {
        if (q + 2 < nz) {
            fill(q + 2);
            if (q + 3 < nz) fetch(q + 3);
            if (q + 5 < nz && tid < GW)
                copy_async(geo + ((q + 5) & 7) * GB + 4 * tid, reinterpret_cast<const int *>(G + q + 5) + tid);
        }
        if (!EMG && Lg > 1 && q >= 1) add_totals(q - 1);
    };

    // EMERGENT: a point's Stokes vectors at the frequencies of a unit, row jd of (direction,
    // frequency), to the reverse mode's store and, at the last plane, to the output
    auto emit = [&](int q, int jd, int v, const X *r) {
        const int w1 = min(XW, (m + 1) * a.nnu - jd);
#pragma unroll
        for (int w = 0; w < XW; ++w) {
            if (w >= w1) break;
            Real o[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) o[s] = xlane(r[s], w);
            if (a.store) {
                Real *d = a.store + ((long long)(jd + w) * nvox + v) * NS;
                if constexpr (NS == 1) {
                    *d = o[0];
                } else {
                    using V = typename V16<Real>::T;
#pragma unroll
                    for (int h = 0; h < 4 / W::per; ++h) chunk_put<Real>(reinterpret_cast<V *>(d) + h, o + h * W::per);
                }
            }
            if (q == nz - 1) {
                int kz;
                lds(geo + (q & 7) * GB + 8, kz);
                double *d = a.out + ((long long)(jd + w) * nx * ny + (v - vox0 - kz * nx * ny)) * NS;
#pragma unroll
                for (int s = 0; s < NS; ++s) d[s] = (double)o[s];
            }
        }
    };

    // One plane of updates (q >= 1). The bilinear weights are used relative to the first
    // one, v_M = w_M (v_00 + u_x v_01 + u_y v_10 + u_x u_y v_11), u = t / (1 - t): w_M cancels
    // in S = eps / eta; those of P are the next plane's. A corner's address is its node's offset, fixed for the sweep, plus a
    // base that is the same for all threads (array, slot, unit). The order of the steps and
    // what is held (the upwind corners' weighted sources; the downwind ones are read again
    // for every unit) keep an FP32 thread within 128 registers: a spilled value would come
    // back from L2, the halo waits' acquire invalidating L1.
    const unsigned ibuf_prev = map_rank(sbase + sm.ibuf, prev_owner);
    const unsigned full_prev = map_rank(bars.full, prev_owner);
    const unsigned row = nx * CB;
    const unsigned chS = nodes * 16, chI = ipts * 16;    // second 16-byte chunks: source (FP64), Stokes
    auto points = [&](auto HASP, int q) {
        constexpr bool has_p = decltype(HASP)::value;
        const unsigned pC = FX * sm.cplane, pS = W::s_words * nodes * SZ, pI = FX * sm.iplane;
        const unsigned stepC = Lg * sm.cplane, stepI = Lg * sm.iplane;
        const int bI = (q + 1) & 1, bW = q & 1;
        const unsigned opc = geo + (q & 7) * GB + 16, opp = geo + ((q + 1) & 7) * GB + 16;   // ux, uy, wM, dsM
        for (int pb = 0; pb < npts && fg < Lg; pb += pw) {
            // lanes beyond the last point repeat it without storing
            const bool active = pb + ptid < npts;
            const int p = min(pb + ptid, npts - 1);
            const int l = pb == 0 ? l_own : p / nx, c = pb == 0 ? c_own : p - l * nx;
            if (C > 1) {
                // the row after the strip's last one comes from the next CTA; the halo row of
                // this parity was read by the CTA before in its last phase
                if (l + 1 == R) bar_wait(bars.full + 8 * bI, ((bI ? ph.full1 : ph.full0) + (unsigned)((q - 1) >> 1)) & 1u, bars.dead, a.jerr);
                if (l == 0 && has_p && q >= 2)
                    bar_wait(bars.freed + 8 * bW, ((bW ? ph.freed1 : ph.freed0) + (unsigned)((q >> 1) - 1)) & 1u, bars.dead, a.jerr);
            }
            // node offsets (a node's coefficients, a Stokes element and, for NS = 4, a source
            // chunk have one size): row before, own row, row after; column before, own, after
            const unsigned n11 = opaque((p + nx) * CB);
            const unsigned n12 = opaque(n11 + (c + 1 == nx ? (unsigned)(1 - nx) : 1u) * CB);
            const unsigned n10 = opaque(n11 + (c == 0 ? (unsigned)(nx - 1) : (unsigned)-1) * CB);
            const unsigned n21 = opaque(n11 + row), n22 = opaque(n12 + row), n01 = opaque(n11 - row), n00 = opaque(n10 - row);
            const unsigned uS_M = sbase + ((q + 3) & 3) * pS, uS_O = sbase + (q & 3) * pS, uS_P = sbase + ((q + 1) & 3) * pS;
            const unsigned c0 = sbase + sm.coef + fg * sm.cplane, i0 = sbase + sm.ibuf + fg * sm.iplane - row;
            unsigned uM = c0 + ((q + 3) & 3) * pC, uO = c0 + (q & 3) * pC, uP = c0 + ((q + 1) & 3) * pC;
            unsigned uI = i0 + bI * pI, uW = i0 + bW * pI;
            unsigned of = sbase + sm.freq + FX * XW * SZ + fg * 8;
            const bool row0 = l == 0 && has_p && active && !(C > 1 && *bars.dead);
            // halo row of the strip before: row prev_R of its Stokes planes
            const unsigned hcol = (prev_R * nx + c) * CB;
            unsigned uH = bW * pI + fg * sm.iplane;
            Real acc[NA];
#pragma unroll
            for (int s = 0; s < NA; ++s) acc[s] = Real(0);
            int vox = 0;
            if constexpr (EMG) lds(sbase + sm.vox + ((q & 3) * nodes + p + nx) * 4, vox);
            // the corners' source vectors (NS = 4: I, Q, U and the S^0_0 that eta_V multiplies)
            auto source = [&](unsigned u, unsigned n, Real *r) {
                if constexpr (NS == 1) lds(u + n / CB * SZ, r[0]);
                else lds4(u + n, chS, r);
            };
            Real m0[NS], m1[NS], m2[NS], m3[NS], SO[NS];
            source(uS_M, n11, m0); source(uS_M, n12, m1); source(uS_M, n21, m2); source(uS_M, n22, m3);
            source(uS_O, n11, SO);
            {
                Real pm[4];
                lds4(opc, 16, pm);
                const Real uxy = pm[0] * pm[1];
#pragma unroll
                for (int s = 0; s < NS; ++s) { m1[s] *= pm[0]; m2[s] *= pm[1]; m3[s] *= uxy; }
            }
            Real p0 = 0, p1 = 0, p2 = 0, p3 = 0;             // NS = 1: the downwind sources
            if constexpr (NS == 1 && has_p) {
                source(uS_P, n11, &p0); source(uS_P, n10, &p1); source(uS_P, n01, &p2); source(uS_P, n00, &p3);
            }
#pragma unroll 1
            for (int f = fg; f < nf; f += Lg) {
                Real pm[4];                                  // ux, uy, wM, dsM
                lds4(opc, 16, pm);
                const Real ux = pm[0], uy = pm[1], uxy = ux * uy, wM = pm[2], dsM = pm[3];
                // a2-a3: transfer coefficients at M, d_M = S_O - eps_M / eta_M, -K'_V at O and M
                X eO, nkM, nkO, S3, eM, dm[NS];
                {
                    X e[NS], k, kM;
                    if constexpr (NS == 1) {
                        lds(n11 + uO, eO);
                        lds(n11 + uM, k);
                        eM = k; e[0] = xms(m0[0], k);
                        lds(n12 + uM, k);
                        eM = xfs(ux, k, eM); e[0] = xfs(m1[0], k, e[0]);
                        lds(n21 + uM, k);
                        eM = xfs(uy, k, eM); e[0] = xfs(m2[0], k, e[0]);
                        lds(n22 + uM, k);
                        eM = xfs(uxy, k, eM); e[0] = xfs(m3[0], k, e[0]);
                    } else {
                        X vO, h;
                        lds2(n11 + uO, eO, vO);
                        nkO = xmul(vO, xnrcp(eO));
                        S3 = xms(-SO[NS - 1], nkO);
                        lds2(n11 + uM, k, h);
                        eM = k; kM = h;
                        e[0] = xms(m0[0], k); e[1] = xms(m0[1], k); e[2] = xms(m0[2], k); e[3] = xms(m0[3], h);
                        lds2(n12 + uM, k, h);
                        eM = xfs(ux, k, eM); kM = xfs(ux, h, kM);
                        e[0] = xfs(m1[0], k, e[0]); e[1] = xfs(m1[1], k, e[1]); e[2] = xfs(m1[2], k, e[2]); e[3] = xfs(m1[3], h, e[3]);
                        lds2(n21 + uM, k, h);
                        eM = xfs(uy, k, eM); kM = xfs(uy, h, kM);
                        e[0] = xfs(m2[0], k, e[0]); e[1] = xfs(m2[1], k, e[1]); e[2] = xfs(m2[2], k, e[2]); e[3] = xfs(m2[3], h, e[3]);
                        lds2(n22 + uM, k, h);
                        eM = xfs(uxy, k, eM); kM = xfs(uxy, h, kM);
                        e[0] = xfs(m3[0], k, e[0]); e[1] = xfs(m3[1], k, e[1]); e[2] = xfs(m3[2], k, e[2]); e[3] = xfs(m3[3], h, e[3]);
                    }
                    const X niM = xnrcp(eM);
#pragma unroll
                    for (int s = 0; s < NS; ++s) dm[s] = xfma(e[s], niM, NS == 4 && s == 3 ? S3 : xset(SO[s]));
                    if constexpr (NS == 4) nkM = xmul(kM, niM);
                }
                // a4, a6: optical path and coefficients of the step
                const X tMO = xms(dsM, xfs(wM, eM, eO));
                const XCoef<X> co = xcoef(tMO);
                [[maybe_unused]] const X ls = has_p ? xadd(co.e0, xneg(co.wm)) : xfs(Real(0.5), co.wc, co.wo);
                // a7: right-hand side of Eq. 7, e I_M + (w_M + w_O + w_C) S_O - w_M d_M - w_C (S_O - c_M),
                // with the upwind Stokes vector over w_M (a3) and K'_V at M coupling I and V
                X r[NS];
                {
                    const X wsum = co.e0, ew = xms(wM, co.e);
                    // without a downwind point c_M = (S_M + S_O) / 2
                    const X nwm = has_p ? xneg(co.wm) : xfs(Real(-0.5), co.wc, xneg(co.wm));
#pragma unroll
                    for (int s = 0; s < NS; ++s)
                        r[s] = xfma(nwm, dm[s], NS == 4 && s == 3 ? xmul(wsum, S3) : xms(SO[s], wsum));
                    if constexpr (NS == 1) {
                        X t, u;
                        lds(n11 + uI, t);
                        lds(n12 + uI, u);
                        t = xfs(ux, u, t);
                        lds(n21 + uI, u);
                        t = xfs(uy, u, t);
                        lds(n22 + uI, u);
                        r[0] = xfma(ew, xfs(uxy, u, t), r[0]);
                    } else {
                        X t0, t1, t2, t3, u0, u1;
                        lds2(n11 + uI, t0, t1);
                        lds2(n12 + uI, u0, u1);
                        t0 = xfs(ux, u0, t0); t1 = xfs(ux, u1, t1);
                        lds2(n21 + uI, u0, u1);
                        t0 = xfs(uy, u0, t0); t1 = xfs(uy, u1, t1);
                        lds2(n22 + uI, u0, u1);
                        t0 = xfs(uxy, u0, t0); t1 = xfs(uxy, u1, t1);
                        lds2(n11 + uI + chI, t2, t3);
                        lds2(n12 + uI + chI, u0, u1);
                        t2 = xfs(ux, u0, t2); t3 = xfs(ux, u1, t3);
                        lds2(n21 + uI + chI, u0, u1);
                        t2 = xfs(uy, u0, t2); t3 = xfs(uy, u1, t3);
                        lds2(n22 + uI + chI, u0, u1);
                        t2 = xfs(uxy, u0, t2); t3 = xfs(uxy, u1, t3);
                        const X pk = xmul(xms(wM, xfs(Real(0.5), co.wc, co.wm)), nkM);
                        r[0] = xfma(pk, t3, xfma(ew, t0, r[0]));
                        r[1] = xfma(ew, t1, r[1]);
                        r[2] = xfma(ew, t2, r[2]);
                        r[3] = xfma(pk, t0, xfma(ew, t3, r[3]));
                    }
                }
                if constexpr (has_p) {
                    // downwind: -d_P = S_O - eps_P / eta_P
                    Real pp[4];                              // vx, vy, wP, dsP
                    lds4(opp, 16, pp);
                    const Real vx = pp[0], vy = pp[1], vxy = vx * vy, wP = pp[2], dsP = pp[3];
                    X eP, e[NS];
                    if constexpr (NS == 1) {
                        X k;
                        lds(n11 + uP, k);
                        eP = k; e[0] = xms(p0, k);
                        lds(n10 + uP, k);
                        k = xms(vx, k); eP = xadd(eP, k); e[0] = xfs(p1, k, e[0]);
                        lds(n01 + uP, k);
                        k = xms(vy, k); eP = xadd(eP, k); e[0] = xfs(p2, k, e[0]);
                        lds(n00 + uP, k);
                        k = xms(vxy, k); eP = xadd(eP, k); e[0] = xfs(p3, k, e[0]);
                    } else {
                        X k, h;
                        Real w[4];
                        lds2(n11 + uP, k, h);
                        lds4(uS_P + n11, chS, w);
                        eP = k;
                        e[0] = xms(w[0], k); e[1] = xms(w[1], k); e[2] = xms(w[2], k); e[3] = xms(w[3], h);
                        lds2(n10 + uP, k, h);
                        lds4(uS_P + n10, chS, w);
                        k = xms(vx, k); h = xms(vx, h); eP = xadd(eP, k);
                        e[0] = xfs(w[0], k, e[0]); e[1] = xfs(w[1], k, e[1]); e[2] = xfs(w[2], k, e[2]); e[3] = xfs(w[3], h, e[3]);
                        lds2(n01 + uP, k, h);
                        lds4(uS_P + n01, chS, w);
                        k = xms(vy, k); h = xms(vy, h); eP = xadd(eP, k);
                        e[0] = xfs(w[0], k, e[0]); e[1] = xfs(w[1], k, e[1]); e[2] = xfs(w[2], k, e[2]); e[3] = xfs(w[3], h, e[3]);
                        lds2(n00 + uP, k, h);
                        lds4(uS_P + n00, chS, w);
                        k = xms(vxy, k); h = xms(vxy, h); eP = xadd(eP, k);
                        e[0] = xfs(w[0], k, e[0]); e[1] = xfs(w[1], k, e[1]); e[2] = xfs(w[2], k, e[2]); e[3] = xfs(w[3], h, e[3]);
                    }
                    const X niP = xnrcp(eP);
                    const X tOP = xms(dsP, xfs(wP, eP, eO));
                    // a5: BESSER control points per Stokes parameter
                    const X hh = xms(Real(0.5), xrcp(xadd(tMO, tOP))), nr = xmul(tMO, xnrcp(tOP));
                    const X na = xmul(xmul(tMO, hh), nr), gb = xmul(tOP, hh), nwc = xneg(co.wc);
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const X ndp = xfma(e[s], niP, NS == 4 && s == 3 ? S3 : xset(SO[s]));
                        r[s] = xfma(nwc, xoffset(dm[s], ndp, na, gb, nr), r[s]);
                    }
                }
                if constexpr (NS == 4) {
                    // kappa^-1 = 1 + psi'_O K'_O (Eq. 8) couples I and V only; psi' = w + w_C / 2.
                    // In FP32 1 / (1 - a^2) as 1 + a^2 / (1 - a^2): the approximate reciprocal of a
                    // number near 1 is 2.5e-8 too large on average, which went into every plane's I
                    // (64 x 64 x 64: J^0_0 of the deep layers 1.8e-8 too large, now 1e-9; the iterates'
                    // error from 64 bits 6.3e-6 -> 4.5e-6)
                    const X nav = xmul(xfs(Real(0.5), co.wc, co.wo), nkO), a2 = xmul(nav, nav);
                    const X idet = xrcp(xadd(xset(Real(1)), xneg(a2)));
                    const X i = xfma(nav, r[3], r[0]), v = xfma(nav, r[0], r[3]);
                    if constexpr (SZ == 4) {
                        const X g = xmul(a2, idet);
                        r[0] = xfma(i, g, i);
                        r[3] = xfma(v, g, v);
                    } else {
                        r[0] = xmul(i, idet);
                        r[3] = xmul(v, idet);
                    }
                }
                if (active) {
                    if constexpr (NS == 1) {
                        sts(n11 + uW, r[0]);
                    } else {
                        sts2(n11 + uW, r[0], r[1]);
                        sts2(n11 + uW + chI, r[2], r[3]);
                    }
                }
                if (row0) {
                    if (C > 1) {
                        const unsigned d = ibuf_prev + hcol + uH, b = full_prev + 8 * bW;
                        if constexpr (NS == 1) {
                            push(d, b, r[0]);
                        } else {
                            push2(d, b, r[0], r[1]);
                            push2(d + chI, b, r[2], r[3]);
                        }
                    } else {
                        const unsigned d = sbase + sm.ibuf + hcol + uH;
                        if constexpr (NS == 1) {
                            sts(d, r[0]);
                        } else {
                            sts2(d, r[0], r[1]);
                            sts2(d + chI, r[2], r[3]);
                        }
                    }
                }
                if constexpr (EMG) {
                    if (active) emit(q, m * a.nnu + j0 + f * XW, vox, r);
                } else {
                    // a8: Lambda* and frequency integration (w_nu phi / N = w_nu eta_I / (chi N))
                    X wt;
                    lds(of, wt);
                    wt = xmul(wt, eO);
#pragma unroll
                    for (int s = 0; s < NA - 1; ++s) acc[s] = xdot(wt, r[s], acc[s]);
                    acc[NA - 1] = xdot(wt, ls, acc[NA - 1]);
                }
                if (PROBE && a.probe_ray == m && active) {
                    const int v = point_voxel(q, l, c);
                    for (int w = 0; w < XW && j0 + f * XW + w < a.nnu; ++w) {
                        const long long pv = (long long)(j0 + f * XW + w) * a.nvox + v;
#pragma unroll
                        for (int s = 0; s < NS; ++s) a.probe[pv * NS + s] = xlane(r[s], w);
                        a.probe_ls[pv] = xlane(ls, w);
                    }
                }
                uM += stepC; uO += stepC; uP += stepC; uI += stepI; uW += stepI; uH += stepI; of += Lg * 8;
            }
            if (!EMG && active) totals(q, p, acc);
        }
    };

    // boundary plane: I = (B, 0, 0, 0) entering at the bottom, 0 at the top; Lambda* = 0
    auto boundary = [&]() {
        Real mu;
        lds(sray, mu);
        const bool upward = mu > Real(0);
        for (int p = ptid; p < npts && fg < Lg; p += pw) {
            const int l = p / nx, c = p - l * nx;
            const int v = point_voxel(0, l, c);
            const X zero = xset(Real(0)), I0 = xset(upward ? a.bpl[v] : Real(0));
            Real acc[NA];
#pragma unroll
            for (int s = 0; s < NA; ++s) acc[s] = Real(0);
            for (int f = fg; f < nf; f += Lg) {
                const unsigned o = sbase + sm.ibuf + f * sm.iplane + p * CB, h = f * sm.iplane + (prev_R * nx + c) * CB;
                if constexpr (NS == 1) {
                    sts(o, I0);
                    if (l == 0) {
                        if (C > 1) push(ibuf_prev + h, full_prev, I0);
                        else sts(sbase + sm.ibuf + h, I0);
                    }
                } else {
                    sts2(o, I0, zero);
                    sts2(o + chI, zero, zero);
                    if (l == 0) {
                        if (C > 1) {
                            push2(ibuf_prev + h, full_prev, I0, zero);
                            push2(ibuf_prev + h + chI, full_prev, zero, zero);
                        } else {
                            sts2(sbase + sm.ibuf + h, I0, zero);
                            sts2(sbase + sm.ibuf + h + chI, zero, zero);
                        }
                    }
                }
                if constexpr (EMG) {
                    X r[NS];
#pragma unroll
                    for (int s = 0; s < NS; ++s) r[s] = s == 0 ? I0 : zero;
                    emit(0, m * a.nnu + j0 + f * XW, v, r);
                } else {
                    X eta, wt;
                    lds(sbase + sm.coef + f * sm.cplane + (p + nx) * CB, eta);
                    lds(sbase + sm.freq + FX * XW * SZ + f * 8, wt);
                    acc[0] = xdot(xmul(wt, eta), I0, acc[0]);
                }
                if (PROBE && a.probe_ray == m) {
                    for (int w = 0; w < XW && j0 + f * XW + w < a.nnu; ++w) {
                        const long long pv = (long long)(j0 + f * XW + w) * a.nvox + v;
#pragma unroll
                        for (int s = 0; s < NS; ++s) a.probe[pv * NS + s] = s == 0 ? xlane(I0, w) : Real(0);
                        a.probe_ls[pv] = Real(0);
                    }
                }
            }
            if (!EMG) totals(0, p, acc);
        }
    };

    // One CTA barrier per plane: in phase q the threads update plane q (reading the nodes
    // of planes q - 1, q, q + 1), fill plane q + 2 and add up plane q - 1. None of these
    // reads what another writes in the same phase, so the warps run them in either order
    // and the waits of one hide behind the arithmetic of another: those of the strip's
    // first rows update first (the CTA before waits for row 0), those of its last rows
    // last (they wait for the CTA after).
    fetch(0);
    fill(0);
    fetch(1);
    fill(1);
    if (nz > 2) fetch(2);
    __syncthreads();
    const bool late = 2 * ((wid * 32 - fg * pw) / nx) >= R;
    const unsigned halo_bytes = (unsigned)(nf * nx * NS) * 8;
    const unsigned freed_next = map_rank(bars.freed, next_owner);
    for (int q = 0; q < nz; ++q) {
        // the halo row of plane q arrives during this plane's update and the next
        if (C > 1 && tid == 0 && R > 0 && q + 1 < nz && !*bars.dead) bar_expect(bars.full + 8 * (q & 1), halo_bytes);
        for (int part = 0; part < 2; ++part) {
            if ((part != 0) != late) {
                aside(q);
                continue;
            }
            if (q == 0) boundary();
            else if (q + 1 < nz) points(std::true_type{}, q);
            else points(std::false_type{}, q);
        }
        __syncthreads();
        // the halo row of plane q - 1 has been read: plane q + 1 may overwrite it (where it does)
        if (C > 1 && tid == 0 && R > 0 && q >= 1 && q + 2 < nz && !*bars.dead) bar_arrive_remote(freed_next + 8 * ((q + 1) & 1));
    }
    // the last plane's sums
    aside(nz);
    __syncthreads();
    if (R > 0) {
        // phases of this item: halo rows of the planes 0 .. nz - 2; those that were overwritten
        ph.full0 += (unsigned)(nz / 2);
        ph.full1 += (unsigned)((nz - 1) / 2);
        ph.freed0 += (unsigned)(nz / 2) - 1u;
        ph.freed1 += nz >= 4 ? (unsigned)((nz - 1) / 2) - 1u : 0u;
    }
}

template <typename Real, int NS, int MODE, bool PACKED>
__global__ void __launch_bounds__(jsweep_max_threads<Real, NS>(), 1) jsweep_kernel(const SweepArgs<Real> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) Real sray[24];
    __shared__ __align__(8) unsigned long long s_bar[4];
    __shared__ int s_dead, s_item[2];
    __shared__ double s_exp[sizeof(Real) == 8 ? 64 : 1];
    profile_table<Real>(s_exp);
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int cid = blockIdx.x / C;
    const int ncl = gridDim.x / C;
    constexpr int XW = jsweep_lanes<Real>();
    const JSmem sm = jsmem<Real, NS>(a.ring_plane, a.ipts_max, a.tots, (a.F + XW - 1) / XW);
    JBars bars;
    bars.full = smem_u32(s_bar);
    bars.freed = smem_u32(s_bar + 2);
    bars.dead = &s_dead;
    JPhase ph = {0, 0, 0, 0};
    if (threadIdx.x == 0) {
        s_dead = 0;
        for (int b = 0; b < 4; ++b) bar_init(smem_u32(s_bar + b));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster.sync();
    // fixed-point sums do not depend on the order of their terms: the frequency groups of a
    // ray are items of their own; per-ray partials add their groups in order in one item
    const int split = a.jacc || MODE == EMERGENT ? a.ngroups : 1;
    const int total = a.nitems * split;
    for (int k = 0, own = cid;; ++k, own += ncl) {
        int item = own;
        if (a.next_item) {
            if (rank == 0 && threadIdx.x == 0) {
                const int it = atomicAdd(a.next_item, 1);
                for (int r = 0; r < C; ++r) *cluster.map_shared_rank(s_item + (k & 1), r) = it;
            }
            cluster.sync();
            item = s_item[k & 1];
        }
        if (item >= total) break;
        const int ray = item / split;
        const int code = a.items ? a.items[ray] : ray;
        const int box = MODE == EMERGENT ? 0 : code / a.nray, m = code - box * a.nray;
        const int g0 = item - ray * split;
        // the ray's constants (mu, ox, oy, oz, T[18], w, pad); the item starts with a barrier
        if (threadIdx.x < 24) sray[threadIdx.x] = reinterpret_cast<const Real *>(a.rays + m)[threadIdx.x];
        for (int g = g0; g < (split > 1 ? g0 + 1 : a.ngroups); ++g) {
            // (a CTA whose wait ran out signals nothing any more)
            if (C == 1 || !*bars.dead)
                jsweep_item<Real, NS, MODE, PACKED>(a, smem_u32(smem_raw), sm, bars, ph, smem_u32(sray), smem_u32(s_exp), box, m, g,
                                                    rank, C);
            // every halo row of the item has been written and read before the next one
            // (whose strips may have other neighbours)
            if (C > 1) cluster.sync();
        }
    }
}

// Before a formal solution: the error flag (where jerr is set) to 0, and the
// fixed-point scale of each voxel: 2^e with e = 46 - ilogb(max(|S^0_0|, |B|)),
// so that a term of the size of the voxel's source function or Planck function
// carries 46 fraction bits and the accumulator has 2^16 of headroom above it
// (an FP32 term then converts without rounding; an FP64 term rounds at 2^-47 of
// the reference value).
// (jacc null: the FP64 form, which has no fixed-point sums; pack null: sweep_jw.cu, or no
// room for them: the inputs are read where they are). The same pass packs each
// voxel's inputs of the sweep next to each other, so that a node's inputs arrive in
// shared memory by 16-byte copies: chi, vel, rho[6], bx, by, bz (NS = 1: chi, vel, rho).
template <typename Real, int NS>
__global__ void jacc_prepare_kernel(const SweepArgs<Real> a, int *jexp, Real *pack)
{
    const long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long nvox = a.nvox;
    if (v >= nvox) return;
    if (v == 0 && a.jerr) *a.jerr = 0;
    using W = JW<Real, NS>;
    if (pack) {
        Real w[W::staged];
        w[0] = a.chi[v];
        w[1] = a.vel[v];
        w[2] = a.rho[v];
        w[W::staged - 1] = Real(0);
        if constexpr (NS == 4) {
#pragma unroll
            for (int k = 1; k < 6; ++k) w[2 + k] = a.rho[k * nvox + v];
            w[8] = a.bx[v];
            w[9] = a.by[v];
            w[10] = a.bz[v];
        }
        using V = typename V16<Real>::T;
#pragma unroll
        for (int h = 0; h < W::staged / W::per; ++h) chunk_put<Real>(reinterpret_cast<V *>(pack + v * W::staged) + h, w + h * W::per);
    }
    if (!a.jacc) return;
    const double ref = fmax(fmax(fabs((double)a.rho[v]), fabs((double)a.bpl[v])), 1e-30);
    // kept within the FP32 exponent range, where the sweep forms 2^e exactly
    jexp[v] = min(max(kJFrac - ilogb(ref), -100), 126);
#pragma unroll
    for (int k = 0; k < W::nacc; ++k) a.jacc[k * nvox + v] = 0ULL;
}

template <int NS>
__global__ void jacc_finalize_kernel(long long nvox, const unsigned long long *jacc, const int *jexp, double *jkq,
                                     double *lstar, const int *err, int *handed)
{
    const long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int flag = v == 0 ? *err : 0;
    if (v >= nvox) return;
    const double inv = ldexp(1.0, -jexp[v]);
    constexpr int NJ = NS == 1 ? 1 : 6;
#pragma unroll
    for (int k = 0; k < NJ; ++k) jkq[v * NJ + k] = (double)(long long)jacc[k * nvox + v] * inv;
    lstar[v] = (double)(long long)jacc[NJ * nvox + v] * inv;
    if (flag) atomicOr(handed, flag);
}

// bar_wait_long on an mbarrier at which nothing arrives
__global__ void halo_wait_kernel(int *err, unsigned long long *ns)
{
    __shared__ __align__(8) unsigned long long s_bar;
    __shared__ int s_dead;
    s_dead = 0;
    bar_init(smem_u32(&s_bar));
    const unsigned long long t0 = global_ns();
    bar_wait_long(smem_u32(&s_bar), 0, &s_dead, err);
    *ns = global_ns() - t0;
}
cudaError_t run_halo_wait(int *err, unsigned long long *ns, cudaStream_t st)
{
    halo_wait_kernel<<<1, 1, 0, st>>>(err, ns);
    return cudaGetLastError();
}

// diagnostic: the coefficients of a unit and the profile as the sweep evaluates them (a thread
// takes a pair in FP32): out[6 i] = e, e0, w_M, w_O, w_C at t[i], exp(-x[i]^2)
template <typename Real>
__global__ void unit_kernel(int n, const double *t, const double *x, double *out)
{
    using X = typename XOf<Real>::X;
    constexpr int XW = jsweep_lanes<Real>();
    __shared__ double s_exp[64];
    profile_table<Real>(s_exp);
    __syncthreads();
    const int i0 = XW * (blockIdx.x * blockDim.x + threadIdx.x), i1 = min(i0 + XW - 1, n - 1);
    if (i0 >= n) return;
    auto put = [](double a, double b) {
        if constexpr (XW == 2) return make_float2((float)a, (float)b);
        else return a;
    };
    const XCoef<X> c = xcoef(put(t[i0], t[i1]));
    const X p = xprofile(put(x[i0], x[i1]), smem_u32(s_exp));
    for (int w = 0; w <= i1 - i0; ++w) {
        const X v[6] = {c.e, c.e0, c.wm, c.wo, c.wc, p};
        for (int k = 0; k < 6; ++k) out[6 * (i0 + w) + k] = (double)xlane(v[k], w);
    }
}
template <typename Real>
cudaError_t run_unit(int n, const double *t, const double *x, double *out, cudaStream_t st)
{
    const int nt = (n + jsweep_lanes<Real>() - 1) / jsweep_lanes<Real>();
    unit_kernel<Real><<<(nt + 127) / 128, 128, 0, st>>>(n, t, x, out);
    return cudaGetLastError();
}
template cudaError_t run_unit<float>(int, const double *, const double *, double *, cudaStream_t);
template cudaError_t run_unit<double>(int, const double *, const double *, double *, cudaStream_t);

template <typename Real, int NS>
cudaError_t launch_jacc_prepare(const SweepArgs<Real> &a, cudaStream_t st)
{
    static_assert(JW<Real, NS>::staged == jpack_words<NS>(), "packed inputs of a voxel");
    const int bs = 256;
    const long long nb = (a.nvox + bs - 1) / bs;
    jacc_prepare_kernel<Real, NS><<<(unsigned)nb, bs, 0, st>>>(a, const_cast<int *>(a.jexp), const_cast<Real *>(a.pack));
    return cudaGetLastError();
}

template <int NS>
cudaError_t launch_jacc_finalize(long long nvox, const unsigned long long *jacc, const int *jexp, double *jkq,
                                 double *lstar, const int *err, int *handed, cudaStream_t st)
{
    const int bs = 256;
    const long long nb = (nvox + bs - 1) / bs;
    jacc_finalize_kernel<NS><<<(unsigned)nb, bs, 0, st>>>(nvox, jacc, jexp, jkq, lstar, err, handed);
    return cudaGetLastError();
}

template <typename Real, int NS, int MODE, bool PACKED>
static cudaError_t jprepare(int cluster, int smem)
{
    void *k = (void *)jsweep_kernel<Real, NS, MODE, PACKED>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (cluster > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <typename Real, int NS>
cudaError_t jsweep_max_active_clusters(int cluster, int smem, int threads, int *out)
{
    cudaError_t e = jprepare<Real, NS, SUMS, true>(cluster, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cluster);
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(out, jsweep_kernel<Real, NS, SUMS, true>, &lc);
}

// the probe variant writes one ray's Stokes vectors and Lambda* at every node and
// frequency (porta_probe_ray); the plain one keeps no trace of that in its loop. A diagnostic,
// it has the form that needs no packed inputs only.
template <typename Real, int NS, int MODE, bool PACKED>
static cudaError_t jlaunch(const SweepArgs<Real> &a, const LaunchCfg &cfg, cudaStream_t st)
{
    cudaError_t e = jprepare<Real, NS, MODE, PACKED>(cfg.cluster, cfg.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cfg.clusters * cfg.cluster);
    lc.blockDim = dim3(cfg.threads);
    lc.dynamicSmemBytes = cfg.smem;
    lc.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cfg.cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    if (cfg.priority != 0) {
        at[1].id = cudaLaunchAttributePriority;
        at[1].val.priority = cfg.priority;
        lc.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&lc, jsweep_kernel<Real, NS, MODE, PACKED>, a);
}

template <typename Real, int NS>
cudaError_t launch_jsweep(const SweepArgs<Real> &a, LaunchCfg &cfg, cudaStream_t st)
{
    if (a.out) return a.pack ? jlaunch<Real, NS, EMERGENT, true>(a, cfg, st) : jlaunch<Real, NS, EMERGENT, false>(a, cfg, st);
    if (a.probe_ray >= 0) return jlaunch<Real, NS, PROBE_RAY, false>(a, cfg, st);
    return a.pack ? jlaunch<Real, NS, SUMS, true>(a, cfg, st) : jlaunch<Real, NS, SUMS, false>(a, cfg, st);
}

#define PORTA_JINST(R, N)                                                                    \
    template int jsweep_smem_bytes<R, N>(int, int, int, int);                                \
    template cudaError_t jsweep_max_active_clusters<R, N>(int, int, int, int *);             \
    template cudaError_t launch_jsweep<R, N>(const SweepArgs<R> &, LaunchCfg &, cudaStream_t);          \
    template cudaError_t launch_jacc_prepare<R, N>(const SweepArgs<R> &, cudaStream_t);
PORTA_JINST(float, 1)
PORTA_JINST(float, 4)
PORTA_JINST(double, 1)
PORTA_JINST(double, 4)
#undef PORTA_JINST
template cudaError_t launch_jacc_finalize<1>(long long, const unsigned long long *, const int *, double *, double *,
                                             const int *, int *, cudaStream_t);
template cudaError_t launch_jacc_finalize<4>(long long, const unsigned long long *, const int *, double *, double *,
                                             const int *, int *, cudaStream_t);

}  // namespace porta
