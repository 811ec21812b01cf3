// Host internals of the C ABI (include/porta.h) shared by its translation
// units: api.cu (contexts, formal solution, Jacobi iteration, frequency bands),
// api_adjoint.cu (emergent Stokes profiles and reverse mode), api_mg.cu
// (multigrid, Sec. 5) and api_ml.cu (multilevel atoms). Error reporting, the
// capped device allocator, the per-ray plane geometry and the sweep's launch
// shape selection.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <limits>
#include <string>
#include <vector>

#include "porta.h"
#include "porta_ctx.h"
#include "porta_internal.cuh"

namespace porta_api {

using namespace porta;

// records msg as the context's last error and returns code
int fail(porta_ctx *c, int code, const std::string &msg);

#define CK(call)                                                                               \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            return fail(c, PORTA_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
    } while (0)

// Device allocations of the library go through pmalloc / pfree, which keep the
// live byte count and honour the process-wide cap of porta_set_device_limit: an
// allocation that would exceed the cap fails with cudaErrorMemoryAllocation
// (reported as PORTA_ENOMEM) without calling the CUDA runtime.
cudaError_t pmalloc_bytes(void **p, size_t bytes);
cudaError_t pfree(void *p);

template <typename T>
cudaError_t pmalloc(T **p, size_t bytes)
{
    void *q = nullptr;
    cudaError_t e = pmalloc_bytes(&q, bytes);
    *p = (T *)q;
    return e;
}

template <typename T>
cudaError_t dalloc(T **p, size_t n)
{
    *p = nullptr;
    if (n == 0) return cudaSuccess;
    return pmalloc(p, n * sizeof(T));
}

// T^K_Q(i, Omega) for i = I, Q, U from the polarization tensors of the ray
// frame: with e_a = dOmega/dtheta and e_b = z x Omega / |z x Omega|, Stokes
// I, Q, U correspond to e_a e_a + e_b e_b, e_a e_a - e_b e_b, e_a e_b + e_b e_a;
// T^0_0 is half the trace and T^2_Q = -sqrt(3)/2 times the spherical
// components of the traceless part (A_0 = sqrt(3/2) A_zz, A_1 = -(A_xz + i A_yz),
// A_2 = (A_xx - A_yy + 2 i A_xy)/2). Output rows of 6 reals per Stokes parameter.
void tkq_tensors(double mu, double chi, double out[18]);

// Gauss-Legendre nodes and weights on (0, 1), n of each, x increasing
void gauss_legendre(int n, double *x, double *w);

// drops the context's captured Jacobi-iteration graph
void drop_graph(porta_ctx *c);
// set c->gsweep = 2 (the global-memory sweep) once, where no shared-memory sweep fits
void check_global_sweep(porta_ctx *c);

inline long long wrapll(long long a, long long n)
{
    if (a >= 0 && a < n) return a;      // (mostly: a division is the longest part of a plane's geometry)
    long long r = a % n;
    return r < 0 ? r + n : r;
}

// plane geometry of one direction in sweep order (see PlaneGeom) for a grid
// nx x ny x nz with periods lx, ly and heights z
template <typename Real>
void plane_geometry(int nx, int ny, int nz, double lx, double ly, const double *z, double mu, double chi,
                    PlaneGeom<Real> *g)
{
    const bool up = mu > 0;
    const double st = std::sqrt(std::max(0.0, 1.0 - mu * mu));
    const double ox = st * std::cos(chi), oy = st * std::sin(chi);
    const double hx = lx / nx, hy = ly / ny, amu = std::fabs(mu);
    long long ax = 0, ay = 0;
    for (int q = 0; q < nz; ++q) {
        int kz = up ? q : nz - 1 - q;
        PlaneGeom<Real> p{};
        p.kz = kz;
        if (q > 0) {
            int ku = up ? kz - 1 : kz + 1;
            double ds = std::fabs(z[kz] - z[ku]) / amu;
            double dx = ds * ox / hx, dy = ds * oy / hy;
            double cx = std::ceil(dx), cy = std::ceil(dy);
            ax = wrapll(ax + (long long)cx, nx);
            ay = wrapll(ay + (long long)cy, ny);
            p.tx = (Real)(cx - dx);
            p.ty = (Real)(cy - dy);
            p.ds = (Real)ds;
        }
        p.ax = (int)ax;
        p.ay = (int)ay;
        g[q] = p;
    }
}

// the next larger or smaller value of a positive normal one
inline float neighbour(float x, bool up)
{
    std::int32_t b;
    std::memcpy(&b, &x, sizeof(b));
    b += up ? 1 : -1;
    std::memcpy(&x, &b, sizeof(b));
    return x;
}
inline double neighbour(double x, bool up)
{
    std::int64_t b;
    std::memcpy(&b, &x, sizeof(b));
    b += up ? 1 : -1;
    std::memcpy(&x, &b, sizeof(b));
    return x;
}

// the same for the J^K_Q sweep, which uses the bilinear weights relative to the first one:
// in place of (tx, ty, ds, pad2) it reads u = t / (1 - t) along x and y, the first weight
// (1 - tx) (1 - ty), and ds / 2, each from FP64.
//
// A point within half a rounding unit of the next node (t = 1: a ray along a grid axis whose
// other component is 1e-17 and not 0) is taken there, t = 0, with the plane's offset ax or ay
// one less from here on. (Held at 1 - t = 2^-24 it moved by that much at every plane: 64 planes,
// the profiles along two axes 37e-7 from their values in Q and U, along the others 3e-7.)
//
// What is rounded goes up or down so that the errors do not gather along a ray: planes of
// equal spacing have equal values, whose errors would add up with one sign. u keeps the sum
// of the point's displacements near 0, and the first weight, which is what makes the rounded
// weights add up to 1, keeps the product of their sums at 1 (a ray through a transparent
// medium would gather their excess, 2e-8 per plane rms, 1e-6 after 64 planes).
template <typename Real>
void relative_geometry(const PlaneGeom<double> *p, int nx, int ny, int nz, PlaneGeom<Real> *r)
{
    const double half = sizeof(Real) == 4 ? 2.98023223876953125e-08 : 5.551115123125783e-17;
    double gathered = 0.0;
    struct Axis {
        double moved = 0.0;     // sum of the displacements so far, in cells
        int back = 0;           // how much less the offset is than the general form's, modulo the cells
    } x, y;
    auto ratio = [&](double t, Axis &a, int n_cell) {
        if (1.0 - t <= half) {
            a.moved += 1.0 - t;
            a.back = a.back + 1 == n_cell ? 0 : a.back + 1;
            return Real(0);
        }
        const double u = t / (1.0 - t), dt = (1.0 - t) * (1.0 - t);      // (dt / du)
        const Real n = (Real)u;
        if (!(n > std::numeric_limits<Real>::min())) return n;
        const Real o = neighbour(n, (double)n < u);
        const double en = a.moved + ((double)n - u) * dt, eo = a.moved + ((double)o - u) * dt;
        const bool swap = std::fabs(eo) < std::fabs(en);
        a.moved = swap ? eo : en;
        return swap ? o : n;
    };
    for (int q = 0; q < nz; ++q) {
        r[q] = {};
        r[q].kz = p[q].kz;
        r[q].tx = ratio(p[q].tx, x, nx);
        r[q].ty = ratio(p[q].ty, y, ny);
        r[q].ax = p[q].ax - x.back + (p[q].ax < x.back ? nx : 0);
        r[q].ay = p[q].ay - y.back + (p[q].ay < y.back ? ny : 0);
        r[q].pad2 = (Real)(0.5 * p[q].ds);
        const Real uxy = r[q].tx * r[q].ty;        // as the sweep forms it
        const double sum = 1.0 + (double)r[q].tx + (double)r[q].ty + (double)uxy;
        const Real w = (Real)(1.0 / sum);
        const double e0 = (double)w * sum - 1.0;
        const Real other = neighbour(w, e0 < 0.0);
        const double e1 = (double)other * sum - 1.0;
        const bool swap = std::fabs(gathered + e1) < std::fabs(gathered + e0);
        r[q].ds = swap ? other : w;
        if (q > 0) gathered += swap ? e1 : e0;
    }
}

// both forms of one direction
template <typename Real>
void plane_geometry(int nx, int ny, int nz, double lx, double ly, const double *z, double mu, double chi,
                    PlaneGeom<Real> *g, PlaneGeom<Real> *rel)
{
    std::vector<PlaneGeom<double>> d(nz);
    plane_geometry(nx, ny, nz, lx, ly, z, mu, chi, d.data());
    for (int q = 0; q < nz; ++q) {
        g[q] = {};
        g[q].ax = d[q].ax;
        g[q].ay = d[q].ay;
        g[q].kz = d[q].kz;
        g[q].tx = (Real)d[q].tx;
        g[q].ty = (Real)d[q].ty;
        g[q].ds = (Real)d[q].ds;
    }
    relative_geometry(d.data(), nx, ny, nz, rel);
}

template <typename Real>
RayDev<Real> ray_dev(double mu, double chi, double w = 0.0)
{
    RayDev<Real> r{};
    r.w = (Real)w;
    double st = std::sqrt(std::max(0.0, 1.0 - mu * mu));
    r.mu = (Real)mu;
    r.ox = (Real)(st * std::cos(chi));
    r.oy = (Real)(st * std::sin(chi));
    r.oz = (Real)mu;
    double t[18];
    tkq_tensors(mu, chi, t);
    for (int i = 0; i < 18; ++i) r.t[i] = (Real)t[i];
    return r;
}

const int kThreads = 512;   // maximum threads per CTA of the sweep kernel
const int kSmemLimit = 220 * 1024;
const int kJSmemLimit = 226 * 1024;   // J^K_Q sweep (its static shared memory stays below 1 KB)

// Shared-memory capacities of a launch with cluster size C over all boxes:
// ring plane (16-byte chunks) and Stokes-plane points, each the maximum over boxes.
template <typename Real, int NS>
void launch_caps(const porta_ctx *c, int C, int &ring_plane, int &ipts_max, bool jk = false)
{
    const int nch = (NS == 1 ? 4 : 8) * (int)sizeof(Real) / 16;
    const bool dich = NS == 4 && c->d_dich != nullptr;
    ring_plane = 0;
    ipts_max = 0;
    for (const BoxDev &b : c->boxes) {
        const int rmax = (b.ny + C - 1) / C;
        const int chunk = (rmax + 2) * b.nx;
        if (jk) {
            // the J^K_Q sweep (sweep_j.cu): ring capacity in nodes, Stokes planes
            ring_plane = std::max(ring_plane, chunk);
            ipts_max = std::max(ipts_max, (rmax + (c->jk_form == 1 ? 1 : 0)) * b.nx);   // (sweep_j.cu: with the halo row)
            continue;
        }
        // with dichroism the slots of a second ring follow the node ring (eta_U / eta_I and the
        // two orientation terms, 3 words per node); an explicit medium keeps K'/eta_I there
        // (6 words per node); the biquadratic stencils need two halo rows on each side instead of one
        const int gchunk = c->interp == 2 && !c->d_kexpl ? (rmax + 4) * b.nx : chunk;
        const int dwords = dich ? 3 : (c->d_kexpl ? 6 : 0);
        const int dchunks = (dwords * ((chunk * (int)sizeof(Real) + 15) / 16 * 16) + 15) / 16;
        ring_plane = std::max(ring_plane, nch * gchunk + dchunks);
        ipts_max = std::max(ipts_max, rmax * b.nx);
    }
}

// The J^K_Q formal solution runs the kernel of sweep_j.cu (per-frequency
// node coefficients in shared memory) unless the lines carry dichroism, which
// only the general sweep (sweep.cu) implements, or a plane is too wide for its
// shared memory: then that of sweep_jw.cu, which needs less per node, or the general
// sweep, which needs less per frequency. jk_form says which of the two kernels.
bool use_jk(const porta_ctx *c);

// The J^K_Q sweep sums an FP32 formal solution into fixed-point accumulators;
// an FP64 one keeps per-ray partial integrals summed in ray order in FP64 (a
// fixed-point scale cannot hold 1e-10 relative precision for quantities that
// span many decades within one voxel, as Lambda-bar* does with optical depth).
bool jfixed(const porta_ctx *c);
// work items of a ray: sweep_j.cu deals out the passes of an FP32 ray separately
int jparts(const porta_ctx *c, int ngroups);

// frequencies of the J^K_Q formal solution (its band, porta_set_freq_range)
int jnu(const porta_ctx *c);

// largest / smallest plane height ny over the context's boxes
int max_ny(const porta_ctx *c);
int min_ny(const porta_ctx *c);

// threads of a J^K_Q sweep CTA (those of the box that needs most) and the entries of its
// totals buffer: as many where some box's strips take several groups of threads, else 0
template <typename Real, int NS>
int jsweep_tots(const porta_ctx *c, int C, int F, int *threads_out)
{
    const int FX = (F + jsweep_lanes<Real>() - 1) / jsweep_lanes<Real>();
    int threads = 64;
    for (const BoxDev &b : c->boxes)
        threads = std::max(threads, jsweep_threads(b.nx, (b.ny + C - 1) / C, FX, jsweep_max_threads<Real, NS>()));
    if (threads_out) *threads_out = threads;
    for (const BoxDev &b : c->boxes)
        // (a strip of the box may have one row less than the largest)
        if (FX > 1 && threads / ((std::max(1, b.ny / C) * b.nx + 31) / 32 * 32) > 1) return threads;
    return 0;
}

// Cycles of one plane of one pass of the J^K_Q sweep in a CTA: a chain of fixed length
// (barrier, geometry, sources of the corners, sums), the units of the points' rounds one
// after the other, a round of the nodes' filling, whose length grows little with the
// frequencies, and a little for the exchange between CTAs (without it two CTAs tie with one on
// 8 x 8 planes: 58 and 50 us per call); in FP64 also the operations of all points and of
// `share` CTAs at 1/64 of the FP32 rate, whichever is longer (smoothly). Fitted to forced
// shapes of boxes from 8 x 8 x 16 to 64 x 64 x 64 (C 1 to 16, every number of passes): the
// shape it picks was the fastest of all, or within 2% of it (FP64: 4%), for each.
template <typename Real, int NS>
double jsweep_plane_cost(int nx, int R, int F, int threads, int share, bool exchange)
{
    const int W = jsweep_lanes<Real>(), FX = (F + W - 1) / W;
    const int pts = R * nx, nodes = (R + 2) * nx;
    const int pw = std::min(threads, (pts + 31) / 32 * 32), Lg = std::min(FX, threads / pw);
    const double units = (double)((pts + pw - 1) / pw) * ((FX + Lg - 1) / Lg);
    const double fills = (nodes + threads - 1) / threads;
    if (sizeof(Real) == 4)
        return (exchange ? 120.0 : 0.0) + (NS == 4 ? 2660.0 + 1106.0 * units + fills * (1190.0 + 151.0 * FX)
                                                   : 3180.0 + 778.0 * units + fills * (339.0 + 6.0 * FX));
    const double chain = NS == 4 ? 5680.0 + 10000.0 * units + fills * (2280.0 + 2330.0 * FX)
                                 : 6720.0 + 5580.0 * units + fills * 2030.0 * FX;
    const double pipe = share * (NS == 4 ? 3930.0 : 2120.0) * ((pts + 31) / 32) * FX;
    // (unevenly shared SMs: the clusters on the fuller ones end last)
    return (NS == 4 && share > 1 ? 1.2 : 1.0) * std::sqrt(std::sqrt(chain * chain * chain * chain + pipe * pipe * pipe * pipe));
}

// Launch shape of the J^K_Q sweep: every cluster size, every number of passes whose
// frequencies fit in shared memory; the (box, ray) items, in FP32 the passes of a ray each,
// spread over the resident clusters.
template <typename Real, int NS>
int choose_jsweep(porta_ctx *c, LaunchCfg &best, int force_c, int force_f, int nitems, int NU, bool emg)
{
    double best_cost = 1e300;
    best = LaunchCfg{};
    const int ny_max = max_ny(c);
    auto even = [&](int g) { return (NU + g - 1) / g; };
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // A forced number of frequencies per pass gives the number of passes, over which they are
    // spread evenly; only where no cluster size holds them, the fewest passes that fit.
    const int g0 = force_f > 0 ? (NU + force_f - 1) / force_f : 1;
    auto search = [&](int g_last) {
        for (int C = 1; C <= std::min(16, ny_max); ++C) {
            if (force_c > 0 && C != force_c) continue;
            int nodes, ipts;
            launch_caps<Real, NS>(c, C, nodes, ipts, true);
            int last_units = 0;
            bool fits = false;
            for (int g = g0; g <= g_last && !(force_f > 0 && fits); ++g) {
                const int F = even(g);
                const int units = (F + jsweep_lanes<Real>() - 1) / jsweep_lanes<Real>();
                if (units == last_units) continue;
                last_units = units;
                int threads = 0;
                const int tots = jsweep_tots<Real, NS>(c, C, F, &threads);
                const int smem = jsweep_smem_bytes<Real, NS>(nodes, ipts, tots, F);
                if (smem > kJSmemLimit) continue;
                const int G = jsweep_groups<Real>(NU, F);
                const int parts = sizeof(Real) == 4 || emg ? G : 1;
                const long long n = (long long)nitems * parts;
                auto cost = [&](int ncl) {
                    const int share = std::max(1, (ncl * C + nsm - 1) / nsm);     // CTAs on one SM
                    double total = 0.0, item_max = 0.0;
                    for (const BoxDev &b : c->boxes) {
                        const double item = (double)b.nz * (G / parts) *
                                            jsweep_plane_cost<Real, NS>(b.nx, (b.ny + C - 1) / C, F, threads, share, C > 1);
                        total += item * c->nray * parts;
                        item_max = std::max(item_max, item);
                    }
                    return c->nbox == 1 || emg ? (double)((n + ncl - 1) / ncl) * item_max : std::max(total / ncl, item_max) * 1.05;
                };
                // no better even with every SM's thread slots taken
                const int per_sm = std::max(1, std::min(2048 / threads, 227 * 1024 / (smem + 1024)));
                double bound = 1e300;
                for (int k = 1; k <= per_sm && bound >= best_cost; ++k) bound = std::min(bound, cost(std::max(1, nsm * k / C)));
                if (best.cluster > 0 && bound >= best_cost) {
                    fits = true;
                    continue;
                }
                int act = 0;
                if (jsweep_max_active_clusters<Real, NS>(C, smem, threads, &act) != cudaSuccess) {
                    cudaGetLastError();
                    continue;
                }
                if (act < 1) continue;
                fits = true;
                const int ncl = (int)std::min<long long>(act, n);
                if (cost(ncl) < best_cost) {
                    best_cost = cost(ncl);
                    best = {C, F, threads, smem, ncl, 0};
                }
            }
        }
    };
    search(force_f > 0 ? g0 : NU);
    if (force_f > 0 && best.cluster == 0) search(NU);
    return best.cluster > 0 ? PORTA_OK : PORTA_EINVAL;
}

// Launch shape of the general sweep: cluster size C (CTAs sharing one ray's plane)
// and frequencies per pass F. Estimated time of a candidate (in units of one
// point update): the (box, ray) work items spread over the resident clusters,
// each item costing, per plane and frequency pass, the thread slots of its
// point updates, the ring fill (halo rows included), the partial-integral
// writes and a barrier.
template <typename Real, int NS>
int choose_sweep(porta_ctx *c, LaunchCfg &best, int force_c, int force_f, int nitems, int NU, bool wide = false)
{
    // accumulated quantities per point (Stokes V too for the polarized lines of a multilevel atom)
    const int NA = NS == 1 ? 2 : (c->d_dich ? 5 : 4);
    double best_cost = 1e300;
    best = LaunchCfg{};
    const int ny_max = max_ny(c);
    for (int C = 1; C <= 16; ++C) {
        if (force_c > 0 && C != force_c) continue;
        if (force_c <= 0 && C > 1 && (C & (C - 1)) != 0 && C != 6 && C != 12) continue;   // heuristic set
        if (C > ny_max) continue;
        // biquadratic stencils reach two rows into the next strip: every CTA needs two rows
        if (c->interp == 2 && !c->d_kexpl && !wide && min_ny(c) / C < 2) continue;
        int ring_plane, ipts_max;
        launch_caps<Real, NS>(c, C, ring_plane, ipts_max, wide);
        int fmax = 0;
        if (wide) {
            // besides the Stokes planes, each frequency of a pass keeps the nodes' coefficients
            // of three planes
            for (int f = NU; f >= 1 && fmax == 0; --f)
                if (jwide_smem_bytes<Real, NS>(ring_plane, ipts_max, f, kThreads) <= kSmemLimit) fmax = f;
            if (fmax == 0) continue;
        } else {
            const long long ring = 3LL * ring_plane * 16;
            const long long per_nu = 2LL * ipts_max * NS * (long long)sizeof(Real);
            const long long scratch = (long long)kThreads * NA * (long long)sizeof(Real);
            if (ring + per_nu + scratch > kSmemLimit) continue;
            fmax = (int)std::min<long long>(NU, (kSmemLimit - ring - scratch) / per_nu);
        }
        if (force_f > 0) {
            if (force_f > fmax) continue;
            fmax = force_f;
        }
        const int G = (NU + fmax - 1) / fmax;
        const int F = (NU + G - 1) / G;
        // threads: the strip's points times the frequency lanes they can use, whole warps, 64..512
        const int threads = std::min(kThreads, std::max(64, (ipts_max * F + 31) / 32 * 32));
        const int smem = wide ? jwide_smem_bytes<Real, NS>(ring_plane, ipts_max, F, threads)
                              : sweep_smem_bytes<Real, NS>(ring_plane, ipts_max, F, threads, NA);
        if (smem > kSmemLimit + 16) continue;
        int act = 0;
        if ((wide ? jwide_max_active_clusters<Real, NS>(C, smem, threads, &act)
                  : max_active_clusters<Real, NS>(C, smem, threads, &act, c->d_dich != nullptr,
                                                  c->interp == 2 && !c->d_kexpl, c->d_kexpl != nullptr)) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (act < 1) continue;
        const int ncl = std::min(act, nitems);
        double total = 0.0, item_max = 0.0;
        for (const BoxDev &b : c->boxes) {
            const int rmax = (b.ny + C - 1) / C;
            const double pts = (double)rmax * b.nx;
            const double slots = std::ceil(pts * F / threads) * kThreads;   // per-SM issue slots per pass
            const double item = b.nz * G * (slots + 0.15 * (rmax + 2) * b.nx + 0.05 * pts + 300.0);
            total += item * c->nray;
            item_max = std::max(item_max, item);
        }
        const double cost = c->nbox == 1 ? std::ceil((double)nitems / ncl) * item_max
                                         : std::max(total / ncl, item_max) * 1.05;
        if (cost < best_cost) {
            best_cost = cost;
            best.cluster = C;
            best.F = F;
            best.threads = threads;
            best.smem = smem;
            best.clusters = ncl;
        }
    }
    return best.cluster > 0 ? PORTA_OK : PORTA_EINVAL;
}

// The shape of a context's sweep (jk: the J^K_Q sweep's; emg: its form for emergent profiles). It follows from sizes and options
// alone and takes some tens of occupancy queries, so the context keeps what it chose.
template <typename Real, int NS>
int choose_launch(porta_ctx *c, LaunchCfg &best, int force_c, int force_f, int nitems, bool jk = false, int nnu = 0,
                  bool emg = false)
{
    const int NU = nnu > 0 ? nnu : c->n_nu;     // frequencies swept
    if (force_f > NU) force_f = NU;
    const std::array<int, 8> key = {force_c, force_f, nitems, jk ? c->jk_form + (emg ? 2 : 0) : 0, NU, c->d_dich != nullptr, c->interp, c->d_kexpl != nullptr};
    for (const auto &s : c->shapes)
        if (s.first == key) {
            best = s.second;
            return PORTA_OK;
        }
    const int rc = jk && c->jk_form == 1 ? choose_jsweep<Real, NS>(c, best, force_c, force_f, nitems, NU, emg)
                                         : choose_sweep<Real, NS>(c, best, force_c, force_f, nitems, NU, jk);
    if (rc == PORTA_OK) {
        if (c->shapes.size() >= 64) c->shapes.clear();
        c->shapes.emplace_back(key, best);
    }
    return rc;
}

// sweep arguments common to every mode: sizes, atmosphere, unknowns, frequencies
template <typename Real>
SweepArgs<Real> base_args(porta_ctx *c)
{
    SweepArgs<Real> a{};
    a.nnu = c->n_nu;
    a.nray = c->nray;
    a.nvox = c->nvox;
    a.boxes = (const BoxDev *)c->d_boxes;
    a.bfac = (Real)(2.0 * c->gbar * c->zeta);
    const Real *atm = (const Real *)c->d_atm;
    a.chi = atm;
    a.vel = atm + c->nvox;
    a.bx = atm + 2 * c->nvox;
    a.by = atm + 3 * c->nvox;
    a.bz = atm + 4 * c->nvox;
    a.bpl = atm + 5 * c->nvox;
    a.rho = (const Real *)c->d_rhoR;
    a.dich = (const Real *)c->d_dich;
    a.xf = (const Real *)c->d_freq;
    a.wf = (const Real *)c->d_freq + c->n_nu;
    a.probe_ray = -1;
    a.interp = c->interp;
    a.kexpl = c->d_kexpl;
    a.sexpl = c->d_sexpl;
    return a;
}

// fill the launch-dependent fields of the arguments
template <typename Real>
void shape_args(porta_ctx *c, SweepArgs<Real> &a, const LaunchCfg &cfg, bool jk = false)
{
    a.F = cfg.F;
    const bool split = jk && c->jk_form == 1;
    a.ngroups = split ? jsweep_groups<Real>(a.nnu, cfg.F) : (a.nnu + cfg.F - 1) / cfg.F;
    if (c->ns == 1)
        launch_caps<Real, 1>(c, cfg.cluster, a.ring_plane, a.ipts_max, jk);
    else
        launch_caps<Real, 4>(c, cfg.cluster, a.ring_plane, a.ipts_max, jk);
    if (jk && !split) {
        a.cstride = jwide_stride(a.ring_plane * (c->ns == 1 ? 1 : 2), (int)sizeof(Real));
        a.istride = jwide_stride(a.ipts_max * c->ns, (int)sizeof(Real));
    }
    if (split)
        a.tots = c->ns == 1 ? jsweep_tots<Real, 1>(c, cfg.cluster, cfg.F, nullptr)
                            : jsweep_tots<Real, 4>(c, cfg.cluster, cfg.F, nullptr);
}

// api.cu
// residual and errors of the formal solutions handed on (synchronizes)
int read_status(porta_ctx *c, double *value);
// the packed inputs of sweep_j.cu, allocated on first use (d_jpack stays null without room)
void ensure_jpack(porta_ctx *c);
void free_all(porta_ctx *c);
bool finite_host(const double *x, long long n);
// copy n doubles from a caller buffer (host or device) into device memory
int copy_in(porta_ctx *c, double *dst, const double *src, long long n, int where);
// number of entries of a device array outside (lo, hi] (NaN counts)
int count_bad(porta_ctx *c, const double *d, long long n, double lo, double hi, unsigned long long *out);
int create_impl(int nbox, const porta_grid *grids, const porta_atom *at, const porta_quad *q, const porta_opts *o,
                porta_ctx **out);

// api_adjoint.cu: emergent Stokes profiles of ndir directions (device pointers)
template <typename Real>
int emergent_t(porta_ctx *c, int ndir, const double *mu, const double *chi, double *dout, int box = 0);
// releases the checkpoints of porta_iterate_ckpt
void it_free(porta_ctx *c);

// api_mg.cu: releases the coarse levels
void mg_free(porta_ctx *c);
// re-derives the sweep's copy of the unknowns after they changed on the device
cudaError_t mg_rho_changed(porta_ctx *L);

// api_ml.cu: line data of every line from the populations
cudaError_t ml_prepare(porta_ctx *c);
// the error counter of the line data and of the rate equations (synchronizes)
int ml_check(porta_ctx *c, const char *what);

}  // namespace porta_api
