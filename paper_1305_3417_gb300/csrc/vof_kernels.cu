// FP64 kernels of libvof: geometry set-up, reconstruction (NAG gradient + Alg. 1
// positioning), point velocities, flux-polyhedron construction and correction,
// phase fluxes by tetrahedral clipping, the conservative update and the
// bounding pass.  Every kernel bounds its loops and reports problems through
// the context status word; none traps.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "vof_internal.h"
#include "vof_device.cuh"

namespace {
using namespace vofd;

// =========================================================== set-up kernels
__global__ void k_face_geom(DevMesh m, double *cf, double *sf, double *nagc)
{
    int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= m.nf) return;
    int b = m.fptr[f], n = m.fptr[f + 1] - b;
    V3 c = mk(0, 0, 0);
    for (int i = 0; i < n; ++i) c = c + ldP(m, m.fpts[b + i]);
    c = c * (1.0 / n);
    V3 S = mk(0, 0, 0);
    if (n == 3) {
        V3 p0 = ldP(m, m.fpts[b]), p1 = ldP(m, m.fpts[b + 1]), p2 = ldP(m, m.fpts[b + 2]);
        S = cross(p1 - p0, p2 - p0) * 0.5;
    } else {
        for (int t = 0; t < n; ++t) {
            V3 a = ldP(m, m.fpts[b + t]) - c, e = ldP(m, m.fpts[b + (t + 1) % n]) - c;
            S = S + cross(a, e) * 0.5;
        }
    }
    // NAG face value (Sec. 2.2.1) as a weighted sum of the point values:
    // phi_f = sum_t w_t (phi' + phi_t + phi_t+1)/3, phi' the point mean, w_t the
    // area share of fan triangle t, so point k weighs (1/n + w_k + w_k-1)/3.
    double A[VOF_MAXFP], sa = 0.0;
    for (int t = 0; t < n; ++t) {
        V3 a = ldP(m, m.fpts[b + t]) - c, e = ldP(m, m.fpts[b + (t + 1) % n]) - c;
        A[t] = 0.5 * norm3(cross(a, e));
        sa += A[t];
    }
    for (int k = 0; k < n; ++k)
        nagc[b + k] = (1.0 / n + A[k] / sa + A[(k + n - 1) % n] / sa) / 3.0;
    st3(cf, m.nf, f, c);
    st3(sf, m.nf, f, S);
}

__global__ void k_cell_geom(DevMesh m, double *cc, double *vc, double *cbox, double *ctvol, unsigned *bad)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.nc) return;
    int p0 = m.cpptr[c], p1 = m.cpptr[c + 1];
    V3 s = mk(0, 0, 0), lo = mk(1e300, 1e300, 1e300), hi = mk(-1e300, -1e300, -1e300);
    for (int i = p0; i < p1; ++i) {
        V3 p = ldP(m, m.cpts[i]);
        s = s + p;
        lo = mk(fmin(lo.x, p.x), fmin(lo.y, p.y), fmin(lo.z, p.z));
        hi = mk(fmax(hi.x, p.x), fmax(hi.y, p.y), fmax(hi.z, p.z));
    }
    V3 ctr = s * (1.0 / (p1 - p0));
    double V = 0.0;
    int k0 = m.ctptr[c];
    for (int k = m.cptr[c]; k < m.cptr[c + 1]; ++k) {
        int code = m.cface[k], f = code >> 1;
        int n = m.fptr[f + 1] - m.fptr[f], nt = n == 3 ? 1 : n;
        for (int t = 0; t < nt; ++t) {
            V3 a, b, e;
            face_tri(m, f, t, code & 1, a, b, e);
            double v = tvol(ctr, a, b, e);
            if (!(v > 0.0)) atomicOr(bad, 1u);
            ctvol[k0++] = v;  // (faces and fan triangles in the order of ctet)
            V += v;
        }
    }
    st3(cc, m.nc, c, ctr);
    vc[c] = V;
    cbox[6 * c + 0] = lo.x; cbox[6 * c + 1] = lo.y; cbox[6 * c + 2] = lo.z;
    cbox[6 * c + 3] = hi.x; cbox[6 * c + 4] = hi.y; cbox[6 * c + 5] = hi.z;
}

// Eq. w_pc: inverse distance from the point to each point-cell centre (on a
// periodic mesh the cell moved next to the point), normalised
__global__ void k_point_weights(DevMesh m, double *pw)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= m.np) return;
    V3 x = ldP(m, p);
    auto centre = [&](int j) {
        V3 c = ld3(m.cc, m.nc, m.pcell[j]);
        return m.pcode ? c + tshift(m, m.pcode[j]) : c;
    };
    double s = 0.0;
    for (int j = m.pptr[p]; j < m.pptr[p + 1]; ++j) s += 1.0 / norm3(x - centre(j));
    for (int j = m.pptr[p]; j < m.pptr[p + 1]; ++j) pw[j] = (1.0 / norm3(x - centre(j))) / s;
}

// wall table: distinct unit normals of the wall faces through each wall point
__global__ void k_wall_table(DevMesh m, const int *wptr, const int *wface, int nrows, double *wallt)
{
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nrows) return;
    int cnt = 0;
    V3 v[2] = {mk(0, 0, 0), mk(0, 0, 0)};
    for (int j = wptr[r]; j < wptr[r + 1]; ++j) {
        int f = wface[j];
        V3 S = ld3(m.sf, m.nf, f);
        V3 u = S * (1.0 / norm3(S));
        bool dup = false;
        for (int k = 0; k < cnt && k < 2; ++k)
            if (fabs(dot(u, v[k])) > 1.0 - 1e-12) dup = true;
        if (dup || cnt >= 3) continue;
        if (cnt < 2) v[cnt] = u;
        ++cnt;
    }
    double *o = wallt + 7 * r;
    o[0] = cnt;
    o[1] = v[0].x; o[2] = v[0].y; o[3] = v[0].z;
    o[4] = v[1].x; o[5] = v[1].y; o[6] = v[1].z;
}

// ====================================================== point velocity (A4)
__device__ __forceinline__ V3 point_velocity(const DevMesh &m, int p, const double *__restrict__ Uc)
{
    V3 u = mk(0, 0, 0);
    for (int j = __ldg(m.pptr + p); j < __ldg(m.pptr + p + 1); ++j) {
        int c = __ldg(m.pcell + j);
        u = u + ld3(Uc, m.nc, c) * __ldg(m.pw + j);
    }
    int r = __ldg(m.pwall + p);
    if (r >= 0) {
        const double *w = m.wallt + 7 * r;
        int cnt = (int)w[0];
        V3 n1 = mk(w[1], w[2], w[3]), n2 = mk(w[4], w[5], w[6]);
        if (cnt == 1) u = u - n1 * dot(u, n1);
        else if (cnt == 2) {
            V3 t = cross(n1, n2);
            t = t * (1.0 / norm3(t));
            u = t * dot(u, t);
        } else if (cnt >= 3) u = mk(0, 0, 0);
    }
    return u;
}

__global__ void k_point_velocity(DevMesh m, const double *__restrict__ Uc, double *Up)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= m.np) return;
    st3(Up, m.np, p, point_velocity(m, p, Uc));
}

// ===================================================== reconstruction (A1-A3)
// G lanes per cell: NAG gradient over the (face, point) entries of the cell,
// then the plane offset, the fill function summed over the cell tetrahedra, KL
// or fewer per lane, each a closed-form cut fraction of its sorted projections.
//
// Bound by the FP64 pipe, which takes one warp instruction in 64 cycles on each
// of an SM's four sub-partitions, whatever the number of active lanes: what counts is FP64 warp
// instructions per cell.  So several cells share a warp, every order and
// threshold test is taken on the integer pipe from the bit patterns, the
// tetrahedra's volumes come from the context, and the fill is evaluated
// without branches and with few divisions (below).

// Reciprocal in FP64 without a full division: the FP32 reciprocal refined by
// one Newton-Raphson step r <- r + r (1 - x r) in FP64, whose relative error is
// about the square of the FP32 one (~4e-15), with exact division where x is
// outside the FP32 range: a conversion pair and two FMAs.
__device__ __noinline__ double exact_rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ double mx_rcp(double x)
{
    const float r0 = __frcp_rn((float)x);
    if (!isfinite(r0) || r0 == 0.0f) return exact_rcp(x);
    const double r = (double)r0;
    return fma(r, fma(-x, r, 1.0), r);
}
// refined once more: FP64 accuracy (the last place may differ)
__device__ __forceinline__ double full_rcp(double x)
{
    const double r = mx_rcp(x), t = fma(r, fma(-x, r, 1.0), r);
    return isfinite(t) ? t : r;
}
__device__ __forceinline__ int hiword(double x) { return __double2hiint(x); }

// Cut fraction of a tetrahedron with sorted projections h0..h3 below a level:
// one vertex below: the product of three edge fractions; one above: one minus
// such a product; two and two: ab + a(1-b)e + (1-a)ce.  The reciprocals of the
// projection differences are formed once (r10 = 1/(h1-h0), ra = 1/(h2-h0),
// rb = 1/(h3-h0), rc = 1/(h2-h1), re = 1/(h3-h1), r32 = 1/(h3-h2)), all three
// forms are evaluated and one is selected by the signs of the level's distances
// to the vertices: 21 FP64 instructions a tetrahedron, where the branches, taken
// one after another by the lanes of a warp, with their divisions were over 200.
// (A difference of zero makes an infinite reciprocal only in a form that is not
// selected.)
struct FillTet { double h0, h1, h2, h3, r10, ra, rb, rc, re, r32; };

__device__ __forceinline__ double fill_below(const FillTet &q, double d)
{
    const double u = d - q.h0, v = d - q.h1, z = q.h2 - d, y = q.h3 - d;
    const double a = u * q.ra, b = u * q.rb, c = v * q.rc, e = v * q.re;
    const double ab = a * b;
    const double mid = fma(fma(-a, c, c), e, fma(fma(-a, b, a), e, ab));
    const double low = (u * q.r10) * ab;
    const double top = 1.0 - (y * q.r32) * (y * q.re) * (y * q.rb);
    double f = hiword(v) <= 0 ? low : hiword(z) <= 0 ? top : mid;
    f = hiword(y) <= 0 ? 1.0 : f;
    return hiword(u) <= 0 ? 0.0 : f;
}

// The same in FP32 with its derivative (the cut area over the volume).  Every
// form is a sum of terms that are not negative, the one for one vertex above
// too: 1 - (1-b)(1-e)(1-g) as b + (1-b)(e + (1-e) g), so that the fill's error is
// relative to the fill and small levels are resolved (one minus a product
// leaves 6e-8 of the tetrahedron: cells of 1e-9 with a normal along the mesh, whose
// tetrahedra have three vertices at the bottom, did not converge on it).
struct FillTetF { float h0, h1, h2, h3, r10, ra, rb, rc, re, r32; };

__device__ __forceinline__ float fill_below(const FillTetF &q, float d, float &df)
{
    const float u = d - q.h0, v = d - q.h1, z = q.h2 - d, y = q.h3 - d;
    const float a = u * q.ra, b = u * q.rb, c = v * q.rc, e = v * q.re;
    const float ab = a * b, b1 = 1.0f - b, a1 = 1.0f - a;
    const float mid = ab + a * b1 * e + a1 * c * e;
    const float dmid = q.ra * b + a * q.rb + q.ra * b1 * e - a * q.rb * e + a * b1 * q.re - q.ra * c * e +
                       a1 * q.rc * e + a1 * c * q.re;
    const float lx = q.r10 * ab, tx = (y * q.re) * (y * q.rb) * q.r32;
    const float low = u * lx, top = fmaf(b1, fmaf(1.0f - e, -z * q.r32, e), b);
    float f = v <= 0.0f ? low : z <= 0.0f ? top : mid;
    df = v <= 0.0f ? 3.0f * lx : z <= 0.0f ? 3.0f * tx : dmid;
    if (y <= 0.0f) { f = 1.0f; df = 0.0f; }
    if (u <= 0.0f) { f = 0.0f; df = 0.0f; }
    return f;
}

// The fill in FP64 with its three derivatives (between two vertex projections
// it is a cubic, so these give it exactly up to the next one); gap is lowered
// to the high word of the least distance of the level to a projection.
__device__ __forceinline__ void fill_taylor(const double h[4], double d, double F[4], int &gap)
{
    const double u = d - h[0], v = d - h[1], z = h[2] - d, y = h[3] - d;
    gap = min(min(gap, hiword(u) & 0x7fffffff), hiword(v) & 0x7fffffff);
    gap = min(min(gap, hiword(z) & 0x7fffffff), hiword(y) & 0x7fffffff);
    F[0] = F[1] = F[2] = F[3] = 0.0;
    if (hiword(u) <= 0) return;
    if (hiword(y) <= 0) { F[0] = 1.0; return; }
    const double d20 = h[2] - h[0], d30 = h[3] - h[0], d31 = h[3] - h[1];
    const bool low = hiword(v) <= 0;
    if (low || hiword(z) <= 0) {
        // k w^3 from the lowest vertex, or one minus that from the highest
        const double w = low ? u : y;
        const double k = mx_rcp(d30 * (low ? (h[1] - h[0]) * d20 : d31 * (h[3] - h[2])));
        const double kw = k * w, kww = kw * w;
        F[0] = low ? kww * w : fma(-kww, w, 1.0);
        F[1] = 3.0 * kww;
        F[2] = (low ? 6.0 : -6.0) * kw;
        F[3] = 6.0 * k;
        return;
    }
    const double ra = mx_rcp(d20), rb = mx_rcp(d30), rc = mx_rcp(h[2] - h[1]), re = mx_rcp(d31);
    const double a = u * ra, b = u * rb, c = v * rc, e = v * re;
    // f = ab + ae + ce - ae (b + c)
    const double s = b + c, rs = rb + rc, ae = a * e, dae = fma(ra, e, a * re), rae = ra * re;
    F[0] = fma(-ae, s, fma(a, b, fma(c, e, ae)));
    F[1] = fma(-ae, rs, fma(-dae, s, fma(ra, b, fma(a, rb, fma(rc, e, fma(c, re, dae))))));
    F[2] = 2.0 * fma(-rae, s, fma(-dae, rs, fma(ra, rb, fma(rc, re, rae))));
    F[3] = -6.0 * rae * rs;
}

struct RcCell {
    int fl, it, it32;
    V3 n;
    double d;
};

// The plane of interface cell c (eps < a = alpha[c] < 1 - eps).
//
// MIXED: the offset is measured from the end of the cell's extent that is
// nearer in volume (target t = a from below, or 1 - a from above), so that
// cells near 0 and 1 keep their relative precision: safeguarded Newton steps (on
// logarithms) in FP32 until the fill's residual is within 1e-5 t (ten times its
// rounding) and one more, then one FP64 evaluation with derivatives, on whose
// cubic the offset is finished when the step stays short of the next vertex
// projection (nearly always: the FP32 offset is good to about 1e-6); else
// safeguarded FP64 Newton steps to the same 1e-13 stop.  (With FP64 Newton
// steps of value and slope there were 2.4 evaluations per cell, up to 14 near 0
// and 1.)  FP64 form: Alg. 1 (secant; bisection once the secant leaves the
// bracket or has not converged in POS_SECANT_MAX steps).
// guess: a start sg (fraction of the extent from below) is given.
template <bool MIXED, int G, int KL>
__device__ __forceinline__ RcCell rc_cell(const DevMesh &m, const double *__restrict__ alpha,
                                          const double *__restrict__ palpha, const double *__restrict__ gin, int c,
                                          double a, bool guess, float sg, unsigned *status)
{
    const int lane = threadIdx.x & (G - 1);
    const unsigned tm = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (threadIdx.x & 31 & ~(G - 1));
    auto tsum = [&](double v) {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(tm, v, o);
        return v;
    };
    RcCell r{VOF_INTERFACE, 0, 0, mk(0, 0, 0), 0.0};
    const double V = m.vc[c];
    const int t0 = __ldg(m.ctptr + c), nt = __ldg(m.ctptr + c + 1) - t0;
    // ---- NAG gradient: lane j handles the j-th (face, point) entry
    // (a given gradient instead, times V: the generalised LSQ one)
    V3 g = mk(0, 0, 0);
    if (gin) {
        if (lane == 0) g = ld3(gin, m.nc, c) * V;
    } else
    for (int j = __ldg(m.ceptr + c) + lane, e1 = __ldg(m.ceptr + c + 1); j < e1; j += G) {
        const int2 en = __ldg(m.cent + j);  // {fpts slot, face code}
        const int f = en.y >> 1, p = __ldg(m.fpts + en.x);
        double ap = 0.0;  // Eq. idwpointphi (precomputed per point when palpha is given)
        if (palpha) ap = __ldg(palpha + p);
        else
            for (int q = __ldg(m.pptr + p); q < __ldg(m.pptr + p + 1); ++q)
                ap += __ldg(m.pw + q) * __ldg(alpha + __ldg(m.pcell + q));
        double w = __ldg(m.nagc + en.x) * ap;
        if (en.y & 1) w = -w;  // Eq. own-nei: the neighbour sees -S_f
        g = g + ld3(m.sf, m.nf, f) * w;
    }
    // g = G / V; the cell is oriented where |g| V^(1/3) > 1e-12, taken
    // as |G|^6 > 1e-72 V^4 (no cube root, square root or division)
    g = mk(tsum(g.x), tsum(g.y), tsum(g.z));
    const double g2 = dot(g, g);
    if (!(g2 * g2 * g2 > 1e-72 * (V * V) * (V * V))) return r;
    const V3 nn = r.n = g * -rsqrt(g2);  // points out of the phase
    r.fl |= VOF_ORIENTED;
    // ---- cell tetrahedra (c_c, outward face triangle), lanes j, j + G, ...:
    // sorted projections and volumes (0: no tetrahedron)
    const double ec = dot(nn, ld3(m.cc, m.nc, c));
    double h[KL][4], vk[KL];
    double lo = 1e300, hi = -1e300;
#pragma unroll
    for (int s = 0; s < KL; ++s) {
        vk[s] = 0.0;
        h[s][0] = h[s][1] = h[s][2] = h[s][3] = 0.0;
        if (lane + G * s >= nt) continue;
        const int4 te = __ldg(m.ctet + t0 + lane + G * s);  // {face code, slot a, slot b, slot c or -1}
        vk[s] = __ldg(m.ctvol + t0 + lane + G * s);
        const V3 p1 = ldP(m, __ldg(m.fpts + te.y)), p2 = ldP(m, __ldg(m.fpts + te.z));
        const V3 p0 = te.w >= 0 ? ldP(m, __ldg(m.fpts + te.w)) : ld3(m.cf, m.nf, te.x >> 1);
        double e0 = ec, e1 = dot(nn, p0), e2 = dot(nn, p1), e3 = dot(nn, p2), t;
#define RC_CS(p, q) if (gt_bits(p, q)) { t = p; p = q; q = t; }
        RC_CS(e0, e1) RC_CS(e2, e3) RC_CS(e0, e2) RC_CS(e1, e3) RC_CS(e1, e2)
#undef RC_CS
        h[s][0] = e0; h[s][1] = e1; h[s][2] = e2; h[s][3] = e3;
        if (gt_bits(lo, e0)) lo = e0;
        if (gt_bits(e3, hi)) hi = e3;
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        const double l2 = __shfl_xor_sync(tm, lo, o), h2 = __shfl_xor_sync(tm, hi, o);
        if (gt_bits(lo, l2)) lo = l2;
        if (gt_bits(h2, hi)) hi = h2;
    }
    const double dmin = lo, dmax = hi, range = dmax - dmin, rV = 1.0 / V;
    int it = 0;
    if constexpr (MIXED) {
        const bool up = gt_pos(a, 0.5);  // measured from above
        const double tgt = up ? 1.0 - a : a;
        FillTetF q[KL];
        float vf[KL];
        const float rr = __frcp_rn((float)range), tf = (float)tgt;
#pragma unroll
        for (int s = 0; s < KL; ++s) {
            if (up) {
                const double x0 = dmax - h[s][3], x1 = dmax - h[s][2], x2 = dmax - h[s][1], x3 = dmax - h[s][0];
                h[s][0] = x0; h[s][1] = x1; h[s][2] = x2; h[s][3] = x3;
            } else {
                h[s][0] -= dmin; h[s][1] -= dmin; h[s][2] -= dmin; h[s][3] -= dmin;
            }
            // in units of the extent; volumes as fractions of the cell's
            const float f0 = (float)h[s][0] * rr, f1 = (float)h[s][1] * rr, f2 = (float)h[s][2] * rr,
                        f3 = (float)h[s][3] * rr;
            q[s] = FillTetF{f0, f1, f2, f3, __fdividef(1.0f, f1 - f0), __fdividef(1.0f, f2 - f0),
                            __fdividef(1.0f, f3 - f0), __fdividef(1.0f, f2 - f1), __fdividef(1.0f, f3 - f1),
                            __fdividef(1.0f, f3 - f2)};
            vf[s] = (float)(vk[s] * rV);
        }
        // start: the fraction itself (or the learned offset), the corner
        // estimate t^(1/3) within 1e-4 of 0 or 1
        float A = 0.0f, B = 1.0f, x;
        if (tf > 1e-4f) x = guess ? (up ? 1.0f - sg : sg) : tf;
        else x = cbrtf(tf);
        while (it < POS_MAXIT) {
            float part = 0.0f, dpart = 0.0f;
#pragma unroll
            for (int s = 0; s < KL; ++s)
                if (vf[s] > 0.0f) {
                    float df;
                    part += vf[s] * fill_below(q[s], x, df);
                    dpart += vf[s] * df;
                }
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) {
                part += __shfl_xor_sync(tm, part, o);
                dpart += __shfl_xor_sync(tm, dpart, o);
            }
            ++it;
            const float gf = part - tf;
            const bool sure = fabsf(gf) > 1e-5f * tf;
            if (sure) {
                if (gf < 0.0f) A = x; else B = x;
            }
            // Newton on log f against log x: near an end the fill is a power of
            // the distance (cube, square or first), where this lands at once
            // and plain steps crawl
            float xn = x * __expf(__fdividef(part * __logf(__fdividef(tf, part)), x * dpart));
            if (!(xn > A && xn < B)) xn = 0.5f * (A + B);
            if (!(xn > A && xn < B)) break;  // bracket at FP32 resolution
            x = xn;
            if (!sure) break;
        }
        r.it32 = it;
        // (the whole extent as the bracket: nothing that FP32 decided is taken over)
        double X = (double)x * range, lo64 = 0.0, hi64 = range;
        while (it < POS_MAXIT) {
            double S[4] = {0.0, 0.0, 0.0, 0.0};
            int gap = 0x7fffffff;
#pragma unroll
            for (int s = 0; s < KL; ++s)
                if (vf[s] > 0.0f) {
                    double F[4];
                    fill_taylor(h[s], X, F, gap);
#pragma unroll
                    for (int k = 0; k < 4; ++k) S[k] = fma(vk[s], F[k], S[k]);
                }
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) {
#pragma unroll
                for (int k = 0; k < 4; ++k) S[k] += __shfl_xor_sync(tm, S[k], o);
                gap = min(gap, __shfl_xor_sync(tm, gap, o));
            }
            ++it;
            const double gx = fma(S[0], rV, -tgt);
            if (le_pos(fabs(gx), POS_TOL)) break;
            if (hiword(gx) < 0) lo64 = X; else hi64 = X;
            if (hi64 - lo64 <= 1e-15 * range) break;
            // chord steps on the cubic gx + f1 s + f2 s^2 + f3 s^3 (the slope
            // sets the rate only: an FP32 reciprocal of it)
            const double f1 = S[1] * rV, f2 = S[2] * (0.5 * rV), f3 = S[3] * ((1.0 / 6.0) * rV);
            const double k1 = (double)__frcp_rn((float)f1);
            const double s1 = -gx * k1;
            auto cubic = [&](double s) { return fma(fma(fma(f3, s, f2), s, f1), s, gx); };
            const double s2 = fma(-cubic(s1), k1, s1);
            const double xn = X + s2;
            if ((hiword(s2) & 0x7fffffff) < gap && le_pos(fabs(cubic(s2)), POS_TOL) && xn > lo64 && xn < hi64) {
                X = xn;
                break;
            }
            X += s1;
            if (!(X > lo64 && X < hi64)) X = 0.5 * (lo64 + hi64);
        }
        r.d = up ? dmax - X : dmin + X;
    } else {
        FillTet q[KL];
#pragma unroll
        for (int s = 0; s < KL; ++s) {
            const double d10 = h[s][1] - h[s][0], d20 = h[s][2] - h[s][0], d30 = h[s][3] - h[s][0];
            const double d21 = h[s][2] - h[s][1], d31 = h[s][3] - h[s][1], d32 = h[s][3] - h[s][2];
            q[s] = FillTet{h[s][0], h[s][1], h[s][2], h[s][3], full_rcp(d10), full_rcp(d20), full_rcp(d30),
                           full_rcp(d21), full_rcp(d31), full_rcp(d32)};
        }
        double A = dmin, B = dmax, x0 = A, g0 = -a, x1 = B, g1 = 1.0 - a, gx = 0.0, x = 0.0;
        const double btol = 1e-15 * range;
        bool bisect = false;
        while (it < POS_MAXIT) {
            if (it >= POS_SECANT_MAX) bisect = true;
            if (!bisect) {
                x = x1 - g1 * (x1 - x0) * mx_rcp(g1 - g0);
                if (!(gt_bits(x, A) && gt_bits(B, x))) bisect = true;
            }
            if (bisect) x = 0.5 * (A + B);
            double part = 0.0;
#pragma unroll
            for (int s = 0; s < KL; ++s)
                if (hiword(vk[s]) > 0) part = fma(vk[s], fill_below(q[s], x), part);
            gx = fma(tsum(part), rV, -a);
            ++it;
            if (hiword(gx) < 0) A = x; else B = x;
            x0 = x1; g0 = g1; x1 = x; g1 = gx;
            if (le_pos(fabs(gx), POS_TOL)) break;
            if (!gt_bits(B - A, btol)) break;
        }
        // The stop leaves a residual of up to 1e-13, whose share of the slope is
        // the offset's error, and which iterate meets the stop hangs on the fill's
        // last bits: the secant through the last two points, not evaluated, takes
        // it off (24^3 to 96^3: rms error 4e-12 .. 5e-11 -> 1e-15 .. 7e-14 of the
        // box).  The step is short, so FP32 conversions on the integer pipe do.
        const double xs = x1 - fd(tf(g1) * __fdividef(tf(x1 - x0), tf(g1 - g0)));
        if (gt_bits(xs, A) && gt_bits(B, xs)) x = xs;
        r.d = x;
    }
    if (it >= POS_MAXIT && lane == 0) atomicOr(status, VOF_ST_POS_NOT_CONVERGED);
    r.it = it;
    return r;
}

struct RcArgs {
    const double *alpha, *palpha, *gin;  // palpha, gin: may be null
    double *n, *d;
    uint8_t *flags;
    int *iters;                  // or null
    unsigned *status;
    unsigned long long *work;    // counting variant
};

constexpr int RC_THREADS = 128;
// blocks per SM (96 registers a thread, 128 with more tetrahedra per lane)
template <int KL> constexpr int rc_resident() { return KL == 1 ? 5 : 4; }

// fill evaluations per cell tetrahedron (FP64, FP32), counted by a cell's first lane
template <int G, bool COUNT>
struct RcCount {
    unsigned nf64 = 0, nf32 = 0;
    __device__ __forceinline__ void add(const DevMesh &m, int c, const RcCell &r)
    {
        if (!COUNT || (threadIdx.x & (G - 1))) return;
        const unsigned nte = __ldg(m.ctptr + c + 1) - __ldg(m.ctptr + c);
        nf32 += r.it32 * nte;
        nf64 += (r.it - r.it32) * nte;
    }
    __device__ __forceinline__ void flush(unsigned long long *work)
    {
        if (!COUNT) return;
        const unsigned r64 = __reduce_add_sync(0xffffffffu, nf64);
        const unsigned r32 = __reduce_add_sync(0xffffffffu, nf32);
        if ((threadIdx.x & 31) == 0) {
            work_add1(work, WK_FILL64, r64);
            work_add1(work, WK_FILL32, r32);
        }
    }
};

// The listed cells; with a counter a lane group takes its next cell as it
// finishes one (cells differ in positioning iterations), else static striding.
template <bool MIXED, int G, int KL, bool COUNT>
__device__ __forceinline__ void rc_list(const DevMesh &m, const RcArgs &q, const int *list, int total, int *maxit,
                                        const float *__restrict__ s0, int s0cap, int *next)
{
    const int lane = threadIdx.x & (G - 1);
    const unsigned tm = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (threadIdx.x & 31 & ~(G - 1));
    const int group = (blockIdx.x * blockDim.x + threadIdx.x) / G, ngroups = (gridDim.x * blockDim.x) / G;
    const double eps = m.eps;
    RcCount<G, COUNT> wk;
    auto take = [&]() {
        int v = 0;
        if (lane == 0) v = atomicAdd(next, 1);
        return __shfl_sync(tm, v, 0, G);
    };
    for (int item = next ? take() : group; item < total; item = next ? take() : item + ngroups) {
        const int c = list[item];
        const double a = q.alpha[c];
        RcCell r{a >= 1.0 - eps ? (int)VOF_FULL : 0, 0, 0, mk(0, 0, 0), 0.0};
        if (a > eps && a < 1.0 - eps) {
            const bool guess = s0 && item < s0cap;
            r = rc_cell<MIXED, G, KL>(m, q.alpha, q.palpha, q.gin, c, a, guess, guess ? s0[item] : 0.0f, q.status);
            wk.add(m, c, r);
        }
        if (lane == 0) {
            st3(q.n, m.nc, c, r.n);
            q.d[c] = r.d;
            q.flags[c] = (uint8_t)r.fl;
            if (q.iters) q.iters[c] = r.it;
            if (maxit && r.it > 0) atomicMax(maxit, r.it);
        }
    }
    wk.flush(q.work);
}

// With no more cells than the launch has warps (in a step), narrow groups would leave most
// warps without one while each cell's chain is as many instructions longer as
// it has tetrahedra per lane: a warp takes a cell then (24^3, 252 cells: the
// reconstruction's share of the step 57 -> 32 us, with the logarithmic steps).
template <bool MIXED, int G, int KL, bool COUNT>
__global__ void __launch_bounds__(RC_THREADS, rc_resident<KL>())
k_reconstruct(DevMesh m, RcArgs q, const int *list, const int *count, int *maxit, const float *__restrict__ s0,
              int s0cap, int *next)
{
    const int total = *count;
    if constexpr (G < 32) {
        if (next && total <= (int)(gridDim.x * blockDim.x) / 32) {
            rc_list<MIXED, 32, (G * KL + 31) / 32, COUNT>(m, q, list, total, maxit, s0, s0cap, next);
            return;
        }
    }
    rc_list<MIXED, G, KL, COUNT>(m, q, list, total, maxit, s0, s0cap, next);
}

// cells per block of k_reconstruct_all: two per lane group, since interface cells come
// in clumps and a block works its own off (mixed 90^3 film: 212 us with 16 a
// group, 99 with 4, 82 with 2)
template <int G> constexpr int rc_chunk() { return 2 * (RC_THREADS / G); }

// Every cell of the mesh: a block writes the defaults (n = 0, d = 0, flags)
// of a chunk of cells, lists the chunk's interface cells in shared memory and
// hands them to its lane groups as they come free.  (One lane group per cell
// of the mesh, nearly all of which are not interface cells: 96^3 FP64 785 us,
// 392 us with the chunks and the evaluation above.)
template <bool MIXED, int G, int KL, bool COUNT>
__global__ void __launch_bounds__(RC_THREADS, rc_resident<KL>()) k_reconstruct_all(DevMesh m, RcArgs q)
{
    constexpr int CHUNK = rc_chunk<G>();
    __shared__ int cells[CHUNK], ncells, taken;
    const int lane = threadIdx.x & (G - 1);
    const unsigned tm = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (threadIdx.x & 31 & ~(G - 1));
    const double eps = m.eps;
    if (threadIdx.x == 0) ncells = taken = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < CHUNK; i += RC_THREADS) {
        const long c = (long)blockIdx.x * CHUNK + i;
        if (c >= m.nc) break;
        const double a = q.alpha[c];
        q.flags[c] = a >= 1.0 - eps ? VOF_FULL : 0;
        st3(q.n, m.nc, (int)c, mk(0, 0, 0));
        q.d[c] = 0.0;
        if (q.iters) q.iters[c] = 0;
        if (a > eps && a < 1.0 - eps) cells[atomicAdd(&ncells, 1)] = (int)c;
    }
    __syncthreads();
    RcCount<G, COUNT> wk;
    const int total = ncells;
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(&taken, 1);
        item = __shfl_sync(tm, item, 0, G);
        if (item >= total) break;
        const int c = cells[item];
        const RcCell r = rc_cell<MIXED, G, KL>(m, q.alpha, q.palpha, q.gin, c, q.alpha[c], false, 0.0f, q.status);
        wk.add(m, c, r);
        if (lane == 0) {
            st3(q.n, m.nc, c, r.n);
            q.d[c] = r.d;
            q.flags[c] = (uint8_t)r.fl;
            if (q.iters) q.iters[c] = r.it;
        }
    }
    wk.flush(q.work);
}

// ======================================== flux polyhedra and correction (A5)
// Cubic V(lambda) = C1 lambda + C2 lambda^2 + C3 lambda^3 of the signed swept
// volume.  Each face triangle (a0,a1,a2), ordered by key (face centre first,
// then global point index, parity par), sweeps to b_k = a_k - lambda w_k and is
// split into the tetrahedra (a0,a1,a2,b2), (a0,a1,b2,b1), (a0,b0,b1,b2), whose
// signed volumes -par*det/6 expand, with E1 = a1-a0, E2 = a2-a0, into
//   k1 = -det(E1,E2,w0+w1+w2),  k2 = det(E1,w2,w1)+det(w0,w1,E2)+det(w0,E1,w2),
//   k3 = -det(w0,w1,w2).
struct Cubic { double c1, c2, c3, s1, s2, s3; };

__device__ __forceinline__ void prism_cubic(V3 a0, V3 a1, V3 a2, V3 w0, V3 w1, V3 w2, long k0,
                                            long k1, long k2, Cubic &q)
{
    int par = 1;
    // sort (a,w,k) triples by key, tracking permutation parity
    if (k1 < k0) { V3 t = a0; a0 = a1; a1 = t; t = w0; w0 = w1; w1 = t; long u = k0; k0 = k1; k1 = u; par = -par; }
    if (k2 < k1) { V3 t = a1; a1 = a2; a2 = t; t = w1; w1 = w2; w2 = t; long u = k1; k1 = k2; k2 = u; par = -par; }
    if (k1 < k0) { V3 t = a0; a0 = a1; a1 = t; t = w0; w0 = w1; w1 = t; long u = k0; k0 = k1; k1 = u; par = -par; }
    // (with det(a,b,c) = a.(b x c): k2 = E1.(w2 x (w0+w1)) + E2.(w0 x w1), k3 = -w2.(w0 x w1))
    const V3 E1 = a1 - a0, E2 = a2 - a0, w01 = w0 + w1, c01 = cross(w0, w1);
    const double f = par > 0 ? -1.0 / 6.0 : 1.0 / 6.0;
    const double t1 = -dot(cross(E1, E2), w01 + w2) * f;
    const double t2 = (dot(E1, cross(w2, w01)) + dot(E2, c01)) * f;
    const double t3 = -dot(w2, c01) * f;
    q.c1 += t1; q.c2 += t2; q.c3 += t3;
    q.s1 += fabs(t1); q.s2 += fabs(t2); q.s3 += fabs(t3);
}

// loads the face's points and per-point displacements w = U_p dt
template <bool IDW>
__device__ __forceinline__ int face_points(const DevMesh &m, int f, const double *__restrict__ U,
                                           double dt, V3 *A, V3 *W, int *id)
{
    int b = __ldg(m.fptr + f), n = __ldg(m.fptr + f + 1) - b;
    for (int i = 0; i < n; ++i) {
        int p = __ldg(m.fpts + b + i);
        id[i] = __ldg(m.fkey + b + i);  // the point's index (its master's on a periodic mesh)
        A[i] = ldP(m, p);
        V3 u = IDW ? point_velocity(m, p, U) : ld3(U, m.np, p);
        W[i] = u * dt;
    }
    return n;
}

// 1/n for the face-centre average (a table: no FP64 division)
__device__ __forceinline__ double inv_n(int n)
{
    return n == 4 ? 0.25 : n == 3 ? 1.0 / 3.0 : n == 5 ? 0.2 : n == 6 ? 1.0 / 6.0 : n == 7 ? 1.0 / 7.0 : 0.125;
}

// face-centre displacement: the mean of the point displacements
__device__ __forceinline__ V3 centre_disp(int n, const V3 *W)
{
    V3 wc = mk(0, 0, 0);
    for (int i = 0; i < n; ++i) wc = wc + W[i];
    return wc * inv_n(n);
}

__device__ __forceinline__ Cubic face_cubic(const DevMesh &m, int f, int n, const V3 *A, const V3 *W,
                                            const int *id)
{
    Cubic q = {0, 0, 0, 0, 0, 0};
    if (n == 3) {
        prism_cubic(A[0], A[1], A[2], W[0], W[1], W[2], id[0], id[1], id[2], q);
    } else {
        V3 c = ld3(m.cf, m.nf, f), wc = centre_disp(n, W);
        for (int t = 0; t < n; ++t) {
            int u = t + 1 == n ? 0 : t + 1;
            prism_cubic(c, A[t], A[u], wc, W[t], W[u], -1, id[t], id[u], q);
        }
    }
    return q;
}

__device__ __forceinline__ double cubic_at(const Cubic &q, double x) { return ((q.c3 * x + q.c2) * x + q.c1) * x; }

// Root of V(lambda) = tau in the first sign-changing interval of the grid
// k*LMAX/NSAMP (the bracket is the same one the secant oracle uses), refined by
// Newton steps that fall back to bisection when they leave the bracket.
// Returns lambda, or -1 (normal-sweep fallback) when no interval brackets a root.
// A flux below 1e-12 of |S_f| max|w| (noise = the rounding of a zero flux, e.g.
// on a wall) gives lambda = 0: no sweep.  The test is taken on squares,
// tau^2 <= 1e-24 |S_f|^2 max|w|^2 (noise2), which needs no square root.
// The sign of V(lambda_k) - tau at a grid point is read from an FP32
// evaluation where that is clearly away from zero (the FP32 conversion of the
// four coefficients and Horner's rounding stay below about 7 units of 2^-24,
// 4.2e-7, of the terms' magnitude B; the test asks for 1e-6 B),
// else from the FP64 one: the same signs, so the same bracket, as FP64
// throughout.  The bracket's end values are FP64.  The Newton step divides by
// the slope through an FP32 reciprocal (the slope sets the rate, not the root).
__device__ double solve_lambda(const Cubic &q, double tau, double noise2, int &its, unsigned &nev)
{
    its = 0;
    if (tau == 0.0) return 0.0;
    if (tau * tau <= 1e-24 * noise2) return 0.0;
    const float c1 = (float)q.c1, c2 = (float)q.c2, c3 = (float)q.c3, tf = (float)tau;
    const float a1 = fabsf(c1), a2 = fabsf(c2), a3 = fabsf(c3), at = fabsf(tf);
    constexpr double STEP = CORR_LMAX / CORR_NSAMP;
    const bool pos0 = -tau > 0.0;
    int klo = 0, khi = 0;
    double rhi = 0.0;
    bool have_rhi = false;
    for (int k = 1; k <= CORR_NSAMP; ++k) {
        const float L = (float)(k * STEP);
        const float r32 = ((c3 * L + c2) * L + c1) * L - tf;
        const float B = ((a3 * L + a2) * L + a1) * L + at;
        bool pos;
        double rk = 0.0;
        const bool sure = fabsf(r32) > 1e-6f * B;
        if (sure) {
            pos = r32 > 0.0f;
        } else {
            rk = cubic_at(q, k * STEP) - tau;
            ++nev;
            if (rk == 0.0) return k * STEP;
            pos = rk > 0.0;
        }
        if (pos != pos0) {
            khi = k;
            rhi = rk;
            have_rhi = !sure;
            break;
        }
        klo = k;
    }
    if (khi == 0) return -1.0;
    double lo = klo * STEP, hi = khi * STEP;
    double rlo = klo == 0 ? -tau : cubic_at(q, lo) - tau;
    nev += klo != 0;
    if (!have_rhi) {
        rhi = cubic_at(q, hi) - tau;
        ++nev;
        if (rhi == 0.0) return hi;
    }
    double x = lo - rlo * (hi - lo) / (rhi - rlo);
    if (!(x > lo && x < hi)) x = 0.5 * (lo + hi);
    while (its < CORR_MAXIT) {
        double r = cubic_at(q, x) - tau;
        ++nev;
        double ax = fabs(x);
        double scale = fmax(fabs(tau), ((q.s3 * ax + q.s2) * ax + q.s1) * ax);
        ++its;
        if ((r > 0) == (rhi > 0)) { hi = x; rhi = r; } else { lo = x; rlo = r; }
        if (fabs(r) <= CORR_TOL * scale) break;
        if (hi - lo <= 1e-15 * hi) break;
        double dr = (3.0 * q.c3 * x + 2.0 * q.c2) * x + q.c1;
        double xn = x - r * (double)__frcp_rn((float)dr);
        if (!(xn > lo && xn < hi)) xn = 0.5 * (lo + hi);
        x = xn;
    }
    return x;
}

__global__ void k_flux_polyhedra(DevMesh m, const double *__restrict__ Up, const double *F,
                                 const double *lambda, double dt, double *V)
{
    int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= m.nf) return;
    V3 A[VOF_MAXFP], W[VOF_MAXFP];
    int id[VOF_MAXFP];
    int n = face_points<false>(m, f, Up, dt, A, W, id);
    double lam = lambda ? lambda[f] : 1.0;
    if (lam < 0.0) {  // normal sweep: uniform translation along S_f
        V3 S = ld3(m.sf, m.nf, f);
        V3 wn = S * (-lam * F[f] * dt / dot(S, S));
        for (int i = 0; i < n; ++i) W[i] = wn;
        lam = 1.0;
    }
    Cubic q = face_cubic(m, f, n, A, W, id);
    V[f] = cubic_at(q, lam);
}

// The correction of one face with points b .. b+n-1 of m.fpts.  N = 3 or 4:
// the face has exactly N points and every array index is static after
// unrolling (registers); N = VOF_MAXFP: any n (local arrays).
template <int N>
__device__ __forceinline__ void correct_face(const DevMesh &m, int f, int b, int n, const double *U,
                                             const double *__restrict__ F, double dt, int item, double *lam_out,
                                             int *it_out, void *disp_out, bool disp32, int *maxit, int *nfallback,
                                             unsigned &ntri, unsigned &nev)
{
    constexpr bool FIXED = N <= 4;
    const int nn = FIXED ? N : n;
    V3 A[N], W[N];
    int id[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (i < nn) {
            int p = __ldg(m.fpts + b + i);
            id[i] = __ldg(m.fkey + b + i);  // the point's index (its master's on a periodic mesh)
            A[i] = ldP(m, p);
            W[i] = mk(U[p], U[m.np + p], U[2 * m.np + p]) * dt;
        }
    }
    const double tau = F[f] * dt;
    Cubic q = {0, 0, 0, 0, 0, 0};
    if (nn == 3) {
        prism_cubic(A[0], A[1], A[2], W[0], W[1], W[2], id[0], id[1], id[2], q);
    } else {
        V3 c = ld3(m.cf, m.nf, f), wc = mk(0, 0, 0);
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i < nn) wc = wc + W[i];
        wc = wc * inv_n(nn);
#pragma unroll
        for (int t = 0; t < N; ++t) {
            if (t < nn) {
                int u = t + 1 == nn ? 0 : t + 1;
                prism_cubic(c, A[t], A[u], wc, W[t], W[u], -1, id[t], id[u], q);
            }
        }
    }
    double w2 = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < nn) w2 = fmax(w2, dot(W[i], W[i]));
    const V3 S = ld3(m.sf, m.nf, f);
    int its = 0;
    ntri += nn == 3 ? 1 : nn;
    const double lam = solve_lambda(q, tau, dot(S, S) * w2, its, nev);
    lam_out[item] = lam;
    if (it_out) it_out[item] = its;
    if (maxit && its > 0) atomicMax(maxit, its);
    if (lam < 0.0 && nfallback) atomicAdd(nfallback, 1);
    if (disp_out) {
        V3 wc = mk(0, 0, 0);
        if (lam < 0.0) {
            wc = S * (-lam * F[f] * dt / dot(S, S));
#pragma unroll
            for (int i = 0; i < N; ++i) W[i] = wc;
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (i < nn) { W[i] = W[i] * lam; wc = wc + W[i]; }
            wc = wc * inv_n(nn);
        }
        // (in the type of the phase flux: converted once here, not by each of
        // its warps' lanes)
        auto put = [&](int i, const V3 &w) {
            if (disp32) {
                float *o = static_cast<float *>(disp_out) + (size_t)item * DISP_STRIDE + i;
                o[0] = (float)w.x; o[1] = (float)w.y; o[2] = (float)w.z;
            } else {
                double *o = static_cast<double *>(disp_out) + (size_t)item * DISP_STRIDE + i;
                o[0] = w.x; o[1] = w.y; o[2] = w.z;
            }
        };
        put(0, wc);
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i < nn) put(3 + 3 * i, W[i]);
    }
}

// One thread per face (LIST: per band slot).  U holds the point velocities.
template <bool LIST>
__global__ void k_correct(DevMesh m, const double *U, const double *__restrict__ F,
                          double dt, const int *list, const int *count, double *lam_out,
                          int *it_out, void *disp_out, bool disp32, int *maxit, int *nfallback, unsigned long long *work,
                          const double *__restrict__ alpha, BandRec *rec)
{
    previous_kernel();
    const int total = LIST ? *count : m.nf;
    unsigned ntri = 0, nev = 0;  // FP64 work: cubic coefficient triangles, cubic evaluations
    for (int item = blockIdx.x * blockDim.x + threadIdx.x; item < total; item += gridDim.x * blockDim.x) {
        const int f = LIST ? list[item] : item;
        const int b = __ldg(m.fptr + f), n = __ldg(m.fptr + f + 1) - b;
        if (n == 4)
            correct_face<4>(m, f, b, n, U, F, dt, item, lam_out, it_out, disp_out, disp32, maxit, nfallback, ntri, nev);
        else if (n == 3)
            correct_face<3>(m, f, b, n, U, F, dt, item, lam_out, it_out, disp_out, disp32, maxit, nfallback, ntri, nev);
        else
            correct_face<VOF_MAXFP>(m, f, b, n, U, F, dt, item, lam_out, it_out, disp_out, disp32, maxit, nfallback, ntri,
                                    nev);
        if (LIST) {
            const long long s0 = __ldg(m.sptr + f);
            const int ns = (int)(__ldg(m.sptr + f + 1) - s0);
            const V3 o = ld3(m.cf, m.nf, f);
            bool decide, comp;
            pf_form(m, F, alpha, f, lam_out[item], ns, decide, comp);
            rec[item] = BandRec{o.x, o.y, o.z, s0, f, b, n, ns, (comp ? 1u : 0u) | (decide ? 2u : 0u), {0u, 0u, 0u}};
        }
    }
    ntri = __reduce_add_sync(0xffffffffu, ntri);
    nev = __reduce_add_sync(0xffffffffu, nev);
    if ((threadIdx.x & 31) == 0) {
        work_add1(work, WK_CTRI, ntri);
        work_add1(work, WK_CEVAL, nev);
    }
}

// Point velocities (Eq. 4 weights, wall projection) of the points of this
// step's band faces, flagged by the classification; each point once, and the
// flag cleared for the next step.
__global__ void k_band_point_velocity(DevMesh m, const double *__restrict__ Uc, uint8_t *flag, double *Up)
{
    next_kernel();
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < m.np; p += gridDim.x * blockDim.x) {
        if (!flag[p]) continue;
        flag[p] = 0;
        st3(Up, m.np, p, point_velocity(m, p, Uc));
    }
}

// ========================================================= phase flux (A6)
struct Tet { V3 v[4]; };

// |T ^ {n_k.x <= d_k, k < np}| by depth-first splitting of T into the
// tetrahedra of its inside parts (1 or 3 per plane); the last plane is applied
// with the closed-form cut fraction.  Bounded stack: 1 + 2(np-1) entries.
__device__ double clip_tet(const Tet &T, const V3 *pn, const double *pd, int np, unsigned *status, WkOn &wk)
{
    wk.add(WK_VOL, 1);
    if (np == 0) return fabs(tvol(T.v[0], T.v[1], T.v[2], T.v[3]));
    Tet st[CLIP_STACK];
    unsigned char lv[CLIP_STACK];
    int sp = 1;
    st[0] = T;
    lv[0] = 0;
    double vol = 0.0;
    while (sp > 0) {
        --sp;
        Tet t = st[sp];
        int k = lv[sp];
        double s[4];
        int nin = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) { s[i] = dot(pn[k], t.v[i]) - pd[k]; nin += s[i] <= 0.0; }
        wk.add(WK_TEST, 1);
        if (nin == 0) continue;
        if (nin == 4) {
            if (k + 1 == np) { vol += fabs(tvol(t.v[0], t.v[1], t.v[2], t.v[3])); wk.add(WK_VOL, 1); }
            else if (sp < CLIP_STACK) { st[sp] = t; lv[sp] = k + 1; ++sp; }
            else atomicOr(status, VOF_ST_CLIP_OVERFLOW);
            continue;
        }
        if (k + 1 == np) {
            wk.add(WK_VOL, 1);
            wk.add(WK_FRAC, 1);
            double h0 = s[0], h1 = s[1], h2 = s[2], h3 = s[3];
            sort4(h0, h1, h2, h3);
            vol += fabs(tvol(t.v[0], t.v[1], t.v[2], t.v[3])) * frac_below(h0, h1, h2, h3, 0.0);
            continue;
        }
        // order vertices: inside ones first
        int ord[4], a = 0, b = 3;
#pragma unroll
        for (int i = 0; i < 4; ++i) { if (s[i] <= 0.0) ord[a++] = i; else ord[b--] = i; }
        V3 P[4];
        double S[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { P[i] = t.v[ord[i]]; S[i] = s[ord[i]]; }
        // point on edge (inside i, outside o), interpolated from the inside end
        auto ep = [&](int i, int o) { return P[i] + (P[o] - P[i]) * (S[i] / (S[i] - S[o])); };
        Tet out[3];
        int nout;
        if (nin == 1) {
            out[0] = Tet{{P[0], ep(0, 1), ep(0, 2), ep(0, 3)}};
            nout = 1;
        } else if (nin == 2) {
            // wedge (P0, p02, p03) -> (P1, p12, p13)
            V3 a0 = P[0], a1 = ep(0, 2), a2 = ep(0, 3), b0 = P[1], b1 = ep(1, 2), b2 = ep(1, 3);
            out[0] = Tet{{a0, a1, a2, b2}};
            out[1] = Tet{{a0, a1, b2, b1}};
            out[2] = Tet{{a0, b0, b1, b2}};
            nout = 3;
        } else {
            // prism (P0, P1, P2) -> (p03, p13, p23)
            V3 a0 = P[0], a1 = P[1], a2 = P[2], b0 = ep(0, 3), b1 = ep(1, 3), b2 = ep(2, 3);
            out[0] = Tet{{a0, a1, a2, b2}};
            out[1] = Tet{{a0, a1, b2, b1}};
            out[2] = Tet{{a0, b0, b1, b2}};
            nout = 3;
        }
        wk.add(WK_EDGE, nin == 2 ? 4 : 3);
        for (int i = 0; i < nout; ++i) {
            if (sp < CLIP_STACK) { st[sp] = out[i]; lv[sp] = k + 1; ++sp; }
            else atomicOr(status, VOF_ST_CLIP_OVERFLOW);
        }
    }
    return vol;
}

// ============================================================ update (A7)
// The cells are taken in segments (contiguous, at most a thousand or a few
// thousand cells of one region: set_bound_regions).  The update leaves, per
// segment, the step's masses and extrema and the sums that the redistribution's
// mesh-wide part needs; the redistribution then only recomputes the segments it
// changes, instead of sweeping every cell twice more.
constexpr int UPD_THREADS = 256;

// Columns of the per-segment table (SD_N columns of nseg values): before the
// redistribution: masses before and after the update, extrema, boundary outflow;
// after it (as before, until changed): mass, extrema; and, filled only where the
// mesh-wide fallback runs, excess and deficit volume, free and phase volume of
// the strictly mixed cells.
enum { SD_MB = 0, SD_MINP, SD_MAXP, SD_OUT, SD_M, SD_MIN, SD_MAX, SD_EP, SD_EM, SD_SP, SD_SM, SD_N };
constexpr int SD_UPD = SD_EP;  // the columns that the update fills
static_assert(SD_N == SEG_COLS && SD_M == SEG_COL_MASS, "the table as its other users see it");

// order of doubles on the integer pipe
__device__ __forceinline__ double min_bits(double a, double b) { return gt_bits(a, b) ? b : a; }
__device__ __forceinline__ double max_bits(double a, double b) { return gt_bits(a, b) ? a : b; }
__device__ __forceinline__ bool is_exc(double a) { return gt_pos(a, 1.0 + BOUND_TOL); }
__device__ __forceinline__ bool is_def(double a) { return lt_neg(a, BOUND_TOL); }
__device__ __forceinline__ bool is_mixed(double a) { return gt_pos(a, BOUND_TOL) && lt_pos(a, 1.0 - BOUND_TOL); }

// a warp's sum of v in a fixed order, skipped where every lane has zero (an
// FP64 add occupies its pipe for many cycles; most segments are empty)
__device__ __forceinline__ double warp_sum_nz(double v)
{
    return __any_sync(0xffffffffu, !is_zero(v)) ? warp_sum(v) : 0.0;
}
__device__ __forceinline__ double warp_min_bits(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min_bits(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ double warp_max_bits(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max_bits(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// A block per segment, a thread per cell.  Bound by HBM (28 B of cell CSR, 16 of
// alpha, 8 of V a cell, each face's flux once) and, on small meshes, by the chain
// of dependent loads.  An empty cell without flux costs no FP64 instruction and
// a full one without flux no division (the FP64 pipe runs at 1/63 of FP32).
__global__ void __launch_bounds__(UPD_THREADS) k_update(DevMesh m, double *alpha, const double *Va,
                                                        const int4 *__restrict__ seg, int nseg, double *sd,
                                                        uint8_t *seg_mixed, int *viol, int *nviol, unsigned *status)
{
    next_kernel();
    previous_kernel();
    __shared__ double sh[UPD_THREADS / 32][SD_UPD];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nb = m.nf - m.ni;
    for (int sgi = blockIdx.x; sgi < nseg; sgi += gridDim.x) {
        const int4 sg = seg[sgi];
        double mb = 0.0, ma = 0.0, out = 0.0, lo = 1e300, hi = -1e300;
        bool special = false;  // some cell beyond [0, 1] or strictly inside
        for (int i0 = sg.y; i0 < sg.z; i0 += UPD_THREADS) {
            const int c = i0 + threadIdx.x;
            bool bad = false;
            if (c < sg.z) {
                // A cell whose face fluxes are all zero (the bulk of either phase
                // away from the band) has s = +0; the FP64 sum runs only where some
                // flux is not zero, so warps of such cells issue no FP64 adds.
                // (six faces everywhere: no offsets to read)
                const int k0 = m.cuse == 6 ? 6 * c : m.cptr[c], k1 = m.cuse == 6 ? k0 + 6 : m.cptr[c + 1];
                const double a0 = alpha[c];
                unsigned nz = 0;
                // (cflux: the cell's faces, a periodic copy read as its face seen
                // from the neighbour; the cell's own faces on other meshes)
#pragma unroll 4
                for (int k = k0; k < k1; ++k) {
                    DBits b = dbits(Va[m.cflux[k] >> 1]);
                    nz |= (unsigned)(b.hi & 0x7fffffff) | b.lo;
                }
                double s = 0.0;
                if (nz)
                    for (int k = k0; k < k1; ++k) {
                        int code = m.cflux[k];
                        double x = Va[code >> 1];
                        s += (code & 1) ? -x : x;
                    }
                double a1 = a0;
                if (!is_zero(s) || !is_pzero(a0)) {  // (an empty cell with no flux: alpha stays +0)
                    const double V = m.vc[c];
                    if (!is_zero(s)) {
                        a1 = a0 - s / V;
                        alpha[c] = a1;
                    }
                    mb = fma(V, a0, mb);
                    ma = fma(V, a1, ma);
                    bad = is_exc(a1) || is_def(a1);
                    special |= bad || is_mixed(a1);
                }
                lo = min_bits(lo, a1);
                hi = max_bits(hi, a1);
            }
            if (viol) warp_append(bad, c, viol, nviol, m.nc, status);
        }
        // boundary faces: a chunk of them goes with each segment
        for (int f = sgi * UPD_THREADS + threadIdx.x; f < nb; f += nseg * UPD_THREADS) {
            const double v = Va[m.ni + f];
            if (!is_zero(v)) out += v;
        }
        double v[SD_UPD];
        v[SD_MB] = warp_sum_nz(mb);
        v[SD_OUT] = warp_sum_nz(out);
        v[SD_M] = warp_sum_nz(ma);
        v[SD_MIN] = v[SD_MINP] = warp_min_bits(lo);
        v[SD_MAX] = v[SD_MAXP] = warp_max_bits(hi);
        if (lane == 0)
#pragma unroll
            for (int i = 0; i < SD_UPD; ++i) sh[w][i] = v[i];
        const int any = __syncthreads_or(special);
        if (threadIdx.x == 0) seg_mixed[sgi] = any != 0;
        if (threadIdx.x < SD_UPD) {
            const int i = threadIdx.x;
            double r = sh[0][i];
            for (int k = 1; k < UPD_THREADS / 32; ++k) {
                const double x = sh[k][i];
                if (i == SD_MIN || i == SD_MINP) r = min_bits(r, x);
                else if (i == SD_MAX || i == SD_MAXP) r = max_bits(r, x);
                else if (!is_zero(x)) r += x;
            }
            sd[(size_t)i * nseg + sgi] = r;
        }
        __syncthreads();
    }
}

// A segment by a whole warp: fn(c, a) for every cell in order (lane-strided), then
// gn(c) for the cells for which fn returned true, 32 at a time in order: the
// few cells that take FP64 arithmetic are gathered first, since an FP64
// instruction costs the warp the same for one lane as for all.
constexpr int SEG_CHUNK = 256;
template <class Fn, class Gn>
__device__ __forceinline__ void seg_cells(const double *alpha, int4 sg, unsigned short *list, Fn fn, Gn gn)
{
    const int lane = threadIdx.x & 31;
    for (int c0 = sg.y; c0 < sg.z; c0 += SEG_CHUNK) {
        const int c1 = min(c0 + SEG_CHUNK, sg.z);
        int cnt = 0;
        double a[SEG_CHUNK / 32];
#pragma unroll
        for (int u = 0; u < SEG_CHUNK / 32; ++u) {
            const int c = c0 + 32 * u + lane;
            a[u] = c < c1 ? alpha[c] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < SEG_CHUNK / 32; ++u) {
            const int c = c0 + 32 * u + lane;
            const bool hit = c < c1 && fn(c, a[u]);
            const unsigned hm = __ballot_sync(0xffffffffu, hit);
            if (hit) list[cnt + __popc(hm & ((1u << lane) - 1u))] = (unsigned short)(c - c0);
            cnt += __popc(hm);
        }
        __syncwarp();
        for (int i = lane; i < cnt; i += 32) gn(c0 + list[i]);
        __syncwarp();
    }
}

// columns SD_M, SD_MIN, SD_MAX again after cells of the segment changed
__device__ __forceinline__ void seg_mass(const DevMesh &m, const double *alpha, int4 sg, int sgi, int nseg, double *sd,
                                         unsigned short *list)
{
    double ma = 0.0, lo = 1e300, hi = -1e300;
    seg_cells(alpha, sg, list,
              [&](int, double a) {
                  lo = min_bits(lo, a);
                  hi = max_bits(hi, a);
                  return !is_pzero(a);
              },
              [&](int c) { ma = fma(m.vc[c], alpha[c], ma); });
    ma = warp_sum_nz(ma);
    lo = warp_min_bits(lo);
    hi = warp_max_bits(hi);
    if ((threadIdx.x & 31) == 0) {
        sd[(size_t)SD_M * nseg + sgi] = ma;
        sd[(size_t)SD_MIN * nseg + sgi] = lo;
        sd[(size_t)SD_MAX * nseg + sgi] = hi;
    }
}

// columns SD_EP .. SD_SM: what the mesh-wide fallback spreads and who takes it
__device__ __forceinline__ void seg_room(const DevMesh &m, const double *alpha, int4 sg, int sgi, int nseg, double *sd,
                                         unsigned short *list)
{
    double ep = 0.0, em = 0.0, sp = 0.0, sm = 0.0;
    seg_cells(alpha, sg, list, [&](int, double a) { return is_exc(a) || is_def(a) || is_mixed(a); },
              [&](int c) {
                  const double a = alpha[c], V = m.vc[c];
                  if (is_exc(a)) ep += (a - 1.0) * V;
                  else if (is_def(a)) em += -a * V;
                  else {
                      sp += (1.0 - a) * V;
                      sm += a * V;
                  }
              });
    const double v[4] = {warp_sum_nz(ep), warp_sum_nz(em), warp_sum_nz(sp), warp_sum_nz(sm)};
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) sd[(size_t)(SD_EP + i) * nseg + sgi] = v[i];
}

// The step's statistics from the segment table (a block of any number of full
// warps, at most 32): a fixed tree.
__device__ void stats_block(const double *sd, int nseg, const int *counters, double *stats, unsigned *status)
{
    __shared__ double sh[32][7];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    constexpr int COL[7] = {SD_MB, SD_OUT, SD_M, SD_MINP, SD_MIN, SD_MAXP, SD_MAX};
    double v[7] = {0.0, 0.0, 0.0, 1e300, 1e300, -1e300, -1e300};
    for (int k = threadIdx.x; k < nseg; k += blockDim.x)
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            const double x = sd[(size_t)COL[i] * nseg + k];
            if (i < 3) { if (!is_zero(x)) v[i] += x; }
            else v[i] = i < 5 ? min_bits(v[i], x) : max_bits(v[i], x);
        }
    auto warp = [&]() {
#pragma unroll
        for (int i = 0; i < 7; ++i) v[i] = i < 3 ? warp_sum_nz(v[i]) : i < 5 ? warp_min_bits(v[i]) : warp_max_bits(v[i]);
    };
    warp();
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < 7; ++i) sh[w][i] = v[i];
    __syncthreads();
    if (w != 0) return;
#pragma unroll
    for (int i = 0; i < 7; ++i) v[i] = lane < nw ? sh[lane][i] : i < 3 ? 0.0 : i < 5 ? 1e300 : -1e300;
    warp();
    if (lane != 0) return;
    stats[VOF_S_MASS_BEFORE] = v[0];
    stats[VOF_S_BOUNDARY_OUT] = v[1];
    stats[VOF_S_MASS_AFTER] = v[2];
    stats[VOF_S_MIN_PRE] = v[3];
    stats[VOF_S_MIN_POST] = v[4];
    stats[VOF_S_MAX_PRE] = v[5];
    stats[VOF_S_MAX_POST] = v[6];
    if (status && (gt_pos(v[6], 1.0 + BOUND_FLAG) || lt_neg(v[4], BOUND_FLAG))) atomicOr(status, VOF_ST_BOUND_RESIDUAL);
    if (counters) {
        stats[VOF_S_N_INTERFACE] = counters[CNT_ICELL];
        stats[VOF_S_N_BAND] = counters[CNT_BAND];
        stats[VOF_S_MAX_POS_IT] = counters[CNT_MAXPOS];
        stats[VOF_S_MAX_CORR_IT] = counters[CNT_MAXCORR];
        stats[VOF_S_N_FALLBACK] = counters[CNT_FALLBACK];
        stats[VOF_S_N_BOUND_SOURCES] = counters[CNT_VIOL0];
        stats[VOF_S_N_BOUND_LEFT] = counters[CNT_VIOL1];
    }
}

constexpr int ST_THREADS = 512;
__global__ void __launch_bounds__(ST_THREADS) k_stats(const double *sd, int nseg, const int *counters, double *stats)
{
    previous_kernel();
    stats_block(sd, nseg, counters, stats, nullptr);
    if (threadIdx.x == 0) stats[VOF_S_BOUND_PASSES] = stats[VOF_S_BOUND_GLOBAL] = 0.0;
}

// ------------------------------------------ redistribution passes (reading R10)
// Sec. 2.3's wisp redistribution, read as passes of a local redistribution:
// a source (alpha > 1 + tol: excess e = (alpha - 1) V; alpha < -tol: deficit
// u = -alpha V) asks each face neighbour r for e w_r / W, where the receiver
// weight w = alpha (1 - alpha) V of an interface cell (tol < alpha < 1 - tol;
// 0 elsewhere, so no bulk cell receives and no wisp is made) and W the sum
// over the source's neighbours; a receiver takes at most its room, (1 - alpha)
// V for excess and alpha V for deficit, and scales all requests to fit, so it
// never leaves [0, 1]; what a source could not place stays with it for the
// next pass.  Passes run while some source has both something left and a
// receiver with room.  Every touched cell's new value is a gather over its
// face neighbours in face order.
// A cell is worked on by BP_LANES lanes, each taking every BP_LANES-th of its
// faces: one short chain of loads an item, and little code -- each phase runs
// once, so its instructions come from L2 as it goes (unrolled over a cell's
// faces, a phase took 10 us on 21 sources).
constexpr int BP_LANES = 8;
template <class Fn>
__device__ __forceinline__ void for_nbrs(const DevMesh &m, int x, Fn fn)
{
#pragma unroll 1
    for (int k = m.cptr[x] + (int)(threadIdx.x & (BP_LANES - 1)), k1 = m.cptr[x + 1]; k < k1; k += BP_LANES) {
        const int nb = m.cnb[k];
        if (nb >= 0) fn(nb);
    }
}
// sum over a cell's lanes, in a fixed order
__device__ __forceinline__ double lanes_sum(double v)
{
    const unsigned gm = ((1u << BP_LANES) - 1u) << (threadIdx.x & 31 & ~(BP_LANES - 1));
#pragma unroll
    for (int o = BP_LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gm, v, o);
    return v;
}
__device__ __forceinline__ double recv_w(double a, double V) { return is_mixed(a) ? a * (1.0 - a) * V : 0.0; }
// a source of a pass.  FP compares, not is_exc / is_def: a NaN fraction is no
// source (it would make its neighbours NaN); it is left to the fallback.
__device__ __forceinline__ bool src_exc(double a) { return a > 1.0 + BOUND_TOL; }
__device__ __forceinline__ bool src_def(double a) { return a < -BOUND_TOL; }

// Grid-wide barrier of a cooperative launch (every block resident): a block
// arrives on the count; the last to arrive resets it and advances the generation
// gen, which the others poll with a growing pause (count and generation sit
// on separate cache lines, so the polls do not hold up the arrivals).  A wait
// gives up after `limit` polls (BAR_SPIN_LIMIT: seconds) and flags VOF_ST_TIMEOUT;
// grid_sync then returns false in every thread of the block, which leaves the
// kernel (the blocks still waiting give up the same way: every wait ends).
constexpr long BAR_SPIN_LIMIT = 4000000;
__device__ bool grid_sync(unsigned *count, unsigned *generation, unsigned *status, long limit = BAR_SPIN_LIMIT)
{
    __shared__ int gave_up;
    __syncthreads();
    if (threadIdx.x == 0) {
        gave_up = 0;
        volatile unsigned *gen = generation;
        const unsigned g = *gen;
        __threadfence();
        if (atomicAdd(count, 1u) == gridDim.x - 1) {
            atomicExch(count, 0u);
            __threadfence();
            atomicAdd(generation, 1u);
        } else {
            long it = 0;
            unsigned pause = 16;
            while (*gen == g) {
                if (++it > limit) {
                    atomicOr(status, VOF_ST_TIMEOUT);
                    gave_up = 1;
                    break;
                }
                if (it <= 16) continue;  // (a barrier usually completes within a few polls)
                __nanosleep(pause);
                if (pause < 1024) pause <<= 1;
            }
        }
        __threadfence();
    }
    __syncthreads();
    return !gave_up;
}

// Numbers that a launch may use to mark cells (a pass each) and segments.  They
// move on where the update group's counters are cleared, before the launch:
// one whose waits ran out leaves no mark that a later launch takes for its own.
constexpr unsigned EPOCH_STEP = BOUND_PASSES_MAX + 2;

// The redistribution of a step: passes over the sources and their receivers,
// the mesh-wide fallback for what no local pass can place (a source none of
// whose face neighbours is an interface cell with room): the total excess
// (deficit) of a region (the whole mesh, or one case of a batch) goes to every
// cell of that region strictly inside (tol, 1-tol) in proportion to its free
// (phase) volume, and sources are set to 1 (0); then the step's statistics.
//
// A pass has three phases with a barrier after each: sources weigh their
// receivers and list them, each once (marked with the pass's own number, so the
// marks need no clearing; EPOCH_STEP); receivers gather their requests, scale them and
// form their new value; sources take off what was placed while the receivers'
// values are written.  The phases are chains of a few dependent loads over
// hundreds of items: barriers, first-time instruction fetches and, where many
// cells are strictly inside, FP64 work on few SMs are the cost.  On meshes up to
// BOUND_CLUSTER_CELLS the kernel is one cluster of eight blocks with the
// hardware's cluster barrier, beyond that one block per SM of a cooperative
// launch: the cluster's barriers are cheaper, and it starts while the update
// ends, until the cells take more than eight SMs (the update and this, in one
// cluster / over all SMs: 32^2 disc 33 / 41 us, 24^3 35 / 42, 24^3 film 37 / 46,
// 16^3 tetrahedra, with a fallback, 71 / 88, 32^3 37 / 47; beyond the line
// 32^3-based octree 69 / 62, 64^3 film 76 / 63, 48^3 tetrahedra, with a fallback,
// 230 / 143, 128^3 114 / 95).  With four barriers a pass over 608 blocks and two
// sweeps over every cell in each step they took 60 us on the 32^2 disc without a
// source (now 19), 94 at 24^3, 135 on the octree, 117 on the film, 153 at 128^3.
struct BoundStep {
    double *alpha;
    int *src;                    // sources (from the update)
    int *nsrc;                   // their count
    int *rl, *nrl;               // receivers of a pass, counts by pass parity
    double *ra;                  // their new values
    double *bs;                  // BS_N doubles per cell
    unsigned *mark;              // per cell: the pass that listed it
    unsigned *segmark;           // per segment: the launch that changed it
    int *dl, *ndl;               // changed segments
    const unsigned *epoch;       // the launch's first number less one (EPOCH_STEP apart)
    int *npass, *act, *left;     // passes that moved something; sources with a receiver, sources left, by pass parity
    int *nleft;                  // out: sources left to the fallback
    const int4 *seg;
    const int *seg_at;           // per SEG_STEP cells: the segment of the first
    int nseg;
    const uint8_t *seg_mixed;    // per segment: cells beyond [0, 1] or strictly inside
    double *sd;
    const int *reg_seg;
    int nreg;
    double *reg_tot;             // REG_TOT per region
    const int *counters;         // or null: no counter statistics
    double *stats;
    unsigned *bar_count;         // grid barrier: arrivals (zero before the launch)
    unsigned *bar_gen;           // and generation (any value)
    unsigned *status;
};
// scratch per cell: source: 1/W (0 where it has no receiver); receiver:
// weight, scales for excess and deficit
enum { BS_RW = 0, BS_W, BS_SP, BS_SM, BS_N = 4 };
// per region: Ep, Em, Sp, Sm and the shares Ep / Sp, Em / Sm of the mesh-wide
// step (0 where none)
constexpr int REG_TOT = 6;
constexpr int BA_THREADS = 1024;
constexpr int BA_CLUSTER = 8;
constexpr int BOUND_CLUSTER_CELLS = 1 << 15;

// region r, by a whole warp; eight segments' flags and sums are read at a time
// (the sums of segments without mixed cells are not kept up and left out)
__device__ void region_totals(const int *reg_seg, int r, const double *sd, const uint8_t *seg_mixed, int nseg,
                              double *totals)
{
    const int lane = threadIdx.x & 31;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    const int k1 = reg_seg[r + 1];
    for (int k = reg_seg[r] + lane; k < k1; k += 8 * 32) {
        unsigned in = 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u) in |= (unsigned)(k + 32 * u < k1 && seg_mixed[k + 32 * u]) << u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = k + 32 * u < k1 ? sd[(size_t)(SD_EP + i) * nseg + k + 32 * u] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) t[i] += in >> u & 1u ? v[u] : 0.0;
        }
    }
    for (int i = 0; i < 4; ++i) t[i] = warp_sum(t[i]);
    if (lane == 0) {
        double *o = totals + REG_TOT * (size_t)r;
        for (int i = 0; i < 4; ++i) o[i] = t[i];
        o[4] = t[0] > 0.0 && t[2] > 0.0 ? t[0] / t[2] : 0.0;
        o[5] = t[1] > 0.0 && t[3] > 0.0 ? t[1] / t[3] : 0.0;
    }
}
__device__ __forceinline__ bool region_applies(const double *tt)
{
    return !((tt[0] == 0.0 && tt[1] == 0.0) || tt[0] > tt[2] || tt[1] > tt[3]);
}

template <bool CLUSTER>
__global__ void __launch_bounds__(BA_THREADS, 1) k_bound_step(DevMesh m, BoundStep a)
{
    previous_kernel();
    // item i goes to block i mod gridDim.x: the few items of a phase spread over
    // every SM of the launch
    const int tl = threadIdx.x * gridDim.x + blockIdx.x, nt = gridDim.x * blockDim.x;
    const int wl = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, nw = nt >> 5;
    const int gl = (threadIdx.x / BP_LANES) * gridDim.x + blockIdx.x, ng = nt / BP_LANES;
    const bool first = (threadIdx.x & (BP_LANES - 1)) == 0;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    auto sync = [&]() -> bool {
        if constexpr (CLUSTER) {
            __syncthreads();
            if (threadIdx.x == 0) __threadfence();
            asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
            if (threadIdx.x == 0) __threadfence();
            __syncthreads();
            return true;
        } else return grid_sync(a.bar_count, a.bar_gen, a.status);
    };
    auto volat = [](const int *p) { return *(const volatile int *)p; };
    __shared__ unsigned short lists[BA_THREADS / 32][SEG_CHUNK];
    unsigned short *list = lists[threadIdx.x >> 5];
    const int n = min(*a.nsrc, m.nc);
    const unsigned e0 = *a.epoch;
    int npass = 0, nleft = n;
    if (n > 0) {
        auto touch = [&](int c) {  // c's segment has changed
            int k = a.seg_at[c / SEG_STEP];
            if (a.nreg > 1)
                while (c >= a.seg[k].z) ++k;
            if (atomicExch(a.segmark + k, e0 + 1) != e0 + 1) a.dl[atomicAdd(a.ndl, 1)] = k;
        };
#pragma unroll 1
        for (int p = 0; p < BOUND_PASSES_MAX; ++p) {
            const unsigned ep = e0 + 1 + p;
            int *act = a.act + (p & 1), *nrl = a.nrl + (p & 1), *left = a.left + (p & 1);
            if (lead) {  // the next pass's counters (last read before the previous pass's last barrier)
                a.act[(p + 1) & 1] = 0;
                a.nrl[(p + 1) & 1] = 0;
            }
            // ---- sources: weight of the receivers around, which are listed
            for (int i = gl; i < n; i += ng) {
                const int c = a.src[i];
                const double as = a.alpha[c];
                double W = 0.0;
                if (src_exc(as) || src_def(as))
                    for_nbrs(m, c, [&](int nb) {
                        const double w = recv_w(a.alpha[nb], m.vc[nb]);
                        if (is_zero(w)) return;
                        W += w;
                        if (atomicExch(a.mark + nb, ep) != ep) a.rl[atomicAdd(nrl, 1)] = nb;
                    });
                W = lanes_sum(W);
                if (first) {
                    a.bs[BS_N * (size_t)c + BS_RW] = W > 0.0 ? 1.0 / W : 0.0;
                    if (W > 0.0) atomicAdd(act, 1);
                }
            }
            if (!sync()) return;
            // (the previous pass's count of sources left was read after its last
            // barrier: it may be cleared only behind this one)
            if (lead) a.left[(p + 1) & 1] = 0;
            if (volat(act) == 0) break;
            npass = p + 1;
            // ---- receivers: requests, scales, new value
            const int nr = volat(nrl);
            for (int i = gl; i < nr; i += ng) {
                const int r = a.rl[i];
                const double ar = a.alpha[r], V = m.vc[r], wr = recv_w(ar, V);
                double Qp = 0.0, Qm = 0.0;
                for_nbrs(m, r, [&](int s) {
                    const double as = a.alpha[s];
                    const bool xe = src_exc(as);
                    if (!xe && !src_def(as)) return;
                    const double q = m.vc[s] * (wr * a.bs[BS_N * (size_t)s + BS_RW]);
                    if (xe) Qp += (as - 1.0) * q;
                    else Qm += -as * q;
                });
                Qp = lanes_sum(Qp);
                Qm = lanes_sum(Qm);
                if (first) {
                    const double Rp = (1.0 - ar) * V, Rm = ar * V;
                    const double sp = Qp > Rp ? Rp / Qp : 1.0, sm = Qm > Rm ? Rm / Qm : 1.0;
                    double *b = a.bs + BS_N * (size_t)r;
                    b[BS_W] = wr;
                    b[BS_SP] = sp;
                    b[BS_SM] = sm;
                    const double dV = Qp * sp - Qm * sm;
                    a.ra[i] = dV != 0.0 ? (ar * V + dV) / V : ar;
                }
            }
            if (!sync()) return;
            // ---- sources take off what was placed; receivers' values
            for (int i = gl; i < n; i += ng) {
                const int c = a.src[i];
                const double as = a.alpha[c];
                const bool xe = src_exc(as);
                if (!xe && !src_def(as)) {
                    if (first && as != as) atomicAdd(left, 1);
                    continue;
                }
                const double rW = a.bs[BS_N * (size_t)c + BS_RW], V = m.vc[c];
                double g = 0.0;
                if (rW > 0.0) {
                    const double e = (xe ? (as - 1.0) * V : -as * V) * rW;
                    for_nbrs(m, c, [&](int nb) {
                        const double *b = a.bs + BS_N * (size_t)nb;
                        if (a.mark[nb] == ep) g += e * b[BS_W] * b[xe ? BS_SP : BS_SM];
                    });
                }
                g = lanes_sum(g);
                if (first) {
                    double an = as;
                    if (g != 0.0) {
                        an = (as * V + (xe ? -g : g)) / V;
                        a.alpha[c] = an;
                        touch(c);
                    }
                    if (src_exc(an) || src_def(an)) atomicAdd(left, 1);
                }
            }
            for (int i = tl; i < nr; i += nt) {
                const int r = a.rl[i];
                a.alpha[r] = a.ra[i];
                touch(r);
            }
            if (!sync()) return;
            nleft = volat(left);
            if (nleft == 0) break;
        }
        if (nleft > 0) {
            for (int k = wl; k < a.nseg; k += nw)
                if (a.seg_mixed[k]) seg_room(m, a.alpha, a.seg[k], k, a.nseg, a.sd, list);
            if (!sync()) return;
            for (int r = wl; r < a.nreg; r += nw)
                region_totals(a.reg_seg, r, a.sd, a.seg_mixed, a.nseg, a.reg_tot);
            if (!sync()) return;
            // a cell strictly inside takes Ep (1 - a) V / Sp and gives Em a V / Sm:
            // a + (Ep / Sp)(1 - a) - (Em / Sm) a, no division per cell
            for (int k = wl; k < a.nseg; k += nw) {
                if (!a.seg_mixed[k]) continue;
                const int4 sg = a.seg[k];
                const double *tt = a.reg_tot + REG_TOT * (size_t)sg.x;
                if (!region_applies(tt)) continue;
                const double sp = tt[4], sm = tt[5];
                seg_cells(a.alpha, sg, list, [&](int, double x) { return is_exc(x) || is_def(x) || is_mixed(x); },
                          [&](int c) {
                              const double x = a.alpha[c];
                              a.alpha[c] = is_exc(x) ? 1.0 : is_def(x) ? 0.0 : x + sp * (1.0 - x) - sm * x;
                          });
                seg_mass(m, a.alpha, sg, k, a.nseg, a.sd, list);
            }
        }
        if (npass > 0) {
            // (a segment changed by a pass and by the fallback is summed twice,
            // by whichever warps: the same sums)
            const int nd = volat(a.ndl);
            if (nleft > 0 && !sync()) return;
            for (int i = wl; i < nd; i += nw) seg_mass(m, a.alpha, a.seg[a.dl[i]], a.dl[i], a.nseg, a.sd, list);
        }
        if (!sync()) return;
    }
    if (blockIdx.x != 0) return;
    if (lead) *a.nleft = nleft;
    __syncthreads();
    stats_block(a.sd, a.nseg, a.counters, a.stats, a.status);
    if (lead) {
        *a.npass = npass;
        double gv = 0.0;  // volume the fallback moved (regions where it applied)
        if (nleft > 0)
            for (int r = 0; r < a.nreg; ++r) {
                const double *tt = a.reg_tot + REG_TOT * (size_t)r;
                if (region_applies(tt)) gv += tt[0] + tt[1];
            }
        a.stats[VOF_S_BOUND_PASSES] = npass;
        a.stats[VOF_S_BOUND_GLOBAL] = gv;
    }
}

// The barrier's own check (a cooperative launch): every block passes `rounds`
// barriers, except block `skip`, which leaves at once, so that the others'
// waits run out after `limit` polls and flag VOF_ST_TIMEOUT (skip < 0: none
// leaves and nothing is flagged).
__global__ void k_barrier_probe(unsigned *count, unsigned *generation, unsigned *status, int skip, int rounds,
                                long limit)
{
    if ((int)blockIdx.x == skip) return;
    for (int r = 0; r < rounds; ++r)
        if (!grid_sync(count, generation, status, limit)) return;
}

__global__ void k_zero_int(int *p, int n)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = 0;
}

// the update group's counters (standalone update; a step zeroes them with the rest)
__global__ void k_zero_update(int *cnt)
{
    const int i = threadIdx.x;
    if (i < CNT_UPD_N) cnt[CNT_UPD + i] = 0;
    if (i == CNT_UPD_N) cnt[CNT_BAR] = 0;
    if (i == CNT_UPD_N + 1) cnt[CNT_EPOCH] = (int)((unsigned)cnt[CNT_EPOCH] + EPOCH_STEP);
}

// ============================================== band classification (A2, R9)
// per point: all cells empty (bit 0) / all full (bit 1); for the other points
// (every point of an interface cell is one) the IDW point value of Eq.
// idwpointphi, in the order the reconstruction would sum it
// (and the step's counters, which only later kernels use)
__global__ void k_point_state(DevMesh m, const double *__restrict__ alpha, uint8_t *state, double *palpha, int *cnt)
{
    next_kernel();
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < CNT_LEN) cnt[p] = 0;
    if (p == CNT_LEN) cnt[CNT_BAR] = 0;
    if (p == CNT_LEN + 1) cnt[CNT_EPOCH] = (int)((unsigned)cnt[CNT_EPOCH] + EPOCH_STEP);
    if (p >= m.np) return;
    bool all_e = true, all_f = true;
    const double full = 1.0 - m.eps;
    const int j0 = m.pptr[p], j1 = m.pptr[p + 1];
#pragma unroll 4
    for (int j = j0; j < j1; ++j) {
        double a = __ldg(alpha + m.pcell[j]);
        all_e &= le_pos(a, m.eps);
        all_f &= ge_pos(a, full);
    }
    state[p] = (all_e ? 1 : 0) | (all_f ? 2 : 0);
    if (!all_e && !all_f) {
        double ap = 0.0;
        for (int j = j0; j < j1; ++j) ap += __ldg(m.pw + j) * __ldg(alpha + m.pcell[j]);
        palpha[p] = ap;
    }
}

// (what the previous kernel wrote is not declared __restrict__: this one may have
// begun before, see previous_kernel)
__global__ void k_classify(DevMesh m, const double *__restrict__ alpha, const double *__restrict__ F,
                           double dt, const uint8_t *state, double *Va, int *band, int *nband,
                           int *icell, int *nicell, uint8_t *bpflag, unsigned *status)
{
    previous_kernel();
    const int lim = m.nf > m.nc ? m.nf : m.nc;
    for (int i0 = blockIdx.x * blockDim.x; i0 < lim; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + threadIdx.x;
        bool isband = false, isint = false;
        if (i < m.nf) {
            // the face's points: four at once on a mesh of quadrilaterals (16 of
            // the 24 bytes a face that the mesh costs otherwise, and one load
            // less in the chain); the flux only where some point has phase
            // (128^3: 54 -> 35 us)
            unsigned st = 3u;
            int4 q = make_int4(0, 0, 0, 0);
            int k0 = 0, k1 = 0;
            if (m.fuse == 4) {
                q = __ldg(reinterpret_cast<const int4 *>(m.fpts) + i);
                st = state[q.x] & state[q.y] & state[q.z] & state[q.w];
            } else {
                k0 = m.fptr[i];
                k1 = m.fptr[i + 1];
#pragma unroll 4
                for (int k = k0; k < k1; ++k) st &= state[m.fpts[k]];
            }
            double v = 0.0;
            if (!(st & 1u)) {
                const double Ff = F[i];
                // (a periodic face's copy carries no flux)
                if (!is_zero(Ff) && !(i >= m.ni && (dbits(Ff).hi < 0 || (m.fimg && m.fimg[i - m.ni] >= 0)))) {
                    if (st & 2u) v = Ff * dt;
                    else {
                        isband = true;
                        if (m.fuse == 4) bpflag[q.x] = bpflag[q.y] = bpflag[q.z] = bpflag[q.w] = 1;
                        else
                            for (int k = k0; k < k1; ++k) bpflag[m.fpts[k]] = 1;
                    }
                }
            }
            Va[i] = v;
        }
        if (i < m.nc) {
            double a = alpha[i];
            isint = gt_pos(a, m.eps) && lt_pos(a, 1.0 - m.eps);
        }
        warp_append(isband, i, band, nband, m.nf, status);
        warp_append(isint, i, icell, nicell, m.nc, status);
    }
}

inline int cdiv(long a, long b) { return (int)((a + b - 1) / b); }

}  // namespace

// ================================================================ launchers
#define LAUNCH_CHECK()                                            \
    do {                                                          \
        cudaError_t e_ = cudaGetLastError();                      \
        if (e_ != cudaSuccess) return VOF_ERR_CUDA;               \
    } while (0)

static int g_sms = 0;
static int num_sms(int dev)
{
    if (g_sms == 0) {
        int v = 0;
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        g_sms = v > 0 ? v : 148;
    }
    return g_sms;
}
int launch_setup_geometry(vof_ctx *c, cudaStream_t s)
{
    DevMesh &m = c->m;
    k_face_geom<<<cdiv(m.nf, 256), 256, 0, s>>>(m, (double *)m.cf, (double *)m.sf, (double *)m.nagc);
    LAUNCH_CHECK();
    unsigned *bad = c->status;
    k_cell_geom<<<cdiv(m.nc, 256), 256, 0, s>>>(m, (double *)m.cc, (double *)m.vc, (double *)m.cbox,
                                                    (double *)m.ctvol, bad);
    LAUNCH_CHECK();
    k_point_weights<<<cdiv(m.np, 256), 256, 0, s>>>(m, (double *)m.pw);
    LAUNCH_CHECK();
    return VOF_OK;
}

int launch_wall_table(vof_ctx *c, const int *wptr, const int *wface, int nrows, cudaStream_t s)
{
    if (nrows == 0) return VOF_OK;
    k_wall_table<<<cdiv(nrows, 256), 256, 0, s>>>(c->m, wptr, wface, nrows, (double *)c->m.wallt);
    LAUNCH_CHECK();
    return VOF_OK;
}

int launch_point_velocity(vof_ctx *c, const double *Uc, double *Up, cudaStream_t s)
{
    k_point_velocity<<<cdiv(c->np, 256), 256, 0, s>>>(c->m, Uc, Up);
    LAUNCH_CHECK();
    return VOF_OK;
}

// ===================================== generalised LSQ gradient (Sec. 2.2.1)
// Per cell the gradient minimising sum_k w^2 (phi_k - phi_c - g.d)^2 over the
// cells k sharing a point with c (d = x_k - x_c, w = 1/|d|, the inverse
// distance of Eq. generalizedLSQminimize): the 3x3 normal equations solved by
// the adjugate of their symmetric matrix (g = 0 where it is singular).
template <bool LIST>
__global__ void k_lsq_gradient(DevMesh m, const double *__restrict__ alpha, const int *list, const int *count,
                               const int *__restrict__ lptr, const int *__restrict__ lcell,
                               const uint8_t *__restrict__ lcode, double *grad)
{
    const int total = LIST ? *count : m.nc;
    for (int item = blockIdx.x * blockDim.x + threadIdx.x; item < total; item += gridDim.x * blockDim.x) {
        const int c = LIST ? list[item] : item;
        const V3 xc = ld3(m.cc, m.nc, c);
        const double pc = alpha[c];
        double a00 = 0, a01 = 0, a02 = 0, a11 = 0, a12 = 0, a22 = 0, b0 = 0, b1 = 0, b2 = 0;
        for (int k = __ldg(lptr + c), k1 = __ldg(lptr + c + 1); k < k1; ++k) {
            const int q = __ldg(lcell + k);
            const V3 dd = (lcode ? ld3(m.cc, m.nc, q) + tshift(m, __ldg(lcode + k)) : ld3(m.cc, m.nc, q)) - xc;
            const double w2 = 1.0 / dot(dd, dd), dp = (alpha[q] - pc) * w2;
            const V3 wd = dd * w2;
            a00 += wd.x * dd.x; a01 += wd.x * dd.y; a02 += wd.x * dd.z;
            a11 += wd.y * dd.y; a12 += wd.y * dd.z; a22 += wd.z * dd.z;
            b0 += dp * dd.x; b1 += dp * dd.y; b2 += dp * dd.z;
        }
        const double c00 = a11 * a22 - a12 * a12, c01 = a02 * a12 - a01 * a22, c02 = a01 * a12 - a02 * a11;
        const double c11 = a00 * a22 - a02 * a02, c12 = a01 * a02 - a00 * a12, c22 = a00 * a11 - a01 * a01;
        const double det = a00 * c00 + a01 * c01 + a02 * c02;
        V3 g = mk(0, 0, 0);
        if (det != 0.0) {
            const double r = 1.0 / det;
            g = mk((c00 * b0 + c01 * b1 + c02 * b2) * r, (c01 * b0 + c11 * b1 + c12 * b2) * r,
                   (c02 * b0 + c12 * b1 + c22 * b2) * r);
        }
        st3(grad, m.nc, c, g);
    }
}

int launch_lsq_gradient(vof_ctx *c, const double *alpha, const int *list, const int *count, double *grad,
                        cudaStream_t s)
{
    if (list)
        k_lsq_gradient<true><<<num_sms(c->device) * 8, 128, 0, s>>>(c->m, alpha, list, count, c->lptr, c->lcell,
                                                                    c->lcode, grad);
    else
        k_lsq_gradient<false><<<cdiv(c->nc, 128), 128, 0, s>>>(c->m, alpha, nullptr, nullptr, c->lptr, c->lcell,
                                                                c->lcode, grad);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

// ======================================= reconstruction error E_vsd (Sec. 4.1)
// The true phase is a ball (centre bc, radius R), resolved as the paper's tool
// mesh resolves a geometry: each cell tetrahedron is split into eight (edge
// midpoints; the inner octahedron about the diagonal joining the midpoints of
// edges ab and cd) down to `levels`; a piece is wholly in the ball (its four
// vertices in the closed ball), wholly outside (centroid distance less the
// largest vertex distance to the centroid at least R), or, undecided at the
// last level, cut by the plane tangent to the sphere at the point nearest its
// centroid.  A piece S with true phase P and reconstructed phase H adds
// |P| + |S ^ H| - 2 |P ^ H| (E_vsd^- + E_vsd^+).  The decisions use
// round-to-nearest operations without contraction, so that every piece is
// decided as the plain definition decides it.
constexpr int EVSD_MAX_LEVELS = 6;
constexpr int EVSD_STACK = 7 * EVSD_MAX_LEVELS + 1;

__device__ __forceinline__ V3 ev_sub(V3 a, V3 b) { return mk(__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y), __dsub_rn(a.z, b.z)); }
__device__ __forceinline__ double ev_d2(V3 a, V3 b)
{
    const V3 t = ev_sub(a, b);
    return __dadd_rn(__dadd_rn(__dmul_rn(t.x, t.x), __dmul_rn(t.y, t.y)), __dmul_rn(t.z, t.z));
}
__device__ __forceinline__ V3 ev_mid(V3 a, V3 b)
{
    return mk(__dmul_rn(__dadd_rn(a.x, b.x), 0.5), __dmul_rn(__dadd_rn(a.y, b.y), 0.5), __dmul_rn(__dadd_rn(a.z, b.z), 0.5));
}

struct EvPiece { V3 v[4]; int lev; };

__device__ double evsd_tet(const Tet &T0, int levels, V3 bc, double R, int hmode, V3 hn, double hd, unsigned *status)
{
    WkOn wk;  // counts nothing here; clip_tet's bookkeeping
    EvPiece st[EVSD_STACK];
    int sp = 0;
    st[sp++] = EvPiece{{T0.v[0], T0.v[1], T0.v[2], T0.v[3]}, 0};
    const double R2 = __dmul_rn(R, R);
    double e = 0.0;
    while (sp > 0) {
        const EvPiece q = st[--sp];
        const V3 a = q.v[0], b = q.v[1], c = q.v[2], d = q.v[3];
        const V3 g = mk(__dmul_rn(__dadd_rn(__dadd_rn(a.x, b.x), __dadd_rn(c.x, d.x)), 0.25),
                        __dmul_rn(__dadd_rn(__dadd_rn(a.y, b.y), __dadd_rn(c.y, d.y)), 0.25),
                        __dmul_rn(__dadd_rn(__dadd_rn(a.z, b.z), __dadd_rn(c.z, d.z)), 0.25));
        const bool inside = ev_d2(a, bc) <= R2 && ev_d2(b, bc) <= R2 && ev_d2(c, bc) <= R2 && ev_d2(d, bc) <= R2;
        double rt = sqrt(ev_d2(a, g));
        rt = fmax(rt, sqrt(ev_d2(b, g)));
        rt = fmax(rt, sqrt(ev_d2(c, g)));
        rt = fmax(rt, sqrt(ev_d2(d, g)));
        const double dist = sqrt(ev_d2(g, bc));
        const Tet S{{a, b, c, d}};
        const bool outside = !inside && __dsub_rn(dist, rt) >= R;
        if (inside || outside || q.lev >= levels) {
            const double vS = fabs(tvol(a, b, c, d));
            const double SH = hmode == 0 ? 0.0 : hmode == 1 ? vS : clip_tet(S, &hn, &hd, 1, status, wk);
            if (inside) { e += vS - SH; continue; }
            if (outside) { e += SH; continue; }
            V3 pn[2];
            double pd[2];
            const V3 u = dist > 0.0 ? (g - bc) * (1.0 / dist) : mk(1, 0, 0);
            pn[0] = u; pd[0] = dot(u, bc) + R;
            const double P = clip_tet(S, pn, pd, 1, status, wk);
            double PH = 0.0;
            if (hmode == 1) PH = P;
            else if (hmode == 2) { pn[1] = hn; pd[1] = hd; PH = clip_tet(S, pn, pd, 2, status, wk); }
            e += P + SH - 2.0 * PH;
            continue;
        }
        if (sp + 8 > EVSD_STACK) { atomicOr(status, VOF_ST_CAPACITY); continue; }
        const V3 ab = ev_mid(a, b), ac = ev_mid(a, c), ad = ev_mid(a, d), bm = ev_mid(b, c), bd = ev_mid(b, d),
                 cd = ev_mid(c, d);
        const int l = q.lev + 1;
        st[sp++] = EvPiece{{a, ab, ac, ad}, l};
        st[sp++] = EvPiece{{b, ab, bm, bd}, l};
        st[sp++] = EvPiece{{c, ac, bm, cd}, l};
        st[sp++] = EvPiece{{d, ad, bd, cd}, l};
        st[sp++] = EvPiece{{ab, cd, ac, ad}, l};
        st[sp++] = EvPiece{{ab, cd, ad, bd}, l};
        st[sp++] = EvPiece{{ab, cd, bd, bm}, l};
        st[sp++] = EvPiece{{ab, cd, bm, ac}, l};
    }
    return e;
}

// one warp per cell, a lane per cell tetrahedron; the lanes' sums in a fixed order
__global__ void k_evsd(DevMesh m, const uint8_t *flags, const double *n, const double *d, double bx, double by,
                       double bz, double R, int levels, double *out, unsigned *status)
{
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const V3 bc = mk(bx, by, bz);
    for (int c = warp; c < m.nc; c += nw) {
        int hmode = 0;
        V3 hn = mk(0, 0, 0);
        double hd = 0.0;
        if (flags) {
            const uint8_t f = flags[c];
            if (f & VOF_FULL) hmode = 1;
            else if ((f & VOF_INTERFACE) && (f & VOF_ORIENTED)) { hmode = 2; hn = ld3(n, m.nc, c); hd = d[c]; }
        }
        const V3 ctr = ld3(m.cc, m.nc, c);
        double e = 0.0;
        for (int tj = __ldg(m.ctptr + c) + lane; tj < __ldg(m.ctptr + c + 1); tj += 32) {
            const int4 te = __ldg(m.ctet + tj);
            V3 t0, t1, t2;
            if (te.w >= 0) {
                t0 = ldP(m, __ldg(m.fpts + te.y)); t1 = ldP(m, __ldg(m.fpts + te.z)); t2 = ldP(m, __ldg(m.fpts + te.w));
            } else {
                t0 = ld3(m.cf, m.nf, te.x >> 1); t1 = ldP(m, __ldg(m.fpts + te.y)); t2 = ldP(m, __ldg(m.fpts + te.z));
            }
            e += evsd_tet(Tet{{ctr, t0, t1, t2}}, levels, bc, R, hmode, hn, hd, status);
        }
        e = warp_sum(e);
        if (lane == 0) out[c] = e;
    }
}

int launch_evsd(vof_ctx *c, const uint8_t *flags, const double *n, const double *d, const double ball[4],
                int levels, double *out, cudaStream_t s)
{
    if (levels < 0 || levels > EVSD_MAX_LEVELS) return VOF_ERR_INVALID_ARG;
    k_evsd<<<num_sms(c->device) * 16, 128, 0, s>>>(c->m, flags, n, d, ball[0], ball[1], ball[2], ball[3], levels,
                                                   out, c->status);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

// ============================= geometric mapping for AMR (Sec. 3, Alg. 2)
// Per destination cell (one warp) the phase volume over its cell pairs
// (source cells sharing volume with it; nested cells): the same cell carries
// alpha_s V; a destination inside an oriented interface source takes its
// cell tetrahedra below the source's plane (lane per tetrahedron, closed-form
// cut fraction); inside any other source alpha_s V_dst; a source inside the
// destination adds alpha_s V_s.  Cells count as the same where their volumes
// agree to 1e-9.
__global__ void k_remap(DevMesh dm, const double *__restrict__ svc, int snc, const double *__restrict__ as,
                        const double *__restrict__ ns, const double *__restrict__ ds, const uint8_t *__restrict__ fs,
                        const int *__restrict__ pptr, const int *__restrict__ psrc, double *ad)
{
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int c = warp; c < dm.nc; c += nw) {
        const double Vc = dm.vc[c];
        const int q0 = __ldg(pptr + c), q1 = __ldg(pptr + c + 1);
        double acc = 0.0;
        if (q1 - q0 == 1) {
            const int s = __ldg(psrc + q0);
            const double Vs = svc[s], a = as[s];
            const uint8_t f = fs[s];
            if (fabs(Vc - Vs) <= 1e-9 * Vs) acc = lane == 0 ? a * Vc : 0.0;
            else if (Vc < Vs && (f & VOF_INTERFACE) && (f & VOF_ORIENTED)) {
                const V3 n = ld3(ns, snc, s);
                const double d = ds[s];
                const V3 ctr = ld3(dm.cc, dm.nc, c);
                for (int tj = __ldg(dm.ctptr + c) + lane; tj < __ldg(dm.ctptr + c + 1); tj += 32) {
                    const int4 te = __ldg(dm.ctet + tj);
                    V3 t0, t1, t2;
                    if (te.w >= 0) {
                        t0 = ldP(dm, __ldg(dm.fpts + te.y)); t1 = ldP(dm, __ldg(dm.fpts + te.z));
                        t2 = ldP(dm, __ldg(dm.fpts + te.w));
                    } else {
                        t0 = ld3(dm.cf, dm.nf, te.x >> 1); t1 = ldP(dm, __ldg(dm.fpts + te.y));
                        t2 = ldP(dm, __ldg(dm.fpts + te.z));
                    }
                    double h0 = dot(n, ctr), h1 = dot(n, t0), h2 = dot(n, t1), h3 = dot(n, t2);
                    sort4(h0, h1, h2, h3);
                    acc += fabs(tvol(ctr, t0, t1, t2)) * frac_below(h0, h1, h2, h3, d);
                }
            } else if (Vc < Vs) acc = lane == 0 ? a * Vc : 0.0;
            else acc = lane == 0 ? a * Vs : 0.0;
        } else {
            // several sources: each inside the destination (un-refined)
            for (int q = q0 + lane; q < q1; q += 32) {
                const int s = __ldg(psrc + q);
                acc += as[s] * svc[s];
            }
        }
        acc = warp_sum(acc);
        if (lane == 0) ad[c] = acc / Vc;
    }
}

int launch_remap(vof_ctx *dst, const vof_ctx *src, const double *alpha_src, const double *n_src,
                 const double *d_src, const uint8_t *flags_src, const int *pair_ptr, const int *pair_src,
                 double *alpha_dst, cudaStream_t s)
{
    k_remap<<<num_sms(dst->device) * 16, 128, 0, s>>>(dst->m, src->m.vc, src->nc, alpha_src, n_src, d_src,
                                                       flags_src, pair_ptr, pair_src, alpha_dst);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

// The reconstruction of the listed cells (list) or of every cell, with the
// context's lanes per cell and tetrahedra per lane (set by the largest cell's
// tetrahedra at creation); the instrumented variant while work counting is on.
template <bool MIXED, bool COUNT, int G, int KL>
static void rc_go(vof_ctx *c, const RcArgs &q, const int *list, const int *count, int *maxit, int *next, cudaStream_t s)
{
    if (list)
        k_reconstruct<MIXED, G, KL, COUNT><<<num_sms(c->device) * rc_resident<KL>(), RC_THREADS, 0, s>>>(
            c->m, q, list, count, maxit, c->mlp_s0, mlp_cap(c), next);
    else
        k_reconstruct_all<MIXED, G, KL, COUNT><<<cdiv(c->nc, rc_chunk<G>()), RC_THREADS, 0, s>>>(c->m, q);
}

template <bool MIXED, bool COUNT>
static void rc_shape(vof_ctx *c, const RcArgs &q, const int *list, const int *count, int *maxit, int *next,
                     cudaStream_t s)
{
    if (c->rc_g == 4) rc_go<MIXED, COUNT, 4, 1>(c, q, list, count, maxit, next, s);
    else if (c->rc_g == 8 && c->rc_k <= 2) rc_go<MIXED, COUNT, 8, 2>(c, q, list, count, maxit, next, s);
    else if (c->rc_g == 8) rc_go<MIXED, COUNT, 8, 3>(c, q, list, count, maxit, next, s);
    else if (c->rc_k == 1) rc_go<MIXED, COUNT, 32, 1>(c, q, list, count, maxit, next, s);
    else if (c->rc_k == 2) rc_go<MIXED, COUNT, 32, 2>(c, q, list, count, maxit, next, s);
    else rc_go<MIXED, COUNT, 32, 3>(c, q, list, count, maxit, next, s);
}

static void rc_launch(vof_ctx *c, const double *alpha, const double *palpha, const int *list, const int *count,
                      double *n, double *d, uint8_t *flags, int *iters, int *maxit, cudaStream_t s,
                      int *next = nullptr)
{
    // the generalised LSQ gradient of the cells first, where selected
    const double *gin = nullptr;
    if (c->grad_kind == VOF_GRAD_LSQ) {
        launch_lsq_gradient(c, alpha, list, count, c->grad, s);
        gin = c->grad;
    }
    const RcArgs q{alpha, palpha, gin, n, d, flags, iters, c->status, c->work_on ? c->work : nullptr};
    if (c->precision == VOF_MIXED) {
        if (c->work_on) rc_shape<true, true>(c, q, list, count, maxit, next, s);
        else rc_shape<true, false>(c, q, list, count, maxit, next, s);
    } else {
        if (c->work_on) rc_shape<false, true>(c, q, list, count, maxit, next, s);
        else rc_shape<false, false>(c, q, list, count, maxit, next, s);
    }
}

// defaults of every cell (n = 0, d = 0, flags FULL or 0, iterations 0), and
// the interface cells appended to a list
__global__ void k_fill_list(int nc, double eps, const double *__restrict__ alpha, double *n, double *d,
                            uint8_t *flags, int *iters, int *list, int *count, unsigned *status)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    bool isint = false;
    if (c < nc) {
        const double a = alpha[c];
        flags[c] = a >= 1.0 - eps ? VOF_FULL : 0;
        n[c] = 0.0; n[nc + c] = 0.0; n[2 * nc + c] = 0.0;
        d[c] = 0.0;
        if (iters) iters[c] = 0;
        isint = a > eps && a < 1.0 - eps;
    }
    warp_append(isint, c, list, count, nc, status);
}

int launch_reconstruct(vof_ctx *c, const double *alpha, double *n, double *d, uint8_t *flags, int *iters,
                       const int *list, const int *count, cudaStream_t s)
{
    const bool mx = c->precision == VOF_MIXED;
    if (mx && c->mlp && !list) {
        // the guess is indexed by list position: list the interface cells first
        k_zero_int<<<1, 32, 0, s>>>(c->counters + CNT_ICELL, 1);
        k_fill_list<<<cdiv(c->nc, 256), 256, 0, s>>>(c->nc, c->eps, alpha, n, d, flags, iters, c->icell,
                                                     c->counters + CNT_ICELL, c->status);
        list = c->icell;
        count = c->counters + CNT_ICELL;
    }
    if (mx && c->mlp) {
        int r = launch_mlp_guess(c, alpha, list, count, c->nc, s);
        if (r) return r;
    }
    rc_launch(c, alpha, nullptr, list, count, n, d, flags, iters, list ? c->counters + CNT_MAXPOS : nullptr, s);
    LAUNCH_CHECK();
    return VOF_OK;
}

int launch_flux_polyhedra(vof_ctx *c, const double *Up, const double *F, const double *lambda, double dt,
                          double *V, cudaStream_t s)
{
    k_flux_polyhedra<<<cdiv(c->nf, 128), 128, 0, s>>>(c->m, Up, F, lambda, dt, V);
    LAUNCH_CHECK();
    return VOF_OK;
}

int launch_correct_all(vof_ctx *c, const double *Up, const double *F, double dt, double *lambda, int *iters,
                       cudaStream_t s)
{
    k_correct<false><<<cdiv(c->nf, 128), 128, 0, s>>>(c->m, Up, F, dt, nullptr, nullptr, lambda, iters,
                                                             nullptr, false, nullptr, nullptr, c->work_on ? c->work : nullptr,
                                                             nullptr, nullptr);
    LAUNCH_CHECK();
    return VOF_OK;
}

int launch_phase_flux_all(vof_ctx *c, const double *alpha, const double *n, const double *d, const uint8_t *flags,
                          const double *Up, const double *F, const double *lambda, double dt, double *Va, cudaStream_t s)
{
    return launch_pf_all(c, alpha, n, d, flags, Up, F, lambda, dt, Va, s);
}

// The update, then the redistribution with the statistics (or the statistics
// alone); counters: the step's, or null.
static int launch_update_group(vof_ctx *c, double *alpha, const double *Va, const int *counters, double *stats,
                               cudaStream_t s)
{
    int *cnt = c->counters;
    if (launch_after(k_update, std::min(c->nseg, num_sms(c->device) * 8), UPD_THREADS, 0, s, c->m, alpha, Va, c->seg,
                     c->nseg, c->sd, c->seg_mixed, c->bound ? c->viol : nullptr, cnt + CNT_VIOL0, c->status))
        return VOF_ERR_CUDA;
    LAUNCH_CHECK();
    if (!c->bound) {
        return launch_after(k_stats, 1, ST_THREADS, 0, s, c->sd, c->nseg, counters, stats);
    }
    const BoundStep a{alpha, c->viol, cnt + CNT_VIOL0, c->rl, cnt + CNT_NRL0, c->ra, c->bscr, c->cmark, c->segmark,
                      c->dl, cnt + CNT_NDL, reinterpret_cast<unsigned *>(cnt + CNT_EPOCH), cnt + CNT_BPASS,
                      cnt + CNT_BACT0, cnt + CNT_LEFT0, cnt + CNT_VIOL1, c->seg, c->seg_at, c->nseg, c->seg_mixed, c->sd, c->reg_seg,
                      c->nreg, c->reg_tot, counters, stats, reinterpret_cast<unsigned *>(cnt + CNT_BAR),
                      reinterpret_cast<unsigned *>(cnt + CNT_BARGEN), c->status};
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(BA_THREADS);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (c->nc <= BOUND_CLUSTER_CELLS) {
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.numAttrs = 2;
        cfg.gridDim = dim3(BA_CLUSTER);
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = BA_CLUSTER;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        return cudaLaunchKernelEx(&cfg, k_bound_step<true>, c->m, a) == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
    }
    cfg.gridDim = dim3(num_sms(c->device));
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    return cudaLaunchKernelEx(&cfg, k_bound_step<false>, c->m, a) == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

int launch_barrier_probe(vof_ctx *c, int skip, cudaStream_t s)
{
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_barrier_probe, 128, 0) != cudaSuccess || occ < 1)
        return VOF_ERR_CUDA;
    const int blocks = num_sms(c->device) * std::min(occ, 2);
    if (skip >= blocks) return VOF_ERR_INVALID_ARG;
    unsigned *cnt = reinterpret_cast<unsigned *>(c->counters + CNT_BAR);
    unsigned *gen = reinterpret_cast<unsigned *>(c->counters + CNT_BARGEN);
    if (cudaMemsetAsync(cnt, 0, sizeof(unsigned), s) != cudaSuccess) return VOF_ERR_CUDA;
    int rounds = 4;
    long limit = 2000;  // with the pauses (up to ~1 us) a few milliseconds
    void *args[] = {&cnt, &gen, &c->status, &skip, &rounds, &limit};
    if (cudaLaunchCooperativeKernel((const void *)k_barrier_probe, dim3(blocks), dim3(128), args, 0, s) != cudaSuccess)
        return VOF_ERR_CUDA;
    return VOF_OK;
}

// Courant number: the largest (1/2) sum |F_f| dt / V_c over the cells, the
// block maxima combined by an atomic max on the bit patterns (non-negative
// doubles order as their 64-bit integers)
__global__ void k_courant(DevMesh m, const double *__restrict__ F, double dt, unsigned long long *co)
{
    __shared__ double red[8];
    double v = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < m.nc; c += gridDim.x * blockDim.x) {
        double sum = 0.0;
        for (int k = m.cptr[c]; k < m.cptr[c + 1]; ++k) sum += fabs(F[m.cflux[k] >> 1]);
        v = fmax(v, 0.5 * sum * dt / m.vc[c]);
    }
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = fmax(v, red[w]);
        atomicMax(co, (unsigned long long)__double_as_longlong(v));
    }
}

int launch_courant(vof_ctx *c, const double *F, double dt, double *co, cudaStream_t s)
{
    if (cudaMemsetAsync(co, 0, sizeof(double), s) != cudaSuccess) return VOF_ERR_CUDA;
    k_courant<<<num_sms(c->device) * 4, 256, 0, s>>>(c->m, F, dt, reinterpret_cast<unsigned long long *>(co));
    LAUNCH_CHECK();
    return VOF_OK;
}

int launch_update(vof_ctx *c, double *alpha, const double *Va, double *stats, cudaStream_t s)
{
    k_zero_update<<<1, 32, 0, s>>>(c->counters);
    LAUNCH_CHECK();
    c->launches = 3;
    return launch_update_group(c, alpha, Va, nullptr, stats ? stats : c->stats_dev, s);
}

int launch_advect(vof_ctx *c, double *alpha, const double *Uc, const double *F, double dt, double *stats,
                  cudaStream_t s, cudaEvent_t wait_before_correct)
{
    DevMesh &m = c->m;
    int sms = num_sms(c->device);
    int *cnt = c->counters;
    int launches = 0;
    cudaEvent_t *ev = nullptr;
    if (c->prof_ev && c->prof_steps < c->prof_max) ev = c->prof_ev + (size_t)c->prof_steps++ * (VOF_PROF_GROUPS + 1);
#define MARK(i) do { if (ev) cudaEventRecord(ev[i], s); } while (0)
    MARK(0);
    k_point_state<<<cdiv(m.np, 256), 256, 0, s>>>(m, alpha, c->pstate, c->palpha, cnt);
    if (launch_after(k_classify, sms * 16, 256, 0, s, m, alpha, F, dt, c->pstate, c->Va, c->band, cnt + CNT_BAND,
                     c->icell, cnt + CNT_ICELL, c->bpflag, c->status))
        return VOF_ERR_CUDA;
    launches += 2;
    LAUNCH_CHECK();
    MARK(1);
    // The correction (band point velocities, then lambda per band face) needs
    // the band list and the velocities, the reconstruction the interface list:
    // the two run side by side, the correction on the context's second stream,
    // joined before the phase flux.  The first use of Uc is there, so a
    // velocity copy still in flight on another stream is waited for there.
    if (cudaEventRecord(c->ev_fork, s) != cudaSuccess || cudaStreamWaitEvent(c->s_aux, c->ev_fork, 0) != cudaSuccess)
        return VOF_ERR_CUDA;
    if (wait_before_correct && cudaStreamWaitEvent(c->s_aux, wait_before_correct, 0) != cudaSuccess)
        return VOF_ERR_CUDA;
    k_band_point_velocity<<<cdiv(m.np, 256), 256, 0, c->s_aux>>>(m, Uc, c->bpflag, c->upb);
    if (launch_after(k_correct<true>, sms * 8, 128, 0, c->s_aux, m, c->upb, F, dt, c->band, cnt + CNT_BAND, c->lam_b,
                     c->it_b, c->disp_b, c->precision == VOF_MIXED, cnt + CNT_MAXCORR, cnt + CNT_FALLBACK,
                     c->work_on ? c->work : nullptr, alpha, c->pf_rec))
        return VOF_ERR_CUDA;
    LAUNCH_CHECK();
    if (cudaEventRecord(c->ev_join, c->s_aux) != cudaSuccess) return VOF_ERR_CUDA;
    if (c->precision == VOF_MIXED && c->mlp) {
        int r = launch_mlp_guess(c, alpha, c->icell, cnt + CNT_ICELL, c->nc, s);
        if (r) return r;
        ++launches;
    }
    rc_launch(c, alpha, c->palpha, c->icell, cnt + CNT_ICELL, c->n, c->d, c->flags, nullptr, cnt + CNT_MAXPOS, s,
              cnt + CNT_RCNEXT);
    MARK(2);
    if (cudaStreamWaitEvent(s, c->ev_join, 0) != cudaSuccess) return VOF_ERR_CUDA;
    MARK(3);
    {
        int r = launch_pf_list(c, alpha, F, dt, sms, s);
        if (r) return r;
    }
    launches += 6;  // reconstruct, band point velocities, correct, phase flux (pairs, clips, sums)
    LAUNCH_CHECK();
    MARK(4);
    // update + bounding + stats
    {
        int r = launch_update_group(c, alpha, c->Va, cnt, stats ? stats : c->stats_dev, s);
        if (r) return r;
    }
    launches += 2;
    MARK(5);
#undef MARK
    c->launches = launches;
    return VOF_OK;
}
