// Phase flux (A6, Eqs. S'_f, S''_f): the flux-polyhedron tetrahedra T of a
// band face, the cell tetrahedra K of its stencil cells and their PLIC planes
// are taken to a frame centred on the face centre and intersected there: in a
// step by three launches over the band faces (pairs, clips, sums; below), in
// the standalone call by a warp per face of the mesh.  One source for both forms:
//  - mixed (R = float): FP32 clipping, pieces summed per lane with TwoSum
//    compensation and finished in FP64 (reading R13 on the on-plane band);
//  - plain (R = double): the same structure in FP64 (what FP32 decides beyond
//    its roundings, it decides).
//
// Only the frame shift of a stencil cell (its centre minus the face centre) and
// of its plane offset are formed in FP64; the cell's own geometry comes from
// offsets to the cell centre computed once at context creation, so the
// rounding of a coordinate is relative to the cell size, not to its position.
#include <cuda_runtime.h>

#include <type_traits>
#include <math.h>
#include <stdint.h>

#include "vof_device.cuh"
#include "vof_internal.h"

namespace {
using namespace vofd;

// ------------------------------------------------------------ real types
template <class R>
struct R3 { R x, y, z; };
struct __align__(16) D4 { double x, y, z, w; };
template <class R> struct Q4;
template <> struct Q4<float> { using T = float4; };
template <> struct Q4<double> { using T = D4; };
template <class R> using R4 = typename Q4<R>::T;

template <class R> __device__ __forceinline__ R3<R> r3(R x, R y, R z) { return R3<R>{x, y, z}; }
template <class R> __device__ __forceinline__ R3<R> operator+(R3<R> a, R3<R> b) { return r3(a.x + b.x, a.y + b.y, a.z + b.z); }
template <class R> __device__ __forceinline__ R3<R> operator-(R3<R> a, R3<R> b) { return r3(a.x - b.x, a.y - b.y, a.z - b.z); }
template <class R> __device__ __forceinline__ R3<R> operator*(R3<R> a, R s) { return r3(a.x * s, a.y * s, a.z * s); }
template <class R> __device__ __forceinline__ R rdot(R3<R> a, R3<R> b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
template <class R> __device__ __forceinline__ R3<R> rcross(R3<R> a, R3<R> b)
{
    return r3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
template <class R> __device__ __forceinline__ R rvol6(R3<R> a, R3<R> b, R3<R> c, R3<R> d)
{
    return rdot(b - a, rcross(c - a, d - a));
}
__device__ __forceinline__ float rmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double rmin(double a, double b) { return fmin(a, b); }
__device__ __forceinline__ float rmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double rmax(double a, double b) { return fmax(a, b); }
__device__ __forceinline__ float rabs(float a) { return fabsf(a); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float rmuladd(float a, float b, float c) { return __fadd_rn(__fmul_rn(a, b), c); }
__device__ __forceinline__ float rnext(float a, float b) { return nextafterf(a, b); }
__device__ __forceinline__ double rnext(double a, double b) { return nextafter(a, b); }
__device__ __forceinline__ double rabs(double a) { return fabs(a); }
// divisions of the clip: the fast FP32 reciprocal-multiply (2 ulp, far inside
// the mixed form's rounding), or FP64 by the FP32 reciprocal of the truncated
// divisor refined twice (error squared each time: to the last place or so),
// four FP64 instructions; the full division where the divisor leaves the FP32 range
__device__ __forceinline__ float rdiv(float a, float b) { return __fdividef(a, b); }
__device__ __noinline__ double full_div(double a, double b) { return a / b; }
__device__ __forceinline__ double rdiv(double a, double b)
{
    const float f = tf(b), r0 = __fdividef(1.0f, f);
    if (!(fabsf(f) > 1e-30f && fabsf(f) < 1e30f)) return full_div(a, b);
    const double r1 = fd(r0), r2 = fma(r1, fma(-b, r1, 1.0), r1), q = a * r2;
    return fma(r2, fma(-b, q, a), q);
}

template <class R> __device__ __forceinline__ R4<R> mk4(R x, R y, R z, R w);
template <> __device__ __forceinline__ float4 mk4<float>(float x, float y, float z, float w) { return make_float4(x, y, z, w); }
template <> __device__ __forceinline__ D4 mk4<double>(double x, double y, double z, double w) { return D4{x, y, z, w}; }
__device__ __forceinline__ float4 ldg4(const float4 *p, long i) { return __ldg(p + i); }
__device__ __forceinline__ D4 ldg4(const D4 *p, long i)
{
    const double2 *q = reinterpret_cast<const double2 *>(p + i);
    const double2 a = __ldg(q), b = __ldg(q + 1);
    return D4{a.x, a.y, b.x, b.y};
}
template <class R> __device__ __forceinline__ R3<R> ld43(const R4<R> *p, long i)
{
    const R4<R> v = ldg4(p, i);
    return r3<R>(v.x, v.y, v.z);
}

// Threshold, sign and order tests of distances (tol >= 0).  FP32: the native
// compares.  FP64: integer compares of the bit patterns (dbits), the same
// decisions for every value that is not NaN: this part's FP64 pipe runs at
// 1/63 of the FP32 rate, and an FP64 compare or min/max holds it as long as
// an FMA.
__device__ __forceinline__ bool rpos(float v) { return v > 0.0f; }
__device__ __forceinline__ bool rneg(float v) { return v < 0.0f; }
__device__ __forceinline__ bool rgt(float a, float b) { return a > b; }
__device__ __forceinline__ bool rabove(double v, double t) { return gt_pos(v, t); }   // v > t
__device__ __forceinline__ bool rbelow(double v, double t) { return lt_neg(v, t); }   // v < -t
__device__ __forceinline__ bool rpos(double v) { return gt_pos(v, 0.0); }
__device__ __forceinline__ bool rneg(double v) { return lt_neg(v, 0.0); }
__device__ __forceinline__ bool rgt(double a, double b) { return gt_bits(a, b); }

// fraction of a tetrahedron below level 0 for sorted vertex values h0..h3
template <class R>
__device__ __forceinline__ R rfrac_below(R h0, R h1, R h2, R h3)
{
    if (!rneg(h0)) return R(0);
    if (!rpos(h3)) return R(1);
    // one division per case
    if constexpr (std::is_same<R, double>::value) {
        // one vertex below or one above: the same cut seen from either end
        const bool low = !rneg(h1);
        if (low || !rpos(h2)) {
            const R x = low ? -h0 : h3, d30 = h3 - h0;
            const R e1 = low ? h1 - h0 : h3 - h1, e2 = low ? h2 - h0 : h3 - h2;
            const R q = rdiv(x * x * x, d30 * e1 * e2);
            return low ? q : R(1) - q;
        }
    }
    if (!rneg(h1)) {
        const R x = -h0;
        return rdiv(x * x * x, (h1 - h0) * (h2 - h0) * (h3 - h0));
    }
    if (!rpos(h2)) {
        const R y = h3;
        return R(1) - rdiv(y * y * y, (h3 - h0) * (h3 - h1) * (h3 - h2));
    }
    const R d1 = h2 - h0, d2 = h3 - h0, d3 = h2 - h1, d4 = h3 - h1;
    const R p12 = d1 * d2, p123 = p12 * d3, q = rdiv(R(1), p123 * d4);
    const R r4 = q * p123, q3 = q * d4, r3 = q3 * p12, q2 = q3 * d3, r1 = q2 * d2, r2 = q2 * d1;
    const R a = -h0 * r1, b = -h0 * r2, c = -h1 * r3, e = -h1 * r4;
    return a * b + a * (R(1) - b) * e + (R(1) - a) * c * e;
}

template <class R>
__device__ __forceinline__ void rsort4(R &a, R &b, R &c, R &d)
{
    R t;
#define CS(p, q)                                                              \
    if constexpr (sizeof(R) == 4) { t = rmin(p, q); q = rmax(p, q); p = t; }  \
    else if (rgt(p, q)) { t = p; p = q; q = t; }
    CS(a, b) CS(c, d) CS(a, c) CS(b, d) CS(b, c)
#undef CS
}

template <class R> struct RTet { R3<R> v[4]; };

// Running sum of the pieces (6 |volume| times sign and weight): FP32 with
// TwoSum (Knuth) compensation, s + c carrying the sum up to the rounding of
// the compensation (no multiplications, so no fused operation can change it);
// FP64 plainly.  (A 64-bit fixed-point sum, exact and order-independent, cost
// 6 % of the kernel's time in its conversions.)
template <class R> struct Acc { R s = R(0), c = R(0); };
__device__ __forceinline__ void acc_add(Acc<float> &a, float x)
{
    const float t = a.s + x;
    const float bp = t - a.s;
    a.c += (a.s - (t - bp)) + (x - bp);
    a.s = t;
}
__device__ __forceinline__ void acc_add(Acc<double> &a, double x) { a.s += x; }

constexpr int MX_MAXT = 3 * VOF_MAXFP;
static_assert(MX_MAXT <= 32, "one flux-polyhedron tetrahedron per lane");

struct MXArgs {
    const double *alpha, *n, *d;
    const uint8_t *flags;
    const double *Up, *F, *lambda;
    double dt;
    double *Va;
    const int *list, *count;
    const void *disp;         // list form: displacements of a face's centre and points, in the form's type
    unsigned *status;
    unsigned long long *work;
    const void *fpl, *cbl, *ktl;  // the context's tables (R4 of the form's type)
    const int *ctptr;
};

constexpr int MX_CAND = 32;    // candidate cell tetrahedra buffered per warp: one per lane
constexpr int MX_QUEUE = MX_MAXT * MX_CAND;  // clip jobs: one per (T, K) pair at most
// pieces of clip jobs waiting for their next plane, per warp (the stack depth
// S is a launch choice: 92 commits more lanes per split step, 56 leaves room
// for more resident warps)
constexpr int MX_STACK_WIDE = 92, MX_STACK_SLIM = 56;

// Shared memory of a warp, by stage.
// the flux polyhedron: its prisms (one per face triangle swept) and tetrahedra
template <class R, class B = R>
struct __align__(16) PolyShared {
    R4<R> P6[VOF_MAXFP][5];  // per prism: a0 a1 a2 b0 b1 b2, 18 values in 20
    B Pb[VOF_MAXFP][6];      // prism box
    R4<B> Pc[VOF_MAXFP][2];  // its centre and half extents
    R Tv6[MX_MAXT];          // |6 vol(T)|
    R Tsg[MX_MAXT];          // sign of T in the flux polyhedron
};
// stencil cells of the current chunk that reach the polyhedron's box
template <class R>
struct __align__(16) CellShared {
    R4<R> CH[32];            // phase (or void) half-space
    R4<R> Cd[32];            // cell centre - face centre; w (as bits): first tetrahedron less the
                             // chunk's tetrahedra before it
    R Cw[32];
    int Cend[32];            // running count of tetrahedra, inclusive
    unsigned char CuseH[32];
};
// buffered candidate cell tetrahedra, their pairs with the prisms and the clip jobs
template <class R>
struct __align__(16) CandShared {
    R4<R> Kp[MX_CAND][5];    // outward unit-normal planes of the candidate cell tetrahedra, then
                             // the cell's phase (or void) half-space; 80-byte rows (FP32): a warp's
                             // float4 reads of different rows are conflict-free
    R Kw[MX_CAND];           // weight: 1, or alpha (1-alpha) of an unoriented cell
    unsigned short Q[MX_QUEUE];              // clip job: t | k << 5 | plane mask << 10
    unsigned short PQ[VOF_MAXFP * MX_CAND];  // (prism, candidate) pairs with overlapping boxes
    unsigned char KuseH[MX_CAND];
};
// the clip queue's pieces; in FP32 the 48-byte tetrahedra are moved as three
// float4 (conflict-free across a warp)
template <class R, int MX_STACK>
struct __align__(16) StackShared {
    RTet<R> S[MX_STACK];     // pieces
    RTet<R> T[MX_MAXT];      // flux-polyhedron tetrahedra
    unsigned short Sm[MX_STACK];  // piece: t | k << 5 | planes still to clip << 10
};
// the whole flux of a face in one warp
template <class R, int MX_STACK_>
struct __align__(16) MXShared : PolyShared<R>, CellShared<R>, CandShared<R>, StackShared<R, MX_STACK_> {
    static constexpr int MX_STACK = MX_STACK_;
    R Kb[MX_CAND][6];
};

__device__ __forceinline__ RTet<float> ldT(const RTet<float> &t)
{
    const float4 *p = reinterpret_cast<const float4 *>(&t);
    const float4 a = p[0], b = p[1], c = p[2];
    return RTet<float>{{r3(a.x, a.y, a.z), r3(a.w, b.x, b.y), r3(b.z, b.w, c.x), r3(c.y, c.z, c.w)}};
}
__device__ __forceinline__ RTet<double> ldT(const RTet<double> &t) { return t; }

__device__ __forceinline__ void stT(RTet<float> &t, const RTet<float> &v)
{
    float4 *p = reinterpret_cast<float4 *>(&t);
    p[0] = make_float4(v.v[0].x, v.v[0].y, v.v[0].z, v.v[1].x);
    p[1] = make_float4(v.v[1].y, v.v[1].z, v.v[2].x, v.v[2].y);
    p[2] = make_float4(v.v[2].z, v.v[3].x, v.v[3].y, v.v[3].z);
}
__device__ __forceinline__ void stT(RTet<double> &t, const RTet<double> &v) { t = v; }

// an int kept in the unused component of a vector
template <class R> __device__ __forceinline__ R int_bits(int i)
{
    if constexpr (std::is_same<R, float>::value) return __int_as_float(i);
    else return __hiloint2double(0x3ff00000, i);
}
__device__ __forceinline__ int bits_int(float x) { return __float_as_int(x); }
__device__ __forceinline__ int bits_int(double x) { return __double2loint(x); }

__device__ __forceinline__ float tof(float x) { return x; }
__device__ __forceinline__ float tof(double x) { return tf(x); }

// signed distance to plane p (FP64: three instructions, not four, of a pipe that
// issues one in many cycles)
__device__ __forceinline__ float pdist(float4 p, R3<float> v) { return p.x * v.x + p.y * v.y + p.z * v.z - p.w; }
__device__ __forceinline__ double pdist(D4 p, R3<double> v) { return fma(p.x, v.x, fma(p.y, v.y, fma(p.z, v.z, -p.w))); }

// signed distances of the vertices to plane p, those within tol taken as 0;
// nin / nup count the vertices strictly below / above
template <class R>
__device__ __forceinline__ void fdist(const RTet<R> &t, R4<R> p, R tol, R s[4], int &nin, int &nup)
{
    nin = 0;
    nup = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        R v = pdist(p, t.v[i]);
        if constexpr (std::is_same<R, double>::value) {  // integer tests
            const bool up = rabove(v, tol), dn = rbelow(v, tol);
            s[i] = (up || dn) ? v : R(0);
            nin += dn;
            nup += up;
        } else {
            if (rabs(v) <= tol) v = R(0);
            s[i] = v;
            nin += v < R(0);
            nup += v > R(0);
        }
    }
}

// The part of t below the plane (distances s, 1 <= nin <= 3 vertices strictly
// below, at least one strictly above) as the tetrahedra (a0, a1, a2, b2) and,
// for nin > 1, (a0, a1, b2, b1) and (a0, b0, b1, b2) of the points c[0..5] = a0 a1 a2
// b0 b1 b2.  Vertices are ordered below-first by a compare-exchange network so
// that every index stays static; the three cases (one, two or three below) run
// as one with selected ends of the cut edges, not as three branches that the
// lanes of a warp take one after another.
template <class R>
__device__ __forceinline__ void fsplit(const RTet<R> &t, const R s[4], int nin, R3<R> c[6])
{
    using V = R3<R>;
    V P0 = t.v[0], P1 = t.v[1], P2 = t.v[2], P3 = t.v[3];
    R S0 = s[0], S1 = s[1], S2 = s[2], S3 = s[3];
#define MX_CX(a, b)                                                   \
    if (!rneg(S##a) && rneg(S##b)) {                                  \
        V tp = P##a; P##a = P##b; P##b = tp;                          \
        R ts = S##a; S##a = S##b; S##b = ts;                          \
    }
    MX_CX(0, 1) MX_CX(2, 3) MX_CX(0, 2) MX_CX(1, 3) MX_CX(1, 2)
#undef MX_CX
    // cut edges from f (below) to g: (0,1) (0,2) (0,3) | (0,2) (0,3) (1,2) (1,3) | (0,3) (1,3) (2,3)
    const bool n1 = nin == 1, n2 = nin == 2, n3 = nin == 3;
    auto sel = [](bool p, V x, V y) { return V{p ? x.x : y.x, p ? x.y : y.y, p ? x.z : y.z}; };
    const V g0 = sel(n1, P1, sel(n2, P2, P3)), f1 = sel(n3, P1, P0), g1 = sel(n1, P2, P3);
    const V f2 = sel(n1, P0, sel(n2, P1, P2)), g2 = sel(n2, P2, P3);
    const R sg0 = n1 ? S1 : n2 ? S2 : S3, sf1 = n3 ? S1 : S0, sg1 = n1 ? S2 : S3;
    const R sf2 = n1 ? S0 : n2 ? S1 : S2, sg2 = n2 ? S2 : S3;
    // the edge parameters sf / (sf - sg) from one division (the reciprocal of
    // the denominators' product, then products): the divisions hold the FP64
    // pipe longest, and FP32 saves issue slots
    const R d1 = S0 - sg0, d2 = sf1 - sg1, d3 = sf2 - sg2, d4 = n2 ? S1 - S3 : R(1);
    const R p12 = d1 * d2, p123 = p12 * d3, q = rdiv(R(1), p123 * d4);
    const R r4 = q * p123, q3 = q * d4, r3 = q3 * p12, q2 = q3 * d3, r1 = q2 * d2, r2 = q2 * d1;
    // (fused explicitly: the selects below let the compiler take the sums apart)
    auto ept = [](V a, V b, R t) { return V{rfma(b.x - a.x, t, a.x), rfma(b.y - a.y, t, a.y), rfma(b.z - a.z, t, a.z)}; };
    const V e0 = ept(P0, g0, S0 * r1), e1 = ept(f1, g1, sf1 * r2), e2 = ept(f2, g2, sf2 * r3);
    const V e3 = ept(P1, P3, S1 * r4);
    c[0] = P0;
    c[1] = sel(n3, P1, e0);
    c[2] = sel(n3, P2, e1);
    c[3] = sel(n3, e0, P1);
    if constexpr (std::is_same<R, double>::value) c[4] = sel(n3, e1, e2);
    else {
        // (this point's product is rounded before the sum: so it always was in
        // the mixed form, its two cases' sums having been one after their branches)
        const V dd = sel(n3, g1 - f1, g2 - f2);
        const R tt = n3 ? sf1 * r2 : sf2 * r3;
        c[4] = V{rmuladd(dd.x, tt, P1.x), rmuladd(dd.y, tt, P1.y), rmuladd(dd.z, tt, P1.z)};
    }
    c[5] = sel(n2, e3, e2);
}

// What an FP32 distance of a point of the flux polyhedron (box pb, M its largest
// coordinate) to a unit-normal plane has to exceed for the point to lie above
// the plane: truncated operands and four roundings err by 8.4e-7 M + 3.6e-7 |w|
// at most, w the plane's offset, which is below 1.8 M where the plane can cut
// the polyhedron; 2e-6 M is above that.  It goes with the polyhedron's extent, not
// with the face's: along a needle cell the sweep is hundreds of face sizes long.
template <class B>
__device__ __forceinline__ float drop_slack(const B pb[6])
{
    float v = 0.0f;
#pragma unroll
    for (int i = 0; i < 6; ++i) v = fmaxf(v, fabsf(tof(pb[i])));
    return 2e-6f * v;
}

// The queued clip jobs, worked through by the whole warp, one piece per lane
// and step.  Pieces with one plane left (leaves) stack up from the bottom of S,
// the others down from its top, and a step works on one kind only, so that the
// lanes run the same code:
//  - leaf step: a piece adds its volume below its last plane (closed-form cut
//    fraction);
//  - split step: a piece from the other stack (else a new job) is cut by its
//    next plane and the parts below are pushed, to the leaves if one plane is
//    left; a new job with one plane goes to the leaves whole (no leaf work in
//    a split step: a step's lanes never mix the two kinds of work).  A
//    part none of whose points is below the plane after is dropped at once (the
//    parts share six points, so this takes six distances, not a push, a pop
//    and a step's share each).
// A split step commits the longest prefix of lanes that leaves the two stacks
// at most MX_STACK - 6 full; if none does, the top piece alone when it fits,
// else a leaf step runs first (leaves need no room).  Every part of a split
// piece has at most 4 planes to go, so the split pieces keep i + 1 + 2 (r - 1)
// <= MX_STACK for depth i and r planes to go: the top one alone always fits
// once the leaves are gone, and the stacks cannot overflow.
template <class R, class Sh, class Wk>
__device__ __forceinline__ void mx_clip(Sh &sh, const unsigned short *Q, int nq, R tol, float drop, Acc<R> &acc, Wk &wk)
{
    constexpr int MX_STACK = Sh::MX_STACK;
    const int lane = threadIdx.x & 31;
    const unsigned le = ((1u << lane) << 1) - 1u;
    __syncwarp();
    int nl = 0, nn = 0, qn = 0;
    bool force_leaf = false;
    for (;;) {
        const bool more = nn > 0 || qn < nq;
        if (!more && nl == 0) break;
        if (force_leaf || nl >= 32 || !more) {
            // ---- leaf step
            force_leaf = false;
            const int p = min(nl, 32);
            if (lane < p) {
                const RTet<R> t = ldT(sh.S[nl - 1 - lane]);
                const unsigned meta = sh.Sm[nl - 1 - lane];
                const int ti = meta & 31, k = (meta >> 5) & 31, j = __ffs(meta >> 10) - 1;
                R sd[4];
                int nin, nup;
                fdist(t, sh.Kp[k][j], tol, sd, nin, nup);
                wk.add(WK_TEST, 1);
                R v6 = R(0);
                if (nin > 0) {
                    v6 = rabs(rvol6(t.v[0], t.v[1], t.v[2], t.v[3]));
                    wk.add(WK_VOL, 1);
                    if (nup > 0) {
                        wk.add(WK_FRAC, 1);
                        R h0 = sd[0], h1 = sd[1], h2 = sd[2], h3 = sd[3];
                        rsort4(h0, h1, h2, h3);
                        v6 *= rfrac_below(h0, h1, h2, h3);
                    }
                }
                if (rpos(v6)) acc_add(acc, sh.Tsg[ti] * sh.Kw[k] * v6);  // (v6 >= 0)
            }
            nl -= p;
            __syncwarp();
            continue;
        }
        // ---- split step
        const int p = min(nn, 32), r = min(32 - p, nq - qn);
        const bool act = lane < p + r;
        RTet<R> t;
        unsigned meta = 0;
        if (act) {
            const RTet<R> *src;
            if (lane < p) {
                meta = sh.Sm[MX_STACK - nn + lane];
                src = &sh.S[MX_STACK - nn + lane];
            } else {
                meta = Q[qn + lane - p];
                src = &sh.T[meta & 31];
            }
            t = ldT(*src);
        }
        __syncwarp();  // every piece read before the pushes reuse the slots
        int nin = 0, nup = 0, ti = 0, k = 0;
        unsigned rem = 0, keep = 0;  // keep: parts to push
        R sd[4];
        bool cut = false, single = false;
        R3<R> c[6];
        int ndrop = 0;
        if (act) {
            ti = meta & 31;
            k = (meta >> 5) & 31;
            rem = meta >> 10;
            single = (rem & (rem - 1)) == 0;
            if (single) keep = 1;  // a job with one plane goes to the leaves whole
            else {
                const int j = __ffs(rem) - 1;
                rem &= rem - 1;
                fdist(t, sh.Kp[k][j], tol, sd, nin, nup);
                if (nin > 0) {
                    cut = nup > 0;
                    keep = cut && nin > 1 ? 7 : 1;
                }
            }
            c[0] = t.v[0]; c[1] = t.v[1]; c[2] = t.v[2]; c[5] = t.v[3];
            if (cut) fsplit(t, sd, nin, c);
            if (keep && !single) {
                // the points below the plane after (FP64: those not above it
                // by an FP32 distance beyond its roundings (drop_slack); a part
                // kept for nothing is dropped when its own turn comes)
                const R4<R> pn = sh.Kp[k][__ffs(rem) - 1];
                const float4 pf = make_float4(tof(pn.x), tof(pn.y), tof(pn.z), tof(pn.w));
                auto below = [&](int i) {
                    if constexpr (std::is_same<R, float>::value) return pdist(pn, c[i]) < -tol;
                    else return pdist(pf, r3(tof(c[i].x), tof(c[i].y), tof(c[i].z))) < drop;
                };
                const bool z0 = below(0), z1 = below(1), z2 = below(2), z5 = below(5);
                ndrop = __popc(keep);
                unsigned kept = z0 || z1 || z2 || z5 ? 1u : 0u;
                if (keep & 2u) {
                    const bool z3 = below(3), z4 = below(4);
                    kept |= z0 || z1 || z5 || z4 ? 2u : 0u;
                    kept |= z0 || z3 || z4 || z5 ? 4u : 0u;
                }
                keep = kept;
                ndrop -= __popc(kept);
            }
        }
        const int nch = __popc(keep);
        const bool toleaf = single || (rem & (rem - 1)) == 0;  // one plane left after this one
        const unsigned b0 = __ballot_sync(0xffffffffu, nch & 1), b1 = __ballot_sync(0xffffffffu, nch & 2);
        const unsigned bl = __ballot_sync(0xffffffffu, toleaf);
        const int inc = __popc(b0 & le) + 2 * __popc(b1 & le);
        const bool fits = act && nl + nn - min(lane + 1, p) + inc <= MX_STACK - 6;
        const unsigned fm = __ballot_sync(0xffffffffu, fits);
        int L = fm ? 32 - __clz(fm) : 0;
        if (L == 0) {
            const int nch0 = __shfl_sync(0xffffffffu, nch, 0);
            if (nl + nn - (p > 0 ? 1 : 0) + nch0 <= MX_STACK) L = 1;
            else { force_leaf = true; continue; }  // nothing written: the leaves first
        }
        const unsigned lm = L >= 32 ? 0xffffffffu : (1u << L) - 1u;
        const int top = MX_STACK - nn + min(L, p);  // the split stack's top after the pops
        if (lane < L) {
            // work of the committed lanes (the others redo theirs later); a
            // dropped part counts as tested
            wk.add(WK_TEST, !single + ndrop);
            if (cut) wk.add(WK_EDGE, nin == 2 ? 4 : 3);
            if (nch > 0) {
                const unsigned cm = (unsigned)ti | ((unsigned)k << 5) | (rem << 10);
                // parts of the lanes before this one that go the same way
                const unsigned same = (toleaf ? bl : ~bl) & ((1u << lane) - 1u);
                const int before = __popc(b0 & same) + 2 * __popc(b1 & same);
                int at = toleaf ? nl + before : top - 1 - before;
                const int step = toleaf ? 1 : -1;
                auto put = [&](const RTet<R> &x) {
                    stT(sh.S[at], x);
                    sh.Sm[at] = (unsigned short)cm;
                    at += step;
                };
                if (keep & 1u) put(RTet<R>{{c[0], c[1], c[2], c[5]}});
                if (keep & 2u) put(RTet<R>{{c[0], c[1], c[5], c[4]}});
                if (keep & 4u) put(RTet<R>{{c[0], c[3], c[4], c[5]}});
            }
        }
        nl += __popc(b0 & bl & lm) + 2 * __popc(b1 & bl & lm);
        nn = MX_STACK - top + __popc(b0 & ~bl & lm) + 2 * __popc(b1 & ~bl & lm);
        qn += max(0, L - p);
        __syncwarp();
    }
}

// rounding allowance of the box tests: coordinates within the polyhedron's box pb
// (and the planes' offsets, of that size) carry a few roundings each, well
// below a quarter of the on-plane band
template <class R>
__device__ __forceinline__ R box_slack(const R pb[6])
{
    R v = R(0);
#pragma unroll
    for (int i = 0; i < 6; ++i) v = rmax(v, rabs(pb[i]));
    return v * (sizeof(R) == 4 ? R(5e-7) : R(1e-15));
}

// a box (centre, half extents) lies wholly outside a plane, by slack
template <class R>
__device__ __forceinline__ bool beyond(R4<R> p, R4<R> ce, R4<R> he, R slack)
{
    const R s = rfma(p.x, ce.x, rfma(p.y, ce.y, rfma(p.z, ce.z, -p.w)));
    const R r = rfma(rabs(p.x), he.x, rfma(rabs(p.y), he.y, rfma(rabs(p.z), he.z, slack)));
    return s >= r;
}

// All (T, K) pairs of the buffered candidates, taken a prism (the three
// tetrahedra of one swept face triangle) at a time.  First lane k tests
// candidate k's box against each prism's box and the overlapping (prism, K)
// pairs are listed; then each listed pair, one per lane, gets the signed
// distances of the prism's six points to K's planes, from which each of its
// three tetrahedra is classified: outside a plane, inside every plane (adds
// |T| at once), or a clip job.  kb: the box of candidate 'lane'.  Returns the
// number of jobs; used gets the candidates that have any.
// FP32: a prism whose box lies wholly beyond a plane of the candidate (by slack,
// which covers the roundings: its points then all classify as outside) is not
// paired; a box against a plane takes 7 instructions, a pair about 60 a plane.
template <class R, class Sh, class Wk>
__device__ __forceinline__ int mx_pairs(Sh &sh, int nt, int ncand, const R kb[6], R tol, R slack, Acc<R> &acc,
                                        unsigned &used, Wk &wk)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int nprism = nt / 3;
    int total = 0;
    {
        constexpr bool CULL = std::is_same<R, float>::value;
        R4<R> pl[5];
        if constexpr (CULL) {
#pragma unroll
            for (int q = 0; q < 5; ++q) pl[q] = sh.Kp[lane][q];
            if (lane >= ncand || !sh.KuseH[lane]) pl[4] = mk4<R>(R(0), R(0), R(0), R(1));
        }
        for (int pr = 0; pr < nprism; ++pr) {
            const R *tb = sh.Pb[pr];
            const bool live = sh.Tsg[3 * pr] != R(0) || sh.Tsg[3 * pr + 1] != R(0) || sh.Tsg[3 * pr + 2] != R(0);
            bool ov = lane < ncand && live &&
                      !(rgt(kb[0], tb[3]) || rgt(tb[0], kb[3]) || rgt(kb[1], tb[4]) || rgt(tb[1], kb[4]) ||
                        rgt(kb[2], tb[5]) || rgt(tb[2], kb[5]));
            if constexpr (CULL) {
                const R4<R> ce = sh.Pc[pr][0], he = sh.Pc[pr][1];
#pragma unroll
                for (int q = 0; q < 5; ++q) ov = ov && !beyond<R>(pl[q], ce, he, slack);
            }
            const unsigned bm = __ballot_sync(0xffffffffu, ov);
            if (ov) sh.PQ[total + __popc(bm & lt)] = (unsigned short)(pr | lane << 3);
            total += __popc(bm);
        }
    }
    __syncwarp();
    int nq = 0;
    used = 0u;
    for (int pb = 0; pb < total; pb += 32) {
        const int pi = pb + lane;
        unsigned code[3] = {0u, 0u, 0u};
        bool job[3] = {false, false, false};
        if (pi < total) {
            const unsigned pc = sh.PQ[pi];
            const int pr = pc & 7, k = pc >> 3;
            R v[20];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const R4<R> q = sh.P6[pr][i];
                v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
            }
            const int npl = sh.KuseH[k] ? 5 : 4;
            wk.add(WK_PRISM, npl);
            unsigned mask[3] = {0u, 0u, 0u};
            bool outside[3] = {false, false, false};
            // a point within tol of a plane is on it: a tetrahedron is outside
            // when none of its points is clearly inside a plane, and a plane cuts
            // it only when its points lie clearly on both sides.  FP64: a rolled
            // loop over the pair's planes (the unrolled body's instruction
            // footprint cost 13 % of the launch); FP32: unrolled over five
            constexpr bool F64 = std::is_same<R, double>::value;
#pragma unroll(F64 ? 1 : 5)
            for (int q = 0; q < (F64 ? npl : 5); ++q) {
                const R4<R> pl = sh.Kp[k][q];
                R d[6];
#pragma unroll
                for (int i = 0; i < 6; ++i)
                    d[i] = rfma(pl.x, v[3 * i], rfma(pl.y, v[3 * i + 1], rfma(pl.z, v[3 * i + 2], -pl.w)));
                // T0 = a0 a1 a2 b2, T1 = a0 a1 b2 b1, T2 = a0 b0 b1 b2
                if constexpr (std::is_same<R, double>::value) {
                    // the points not clearly inside the plane (ge) and those
                    // clearly outside it (gt) as bits 0..5 = a0 a1 a2 b0 b1 b2,
                    // from integer tests (no FP64 compare or min/max)
                    unsigned ge = 0u, gt = 0u;
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        ge |= (unsigned)!rbelow(d[i], tol) << i;
                        gt |= (unsigned)rabove(d[i], tol) << i;
                    }
                    constexpr unsigned M0 = 0x27u, M1 = 0x33u, M2 = 0x39u;
                    if (q < npl) {
                        outside[0] |= (ge & M0) == M0; outside[1] |= (ge & M1) == M1; outside[2] |= (ge & M2) == M2;
                        if (gt & M0) mask[0] |= 1u << q;
                        if (gt & M1) mask[1] |= 1u << q;
                        if (gt & M2) mask[2] |= 1u << q;
                    }
                } else {
                    const R l01 = rmin(d[0], d[1]), h01 = rmax(d[0], d[1]);
                    const R lo0 = rmin(l01, rmin(d[2], d[5])), hi0 = rmax(h01, rmax(d[2], d[5]));
                    const R lo1 = rmin(l01, rmin(d[5], d[4])), hi1 = rmax(h01, rmax(d[5], d[4]));
                    const R lo2 = rmin(rmin(d[0], d[3]), rmin(d[4], d[5])), hi2 = rmax(rmax(d[0], d[3]), rmax(d[4], d[5]));
                    if (q < npl) {
                        outside[0] |= lo0 >= -tol; outside[1] |= lo1 >= -tol; outside[2] |= lo2 >= -tol;
                        if (hi0 > tol) mask[0] |= 1u << q;
                        if (hi1 > tol) mask[1] |= 1u << q;
                        if (hi2 > tol) mask[2] |= 1u << q;
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int t = 3 * pr + j;
                const R sg = sh.Tsg[t];
                if (sg != R(0) && !outside[j]) {
                    if (mask[j] == 0) acc_add(acc, sg * sh.Kw[k] * sh.Tv6[t]);
                    else { job[j] = true; code[j] = (unsigned)t | ((unsigned)k << 5) | (mask[j] << 10); }
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const unsigned bm = __ballot_sync(0xffffffffu, job[j]);
            if (job[j]) sh.Q[nq + __popc(bm & lt)] = (unsigned short)code[j];
            nq += __popc(bm);
        }
        used |= __reduce_or_sync(0xffffffffu, (job[0] ? 1u << (code[0] >> 5 & 31) : 0u) |
                                                  (job[1] ? 1u << (code[1] >> 5 & 31) : 0u) |
                                                  (job[2] ? 1u << (code[2] >> 5 & 31) : 0u));
    }
    return nq;
}

// the pairs of the buffered candidates and the clipping of their jobs
template <class R, class Sh, class Wk>
__device__ __forceinline__ void mx_flush(Sh &sh, int nt, int ncand, R tol, R slack, float drop, Acc<R> &acc, Wk &wk)
{
    const int lane = threadIdx.x & 31;
    R kb[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) kb[q] = lane < ncand ? sh.Kb[lane][q] : R(0);
    unsigned used;
    const int nq = mx_pairs(sh, nt, ncand, kb, tol, slack, acc, used, wk);
    if (nq > 0) mx_clip(sh, sh.Q, nq, tol, drop, acc, wk);
    __syncwarp();
}

template <class R> __device__ __forceinline__ R rconv(double v) { return (R)v; }

// over the warp in one instruction (ten for a shuffle tree; pair stage 1 % faster)
__device__ __forceinline__ float warp_min(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// The flux polyhedron of face f (band slot item of a LIST form; points b .. b +
// n - 1 of the face-point arrays) in the frame of the face centre: prisms with
// their boxes, tetrahedra (a lane each) with signs and volumes in shared
// memory (their vertices with KEEP_T), and the box pb of the whole.
// B = float in an FP64 form: prism points and boxes in FP32 too (for the pair
// stage's FP32 tests), the boxes widened over the truncation.
template <class R, bool LIST, bool KEEP_T, class B, class Sh>
__device__ __forceinline__ void mx_poly(const DevMesh &m, const MXArgs &a, Sh &sh, int item, int f, int b, int n, int nt,
                                        B pb[6])
{
    using V = R3<R>;
    constexpr bool F32BOX = !std::is_same<R, B>::value;
    auto box = [](R v) -> B { if constexpr (std::is_same<R, B>::value) return v; else return tf(v); };
    const R4<R> *fpl = static_cast<const R4<R> *>(a.fpl);
    const int lane = threadIdx.x & 31;
    // ---- flux polyhedron tetrahedra in the face frame
    B bx[6] = {B(3e38), B(3e38), B(3e38), B(-3e38), B(-3e38), B(-3e38)};
    if (lane < nt) {
        int pr = lane / 3, j = lane % 3;
        auto disp = [&](int i) -> V {  // i < 0: face centre
            V3 w;
            if (LIST) {
                const R *q = static_cast<const R *>(a.disp) + (size_t)item * DISP_STRIDE + (i < 0 ? 0 : 3 + 3 * i);
                return r3(q[0], q[1], q[2]);
            } else {
                double lam = a.lambda[f];
                if (lam < 0.0) {
                    V3 S = ld3(m.sf, m.nf, f);
                    w = S * (-lam * a.F[f] * a.dt / dot(S, S));
                } else if (i >= 0) {
                    w = ld3(a.Up, m.np, __ldg(m.fpts + b + i)) * (a.dt * lam);
                } else {
                    w = mk(0, 0, 0);
                    for (int q = 0; q < n; ++q) w = w + ld3(a.Up, m.np, __ldg(m.fpts + b + q)) * (a.dt * lam);
                    w = w * (1.0 / n);
                }
            }
            return r3(rconv<R>(w.x), rconv<R>(w.y), rconv<R>(w.z));
        };
        V a0, a1, a2, w0, w1, w2;
        long k0, k1, k2;
        if (n == 3) {
            k0 = __ldg(m.fkey + b); k1 = __ldg(m.fkey + b + 1); k2 = __ldg(m.fkey + b + 2);
            a0 = ld43<R>(fpl, b); a1 = ld43<R>(fpl, b + 1); a2 = ld43<R>(fpl, b + 2);
            w0 = disp(0); w1 = disp(1); w2 = disp(2);
        } else {
            int u = pr + 1 == n ? 0 : pr + 1;
            k0 = -1; k1 = __ldg(m.fkey + b + pr); k2 = __ldg(m.fkey + b + u);
            a0 = r3(R(0), R(0), R(0)); a1 = ld43<R>(fpl, b + pr); a2 = ld43<R>(fpl, b + u);
            w0 = disp(-1); w1 = disp(pr); w2 = disp(u);
        }
        int par = 1;
        if (k1 < k0) { V t = a0; a0 = a1; a1 = t; t = w0; w0 = w1; w1 = t; long q = k0; k0 = k1; k1 = q; par = -par; }
        if (k2 < k1) { V t = a1; a1 = a2; a2 = t; t = w1; w1 = w2; w2 = t; long q = k1; k1 = k2; k2 = q; par = -par; }
        if (k1 < k0) { V t = a0; a0 = a1; a1 = t; t = w0; w0 = w1; w1 = t; long q = k0; k0 = k1; k1 = q; par = -par; }
        V b0 = a0 - w0, b1 = a1 - w1, b2 = a2 - w2;
        RTet<R> T;
        if (j == 0) T = RTet<R>{{a0, a1, a2, b2}};
        else if (j == 1) T = RTet<R>{{a0, a1, b2, b1}};
        else T = RTet<R>{{a0, b0, b1, b2}};
        R v6 = rvol6(T.v[0], T.v[1], T.v[2], T.v[3]);
        R sv = R(-par) * v6;
        if constexpr (KEEP_T) stT(sh.T[lane], T);
        sh.Tsg[lane] = sv > R(0) ? R(1) : (sv < R(0) ? R(-1) : R(0));
        sh.Tv6[lane] = rabs(v6);
        if (j == 0) {
            // (the prism's points are its tetrahedra's: its box is theirs together)
            R *q = reinterpret_cast<R *>(sh.P6[pr]);
            const V pv[6] = {a0, a1, a2, b0, b1, b2};
            B px[6], py[6], pz[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                q[3 * i] = pv[i].x; q[3 * i + 1] = pv[i].y; q[3 * i + 2] = pv[i].z;
                px[i] = box(pv[i].x); py[i] = box(pv[i].y); pz[i] = box(pv[i].z);
            }
            if constexpr (F32BOX) {
                float *qf = reinterpret_cast<float *>(sh.P6f[pr]);
#pragma unroll
                for (int i = 0; i < 6; ++i) { qf[3 * i] = px[i]; qf[3 * i + 1] = py[i]; qf[3 * i + 2] = pz[i]; }
            }
            bx[0] = bx[3] = px[0]; bx[1] = bx[4] = py[0]; bx[2] = bx[5] = pz[0];
#pragma unroll
            for (int i = 1; i < 6; ++i) {
                bx[0] = rmin(bx[0], px[i]); bx[1] = rmin(bx[1], py[i]); bx[2] = rmin(bx[2], pz[i]);
                bx[3] = rmax(bx[3], px[i]); bx[4] = rmax(bx[4], py[i]); bx[5] = rmax(bx[5], pz[i]);
            }
            if constexpr (F32BOX) {
                B w = B(0);
#pragma unroll
                for (int i = 0; i < 6; ++i) w = rmax(w, rabs(bx[i]));
                w *= B(2.5e-7);
#pragma unroll
                for (int i = 0; i < 3; ++i) { bx[i] -= w; bx[3 + i] += w; }
            }
            for (int i = 0; i < 6; ++i) sh.Pb[pr][i] = bx[i];
            const B hf = B(0.5);
            sh.Pc[pr][0] = mk4<B>(hf * (bx[0] + bx[3]), hf * (bx[1] + bx[4]), hf * (bx[2] + bx[5]), B(0));
            sh.Pc[pr][1] = mk4<B>(hf * (bx[3] - bx[0]), hf * (bx[4] - bx[1]), hf * (bx[5] - bx[2]), B(0));
        }
    }
    // bounding box of the whole polyhedron
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        if constexpr (std::is_same<B, float>::value) pb[i] = i < 3 ? warp_min(bx[i]) : warp_max(bx[i]);
        else {
            B v = bx[i];
#pragma unroll
            for (int o2 = 16; o2 > 0; o2 >>= 1) {
                B w = __shfl_xor_sync(0xffffffffu, v, o2);
                v = i < 3 ? rmin(v, w) : rmax(v, w);
            }
            pb[i] = v;
        }
    }
    __syncwarp();
}

// A chunk of 32 stencil cells of face f, a lane each, from entry sc: those that
// reach the polyhedron's box pb and carry phase (void, where comp) go to shared
// memory with their half-space, frame shift and tetrahedron range; ntot gets
// the chunk's tetrahedra, ncell its cells.  decide: the stencil is this one
// chunk, and comp is chosen here by which form leaves fewer cells.
// B = float in an FP64 form: box tests in FP32, wide by its roundings.
template <class R, class B, class Sh>
__device__ __forceinline__ void mx_chunk(const DevMesh &m, const MXArgs &a, Sh &sh, long long sc, long long s1,
                                         const V3 &o, const B pb[6], bool decide, bool &comp, int &ntot, int &ncell)
{
    using V = R3<R>;
    const R4<R> *cbl = static_cast<const R4<R> *>(a.cbl);
    const int lane = threadIdx.x & 31;
    const double eps = m.eps;
    const long long s = sc + lane;
    bool pass = false;
    double al = 0.0, d = 0.0;
    V dc = r3(R(0), R(0), R(0));
    V3 hn = mk(0, 0, 0);
    int t0 = 0, t1 = 0, fl = 0;
    // the face centre in the cell's frame: on a periodic mesh
    // the cell sits next to the face moved by its stencil
    // translation t, and the cell, its tetrahedra and its
    // plane are taken relative to o - t
    V3 oc = o;
    bool emp = false, ful = false;
    if (s < s1) {
        // everything about the cell in one round trip (its plane is read for
        // nothing where the cell is dropped)
        const int c = __ldg(m.scell + s);
        al = a.alpha[c];
        const V3 cc = ld3(m.cc, m.nc, c);
        const R4<R> cb0 = ldg4(cbl, 2 * (long)c), cb1 = ldg4(cbl, 2 * (long)c + 1);
        t0 = __ldg(a.ctptr + c);
        t1 = __ldg(a.ctptr + c + 1);
        fl = a.flags[c];
        hn = mk(a.n[c], a.n[m.nc + c], a.n[2 * m.nc + c]);
        d = a.d[c];
        if (m.scode) oc = o - tshift(m, __ldg(m.scode + s));
        // an empty cell carries no phase, a full cell no void
        // thresholds on the integer pipe (bit-pattern order of doubles)
        emp = le_pos(al, eps);
        ful = ge_pos(al, 1.0 - eps);
        if (decide || !(comp ? ful : emp)) {
            dc = r3(rconv<R>(cc.x - oc.x), rconv<R>(cc.y - oc.y), rconv<R>(cc.z - oc.z));
            if constexpr (std::is_same<R, B>::value)
                pass = !(rgt(pb[0], cb1.x + dc.x) || rgt(cb0.x + dc.x, pb[3]) || rgt(pb[1], cb1.y + dc.y) ||
                         rgt(cb0.y + dc.y, pb[4]) || rgt(pb[2], cb1.z + dc.z) || rgt(cb0.z + dc.z, pb[5]));
            else {
                auto apart = [](float l, float h, double c0, double c1, double s) {
                    const float d = tf(s), f0 = tf(c0), f1 = tf(c1);
                    const float w = 5e-7f * (fabsf(d) + fabsf(f0) + fabsf(f1));
                    return l > f1 + d + w || f0 + d - w > h;
                };
                pass = !(apart(pb[0], pb[3], cb0.x, cb1.x, dc.x) || apart(pb[1], pb[4], cb0.y, cb1.y, dc.y) ||
                         apart(pb[2], pb[5], cb0.z, cb1.z, dc.z));
            }
        }
    }
    if (decide) {  // the whole stencil is this chunk
        const int nful = __popc(__ballot_sync(0xffffffffu, pass && ful));
        const int nemp = __popc(__ballot_sync(0xffffffffu, pass && emp));
        if (nful != nemp) comp = nful > nemp;
    }
    pass = pass && !(comp ? ful : emp);
    const int nkt = pass ? t1 - t0 : 0;
    R wgt = R(1);
    bool useH = false;
    R4<R> H = mk4<R>(R(0), R(0), R(0), R(0));
    if (pass && !emp && !ful) {
        if (fl & VOF_ORIENTED) {
            const double hd = d - dot(hn, oc);
            // phase side n.x <= d; the void side is -n.x <= -d
            R sg = comp ? R(-1) : R(1);
            H = mk4<R>(sg * rconv<R>(hn.x), sg * rconv<R>(hn.y), sg * rconv<R>(hn.z),
                       sg * rconv<R>(hd));
            useH = true;
        } else wgt = comp ? rconv<R>(1.0 - al) : rconv<R>(al);
    }
    int inc = nkt;
#pragma unroll
    for (int o2 = 1; o2 < 32; o2 <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o2);
        if (lane >= o2) inc += v;
    }
    const unsigned pm = __ballot_sync(0xffffffffu, pass);
    if (pass) {
        const int r = __popc(pm & ((1u << lane) - 1u));
        sh.CH[r] = H;
        sh.Cd[r] = mk4<R>(dc.x, dc.y, dc.z, int_bits<R>(t0 - (inc - nkt)));
        sh.Cw[r] = wgt;
        sh.CuseH[r] = useH;
        sh.Cend[r] = inc;
    }
    ntot = __shfl_sync(0xffffffffu, inc, 31);
    ncell = __popc(pm);
    __syncwarp();
}

// lane sums (and their compensations) merged across the warp
template <class R>
__device__ __forceinline__ void mx_merge(Acc<R> &acc)
{
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
        const R xs = __shfl_xor_sync(0xffffffffu, acc.s, o2), xc = __shfl_xor_sync(0xffffffffu, acc.c, o2);
        acc_add(acc, xs);
        acc.c += xc;
    }
}

template <class R, int MX_STACK, class Wk>
__device__ __forceinline__ void phase_flux_body(const DevMesh &m, const MXArgs &a, MXShared<R, MX_STACK> &sh)
{
    using V = R3<R>;
    const R4<R> *fpl = static_cast<const R4<R> *>(a.fpl);
    const R4<R> *ktl = static_cast<const R4<R> *>(a.ktl);
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const double eps = m.eps;
    Wk wk;
    for (int f = warp; f < m.nf; f += nwarps) {
        const long long s0 = __ldg(m.sptr + f), s1 = __ldg(m.sptr + f + 1);
        {
            double Ff = a.F[f];
            bool all_e = true, all_f = true;
            for (long long s = s0 + lane; s < s1; s += 32) {
                double al = a.alpha[__ldg(m.scell + s)];
                all_e &= al <= eps;
                all_f &= al >= 1.0 - eps;
            }
            all_e = __all_sync(0xffffffffu, all_e);
            all_f = __all_sync(0xffffffffu, all_f);
            double triv = 0.0;
            bool done = true;
            // (inflow through a boundary face brings nothing; a periodic face's
            // copy carries no flux)
            if (Ff == 0.0 || (f >= m.ni && (Ff < 0.0 || (m.fimg && m.fimg[f - m.ni] >= 0))) || all_e) triv = 0.0;
            else if (all_f) triv = Ff * a.dt;
            else done = false;
            if (done) {
                if (lane == 0) a.Va[f] = triv;
                continue;
            }
        }
        const V3 o = ld3(m.cf, m.nf, f);
        const int b = __ldg(m.fptr + f), n = __ldg(m.fptr + f + 1) - b;
        bool decide, comp;
        pf_form(m, a.F, a.alpha, f, a.lambda[f], s1 - s0, decide, comp);
        const int nt = n == 3 ? 3 : 3 * n;
        // signed distances (to unit-normal planes) within the on-plane band of
        // the face (FP32: 2e-6 of the face size, FP64: 1e-14) are taken as zero:
        // points shared by the polyhedron and the cell tetrahedra come out of
        // different roundings and would otherwise look like cuts
        const R tol = ldg4(fpl, b).w;
        R pb[6];
        mx_poly<R, false, true, R>(m, a, sh, 0, f, b, n, nt, pb);
        Acc<R> acc;
        wk.add(WK_VOL, lane < nt);  // the flux polyhedron's tetrahedra
        wk.face();
        int ncand = 0;
        // The stencil is taken 32 cells at a time, one per lane: the cells that
        // reach the polyhedron's box are kept (with their half-space) in shared
        // memory, then their tetrahedra come 32 at a time into the candidate
        // buffer. A batch that does not fit is produced again after the buffer
        // has been processed, so that the buffer is processed at one place and
        // no candidate is held across it.
        long long sc = s0 - 32;
        int tb = 0, ntot = 0, ncell = 0;
        for (;;) {
            if (tb >= ntot) {  // the chunk's tetrahedra are done: next chunk
                sc += 32;
                tb = 0;
                ntot = 0;
                if (sc < s1) {
                    mx_chunk<R, R>(m, a, sh, sc, s1, o, pb, decide, comp, ntot, ncell);
                    continue;
                }
            }
            const bool fin = sc >= s1;
            bool cand = false;
            int ci = 0;
            R4<R> kp[4];
            R kbx[6];
            if (!fin) {
                // the cell of tetrahedron tb + lane: the cells that end at or
                // before tb, plus one for each cell that ends inside the batch at
                // or before this lane (cell 'lane' ends rel tetrahedra after tb)
                const int rel = lane < ncell ? sh.Cend[lane] - tb : 0x7fffffff;
                const unsigned ends = __reduce_or_sync(0xffffffffu, rel > 0 && rel < 32 ? 1u << rel : 0u);
                ci = __popc(__ballot_sync(0xffffffffu, rel <= 0)) + __popc(ends & (((1u << lane) << 1) - 1u));
            }
            if (!fin && tb + lane < ntot) {
                // this lane's tetrahedron: planes and box move from the cell frame
                // to the face frame by the shift dc
                const R4<R> dc = sh.Cd[ci];
                const size_t j = bits_int(dc.w) + tb + lane;
                // box and planes in one round trip to L2 (the planes of the
                // tetrahedra the box test drops are read for nothing)
                const R4<R> b0 = ldg4(ktl, 6 * j + 4), b1 = ldg4(ktl, 6 * j + 5);
#pragma unroll
                for (int i = 0; i < 4; ++i) kp[i] = ldg4(ktl, 6 * j + i);
                kbx[0] = b0.x + dc.x; kbx[1] = b0.y + dc.y; kbx[2] = b0.z + dc.z;
                kbx[3] = b1.x + dc.x; kbx[4] = b1.y + dc.y; kbx[5] = b1.z + dc.z;
                cand = !(rgt(pb[0], kbx[3]) || rgt(kbx[0], pb[3]) || rgt(pb[1], kbx[4]) || rgt(kbx[1], pb[4]) ||
                         rgt(pb[2], kbx[5]) || rgt(kbx[2], pb[5]));
                if (cand) {
                    wk.add(WK_SHIFT, 4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const R4<R> pl = kp[i];
                        kp[i] = mk4<R>(pl.x, pl.y, pl.z, pl.w + (pl.x * dc.x + pl.y * dc.y + pl.z * dc.z));
                    }
                }
            }
            const unsigned cmask = __ballot_sync(0xffffffffu, cand);
            if (fin ? ncand > 0 : ncand + __popc(cmask) > MX_CAND) {
                mx_flush(sh, nt, ncand, tol, box_slack<R>(pb), drop_slack(pb), acc, wk);
                ncand = 0;
                continue;  // the batch again (or the end)
            }
            if (fin) break;
            if (cand) {
                int r = ncand + __popc(cmask & ((1u << lane) - 1u));
                for (int q = 0; q < 4; ++q) sh.Kp[r][q] = kp[q];
                for (int q = 0; q < 6; ++q) sh.Kb[r][q] = kbx[q];
                sh.Kp[r][4] = sh.CH[ci];
                sh.Kw[r] = sh.Cw[ci];
                sh.KuseH[r] = sh.CuseH[ci];
            }
            ncand += __popc(cmask);
            tb += 32;
            __syncwarp();
        }
        mx_merge(acc);  // then the 1/6 of the volumes in FP64
        double va = ((double)acc.s + (double)acc.c) * (1.0 / 6.0);
        if (comp) va = a.F[f] * a.dt - va;
        if (lane == 0) a.Va[f] = va;
        __syncwarp();
    }
    wk.flush(a.work, lane);
}

// every face of the mesh (the standalone call): a warp per face does it all.
// Seven blocks of two warps an SM as the bound in FP32: 128 registers, as eight
// give, in a schedule that is 2 to 7 % faster (64^2 disc 54.1 -> 50.4 us, 64^3
// film 1354 -> 1318); six give 160 and fewer warps (47.9, 1540).
template <class R, int W, class Wk>
__global__ void __launch_bounds__(W * 32, 7) k_phase_flux(DevMesh m, MXArgs a)
{
    extern __shared__ __align__(16) unsigned char pf_smem[];
    phase_flux_body<R, MX_STACK_WIDE, Wk>(m, a, reinterpret_cast<MXShared<R, MX_STACK_WIDE> *>(pf_smem)[threadIdx.x >> 5]);
}


// ================================================ the step's three launches
// The fluxes of a step's band faces: pairs, clips, sums.
//  - pairs (k_pf_pairs): a warp per band face, or per part of one where there
//    are few, builds the flux polyhedron, finds the candidate cell tetrahedra
//    and classifies the (prism, K) pairs; the clip jobs of up to 32 candidates
//    go to the context's queue as one batch with what their clipping reads
//    (planes, prism points), the tetrahedra inside every plane are summed here;
//  - clips (k_pf_clip): a warp per batch works the jobs' pieces off;
//  - sums (k_pf_finish): a lane per unit of work adds its batches, the units of a
//    face make its V_alpha; faces whose batches found no room in the queue go through the pair
//    stage again there, a warp each, which clips every batch at once: the same
//    batches, pieces and sums, so which faces found room changes no bit.
// One launch that did all of it per face kept 16 warps on an SM (128 registers,
// 13.6 KB of shared memory a warp) at 54 % of the issue slots, and took as long
// as its slowest face where there are fewer faces than warps; the stages by
// themselves keep 24, the clip work of a face spreads over several warps, and a
// face's candidates too where the chip would be idle.  The pieces, their order
// and their arithmetic are those of the one-launch form (the sums differ in
// the order of compensated additions).
struct PfQueue {
    const uint4 *rec;             // per band slot: its face's record (BandRec)
    uint4 *arena;                 // batches, in units of 16 bytes
    unsigned cap;                 // units
    unsigned long long *ctr;      // units taken (low word), batches (high word)
    unsigned *boff;               // per batch: first unit, or PF_NONE
    int *bnext;                   // per batch: the unit's next batch, -1
    double *part;                 // per batch: 6 x its volume
    int bcap;
    double *base;                 // per unit of work: 6 x the volume summed by the pair stage
    int2 *head;                   // per unit: first batch (-1 none, PF_FAIL), complement form
    int *ovf, *novf;              // units without room
    int *next_pair, *next_clip, *next_ovf;
    int pair_warps;               // warps of the pair launch
};
constexpr unsigned PF_NONE = 0xffffffffu;
constexpr int PF_FAIL = -2;
constexpr int PF_OVER = 2;        // parts per warp of the launch at most
constexpr int PF_SPLIT = 4;       // a face in up to 2^4 parts

// log2 of the parts a face is dealt into: as many as leave no part waiting for
// a warp (parts repeat the polyhedron's set-up and the stencil pass, 15 % of a
// face's work, so they pay only where warps would be idle)
__device__ __forceinline__ int pf_split(int total, int warps)
{
    int ls = 0;
    while (ls < PF_SPLIT && ((long long)total << (ls + 1)) <= PF_OVER * (long long)warps) ++ls;
    return ls;
}

// layout of a batch in 16-byte units: header (2), prism points, planes (five a
// candidate), weights, job codes
template <class R>
struct PfLayout {
    static constexpr unsigned RW = sizeof(R4<R>) / 16;
    unsigned P, K, W, Q, end;
    __device__ __forceinline__ PfLayout(unsigned nprism, unsigned nk, unsigned nq)
    {
        P = 2;
        K = P + nprism * 5 * RW;
        W = K + nk * 5 * RW;
        Q = W + (nk * (unsigned)sizeof(R) + 15) / 16;
        end = Q + (nq * 2 + 15) / 16;
    }
};

constexpr int PF_RING = 64;       // cell tetrahedra between the box test and their planes
constexpr int PO_LANE = 8;        // open (plane, point) of a pair decided at a time
constexpr int PF_FLUSH = 24;      // candidates from which the pairs are taken (at most MX_CAND)
template <class R>
struct __align__(16) PairShared : PolyShared<R>, CellShared<R>, CandShared<R> {
    R Kb[MX_CAND][6];
    R4<R> X[4];                   // the polyhedron's box: low (w: slack), high (w: tol), centre, half extents
    double o[3];                  // face centre
    int Cj[PF_RING];              // cell tetrahedron
    unsigned char Cc[PF_RING];    // its cell in the chunk
    unsigned char Kmap[MX_CAND];
};

// The FP64 form classifies in FP32 wherever that is clear of its roundings and
// in FP64 only the planes that are not (the FP64 pipe issues one warp
// instruction in about 64 cycles on its sub-partition): boxes, prism points and
// shifted planes are held in FP32 as well, with each candidate's rounding
// allowance; the FP64 planes stay in the cell's frame until then.  Every
// decision is the one FP64 throughout takes.
template <>
struct __align__(16) PairShared<double> : PolyShared<double, float>, CellShared<double> {
    float4 P6f[VOF_MAXFP][5];
    D4 Kp[MX_CAND][5];            // planes (in the cell frame until the pairs are taken) and the half-space
    double Kdc[MX_CAND][3];       // cell centre - face centre
    double Kw[MX_CAND];
    float4 Kf[MX_CAND][5];        // planes and half-space in the face frame, FP32
    float Kb[MX_CAND][6];
    float Km[MX_CAND];            // rounding allowance of the FP32 distances
    float4 X[4];
    double o[3];
    int Cj[PF_RING];
    unsigned short Q[MX_QUEUE], PQ[VOF_MAXFP * MX_CAND];
    unsigned short O[32 * PO_LANE];  // open (plane, point) of the pairs at hand: 6 plane + point | pair << 5
    unsigned Oin[32], Oout[32];   // (plane, point) bits of the pairs at hand
    unsigned char Cc[PF_RING];
    unsigned char KuseH[MX_CAND], Kmap[MX_CAND];
};

// all (T, K) pairs of the candidates, as mx_pairs
template <class Wk>
__device__ __forceinline__ int pf_pairs64(PairShared<double> &sh, int nt, int ncand, double tol, Acc<double> &acc,
                                          unsigned &used, Wk &wk)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int nprism = nt / 3;
    int total = 0;
    {
        const bool live0 = lane < ncand;
        float4 pl[5];
        float kb[6], mg = 0.0f;
        if (live0) {
            mg = sh.Km[lane];
#pragma unroll
            for (int q = 0; q < 5; ++q) pl[q] = sh.Kf[lane][q];
#pragma unroll
            for (int q = 0; q < 6; ++q) kb[q] = sh.Kb[lane][q];
        }
        for (int pr = 0; pr < nprism; ++pr) {
            const float *tb = sh.Pb[pr];
            const bool live = sh.Tsg[3 * pr] != 0.0 || sh.Tsg[3 * pr + 1] != 0.0 || sh.Tsg[3 * pr + 2] != 0.0;
            bool ov = live0 && live;
            if (ov) {
                ov = !(kb[0] > tb[3] + mg || tb[0] > kb[3] + mg || kb[1] > tb[4] + mg || tb[1] > kb[4] + mg ||
                       kb[2] > tb[5] + mg || tb[2] > kb[5] + mg);
                const float4 ce = sh.Pc[pr][0], he = sh.Pc[pr][1];
#pragma unroll
                for (int q = 0; q < 5; ++q) ov = ov && !beyond<float>(pl[q], ce, he, mg);
            }
            const unsigned bm = __ballot_sync(0xffffffffu, ov);
            if (ov) sh.PQ[total + __popc(bm & lt)] = (unsigned short)(pr | lane << 3);
            total += __popc(bm);
        }
    }
    __syncwarp();
    // The planes into the face frame, in FP64 (12 instructions of its pipe).
    if (lane < ncand) {
        const double *dc = sh.Kdc[lane];
        wk.add(WK_SHIFT, 4);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            D4 &pl = sh.Kp[lane][q];
            pl.w = pl.w + (pl.x * dc[0] + pl.y * dc[1] + pl.z * dc[2]);
        }
    }
    __syncwarp();
    // A pair a lane: FP32 distances of the prism's six points to the planes give
    // for each (plane, point) clearly inside (bit 6 q + i of in), clearly outside
    // (out) or open; of the open ones those that can change what becomes of one
    // of the prism's tetrahedra are listed, dense over the warp, and decided in
    // FP64, a (plane, point) a lane.  (A tetrahedron's open planes decided by
    // its own lane, four points at a time, took ten times the FP64 instructions:
    // the planes shared by a face's cells and polyhedron are open everywhere,
    // most others nowhere; pairs of 64^3 hexahedra 402 -> 370 us, and 317
    // with the loops over the planes rolled: the launch waited for instructions;
    // 281 since.)
    constexpr unsigned M[3] = {0x27u, 0x33u, 0x39u};  // T0 = a0 a1 a2 b2, T1 = a0 a1 b2 b1, T2 = a0 b0 b1 b2
    int nq = 0;
    used = 0u;
    for (int pb = 0; pb < total; pb += 32) {
        const int pi = pb + lane;
        unsigned in = 0u, out = 0u, open = 0u, live = 0u, pc = 0u;
        int npl = 0;
        if (pi < total) {
            pc = sh.PQ[pi];
            const int pr = pc & 7, k = pc >> 3;
            float v[20];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const float4 x = sh.P6f[pr][i];
                v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
            }
            npl = sh.KuseH[k] ? 5 : 4;
            const float mg = sh.Km[k];
#pragma unroll
            for (int j = 0; j < 3; ++j) live |= (unsigned)(sh.Tsg[3 * pr + j] != 0.0) << j;
#pragma unroll 1
            for (int q = 0; q < npl; ++q) {
                const float4 pl = sh.Kf[k][q];
                unsigned lo = 0u, hi = 0u;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    const float d = fmaf(pl.x, v[3 * i], fmaf(pl.y, v[3 * i + 1], fmaf(pl.z, v[3 * i + 2], -pl.w)));
                    lo |= (unsigned)(d < -mg) << i;
                    hi |= (unsigned)(d > mg) << i;
                }
                in |= lo << 6 * q;
                out |= hi << 6 * q;
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if ((hi & M[j]) == M[j]) live &= ~(1u << j);
            }
#pragma unroll 1
            for (int q = 0; q < npl; ++q) {
                const unsigned lo = in >> 6 * q & 63u, hi = out >> 6 * q & 63u;
                unsigned need = 0u;
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if ((live >> j & 1u) && (!(lo & M[j]) || !(hi & M[j]))) need |= M[j];
                open |= (need & ~(lo | hi)) << 6 * q;
            }
        }
        while (__any_sync(0xffffffffu, open != 0u)) {
            // up to PO_LANE of each lane's
            const int c = min(__popc(open), PO_LANE);
            int at = c;
#pragma unroll
            for (int o2 = 1; o2 < 32; o2 <<= 1) {
                const int w = __shfl_up_sync(0xffffffffu, at, o2);
                if (lane >= o2) at += w;
            }
            const int n = __shfl_sync(0xffffffffu, at, 31);
            at -= c;
            for (int i = 0; i < c; ++i) {
                sh.O[at + i] = (unsigned short)((__ffs(open) - 1) | lane << 5);
                open &= open - 1;
            }
            sh.Oin[lane] = in;
            sh.Oout[lane] = out;
            __syncwarp();
            for (int i = lane; i < n; i += 32) {
                const unsigned w = sh.O[i], bit = w & 31, l = w >> 5, pk = sh.PQ[pb + l], q = bit / 6, x = bit % 6;
                const D4 pl = sh.Kp[pk >> 3][q];
                const double *p = reinterpret_cast<const double *>(sh.P6[pk & 7]) + 3 * x;
                wk.add(WK_TEST, !(i & 3));  // (four distances make a test)
                const double d = fma(pl.x, p[0], fma(pl.y, p[1], fma(pl.z, p[2], -pl.w)));
                if (rbelow(d, tol)) atomicOr(&sh.Oin[l], 1u << bit);
                if (rabove(d, tol)) atomicOr(&sh.Oout[l], 1u << bit);
            }
            __syncwarp();
            in = sh.Oin[lane];
            out = sh.Oout[lane];
        }
        // outside (no point inside some plane), inside every plane (summed) or a
        // clip job
        const int pr = pc & 7, k = pc >> 3;
#pragma unroll 1
        for (int j = 0; j < 3; ++j) {
            const unsigned mj = 0x393327u >> 8 * j & 63u;
            unsigned mask = 0u;
            bool outside = !(live >> j & 1u);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                if (q < npl) {
                    if (!(in >> 6 * q & mj)) outside = true;
                    if (out >> 6 * q & mj) mask |= 1u << q;
                }
            }
            const int t = 3 * pr + j;
            if (!outside && mask == 0u) acc_add(acc, sh.Tsg[t] * sh.Kw[k] * sh.Tv6[t]);
            const bool job = !outside && mask != 0u;
            const unsigned bm = __ballot_sync(0xffffffffu, job);
            if (job) sh.Q[nq + __popc(bm & lt)] = (unsigned short)((unsigned)t | (unsigned)k << 5 | mask << 10);
            nq += __popc(bm);
            used |= __reduce_or_sync(0xffffffffu, job ? 1u << k : 0u);
        }
    }
    return nq;
}

// a sum and its compensation in 8 bytes: in FP32 side by side, added in FP64
// where they are read (a thread per face there, one lane of 32 here)
__device__ __forceinline__ void put_sum(double *a, int i, const Acc<float> &v)
{
    reinterpret_cast<float2 *>(a)[i] = make_float2(v.s, v.c);
}
__device__ __forceinline__ void put_sum(double *a, int i, const Acc<double> &v) { a[i] = v.s + v.c; }
template <class R> __device__ __forceinline__ double get_sum(const double *a, int i)
{
    if constexpr (std::is_same<R, float>::value) {
        const float2 v = reinterpret_cast<const float2 *>(a)[i];
        return (double)v.x + (double)v.y;
    } else return a[i];
}

// a band face's record, a quarter in each of the first four lanes
struct PfFace {
    int f, b, n, nt;
    long long s0, s1;
    bool decide, comp;
};
// (what only some stages need waits in shared memory, not in registers; lane 0
// of the record holds ox and oy, lane 1 oz)
template <class R>
__device__ __forceinline__ PfFace pf_face(const uint4 &rec, PairShared<R> &sh)
{
    const int lane = threadIdx.x & 31;
    auto word = [&](unsigned v, int l) { return __shfl_sync(0xffffffffu, v, l); };
    if (lane < 2) {
        sh.o[2 * lane] = __hiloint2double((int)rec.y, (int)rec.x);
        if (lane == 0) sh.o[1] = __hiloint2double((int)rec.w, (int)rec.z);
    }
    PfFace p;
    p.s0 = (long long)((unsigned long long)word(rec.w, 1) << 32 | word(rec.z, 1));
    p.f = (int)word(rec.x, 2);
    p.b = (int)word(rec.y, 2);
    p.n = (int)word(rec.z, 2);
    p.s1 = p.s0 + (int)word(rec.w, 2);
    const unsigned form = word(rec.x, 3);
    p.decide = form & 2u;
    p.comp = form & 1u;
    p.nt = p.n == 3 ? 3 : 3 * p.n;
    return p;
}

// its flux polyhedron, and the box's numbers
template <class R>
__device__ __forceinline__ void pf_poly(const DevMesh &m, const MXArgs &a, PairShared<R> &sh, int item, const PfFace &p)
{
    using B = float;
    const R tol = ldg4(static_cast<const R4<R> *>(a.fpl), p.b).w;
    B pb[6];
    mx_poly<R, true, false, B>(m, a, sh, item, p.f, p.b, p.n, p.nt, pb);
    if ((threadIdx.x & 31) == 0) {
        const B hf = B(0.5);
        sh.X[0] = mk4<B>(pb[0], pb[1], pb[2], box_slack<B>(pb));
        sh.X[1] = mk4<B>(pb[3], pb[4], pb[5], (B)tol);
        sh.X[2] = mk4<B>(hf * (pb[0] + pb[3]), hf * (pb[1] + pb[4]), hf * (pb[2] + pb[5]), B(0));
        sh.X[3] = mk4<B>(hf * (pb[3] - pb[0]), hf * (pb[4] - pb[1]), hf * (pb[5] - pb[2]), B(0));
    }
}
template <class R>
__device__ __forceinline__ float pf_drop(const PairShared<R> &sh)
{
    const float4 lo = sh.X[0], hi = sh.X[1];
    const float box[6] = {lo.x, lo.y, lo.z, hi.x, hi.y, hi.z};
    return drop_slack(box);
}

// The pairs of part 'part' of 2^ls of a face: volumes inside every plane go to
// acc, and sink(nq, used, tol) gets the clip jobs of up to 32 candidates at a time
// (sh.Q, nq of them; used: the candidates that have any; sh.Kp, sh.Kw).
template <class R, class Wk, class Sink>
__device__ __forceinline__ void pf_stencil(const DevMesh &m, const MXArgs &a, PairShared<R> &sh, const PfFace &p, int part,
                                           int ls, bool &comp, Acc<R> &acc, Wk &wk, Sink sink)
{
    constexpr bool F64 = std::is_same<R, double>::value;
    using B = float;  // boxes
    const R4<R> *fpl = static_cast<const R4<R> *>(a.fpl);
    const R4<R> *ktl = static_cast<const R4<R> *>(a.ktl);
    const int lane = threadIdx.x & 31, msk = (1 << ls) - 1;
    const unsigned lt = (1u << lane) - 1u;
    const long long s0 = p.s0, s1 = p.s1;
    const int b = p.b, nt = p.nt;
    const bool decide = p.decide;
    // The stencil is taken 32 cells at a time, one per lane, then the
    // tetrahedra of those that reach the polyhedron, 32 at a time (a part
    // takes every 2^ls-th such batch): those whose boxes reach it go to a
    // ring; from the ring, 32 lanes wide, a tetrahedron gets its planes, is
    // dropped where the polyhedron's box lies beyond one, and else becomes a
    // candidate; from PF_FLUSH candidates on the pairs are classified.
    long long sc = s0 - 32;
    int tb = 0, ntot = 0, ncell = 0, bt = 0;
    int base = 0, cnt = 0, nk = 0;  // ring: first entry, entries; candidates
    for (;;) {
        const bool cdone = tb >= ntot;
        if (cnt >= 32 || (cdone && cnt > 0)) {
            // ---- planes of the ring's first tetrahedra
            const int nr = min(cnt, MX_CAND - nk);
            bool keep = false;
            R4<R> kp[4], H;
            B kbx[6];
            float4 kf[4], hf4;
            float mg = 0.0f;
            int ci = 0;
            if (lane < nr) {
                const int e = (base + lane) & (PF_RING - 1);
                ci = sh.Cc[e];
                const size_t j = sh.Cj[e];
                const R4<R> dc = sh.Cd[ci];
                const R3<float> df = r3(tof(dc.x), tof(dc.y), tof(dc.z));
                H = sh.CH[ci];
                const bool useH = sh.CuseH[ci];
                const R4<R> b0 = ldg4(ktl, 6 * j + 4), b1 = ldg4(ktl, 6 * j + 5);
#pragma unroll
                for (int i = 0; i < 4; ++i) kp[i] = ldg4(ktl, 6 * j + i);
                kbx[0] = tof(b0.x) + df.x; kbx[1] = tof(b0.y) + df.y; kbx[2] = tof(b0.z) + df.z;
                kbx[3] = tof(b1.x) + df.x; kbx[4] = tof(b1.y) + df.y; kbx[5] = tof(b1.z) + df.z;
                const float4 pce = sh.X[2], phe = sh.X[3];
                keep = true;
                if constexpr (F64) {
                    // allowance: a few FP32 roundings of what enters a distance
                    const float rs = sh.X[0].w * 2e6f + fmaxf(fabsf(df.x), fmaxf(fabsf(df.y), fabsf(df.z))) +
                                     fmaxf(fabsf(tof(kp[3].w)), fabsf(tof(H.w)));
                    mg = 2e-6f * rs;
                } else mg = sh.X[0].w;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const R4<R> pl = kp[i];
                    if constexpr (F64) {
                        kf[i] = make_float4(tof(pl.x), tof(pl.y), tof(pl.z), 0.0f);
                        kf[i].w = tof(pl.w) + (kf[i].x * df.x + kf[i].y * df.y + kf[i].z * df.z);
                        keep = keep && !beyond<float>(kf[i], pce, phe, mg);
                    } else {
                        wk.add(WK_SHIFT, 1);
                        kp[i] = mk4<R>(pl.x, pl.y, pl.z, pl.w + (pl.x * dc.x + pl.y * dc.y + pl.z * dc.z));
                        keep = keep && !beyond<R>(kp[i], pce, phe, mg);
                    }
                }
                hf4 = make_float4(tof(H.x), tof(H.y), tof(H.z), tof(H.w));
                keep = keep && !(useH && beyond<float>(hf4, pce, phe, mg));
                if (!useH) hf4 = make_float4(0.0f, 0.0f, 0.0f, 1.0f);  // (nothing is beyond it)
            }
            const unsigned km = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int r = nk + __popc(km & lt);
#pragma unroll
                for (int i = 0; i < 4; ++i) sh.Kp[r][i] = kp[i];
                sh.Kp[r][4] = H;
#pragma unroll
                for (int i = 0; i < 6; ++i) sh.Kb[r][i] = kbx[i];
                if constexpr (F64) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) sh.Kf[r][i] = kf[i];
                    sh.Kf[r][4] = hf4;
                    sh.Km[r] = mg;
                    const D4 dc = sh.Cd[ci];
                    sh.Kdc[r][0] = dc.x; sh.Kdc[r][1] = dc.y; sh.Kdc[r][2] = dc.z;
                }
                sh.Kw[r] = sh.Cw[ci];
                sh.KuseH[r] = sh.CuseH[ci];
            }
            nk += __popc(km);
            base = (base + nr) & (PF_RING - 1);
            cnt -= nr;
            __syncwarp();
            if (nk < PF_FLUSH) continue;
        } else if (!cdone) {
            // ---- boxes of the part's next batch of 32 tetrahedra
            // the cell of tetrahedron tb + lane: the cells that end at or
            // before tb, plus one for each cell that ends inside the batch at
            // or before this lane (cell 'lane' ends rel tetrahedra after tb)
            const int rel = lane < ncell ? sh.Cend[lane] - tb : 0x7fffffff;
            const unsigned ends = __reduce_or_sync(0xffffffffu, rel > 0 && rel < 32 ? 1u << rel : 0u);
            const int ci = __popc(__ballot_sync(0xffffffffu, rel <= 0)) + __popc(ends & (((1u << lane) << 1) - 1u));
            bool cand = false;
            int j = 0;
            if (tb + lane < ntot) {
                const R4<R> dc = sh.Cd[ci];
                j = bits_int(dc.w) + tb + lane;
                const R4<R> b0 = ldg4(ktl, 6 * (size_t)j + 4), b1 = ldg4(ktl, 6 * (size_t)j + 5);
                const float4 lo = sh.X[0], hi = sh.X[1];
                if constexpr (F64) {
                    auto apart = [](float l, float h, double c0, double c1, double s) {
                        const float d = tf(s), f0 = tf(c0), f1 = tf(c1);
                        const float w = 5e-7f * (fabsf(d) + fabsf(f0) + fabsf(f1));
                        return l > f1 + d + w || f0 + d - w > h;
                    };
                    cand = !(apart(lo.x, hi.x, b0.x, b1.x, dc.x) || apart(lo.y, hi.y, b0.y, b1.y, dc.y) ||
                             apart(lo.z, hi.z, b0.z, b1.z, dc.z));
                } else
                    cand = !(rgt(lo.x, b1.x + dc.x) || rgt(b0.x + dc.x, hi.x) || rgt(lo.y, b1.y + dc.y) ||
                             rgt(b0.y + dc.y, hi.y) || rgt(lo.z, b1.z + dc.z) || rgt(b0.z + dc.z, hi.z));
            }
            const unsigned cmask = __ballot_sync(0xffffffffu, cand);
            if (cand) {
                const int e = (base + cnt + __popc(cmask & lt)) & (PF_RING - 1);
                sh.Cj[e] = j;
                sh.Cc[e] = (unsigned char)ci;
            }
            cnt += __popc(cmask);
            tb += 32 << ls;
            __syncwarp();
            continue;
        } else {
            // ---- next chunk
            sc += 32;
            bt += (ntot + 31) >> 5;
            tb = ((part - bt) & msk) << 5;
            ntot = 0;
            if (sc < s1) {
                const float4 lo = sh.X[0], hi = sh.X[1];
                const B pb[6] = {lo.x, lo.y, lo.z, hi.x, hi.y, hi.z};
                mx_chunk<R, B>(m, a, sh, sc, s1, mk(sh.o[0], sh.o[1], sh.o[2]), pb, decide, comp, ntot, ncell);
                continue;
            }
        }
        // ---- pairs and clip jobs of the candidates
        if (nk > 0) {
            unsigned used;
            int nq;
            R tol;
            if constexpr (F64) tol = ldg4(fpl, b).w;
            else tol = sh.X[1].w;
            if constexpr (F64) nq = pf_pairs64(sh, nt, nk, tol, acc, used, wk);
            else {
                R kb[6];
#pragma unroll
                for (int i = 0; i < 6; ++i) kb[i] = lane < nk ? sh.Kb[lane][i] : R(0);
                nq = mx_pairs(sh, nt, nk, kb, tol, sh.X[0].w, acc, used, wk);
            }
            if (nq > 0) sink(nq, used, tol);
            nk = 0;
            __syncwarp();
        }
        if (cdone && cnt == 0 && sc >= s1) break;
    }
}

template <class R, class Wk>
__device__ __forceinline__ void pf_pairs_body(const DevMesh &m, const MXArgs &a, const PfQueue &q, PairShared<R> &sh)
{
    constexpr bool F64 = std::is_same<R, double>::value;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int total = *a.count, ls = pf_split(total, q.pair_warps), units = total << ls;
    // the next unit is taken, and its record read (16 bytes by each of four
    // lanes), while the current one is worked on; with few units a warp takes it
    // when it is done, not ahead of a warp that is free (24^3 hexahedra, 1.6
    // units a warp: 42 -> 34 us); in FP64 always, where a unit takes many times
    // as long as the wait and the record's registers spill
    const bool ahead = !F64 && units > 4 * q.pair_warps;
    auto take = [&]() { return lane == 0 ? atomicAdd(q.next_pair, 1) : 0; };
    auto record = [&](int u) {
        return lane < 4 && u < units ? q.rec[4 * (size_t)(u >> ls) + lane] : make_uint4(0u, 0u, 0u, 0u);
    };
    Wk wk;
    int unit = __shfl_sync(0xffffffffu, take(), 0);
    uint4 rec = record(unit);
    while (unit < units) {
        const int item = unit >> ls, part = unit & ((1 << ls) - 1);
        const Wk wk0 = wk;
        const PfFace p = pf_face(rec, sh);
        const int taken = ahead ? take() : 0;
        pf_poly(m, a, sh, item, p);
        int next = __shfl_sync(0xffffffffu, taken, 0);
        if (ahead) rec = record(next);
        __syncwarp();
        Acc<R> acc;
        if (part == 0) {
            wk.add(WK_VOL, lane < p.nt);  // the flux polyhedron's tetrahedra
            wk.face();
        }
        bool comp = p.comp;
        int last = -1;
        pf_stencil(m, a, sh, p, part, ls, comp, acc, wk, [&](int nq, unsigned used, R tol) {
            if (last == PF_FAIL) return;
            const int nt = p.nt, nprism = nt / 3;
            // the jobs, as a batch of the queue (a warp that found no room once
            // takes no more units on: the counter stays near the capacity, far
            // from overflowing its halves)
            const int nu = __popc(used);
            const PfLayout<R> L(nprism, nu, nq);
            unsigned off = PF_NONE;
            int bi = -1;
            if (lane == 0) {
                const unsigned long long old = atomicAdd(q.ctr, (1ull << 32) | L.end);
                off = (unsigned)old;
                bi = (int)(old >> 32);
                if (bi >= q.bcap) bi = -1;
                else if (off > q.cap || L.end > q.cap - off) { q.boff[bi] = PF_NONE; bi = -1; }
                else {
                    q.boff[bi] = off;
                    q.bnext[bi] = -1;
                    if (last < 0) q.head[unit].x = bi;
                    else q.bnext[last] = bi;
                }
            }
            if (used >> lane & 1u) sh.Kmap[__popc(used & lt)] = (unsigned char)lane;
            __syncwarp();  // the map and the job codes are read by other lanes below
            const R sg = lane < nt ? sh.Tsg[lane] : R(0);
            const unsigned pos = __ballot_sync(0xffffffffu, sg > R(0)), neg = __ballot_sync(0xffffffffu, sg < R(0));
            off = __shfl_sync(0xffffffffu, off, 0);
            bi = __shfl_sync(0xffffffffu, bi, 0);
            if (bi < 0 && lane == 0 && last >= 0)  // the unit's batches so far are not clipped
                for (int k = q.head[unit].x; k >= 0; k = q.bnext[k]) q.boff[k] = PF_NONE;
            last = bi < 0 ? PF_FAIL : bi;
            if (bi >= 0) {
                uint4 *ob = q.arena + off;
                if (lane == 0) {
                    ob[0] = make_uint4((unsigned)nq | (unsigned)nu << 16 | (unsigned)nprism << 24, pos, neg, 0u);
                    if constexpr (F64) {
                        const DBits t = dbits(tol);
                        ob[1] = make_uint4(t.lo, (unsigned)t.hi, __float_as_uint(pf_drop(sh)), 0u);
                    } else ob[1] = make_uint4(__float_as_uint(tol), 0u, 0u, 0u);
                }
                const uint4 *ps = reinterpret_cast<const uint4 *>(sh.P6);
                for (unsigned i = lane; i < nprism * 5 * L.RW; i += 32) ob[L.P + i] = ps[i];
                R4<R> *ok = reinterpret_cast<R4<R> *>(ob + L.K);
                for (int i = lane; i < nu * 5; i += 32) {
                    const int k = sh.Kmap[i / 5], c = i % 5;
                    ok[i] = sh.Kp[k][c];
                }
                if (lane < nu) reinterpret_cast<R *>(ob + L.W)[lane] = sh.Kw[sh.Kmap[lane]];
                auto code = [&](int i) -> unsigned {  // candidates renumbered among those used
                    if (i >= nq) return 0u;
                    const unsigned v = sh.Q[i], k = v >> 5 & 31;
                    return (v & ~(31u << 5)) | (unsigned)__popc(used & ((1u << k) - 1u)) << 5;
                };
                unsigned *oq = reinterpret_cast<unsigned *>(ob + L.Q);
                for (int i = lane; 2 * i < nq; i += 32) oq[i] = code(2 * i) | code(2 * i + 1) << 16;
            }
        });
        mx_merge(acc);
        if (last == PF_FAIL) wk = wk0;  // (done, and counted, again)
        if (lane == 0) {
            put_sum(q.base, unit, acc);
            q.head[unit].y = comp;
            if (last < 0) q.head[unit].x = last;
            if (last == PF_FAIL) q.ovf[atomicAdd(q.novf, 1)] = unit;
        }
        __syncwarp();
        if (!ahead) {
            next = __shfl_sync(0xffffffffu, take(), 0);
            rec = record(next);
        }
        unit = next;
        if (last == PF_FAIL) break;
    }
    // no room in the queue any more: the rest is left to the third launch
    for (; unit < units; unit = __shfl_sync(0xffffffffu, take(), 0))
        if (lane == 0) {
            q.head[unit].x = PF_FAIL;
            q.ovf[atomicAdd(q.novf, 1)] = unit;
        }
    next_kernel();
    wk.flush(a.work, lane);
}

template <class R, int MX_STACK_>
struct __align__(16) ClipShared : StackShared<R, MX_STACK_> {
    static constexpr int MX_STACK = MX_STACK_;
    R4<R> Kp[MX_CAND][5];
    R Tsg[MX_MAXT];
    R Kw[MX_CAND];
};

// tetrahedron i of the prisms with points P (20 numbers a prism): T0 = a0 a1 a2 b2,
// T1 = a0 a1 b2 b1, T2 = a0 b0 b1 b2
template <class R>
__device__ __forceinline__ RTet<R> prism_tet(const R *P, int i)
{
    const int j = i % 3;
    const R *p = P + 20 * (i / 3);
    auto at = [&](int k) { return r3(p[k], p[k + 1], p[k + 2]); };
    return RTet<R>{{at(0), at(j == 2 ? 9 : 3), at(j == 0 ? 6 : j == 1 ? 15 : 12), at(j == 1 ? 12 : 15)}};
}

template <class R, int ST, class Wk>
__device__ __forceinline__ void pf_clip_body(const MXArgs &a, const PfQueue &q, ClipShared<R, ST> &sh)
{
    const int lane = threadIdx.x & 31;
    previous_kernel();
    const unsigned long long ctr = *q.ctr;
    const int nb = min((int)(ctr >> 32), q.bcap);
    auto take = [&]() {
        int v = 0;
        if (lane == 0) v = atomicAdd(q.next_clip, 1);
        return __shfl_sync(0xffffffffu, v, 0);
    };
    Wk wk;
    for (int bi = take(); bi < nb; bi = take()) {
        const unsigned off = q.boff[bi];
        if (off == PF_NONE) continue;
        const uint4 *ob = q.arena + off;
        const uint4 h0 = ob[0], h1 = ob[1];
        const int nq = h0.x & 0xffff, nu = h0.x >> 16 & 0xff, nprism = h0.x >> 24;
        const PfLayout<R> L(nprism, nu, nq);
        R tol;
        if constexpr (std::is_same<R, double>::value) tol = __hiloint2double((int)h1.y, (int)h1.x);
        else tol = __uint_as_float(h1.x);
        uint4 *kd = reinterpret_cast<uint4 *>(sh.Kp);
        for (unsigned i = lane; i < nu * 5 * L.RW; i += 32) kd[i] = ob[L.K + i];
        if (lane < nu) sh.Kw[lane] = reinterpret_cast<const R *>(ob + L.W)[lane];
        if (lane < 3 * nprism) {
            stT(sh.T[lane], prism_tet(reinterpret_cast<const R *>(ob + L.P), lane));
            sh.Tsg[lane] = h0.y >> lane & 1u ? R(1) : h0.z >> lane & 1u ? R(-1) : R(0);
        }
        __syncwarp();
        Acc<R> acc;
        mx_clip(sh, reinterpret_cast<const unsigned short *>(ob + L.Q), nq, tol, __uint_as_float(h1.z), acc, wk);
        mx_merge(acc);
        if (lane == 0) put_sum(q.part, bi, acc);
        __syncwarp();
    }
    next_kernel();
    wk.flush(a.work, lane);
}

// V_alpha of a band face from 6 x its volume (rounded step by step: the two
// callers have to agree to the bit)
__device__ __forceinline__ void pf_write(const MXArgs &a, int item, double v6, bool comp)
{
    const int f = a.list[item];
    const double v = __dmul_rn(v6, 1.0 / 6.0);
    a.Va[f] = comp ? fma(a.F[f], a.dt, -v) : v;
}

// The band faces from their parts, in a fixed order: a unit's batches, then what
// its pair stage summed.  A lane a unit (the batches are a chain of reads), the
// units of a face side by side.
template <class R>
__device__ __forceinline__ void pf_sums(const MXArgs &a, const PfQueue &q)
{
    const int total = *a.count, ls = pf_split(total, q.pair_warps), per = 32 >> ls;
    const int lane = threadIdx.x & 31, part = lane & ((1 << ls) - 1);
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int i0 = warp * per; i0 < total; i0 += nw * per) {
        const int item = i0 + (lane >> ls);
        const bool live = item < total;
        int2 h = make_int2(-1, 0);
        double w = 0.0, v = 0.0;
        if (live) {
            const int u = (item << ls) + part;
            h = q.head[u];
            for (int bi = h.x; bi >= 0; bi = q.bnext[bi]) w += get_sum<R>(q.part, bi);
            w += get_sum<R>(q.base, u);
        }
        const unsigned fail = __ballot_sync(0xffffffffu, h.x == PF_FAIL) >> (lane - part) & ((1u << (1 << ls)) - 1u);
        for (int k = 0; k < 1 << ls; ++k) v += __shfl_sync(0xffffffffu, w, lane - part + k);
        if (live && part == 0 && !fail) pf_write(a, item, v, h.y != 0);
    }
}

// The faces without room, a warp each: pairs and clips of a unit in turn, the
// batches as the pair stage forms them and the clips with the clip stage's stack.
template <class R, int ST>
struct __align__(16) RedoShared : PairShared<R>, StackShared<R, ST> {
    static constexpr int MX_STACK = ST;
};
__device__ __forceinline__ double lane_sum(const Acc<float> &v) { return (double)v.s + (double)v.c; }
__device__ __forceinline__ double lane_sum(const Acc<double> &v) { return v.s + v.c; }

template <class R, int ST, class Wk>
__device__ __forceinline__ void pf_redo(const DevMesh &m, const MXArgs &a, const PfQueue &q, RedoShared<R, ST> &sh)
{
    const int lane = threadIdx.x & 31;
    const int ls = pf_split(*a.count, q.pair_warps), n = *q.novf;
    auto take = [&]() {
        int v = 0;
        if (lane == 0) v = atomicAdd(q.next_ovf, 1);
        return __shfl_sync(0xffffffffu, v, 0);
    };
    Wk wk;
    unsigned done = 0;
    for (int i = take(); i < n; i = take()) {
        const int unit = q.ovf[i], item = unit >> ls;
        bool other = false;  // (a face is redone once, for its first part without room)
        for (int u = item << ls; u < unit; ++u) other |= q.head[u].x == PF_FAIL;
        if (other) continue;
        ++done;
        const uint4 rec = lane < 4 ? q.rec[4 * (size_t)item + lane] : make_uint4(0u, 0u, 0u, 0u);
        const PfFace p = pf_face<R>(rec, sh);
        pf_poly<R>(m, a, sh, item, p);
        __syncwarp();
        if (q.head[item << ls].x == PF_FAIL) {  // (else counted by its first part)
            wk.add(WK_VOL, lane < p.nt);
            wk.face();
        }
        double v = 0.0;
        bool comp = p.comp;
        for (int part = 0; part < 1 << ls; ++part) {
            double w = 0.0;
            Acc<R> acc;
            comp = p.comp;
            pf_stencil<R>(m, a, sh, p, part, ls, comp, acc, wk, [&](int nq, unsigned, R tol) {
                if (lane < p.nt) stT(sh.T[lane], prism_tet(reinterpret_cast<const R *>(sh.P6), lane));
                Acc<R> cut;
                mx_clip(sh, sh.Q, nq, tol, pf_drop<R>(sh), cut, wk);
                mx_merge(cut);
                w += lane_sum(cut);
            });
            mx_merge(acc);
            v += w + lane_sum(acc);
        }
        if (lane == 0) pf_write(a, item, v, comp);
        __syncwarp();
    }
    if (std::is_same<Wk, WkOn>::value && lane == 0) work_add1(a.work, WK_NOROOM, done);
    wk.flush(a.work, lane);
}

// warps per block of the pair launch, and blocks per SM: FP32 3 / 4 / 5 / 6
// blocks take 434 / 364 / 380 / 410 us at 128^3 hexahedra (fewer leave the issue
// slots idle, more leave the L1 less room and spill); FP64 is held by its shared
// memory
template <class R> constexpr int pp_warps() { return sizeof(R) == 4 ? 4 : 2; }
template <class R> constexpr int pp_resident() { return sizeof(R) == 4 ? 4 : 6; }
template <class R, class Wk>
__global__ void __launch_bounds__(pp_warps<R>() * 32, pp_resident<R>()) k_pf_pairs(DevMesh m, MXArgs a, PfQueue q)
{
    extern __shared__ __align__(16) unsigned char pf_smem[];
    previous_kernel();
    pf_pairs_body<R, Wk>(m, a, q, reinterpret_cast<PairShared<R> *>(pf_smem)[threadIdx.x >> 5]);
}

template <class R> constexpr int pc_resident(int w, int st)
{
    return sizeof(R) == 8 ? 12 / w : st == MX_STACK_WIDE ? 24 / w : 28 / w;
}
template <class R, int W, int ST, class Wk>
__global__ void __launch_bounds__(W * 32, pc_resident<R>(W, ST)) k_pf_clip(MXArgs a, PfQueue q)
{
    extern __shared__ __align__(16) unsigned char pf_smem[];
    pf_clip_body<R, ST, Wk>(a, q, reinterpret_cast<ClipShared<R, ST> *>(pf_smem)[threadIdx.x >> 5]);
}

constexpr int PF_FINISH_WARPS = 2;
template <class R> constexpr int pf_finish_resident() { return sizeof(R) == 4 ? 7 : 3; }  // by its shared memory
template <class R, int ST, class Wk>
__global__ void __launch_bounds__(32 * PF_FINISH_WARPS, pf_finish_resident<R>()) k_pf_finish(DevMesh m, MXArgs a, PfQueue q)
{
    next_kernel();
    previous_kernel();
    extern __shared__ __align__(16) unsigned char pf_smem[];
    pf_sums<R>(a, q);
    if (*q.novf > 0)
        pf_redo<R, ST, Wk>(m, a, q, reinterpret_cast<RedoShared<R, ST> *>(pf_smem)[threadIdx.x >> 5]);
}

// geometry of every cell relative to its centre (context creation): face
// centres and face points, and the cell's box widened by one rounding of R so
// that the boxes stay conservative
template <class R>
__global__ void k_local_geom(DevMesh m, const int *cfpptr, R4<R> *cfl, R4<R> *cfpl, R4<R> *cbl)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.nc) return;
    V3 cc = ld3(m.cc, m.nc, c);
    int o = cfpptr[c];
    for (int k = m.cptr[c]; k < m.cptr[c + 1]; ++k) {
        int g = m.cface[k] >> 1;
        V3 q = ld3(m.cf, m.nf, g) - cc;
        cfl[k] = mk4<R>((R)q.x, (R)q.y, (R)q.z, R(0));
        for (int j = m.fptr[g]; j < m.fptr[g + 1]; ++j) {
            V3 p = ldP(m, m.fpts[j]) - cc;
            cfpl[o++] = mk4<R>((R)p.x, (R)p.y, (R)p.z, R(0));
        }
    }
    const double *b = m.cbox + 6 * (size_t)c;
    auto lo = [](double v) {
        R f = (R)v;
        return (double)f > v ? rnext(f, R(-3e38)) : f;
    };
    auto hi = [](double v) {
        R f = (R)v;
        return (double)f < v ? rnext(f, R(3e38)) : f;
    };
    cbl[2 * c] = mk4<R>(lo(b[0] - cc.x), lo(b[1] - cc.y), lo(b[2] - cc.z), R(0));
    cbl[2 * c + 1] = mk4<R>(hi(b[3] - cc.x), hi(b[4] - cc.y), hi(b[5] - cc.z), R(0));
}

__device__ __forceinline__ float rrsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rrsqrt(double x) { return rsqrt(x); }

// the tetrahedra of every cell (cell centre + fan triangle of a face, in the
// order of the cell's faces and of the face's points) as 4 outward unit-normal
// planes and a box, in the cell frame (context creation)
template <class R>
__global__ void k_cell_tets(DevMesh m, const int *cfpptr, const R4<R> *cfl, const R4<R> *cfpl, const int *ctptr,
                            R4<R> *ktl)
{
    using V = R3<R>;
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.nc) return;
    int o = cfpptr[c], j = ctptr[c];
    for (int k = m.cptr[c]; k < m.cptr[c + 1]; ++k) {
        const int code = m.cface[k], g = code >> 1, gn = m.fptr[g + 1] - m.fptr[g];
        for (int i = 0; i < (gn == 3 ? 1 : gn); ++i, ++j) {
            V k0 = r3(R(0), R(0), R(0)), k1, k2, k3;
            if (gn == 3) {
                k1 = ld43<R>(cfpl, o); k2 = ld43<R>(cfpl, o + 1); k3 = ld43<R>(cfpl, o + 2);
            } else {
                k1 = ld43<R>(cfl, k); k2 = ld43<R>(cfpl, o + i); k3 = ld43<R>(cfpl, o + (i + 1 == gn ? 0 : i + 1));
            }
            if (code & 1) { V t = k2; k2 = k3; k3 = t; }
            V n0 = rcross(k2 - k0, k1 - k0), n1 = rcross(k1 - k0, k3 - k0);
            V n2 = rcross(k3 - k0, k2 - k0), n3 = rcross(k2 - k1, k3 - k1);
            const R tiny = sizeof(R) == 4 ? R(1e-37) : R(1e-300);
            n0 = n0 * rrsqrt(rdot(n0, n0) + tiny); n1 = n1 * rrsqrt(rdot(n1, n1) + tiny);
            n2 = n2 * rrsqrt(rdot(n2, n2) + tiny); n3 = n3 * rrsqrt(rdot(n3, n3) + tiny);
            R4<R> *q = ktl + 6 * (size_t)j;
            q[0] = mk4<R>(n0.x, n0.y, n0.z, R(0));
            q[1] = mk4<R>(n1.x, n1.y, n1.z, R(0));
            q[2] = mk4<R>(n2.x, n2.y, n2.z, R(0));
            q[3] = mk4<R>(n3.x, n3.y, n3.z, rdot(n3, k1));
            q[4] = mk4<R>(rmin(rmin(k0.x, k1.x), rmin(k2.x, k3.x)), rmin(rmin(k0.y, k1.y), rmin(k2.y, k3.y)),
                          rmin(rmin(k0.z, k1.z), rmin(k2.z, k3.z)), R(0));
            q[5] = mk4<R>(rmax(rmax(k0.x, k1.x), rmax(k2.x, k3.x)), rmax(rmax(k0.y, k1.y), rmax(k2.y, k3.y)),
                          rmax(rmax(k0.z, k1.z), rmax(k2.z, k3.z)), R(0));
        }
        o += gn;
    }
}

// face points relative to the face centre; the w of the face's first point
// holds the on-plane band of the clipping: 2e-6 of the face size in FP32
// (reading R13), 1e-14 of it in FP64
template <class R>
__global__ void k_face_local(DevMesh m, R4<R> *fpl)
{
    int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= m.nf) return;
    V3 c = ld3(m.cf, m.nf, f), S = ld3(m.sf, m.nf, f);
    const double band = sizeof(R) == 4 ? 2e-6 : 1e-14;
    const R tol = (R)(band * sqrt(sqrt(dot(S, S))));
    for (int j = m.fptr[f]; j < m.fptr[f + 1]; ++j) {
        V3 p = ldP(m, m.fpts[j]) - c;
        fpl[j] = mk4<R>((R)p.x, (R)p.y, (R)p.z, j == m.fptr[f] ? tol : R(0));
    }
}

inline int cdiv(long a, long b) { return (int)((a + b - 1) / b); }

template <class R>
int setup_tables(vof_ctx *c, cudaStream_t s)
{
    R4<R> *cfl = static_cast<R4<R> *>(c->cfl), *cfpl = static_cast<R4<R> *>(c->cfpl);
    k_local_geom<R><<<cdiv(c->nc, 256), 256, 0, s>>>(c->m, c->cfpptr, cfl, cfpl, static_cast<R4<R> *>(c->cbl));
    k_face_local<R><<<cdiv(c->nf, 256), 256, 0, s>>>(c->m, static_cast<R4<R> *>(c->fpl));
    k_cell_tets<R><<<cdiv(c->nc, 256), 256, 0, s>>>(c->m, c->cfpptr, cfl, cfpl, c->m.ctptr,
                                                    static_cast<R4<R> *>(c->ktl));
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

}  // namespace

size_t phase_flux_table_entry_bytes(int precision)
{
    return precision == VOF_MIXED ? sizeof(float4) : sizeof(D4);
}

static MXArgs mx_args(vof_ctx *c, const double *alpha, const double *n, const double *d, const uint8_t *flags,
                      const double *Up, const double *F, const double *lambda, double dt, double *Va,
                      const int *list, const int *count, const void *disp, unsigned long long *work)
{
    return MXArgs{alpha, n, d, flags, Up, F, lambda, dt, Va, list, count, disp, c->status, work,
                  c->fpl, c->cbl, c->ktl, c->m.ctptr};
}

// the band slots' work queue and counters (zeroed with the step's counters)
static PfQueue pf_queue(vof_ctx *c, int pair_warps)
{
    int *cnt = c->counters;
    return PfQueue{reinterpret_cast<const uint4 *>(c->pf_rec), static_cast<uint4 *>(c->pf_arena), c->pf_cap, reinterpret_cast<unsigned long long *>(cnt + CNT_PFQ),
                   c->pf_boff, c->pf_bnext, c->pf_part, c->pf_bcap, c->pf_base, c->pf_head, c->pf_ovf, cnt + CNT_PFOVF,
                   cnt + CNT_PFNEXT, cnt + CNT_CLNEXT, cnt + CNT_OVNEXT, pair_warps};
}

// the kernels' shared memory (above the default limit), on the current device
template <class K>
static bool pf_smem(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}
template <class R, int W, class Wk>
static bool pf_smem_form()
{
    bool ok = pf_smem(k_phase_flux<R, W, Wk>, W * sizeof(MXShared<R, MX_STACK_WIDE>)) &&
              pf_smem(k_pf_pairs<R, Wk>, pp_warps<R>() * sizeof(PairShared<R>)) &&
              pf_smem(k_pf_finish<R, MX_STACK_WIDE, Wk>, PF_FINISH_WARPS * sizeof(RedoShared<R, MX_STACK_WIDE>)) &&
              pf_smem(k_pf_clip<R, 1, MX_STACK_WIDE, Wk>, sizeof(ClipShared<R, MX_STACK_WIDE>));
    if constexpr (sizeof(R) == 4)
        ok = ok && pf_smem(k_pf_finish<R, MX_STACK_SLIM, Wk>, PF_FINISH_WARPS * sizeof(RedoShared<R, MX_STACK_SLIM>)) &&
             pf_smem(k_pf_clip<R, 2, MX_STACK_WIDE, Wk>, 2 * sizeof(ClipShared<R, MX_STACK_WIDE>)) &&
             pf_smem(k_pf_clip<R, 3, MX_STACK_WIDE, Wk>, 3 * sizeof(ClipShared<R, MX_STACK_WIDE>)) &&
             pf_smem(k_pf_clip<R, 1, MX_STACK_SLIM, Wk>, sizeof(ClipShared<R, MX_STACK_SLIM>)) &&
             pf_smem(k_pf_clip<R, 2, MX_STACK_SLIM, Wk>, 2 * sizeof(ClipShared<R, MX_STACK_SLIM>)) &&
             pf_smem(k_pf_clip<R, 3, MX_STACK_SLIM, Wk>, 3 * sizeof(ClipShared<R, MX_STACK_SLIM>));
    return ok;
}

template <class R, int W, int ST, class Wk>
static int go_clip(const MXArgs &a, const PfQueue &q, int sms, int mult, cudaStream_t s)
{
    constexpr size_t bytes = W * sizeof(ClipShared<R, ST>);
    return launch_after(k_pf_clip<R, W, ST, Wk>, sms * pc_resident<R>(W, ST) * mult, 32 * W, bytes, s, a, q);
}

template <class R, int ST, class Wk>
static int go_finish(vof_ctx *c, const MXArgs &a, const PfQueue &q, int sms, cudaStream_t s)
{
    constexpr size_t bytes = PF_FINISH_WARPS * sizeof(RedoShared<R, ST>);
    return launch_after(k_pf_finish<R, ST, Wk>, sms * pf_finish_resident<R>(), 32 * PF_FINISH_WARPS, bytes, s, c->m, a, q);
}

template <class R, class Wk>
static int go_list(vof_ctx *c, const MXArgs &a, int sms, cudaStream_t s)
{
    const int pblocks = sms * pp_resident<R>();
    const PfQueue q = pf_queue(c, pblocks * pp_warps<R>());
    constexpr size_t pbytes = pp_warps<R>() * sizeof(PairShared<R>);
    k_pf_pairs<R, Wk><<<pblocks, 32 * pp_warps<R>(), pbytes, s>>>(c->m, a, q);
    // launch configuration of the clips (vof_tune): warps per block, stack
    // depth, and grid = SMs x resident blocks x multiplier
    const int w = c->pf_warps >= 1 && c->pf_warps <= 3 ? c->pf_warps : 2;
    const int mult = c->pf_mult >= 1 ? c->pf_mult : 1;
    int r;
    if constexpr (sizeof(R) == 4) {
        if (c->pf_stack == 1)
            r = w == 1 ? go_clip<R, 1, MX_STACK_SLIM, Wk>(a, q, sms, mult, s)
                       : w == 2 ? go_clip<R, 2, MX_STACK_SLIM, Wk>(a, q, sms, mult, s)
                                : go_clip<R, 3, MX_STACK_SLIM, Wk>(a, q, sms, mult, s);
        else
            r = w == 1 ? go_clip<R, 1, MX_STACK_WIDE, Wk>(a, q, sms, mult, s)
                       : w == 2 ? go_clip<R, 2, MX_STACK_WIDE, Wk>(a, q, sms, mult, s)
                                : go_clip<R, 3, MX_STACK_WIDE, Wk>(a, q, sms, mult, s);
    } else r = go_clip<R, 1, MX_STACK_WIDE, Wk>(a, q, sms, 1, s);
    if (r) return r;
    if constexpr (sizeof(R) == 4)
        r = c->pf_stack == 1 ? go_finish<R, MX_STACK_SLIM, Wk>(c, a, q, sms, s) : go_finish<R, MX_STACK_WIDE, Wk>(c, a, q, sms, s);
    else r = go_finish<R, MX_STACK_WIDE, Wk>(c, a, q, sms, s);
    if (r) return r;
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

template <class R, int W, class Wk>
static int go_all(vof_ctx *c, const MXArgs &a, cudaStream_t s)
{
    constexpr size_t bytes = W * sizeof(MXShared<R, MX_STACK_WIDE>);
    k_phase_flux<R, W, Wk><<<cdiv(c->nf, W), 32 * W, bytes, s>>>(c->m, a);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

int launch_pf_all(vof_ctx *c, const double *alpha, const double *n, const double *d, const uint8_t *flags,
                  const double *Up, const double *F, const double *lambda, double dt, double *Va, cudaStream_t s)
{
    const MXArgs a = mx_args(c, alpha, n, d, flags, Up, F, lambda, dt, Va, nullptr, nullptr, nullptr,
                             c->work_on ? c->work : nullptr);
    if (c->precision == VOF_MIXED) return c->work_on ? go_all<float, 2, WkOn>(c, a, s) : go_all<float, 2, WkOff>(c, a, s);
    return c->work_on ? go_all<double, 1, WkOn>(c, a, s) : go_all<double, 1, WkOff>(c, a, s);
}

int launch_pf_list(vof_ctx *c, const double *alpha, const double *F, double dt, int sms, cudaStream_t s)
{
    const MXArgs a = mx_args(c, alpha, c->n, c->d, c->flags, nullptr, F, nullptr, dt, c->Va, c->band,
                             c->counters + CNT_BAND, c->disp_b, c->work_on ? c->work : nullptr);
    if (c->precision == VOF_MIXED) return c->work_on ? go_list<float, WkOn>(c, a, sms, s) : go_list<float, WkOff>(c, a, sms, s);
    return c->work_on ? go_list<double, WkOn>(c, a, sms, s) : go_list<double, WkOff>(c, a, sms, s);
}

int launch_setup_mixed(vof_ctx *c, cudaStream_t s)
{
    const bool ok = c->precision == VOF_MIXED ? pf_smem_form<float, 2, WkOff>() && pf_smem_form<float, 2, WkOn>()
                                              : pf_smem_form<double, 1, WkOff>() && pf_smem_form<double, 1, WkOn>();
    if (!ok) return VOF_ERR_CUDA;
    return c->precision == VOF_MIXED ? setup_tables<float>(c, s) : setup_tables<double>(c, s);
}
