// Evaluation at targets (Algorithms 1-3, step 2 "Calculation").
//
//  near branch  (|x_last| <= c): reduce to the unit cell (step 2c), gather the
//               4^d stencil of the padded grid with separable cubic Lagrange
//               weights (step 2d), add the singular part back in double
//               precision (step 2e), apply the quasi-periodic phase (step 2f).
//               3D evaluations first classify the targets (a far list sorted
//               by |x3| bucket, a near list), then run the near targets from
//               their list in full warps.
//  far branch   (|x_last| > c, step 2b): the eigen-series (ei)/(he) (and its
//               second derivatives for the Maxwell tensor), truncated to
//               |alpha_n|^2 <= k^2 + (T/|x_last|)^2, one thread per target,
//               the 32 lanes of a warp walking the same index set so that the
//               per-index table of beta_n is read by broadcast; for
//               double-precision plans two kernels, the double and float-float
//               core sums and the float tails, run side by side.
#include <math_constants.h>

#include "gf_internal.cuh"

namespace {

constexpr double TWO_PI = 2.0 * GF_PI;
constexpr double INV_TWO_PI = 1.0 / (2.0 * GF_PI);

// floor of the correctly rounded quotient a/b.  The product a * ib (ib = fl(1/b))
// differs from that quotient by a few ulps, so it decides the floor unless it
// lies within 1e-14 max(1, |a/b|) of an integer, where the quotient is formed.
// q receives the value the floor was taken of.
__device__ __forceinline__ double floor_quot(double a, double b, double ib, double &q)
{
    q = __dmul_rn(a, ib);
    const double fq = floor(q), fr = q - fq;
    const double g = 1e-14 * fmax(1.0, fabs(q));
    if (fr < g || fr > 1.0 - g) {
        q = __ddiv_rn(a, b);
        return floor(q);
    }
    return fq;
}

// x = 2 pi m + t, t in [-pi, pi), with explicit round-to-nearest operations
// (no contraction) so that the cell decision is reproducible: m is the floor of
// the correctly rounded (x + pi)/(2 pi).
__device__ __forceinline__ void reduce_period(double x, double &t, double &m)
{
    double q;
    double mm = floor_quot(__dadd_rn(x, GF_PI), TWO_PI, INV_TWO_PI, q);
    double tt = __dsub_rn(x, __dmul_rn(TWO_PI, mm));
    if (tt >= GF_PI) {
        tt = __dsub_rn(tt, TWO_PI);
        mm += 1.0;
    }
    if (tt < -GF_PI) {
        tt = __dadd_rn(tt, TWO_PI);
        mm -= 1.0;
    }
    t = tt;
    m = mm;
}

// stencil origin on an axis: u = (y - y0)/h, i0 = floor(u) clamped to [0, M-1],
// f = u - i0; the padded nodes i0 .. i0+3 hold the stencil nodes i0-1 .. i0+2.
// i0 is the floor of the correctly rounded quotient (ih = fl(1/h)).
__device__ __forceinline__ int stencil_origin(double y, double y0, double h, double ih, int M, double &f)
{
    double u;
    double i0 = floor_quot(__dsub_rn(y, y0), h, ih, u);
    if (i0 > (double)(M - 1)) i0 = (double)(M - 1);
    if (i0 < 0.0) i0 = 0.0;
    f = u - i0;
    return (int)i0;
}

template <typename T>
__device__ __forceinline__ void lagrange4(T f, T w[4])
{
    const T fm1 = f - (T)1, fm2 = f - (T)2, fp1 = f + (T)1;
    w[0] = -f * fm1 * fm2 * (T)(1.0 / 6.0);
    w[1] = fp1 * fm1 * fm2 * (T)0.5;
    w[2] = -fp1 * f * fm2 * (T)0.5;
    w[3] = fp1 * f * fm1 * (T)(1.0 / 6.0);
}

// quasi-periodic lift e^{i 2 pi <alpha . m>} (fractional part taken first)
__device__ __forceinline__ double2 lattice_phase(double a1, double m1, double a2, double m2)
{
    double ph = a1 * m1 + a2 * m2;
    ph -= rint(ph);
    double s, c;
    sincospi(2.0 * ph, &s, &c);
    return make_double2(c, s);
}

__device__ __forceinline__ void store_out(double2 *o, double2 v) { *o = v; }
__device__ __forceinline__ void store_out(float2 *o, double2 v) { *o = make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ void add_out(double2 *o, double2 v)
{
    atomicAdd(&o->x, v.x);
    atomicAdd(&o->y, v.y);
}
__device__ __forceinline__ void add_out_f(float2 *o, float2 v)
{
    atomicAdd(&o->x, v.x);
    atomicAdd(&o->y, v.y);
}
__device__ __forceinline__ void add_c(double2 *o, double2 v) { add_out(o, v); }
__device__ __forceinline__ void add_c(float2 *o, float2 v) { add_out_f(o, v); }

// A far kernel's share (entries v[0 .. ne-1]) of target idx, from row slab `slab`
// of `nslab` of chunk w.  With one slab per chunk, or no slab scratch, it is
// added into the output at once.  Otherwise each slab stores its partials; the
// chunk's last slab to finish (the one that draws the last ticket; nobody waits)
// adds them up in slab order and deposits the total.  The output, zeroed by the
// near pass, then receives one addend per far kernel (two at most), and a sum of
// two terms onto zero is the same in either order: the result does not depend on
// which slab or kernel finishes first.
template <typename C, int NE>
__device__ __forceinline__ void far_deposit(const EvalArgs &a, int kind, int w, int slab, int nslab, int nslot,
                                            bool valid, int idx, int ne, const C (&v)[NE])
{
    C *o = reinterpret_cast<C *>(a.out) + (size_t)idx * ne;
    C *buf = reinterpret_cast<C *>(a.slabbuf[kind]);
    if (nslab <= 1 || buf == nullptr) {
        if (valid)
#pragma unroll
            for (int e = 0; e < NE; ++e)
                if (e < ne) add_c(o + e, v[e]);
        return;
    }
    const int lane = threadIdx.x & 31;
    const size_t slot = (size_t)w * 32 + lane;
    if (valid)
#pragma unroll
        for (int e = 0; e < NE; ++e)
            if (e < ne) buf[((size_t)slab * nslot + slot) * ne + e] = v[e];
    __threadfence();
    __syncwarp();
    int last = 0;
    if (lane == 0) last = atomicAdd(a.slabtick[kind] + w, 1) == nslab - 1;
    last = __shfl_sync(0xffffffffu, last, 0);
    if (!last || !valid) return;
    __threadfence();
#pragma unroll
    for (int e = 0; e < NE; ++e) {
        if (e >= ne) break;
        C sum = __ldcg(buf + slot * ne + e);
#pragma unroll 4
        for (int s = 1; s < nslab; ++s) sum = cadd(sum, __ldcg(buf + ((size_t)s * nslot + slot) * ne + e));
        add_c(o + e, sum);
    }
}

// Row slabs per chunk of a far launch, capped by the slab scratch (kind 0: the
// main far kernel, 1: the float tails).
__device__ __forceinline__ int far_slabs_capped(const EvalArgs &a, int kind, int nch, int S)
{
    if (a.slabbuf[kind] == nullptr || nch <= 0) return S;
    const int64_t fit = a.slabcap / ((int64_t)nch * 32);
    return (int)(fit < 1 ? 1 : (fit < S ? fit : S));
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename R> __device__ __forceinline__ typename cplx_t<R>::T zero_c();
template <> __device__ __forceinline__ double2 zero_c<double>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 zero_c<float>() { return make_float2(0.f, 0.f); }

template <typename R> __device__ __forceinline__ typename cplx_t<R>::T nan_c();
template <> __device__ __forceinline__ double2 nan_c<double>() { return make_double2(CUDART_NAN, CUDART_NAN); }
template <> __device__ __forceinline__ float2 nan_c<float>() { return make_float2(CUDART_NAN_F, CUDART_NAN_F); }

__device__ __forceinline__ double2 ld_grid(const double2 *p) { return __ldg(p); }
__device__ __forceinline__ double2 ld_grid(const float2 *p)
{
    float2 v = __ldg(p);
    return make_double2(v.x, v.y);
}

// entries written per target
__host__ __device__ __forceinline__ int n_entries(int which) { return gf_out_entries(which); }

// Warp-aggregated append of far targets to the scratch list.
__device__ __forceinline__ void push_far(bool isfar, int i, int *list, int *count)
{
    unsigned mask = __ballot_sync(0xffffffffu, isfar);
    if (mask == 0u) return;
    int lane = threadIdx.x & 31;
    int leader = __ffs(mask) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(count, __popc(mask));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (isfar) list[base + __popc(mask & ((1u << lane) - 1u))] = i;
}

// (in float: a double quotient for every far target was half of the classification's time)
__device__ __forceinline__ int far_bucket(double z, double c)
{
    const int b = (int)((float)(GF_FAR_BUCKETS * c) / (float)z);
    return b < GF_FAR_BUCKETS - 1 ? b : GF_FAR_BUCKETS - 1;
}

// ---------------------------------------------------------------------------
// 3D near kernel.  NF = 1: Helmholtz (field L_d).  NF = 7: Maxwell
// (fields 0..5 = (delta_pq - c^p c^q/k^2) L_d, field 6 = L_d).
// R = storage/accumulation type of the grid (double: GF_FP64, float: split).
//
// What the near branch is made of at one target (finite, |x3| <= c; Algorithm 2,
// calculation step): the stencil and the phase (near_lane), the tensor cubic
// interpolation of the stored grid, the lift (store_near), and within 2 eps of
// a source the singular part (near_sing), added to the stored entries.  The
// far-region grid shares all but the last.
// ---------------------------------------------------------------------------

// One target's stencil: offset of its first node in the grid, position within
// the cell on each axis, e^{i alpha . x} and what the exceptions need.
template <typename R>
struct NearLane {
    int64_t off;     // (i3 P2 + i2) P1 + i1
    R f1, f2, f3;
    R lx, ly;        // e^{i alpha . x} = e^{i alpha . t} e^{i 2 pi <alpha . m>}
    int i3n;         // x3 stencil node (near grid)
    bool neg, sing;  // x3 < 0; within 2 eps of a source (a little more)
};

// Node floor(u) and d = u - 1/2 - floor(u) in [-1/2, 1/2] from v = u - 1/2: the sum
// with 1.5 2^52 rounds v to an integer and leaves it (modulo 2^32) in the low
// word.  Where u is an integer either neighbour may be taken, the interpolant is
// the node's value for both.
__device__ __forceinline__ int node_of(double v, double &d)
{
    const double w = v + 6755399441055744.0;
    d = v - (w - 6755399441055744.0);
    return __double2loint(w);
}

// The same for a float position: v in fixed point.  u = v + 1/2 plus 1.5 2^20 has its integer part (modulo 2^20, a
// multiple of every grid's size) in the upper word and 32 bits of its fraction in the lower one, so an axis
// takes two double operations and an integer conversion (a million targets: list 102 -> 96 us, with the far grid 130 ->
// 122 us).  |v| < 2^19 only; distant targets take the double form.
__device__ __forceinline__ int node_fixed(double v, float &f)
{
    const double w = v + 1572864.5;
    f = (float)(unsigned)__double2loint(w) * 0x1p-32f;
    return __double2hiint(w) & 0xFFFFF;  // node + 2^19
}
__device__ __forceinline__ bool fixed_range(double v) { return (__double2hiint(v) & 0x7fffffff) < 0x411f0000; }

// Five double operations an axis and five for the phase, against 23 and 60: the
// double pipe takes a warp instruction in 16 cycles, and bounds the near kernels of
// both precisions.  The stencil coordinate comes from x itself (the in-plane
// axes are periodic in powers of two: the node is its low bits), the lift from
// alpha . x, both good to a rounding of x.
template <typename R, bool FGRID>
__device__ __forceinline__ NearLane<R> near_lane(const EvalArgs &a, double x1, double x2, double x3, bool mirror)
{
    NearLane<R> L;
    const GatherArgs &g = a.ga;
    double d1, d2, d3;
    int i1, i2, i3;
    const double v1 = fma(x1, FGRID ? g.fih1 : g.ih1, FGRID ? g.fo1 : g.o1), v2 = fma(x2, FGRID ? g.fih1 : g.ih2, FGRID ? g.fo1 : g.o2);
    const double ph0 = fma(x1, g.al1, x2 * g.al2);
    if (sizeof(R) == 4) {
        const double v3 = FGRID ? fma(fabs(x3), g.fihz, g.foz) : fma(mirror ? fabs(x3) : x3, g.ih3, g.o3);
        if (fixed_range(v1) && fixed_range(v2) && fixed_range(v3) && fixed_range(ph0)) {
            float f1, f2, f3;
            i1 = node_fixed(v1, f1) & ((FGRID ? a.fM1 : a.M1) - 1);
            i2 = node_fixed(v2, f2) & ((FGRID ? a.fM2 : a.M2) - 1);
            const int n = node_fixed(v3, f3) - (1 << 19), nc = FGRID ? min(max(n, 1), a.fNZ - 3) : min(max(n, 0), a.M3 - 1);
            f3 += (float)(n - nc);
            L.i3n = nc;
            i3 = FGRID ? nc - 1 : nc - a.Q3lo;
            L.off = FGRID ? ((int64_t)i3 * a.fP2 + i2) * a.fP1 + i1 : ((int64_t)i3 * a.P2 + i2) * a.P1 + i1;
            L.f1 = (R)f1;
            L.f2 = (R)f2;
            L.f3 = (R)f3;
            float s, c;
            sincospif((float)__double2loint(ph0 + 1572864.0) * 0x1p-31f, &s, &c);
            L.lx = (R)c;
            L.ly = (R)s;
            L.neg = x3 < 0.0;
            L.sing = false;
            if (!FGRID) {
                const float t1 = fmaf((float)i1 + f1, g.h1, -(float)GF_PI), t2 = fmaf((float)i2 + f2, g.h2, -(float)GF_PI);
                const float t3 = (float)x3;
                L.sing = t1 * t1 + t2 * t2 + t3 * t3 < g.rs2;
            }
            return L;
        }
    }
    i1 = node_of(v1, d1) & ((FGRID ? a.fM1 : a.M1) - 1);
    i2 = node_of(v2, d2) & ((FGRID ? a.fM2 : a.M2) - 1);
    if (FGRID) {
        // planes are not padded: the stencil planes are i3 .. i3 + 3
        const double v = fma(fabs(x3), g.fihz, g.foz);
        const int n = node_of(v, d3), nc = min(max(n, 1), a.fNZ - 3);
        if (nc != n) d3 = v - (double)nc;
        L.i3n = nc;
        i3 = nc - 1;
    } else {
        // stored planes from Q3lo: a Helmholtz grid (even in x3) holds x3 >= -h3 only
        // and is read at |x3|; so is a Maxwell grid that keeps the odd fields' Nyquist
        // planes (nyqgrid), otherwise it holds the slab |x3| <= c
        const double v = fma(mirror ? fabs(x3) : x3, g.ih3, g.o3);
        const int n = node_of(v, d3), nc = min(max(n, 0), a.M3 - 1);
        if (nc != n) d3 = v - (double)nc;
        L.i3n = nc;
        i3 = nc - a.Q3lo;
    }
    L.off = FGRID ? ((int64_t)i3 * a.fP2 + i2) * a.fP1 + i1 : ((int64_t)i3 * a.P2 + i2) * a.P1 + i1;
    L.f1 = (R)d1 + (R)0.5;
    L.f2 = (R)d2 + (R)0.5;
    L.f3 = (R)d3 + (R)0.5;
    const double ph = ph0 - rint(ph0);
    if (sizeof(R) == 4) {
        float s, c;
        sincospif(2.0f * (float)ph, &s, &c);
        L.lx = (R)c;
        L.ly = (R)s;
    } else {
        double s, c;
        sincospi(2.0 * ph, &s, &c);
        L.lx = (R)c;
        L.ly = (R)s;
    }
    L.neg = x3 < 0.0;
    L.sing = false;
    if (!FGRID) {
        const float t1 = fmaf((float)i1 + (float)L.f1, g.h1, -(float)GF_PI), t2 = fmaf((float)i2 + (float)L.f2, g.h2, -(float)GF_PI);
        const float t3 = (float)x3;
        L.sing = t1 * t1 + t2 * t2 + t3 * t3 < g.rs2;
    }
    return L;
}

// (a b) in float, each part by Kahan's two-product difference: 1.5 roundings of the
// result, as a product in double rounded once, without the double pipe.
__device__ __forceinline__ float2 cmul_kahan(float2 a, float2 b)
{
    const float w = a.y * b.y, v = -a.y * b.x;
    return make_float2(fmaf(a.x, b.x, -w) - fmaf(a.y, b.y, -w), fmaf(a.x, b.y, -v) - fmaf(-a.y, b.x, -v));
}
__device__ __forceinline__ float2 lift_mul(float2 a, float2 b) { return cmul_kahan(a, b); }
__device__ __forceinline__ double2 lift_mul(double2 a, double2 b) { return cmul(a, b); }

// Tensor cubic interpolation by one thread: P1, P2 the grid's padded extents.
template <typename R, int NF>
__device__ __forceinline__ void gather_lane(const void *grid, int P1, int P2, const NearLane<R> &L, const R w1[4], const R w2[4],
                                            const R w3[4], R acc[NF][2])
{
    typedef typename cplx_t<R>::T C;
    const C *G = reinterpret_cast<const C *>(grid) + L.off * NF;
#pragma unroll
    for (int e = 0; e < NF; ++e) acc[e][0] = acc[e][1] = (R)0;
#pragma unroll
    for (int d3 = 0; d3 < 4; ++d3) {
#pragma unroll
        for (int d2 = 0; d2 < 4; ++d2) {
            const C *row = G + ((size_t)d3 * P2 + d2) * P1 * NF;
            const R w23 = w3[d3] * w2[d2];
#pragma unroll
            for (int e = 0; e < NF; ++e) {
                R sr = 0, si = 0;
#pragma unroll
                for (int d1 = 0; d1 < 4; ++d1) {
                    C g = __ldg(row + d1 * NF + e);
                    sr = fma(w1[d1], g.x, sr);
                    si = fma(w1[d1], g.y, si);
                }
                acc[e][0] = fma(w23, sr, acc[e][0]);
                acc[e][1] = fma(w23, si, acc[e][1]);
            }
        }
    }
}

// The stencil of x3 < 0 on a half grid is the mirror of the one read at |x3| (nodes
// a' = i3n - 1 .. i3n + 2 <-> M3 - a').  Even fields: the same values.  Odd
// fields (4: xz, 5: yz): L(M3 - a') = -L(a') + 2 (-1)^(M3/2 + a') P(t), so
// the interpolant is -acc + 2 (-1)^(M3/2) (sum_d w3_d (-1)^(a'_d)) P(t),
// P interpolated bicubically from the Nyquist planes.  The factor of P:
template <typename R>
__device__ __forceinline__ R nyq_factor(const EvalArgs &a, int i3n, const R w3[4])
{
    const R sgn = w3[0] - w3[1] + w3[2] - w3[3];
    return (((i3n - 1) ^ (a.M3 >> 1)) & 1) ? (R)-2 * sgn : (R)2 * sgn;
}

template <typename R>
__device__ __forceinline__ void nyq_lane(const EvalArgs &a, const NearLane<R> &L, const R w1[4], const R w2[4], const R w3[4],
                                         R acc[][2])
{
    typedef typename cplx_t<R>::T C;
    const C *NG = reinterpret_cast<const C *>(a.nyqgrid);
    const int i21 = (int)L.off - (L.i3n - a.Q3lo) * a.P2 * a.P1;
    R pr[2] = {0, 0}, pi[2] = {0, 0};
#pragma unroll
    for (int d2 = 0; d2 < 4; ++d2) {
        const C *row = NG + ((size_t)i21 + (size_t)d2 * a.P1) * 2;
        R s4r = 0, s4i = 0, s5r = 0, s5i = 0;
#pragma unroll
        for (int d1 = 0; d1 < 4; ++d1) {
            const C g4 = __ldg(row + 2 * d1), g5 = __ldg(row + 2 * d1 + 1);
            s4r = fma(w1[d1], g4.x, s4r);
            s4i = fma(w1[d1], g4.y, s4i);
            s5r = fma(w1[d1], g5.x, s5r);
            s5i = fma(w1[d1], g5.y, s5i);
        }
        pr[0] = fma(w2[d2], s4r, pr[0]);
        pi[0] = fma(w2[d2], s4i, pi[0]);
        pr[1] = fma(w2[d2], s5r, pr[1]);
        pi[1] = fma(w2[d2], s5i, pi[1]);
    }
    const R two_s = nyq_factor<R>(a, L.i3n, w3);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        acc[4 + q][0] = fma(two_s, pr[q], -acc[4 + q][0]);
        acc[4 + q][1] = fma(two_s, pi[q], -acc[4 + q][1]);
    }
}

// Entries of target i: lift L (the remainder alone for GF_OUT_LD); the Maxwell xz and yz
// entries of the far-region grid change sign with x3.
template <typename R, int NF, bool FGRID>
__device__ __forceinline__ void store_near(const EvalArgs &a, int64_t i, const NearLane<R> &L, const R acc[NF][2])
{
    typedef typename cplx_t<R>::T C;
    const int ne = n_entries(a.which);
    C *o = reinterpret_cast<C *>(a.out) + i * ne;
    const C lift = cmk(L.lx, L.ly);
    if (NF == 1) {
        const C v = cmk(acc[0][0], acc[0][1]);
        o[0] = a.which == GF_OUT_LD ? v : lift_mul(lift, v);
    } else {
#pragma unroll
        for (int e = 0; e < 7; ++e) {
            C v = lift_mul(lift, cmk(acc[e < NF ? e : 0][0], acc[e < NF ? e : 0][1]));
            if (FGRID && (e == 4 || e == 5) && L.neg) v = cmk(-v.x, -v.y);
            if (e < ne) o[e] = v;
        }
    }
}

// *o += v, rounded once (the caller's own entry).
__device__ __forceinline__ void add_near(double2 *o, double2 v) { *o = cadd(*o, v); }
__device__ __forceinline__ void add_near(float2 *o, double2 v)
{
    const float2 u = *o;
    *o = make_float2((float)((double)u.x + v.x), (float)((double)u.y + v.y));
}

// The singular part at target i, e^{i 2pi<alpha.m>} Phi Y (G = lift L + that, K = L + F, F =
// e^{-i alpha.t} Phi Y) and for Maxwell its derivatives, added to the stored entries.
// Not forced inline: one target in sixteen of a uniform slab comes here.
template <typename R, int NF>
__device__ __noinline__ void near_sing(const EvalArgs &a, int64_t i)
{
    typedef typename cplx_t<R>::T C;
    const int ne = n_entries(a.which);
    C *o = reinterpret_cast<C *>(a.out) + i * ne;
    const double x3 = a.x[3 * i + 2];
    double t1, m1, t2, m2;
    reduce_period(a.x[3 * i], t1, m1);
    reduce_period(a.x[3 * i + 1], t2, m2);
    const double r = sqrt(t1 * t1 + t2 * t2 + x3 * x3);
    if (!(r < 2.0 * a.eps)) return;
    const double2 lat = lattice_phase(a.a1, m1, a.a2, m2);
    // Phi(r) = e^{ikr}/(4 pi r) Y_eps(r) and its r-derivatives (Sec. 3.2, Sec. 4)
    double sk, ck;
    sincos(a.k * r, &sk, &ck);
    const double ir = 1.0 / r;
    const double2 g0 = make_double2(ck * ir * (0.25 / GF_PI), sk * ir * (0.25 / GF_PI));
    const double s = (r - a.eps) / a.eps;
    const double Y0 = 1.0 - smooth8(s);
    const double2 PhiY = cscale(g0, Y0);
    if (NF == 1) {
        add_near(o, cmul(lat, PhiY));
        return;
    }
    const double Y1 = -smooth8_d1(s) / a.eps;
    const double Y2 = -smooth8_d2(s) / (a.eps * a.eps);
    const double2 L1 = make_double2(-ir, a.k);                  // ik - 1/r
    const double2 g1 = cmul(g0, L1);
    double2 L2 = cmul(L1, L1);
    L2.x += ir * ir;
    const double2 g2 = cmul(g0, L2);
    const double2 dPhi = cadd(cscale(g1, Y0), cscale(g0, Y1));
    const double2 d2Phi = cadd(cadd(cscale(g2, Y0), cscale(g1, 2.0 * Y1)), cscale(g0, Y2));
    const double ik2 = 1.0 / (a.k * a.k);
    const double xv[3] = {t1, t2, x3};
    const int PP[6] = {0, 1, 2, 0, 0, 1}, QQ[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const double xp = xv[PP[e]] * ir, xq = xv[QQ[e]] * ir;
        const double dl = PP[e] == QQ[e] ? 1.0 : 0.0;
        // delta_pq Phi + k^-2 [Phi'' xp xq + (Phi'/r)(delta_pq - xp xq)]
        double2 v = cadd(cscale(d2Phi, xp * xq), cscale(dPhi, ir * (dl - xp * xq)));
        v = cscale(v, ik2);
        if (dl != 0.0) v = cadd(v, PhiY);
        add_near(o + e, cmul(lat, v));
    }
    if (a.which == GF_OUT_MAXWELL7) add_near(o + 6, cmul(lat, PhiY));
}

// One target by one thread (evaluations without list scratch).
template <typename R, int NF, bool FGRID>
__device__ __forceinline__ void near_point(const EvalArgs &a, int64_t i, double x1, double x2, double x3)
{
    const NearLane<R> L = near_lane<R, FGRID>(a, x1, x2, x3, NF == 1 || a.nyqgrid != nullptr);
    R w1[4], w2[4], w3[4], acc[NF][2];
    lagrange4<R>(L.f1, w1);
    lagrange4<R>(L.f2, w2);
    lagrange4<R>(L.f3, w3);
    gather_lane<R, NF>(FGRID ? a.fargrid : a.grid, FGRID ? a.fP1 : a.P1, FGRID ? a.fP2 : a.P2, L, w1, w2, w3, acc);
    if (NF > 1 && !FGRID && a.nyqgrid != nullptr && L.neg) nyq_lane<R>(a, L, w1, w2, w3, acc);
    store_near<R, NF, FGRID>(a, i, L, acc);
    if (L.sing && a.which != GF_OUT_LD) near_sing<R, NF>(a, i);
}

// ---------------------------------------------------------------------------
// Listed targets, 32 at a time by one warp.
//
// Read by its own thread, a target's stencil costs 64 NF loads of which every lane
// touches another cache line: the L1 takes 32 cycles for each (14,300 a warp with
// seven fields in float; 0.8 of the kernel's time).  Here the lanes that take one row of a
// stencil are neighbours: one field, four lanes a target (x1 nodes), eight targets a load;
// seven fields, 28 lanes (node, field), one target a load.  The products w3 w2 and
// the weights w1 come from the warp's shared memory, the sums over x1 by
// shuffles, and with seven fields the lanes write a target's entries side by side.
// (Seven fields in double stay with one thread a target: there the double pipe
// is the limit, and 28 lanes of 32 and the shuffled sums would cost more of it.)
// The targets next to a source wait in the warp's queue until a full warp of
// them is there: most warps hold one or two, and would all pay for the singular part.
// 600,000 near targets of a million (cold), one thread a target -> this: Helmholtz 128 x 128 x 64
// float 228 -> 103 us, double 534 -> 349 us (170 of its 250 double operations a target are the
// interpolation); Maxwell 256 x 256 x 64 float 802 -> 320 us; with 400,000 more in a 512 x 512 far grid
// 290 -> 130 us; 64 batched pairs, 3.4 million near targets, 1345 -> 342 us.
// ---------------------------------------------------------------------------
constexpr int NEAR_WARPS = 4;
template <typename R> constexpr int near_ws() { return sizeof(R) == 4 ? 20 : 22; }  // w23 [16], w1 [4] (and bank padding)

struct SingItem {
    int pair, i;
};
template <typename R, int NF>
struct NearWarp {
    R w[sizeof(R) == 8 && NF > 1 ? 1 : 32][near_ws<R>()];
    SingItem q[64];
};

template <typename R>
__device__ __forceinline__ void gather_quads(const void *grid, int P1, int P2, int64_t off, const R (*w)[near_ws<R>()], R acc[1][2])
{
    typedef typename cplx_t<R>::T C;
    const int lane = threadIdx.x & 31, d1 = lane & 3;
    const size_t P12 = (size_t)P1 * P2;
    acc[0][0] = acc[0][1] = (R)0;
#pragma unroll 1
    for (int p = 0; p < 4; ++p) {
        const int src = p * 8 + (lane >> 2);
        const C *g = reinterpret_cast<const C *>(grid) + __shfl_sync(0xffffffffu, off, src) + d1;
        const R *ws = w[src];
        R ax = 0, ay = 0;
#pragma unroll
        for (int d3 = 0; d3 < 4; ++d3)
#pragma unroll
            for (int d2 = 0; d2 < 4; ++d2) {
                const C v = __ldg(g + d3 * P12 + d2 * P1);
                const R w23 = ws[d3 * 4 + d2];
                ax = fma(w23, v.x, ax);
                ay = fma(w23, v.y, ay);
            }
        const R w1 = ws[16 + d1];
        ax *= w1;
        ay *= w1;
        ax += __shfl_xor_sync(0xffffffffu, ax, 1);
        ay += __shfl_xor_sync(0xffffffffu, ay, 1);
        ax += __shfl_xor_sync(0xffffffffu, ax, 2);
        ay += __shfl_xor_sync(0xffffffffu, ay, 2);
        const R rx = __shfl_sync(0xffffffffu, ax, (lane & 7) * 4), ry = __shfl_sync(0xffffffffu, ay, (lane & 7) * 4);
        if ((lane >> 3) == p) {
            acc[0][0] = rx;
            acc[0][1] = ry;
        }
    }
}

// Seven float fields: target after target, entries written by lanes 0 .. 6.
template <bool FGRID>
__device__ __forceinline__ void gather_rows(const EvalArgs &a, int i, int cnt, const NearLane<float> &L, float nyqf,
                                            const float (*w)[near_ws<float>()])
{
    const int lane = threadIdx.x & 31, ne = n_entries(a.which), d1 = lane < 28 ? lane / 7 : 3;
    const int P1 = FGRID ? a.fP1 : a.P1, P2 = FGRID ? a.fP2 : a.P2;
    const size_t s2 = (size_t)P1 * 7, s3 = s2 * P2;
    const float2 *G = reinterpret_cast<const float2 *>(FGRID ? a.fargrid : a.grid) + (lane < 28 ? lane : 27);
    const bool half = !FGRID && a.nyqgrid != nullptr;
    const unsigned negs = __ballot_sync(0xffffffffu, L.neg);
    const int P12 = P1 * P2;
#pragma unroll 1
    for (int t = 0; t < cnt; ++t) {
        const int64_t off = __shfl_sync(0xffffffffu, L.off, t);
        const int it = __shfl_sync(0xffffffffu, i, t);
        const float lx = __shfl_sync(0xffffffffu, L.lx, t), ly = __shfl_sync(0xffffffffu, L.ly, t);
        const float2 *g = G + off * 7;
        const float *ws = w[t];
        float ax = 0.f, ay = 0.f;
#pragma unroll
        for (int d3 = 0; d3 < 4; ++d3)
#pragma unroll
            for (int d2 = 0; d2 < 4; ++d2) {
                const float2 v = __ldg(g + d3 * s3 + d2 * s2);
                const float w23 = ws[d3 * 4 + d2];
                ax = fmaf(w23, v.x, ax);
                ay = fmaf(w23, v.y, ay);
            }
        const float w1 = ws[16 + d1];
        ax *= w1;
        ay *= w1;
        ax += __shfl_down_sync(0xffffffffu, ax, 14);
        ay += __shfl_down_sync(0xffffffffu, ay, 14);
        ax += __shfl_down_sync(0xffffffffu, ax, 7);
        ay += __shfl_down_sync(0xffffffffu, ay, 7);
        const bool neg = (negs >> t) & 1;
        if (half && neg) {
            // the Nyquist planes' stencil: lane = (d2, d1, field), and the sum over the nodes
            const int i21 = (int)off % P12;
            const float nf = __shfl_sync(0xffffffffu, nyqf, t);
            const float *wt = ws + 16;
            const float2 v = __ldg(reinterpret_cast<const float2 *>(a.nyqgrid) +
                                   ((size_t)i21 + (size_t)(lane >> 3) * P1 + ((lane >> 1) & 3)) * 2 + (lane & 1));
            // w2[d2] = sum over d3 of w3[d3] w2[d2] (the w3 sum to 1)
            const int q2 = lane >> 3;
            const float w2 = (ws[q2] + ws[4 + q2]) + (ws[8 + q2] + ws[12 + q2]);
            const float ww = w2 * wt[(lane >> 1) & 3];
            float px = ww * v.x, py = ww * v.y;
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) {
                px += __shfl_xor_sync(0xffffffffu, px, o);
                py += __shfl_xor_sync(0xffffffffu, py, o);
            }
            if (lane == 4 || lane == 5) {
                ax = fmaf(nf, px, -ax);
                ay = fmaf(nf, py, -ay);
            }
        }
        if (lane < ne) {
            float2 v = cmul_kahan(make_float2(lx, ly), make_float2(ax, ay));
            if (FGRID && neg && (lane == 4 || lane == 5)) v = make_float2(-v.x, -v.y);
            reinterpret_cast<float2 *>(a.out)[(size_t)it * ne + lane] = v;
        }
    }
}

// 32 targets (cnt of them valid): lane's target is i.  Returns whether the lane's target
// needs the singular part.
template <typename R, int NF, bool FGRID>
__device__ __forceinline__ bool near_warp(const EvalArgs &a, int i, int cnt, NearWarp<R, NF> &sm)
{
    const int lane = threadIdx.x & 31;
    const bool valid = lane < cnt;
    double x1 = 0.0, x2 = 0.0, x3 = a.c;
    if (valid) {
        x1 = a.x[3 * (int64_t)i];
        x2 = a.x[3 * (int64_t)i + 1];
        x3 = a.x[3 * (int64_t)i + 2];
    }
    const NearLane<R> L = near_lane<R, FGRID>(a, x1, x2, x3, NF == 1 || a.nyqgrid != nullptr);
    R w1[4], w2[4], w3[4];
    lagrange4<R>(L.f1, w1);
    lagrange4<R>(L.f2, w2);
    lagrange4<R>(L.f3, w3);
    R acc[NF][2];
    if (sizeof(R) == 8 && NF > 1) {
        gather_lane<R, NF>(FGRID ? a.fargrid : a.grid, FGRID ? a.fP1 : a.P1, FGRID ? a.fP2 : a.P2, L, w1, w2, w3, acc);
        if (!FGRID && a.nyqgrid != nullptr && L.neg) nyq_lane<R>(a, L, w1, w2, w3, acc);
        if (valid) store_near<R, NF, FGRID>(a, i, L, acc);
        return valid && L.sing;
    }
    R *w = sm.w[sizeof(R) == 8 && NF > 1 ? 0 : lane];
    __syncwarp();
#pragma unroll
    for (int d3 = 0; d3 < 4; ++d3)
#pragma unroll
        for (int d2 = 0; d2 < 4; ++d2) w[d3 * 4 + d2] = w3[d3] * w2[d2];
#pragma unroll
    for (int d1 = 0; d1 < 4; ++d1) w[16 + d1] = w1[d1];
    __syncwarp();
    if (NF == 1) {
        gather_quads<R>(FGRID ? a.fargrid : a.grid, FGRID ? a.fP1 : a.P1, FGRID ? a.fP2 : a.P2, L.off, sm.w, acc);
        if (valid) store_near<R, NF, FGRID>(a, i, L, acc);
    } else if constexpr (sizeof(R) == 4 && NF > 1) {
        gather_rows<FGRID>(a, i, cnt, L, nyq_factor<R>(a, L.i3n, w3), sm.w);
    }
    return valid && L.sing;
}

// A warp's queue of targets next to a source: n entries of q.
template <typename R, int NF>
__device__ __forceinline__ void sing_flush(const EvalArgs *args, NearWarp<R, NF> &sm, int &n)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < n) near_sing<R, NF>(args[sm.q[lane].pair], sm.q[lane].i);
    __syncwarp();
    if (n > 32) {
        if (lane < n - 32) sm.q[lane] = sm.q[32 + lane];
        __syncwarp();
    }
    n = n > 32 ? n - 32 : 0;
}

// Tile t of pair p's lists: the near targets' tiles, then the far-grid ones'.
template <typename R, int NF>
__device__ __forceinline__ void near_list_tile(const EvalArgs *args, int p, int t, int nnear, int nfg, NearWarp<R, NF> &sm, int &nq)
{
    const EvalArgs &a = args[p];
    const int lane = threadIdx.x & 31, tn = (nnear + 31) >> 5;
    if (t >= tn) {
        const int j0 = (t - tn) * 32, cnt = min(nfg - j0, 32);
        near_warp<R, NF, true>(a, a.near_idx[a.n - 1 - (j0 + min(lane, cnt - 1))], cnt, sm);
        return;
    }
    const int j0 = t * 32, cnt = min(nnear - j0, 32);
    const int i = a.near_idx[j0 + min(lane, cnt - 1)];
    const bool sing = near_warp<R, NF, false>(a, i, cnt, sm) && a.which != GF_OUT_LD;
    const unsigned m = __ballot_sync(0xffffffffu, sing);
    if (sing) {
        SingItem &q = sm.q[nq + __popc(m & ((1u << lane) - 1u))];
        q.pair = p;
        q.i = i;
    }
    nq += __popc(m);
    if (nq >= 32) sing_flush<R, NF>(args, sm, nq);
}

// Classify every target (far list, bucket histogram, zeroed far outputs, NaN for
// non-finite ones) and evaluate the near ones (and those of the far-region grid)
// here: evaluations without list scratch.
template <typename R, int NF>
__device__ void near3d_tiles(const EvalArgs &a, int64_t base0, int64_t stride, int *hist)
{
    typedef typename cplx_t<R>::T C;
    C *out = reinterpret_cast<C *>(a.out);
    const int ne = n_entries(a.which);
    for (int64_t base = base0; base < a.n; base += stride) {
        const int64_t i = base + threadIdx.x;
        bool valid = i < a.n;
        double x1 = 0, x2 = 0, x3 = 0;
        if (valid) {
            x1 = a.x[3 * i];
            x2 = a.x[3 * i + 1];
            x3 = a.x[3 * i + 2];
        }
        bool finite = isfinite(x1) && isfinite(x2) && isfinite(x3);
        bool isfar = valid && finite && fabs(x3) > a.c;
        const bool only_L = NF == 1 && a.which == GF_OUT_LD;
        if (only_L && isfar) {
            out[i] = nan_c<R>();  // the remainder alone is served on the near region only
            isfar = false;
            valid = false;
        }
        // far targets inside the far-region grid's slab are gathered, not summed
        const bool fgrid = isfar && a.fargrid != nullptr && fabs(x3) <= a.fzmax;
        if (fgrid) isfar = false;
        push_far(isfar, (int)i, a.far_idx, a.far_count);
        C *o = out + i * ne;
        if (fgrid) {
            near_point<R, NF, true>(a, i, x1, x2, x3);
            continue;
        }
        if (isfar) {
            // the far kernels add their row slabs into these entries
            atomicAdd(&hist[far_bucket(fabs(x3), a.c)], 1);
            for (int e = 0; e < ne; ++e) o[e] = zero_c<R>();
            continue;
        }
        if (!valid) continue;
        if (!finite) {
            for (int e = 0; e < ne; ++e) o[e] = nan_c<R>();
            continue;
        }
        near_point<R, NF, false>(a, i, x1, x2, x3);
    }
}

// Classification alone, 512 targets by a CTA of 256: the near targets go to the start of
// a.near_idx and the far-grid ones, backwards, to its end (near3d_list evaluates them in full
// warps), the far ones to a.far_idx (LISTED) or every target's far bucket there
// (else), with their histogram in shared memory.  The CTA takes its places in a list with one
// atomic: with one per warp the list counters' 60,000 serial updates were most of a million
// targets' 51 us (now 15, with the far bucket's quotient in float and the tests on the bits).
constexpr int CLS_THR = 256, CLS_TILE = 2 * CLS_THR;
struct ClassifySmem {
    int hist[GF_FAR_BUCKETS];
    int cnt[3][CLS_THR / 32], base[3][CLS_THR / 32];
};

__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

template <typename R, int NF, bool LISTED>
__device__ void classify_tile(const EvalArgs &a, int64_t j0, int64_t i1, ClassifySmem &sm)
{
    typedef typename cplx_t<R>::T C;
    C *out = reinterpret_cast<C *>(a.out);
    const int ne = n_entries(a.which), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool only_L = NF == 1 && a.which == GF_OUT_LD;
    double x[2][3];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int64_t i = j0 + u * CLS_THR + threadIdx.x;
#pragma unroll
        for (int d = 0; d < 3; ++d) x[u][d] = i < i1 ? a.x[3 * i + d] : CUDART_NAN;
    }
    bool is[3][2];  // near, far grid, far
    unsigned bal[3][2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int64_t i = j0 + u * CLS_THR + threadIdx.x;
        // tests on the bits (non-negative doubles order like them), off the double pipe
        const bool finite = finite_bits(x[u][0]) && finite_bits(x[u][1]) && finite_bits(x[u][2]);
        const double z = fabs(x[u][2]);
        const long long zb = __double_as_longlong(z);
        const bool beyond = finite && zb > __double_as_longlong(a.c);
        is[0][u] = finite && !beyond;
        // far targets inside the far-region grid's slab are gathered, not summed; the remainder
        // alone is served on the near region only
        is[1][u] = beyond && !only_L && a.fargrid != nullptr && zb <= __double_as_longlong(a.fzmax);
        is[2][u] = beyond && !only_L && !is[1][u];
        if (i < i1) {
            int code = -1;
            if (is[2][u]) {
                // the far kernels add their row slabs into these entries
                code = far_bucket(z, a.c);
                atomicAdd(&sm.hist[code], 1);
                for (int e = 0; e < ne; ++e) out[i * ne + e] = zero_c<R>();
            } else if (!is[0][u] && !is[1][u]) {
                for (int e = 0; e < ne; ++e) out[i * ne + e] = nan_c<R>();
            }
            if (!LISTED) a.far_idx[i] = code;
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) bal[l][u] = __ballot_sync(0xffffffffu, is[l][u]);
    }
    if (lane < 3) {
        const int l = lane;
        sm.cnt[l][warp] = l == 0 ? __popc(bal[0][0]) + __popc(bal[0][1])
                          : l == 1 ? __popc(bal[1][0]) + __popc(bal[1][1])
                                   : __popc(bal[2][0]) + __popc(bal[2][1]);
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int l = threadIdx.x;
        int tot = 0;
        for (int w = 0; w < CLS_THR / 32; ++w) tot += sm.cnt[l][w];
        int b = tot ? atomicAdd(a.far_count + (l == 0 ? GF_NEAR_SLOT : l == 1 ? GF_FGRID_SLOT : 0), tot) : 0;
        for (int w = 0; w < CLS_THR / 32; ++w) {
            sm.base[l][w] = b;
            b += sm.cnt[l][w];
        }
    }
    __syncthreads();
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int i = (int)(j0 + u * CLS_THR + threadIdx.x);
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            if (!is[l][u]) continue;
            const int at = sm.base[l][warp] + (u ? __popc(bal[l][0]) : 0) + __popc(bal[l][u] & below);
            if (l == 0) a.near_idx[at] = i;
            if (l == 1) a.near_idx[a.n - 1 - at] = i;
            if (l == 2 && LISTED) a.far_idx[at] = i;
        }
    }
    // (cnt is written again only after every thread has passed the second barrier, base after the
    // next call's first)
}

// Single evaluations: a CTA classifies whole segments and leaves each one's far-bucket counts
// (a.seghist) for the stable far list.
template <typename R, int NF>
__global__ void __launch_bounds__(CLS_THR) classify_segs(const __grid_constant__ EvalArgs a)
{
    __shared__ ClassifySmem sm;
    __shared__ int total[GF_FAR_BUCKETS];
    for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += CLS_THR) total[b] = 0;
    for (int seg = blockIdx.x; seg < a.nseg; seg += gridDim.x) {
        for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += CLS_THR) sm.hist[b] = 0;
        __syncthreads();
        const int64_t i0 = (int64_t)seg * a.segsize, i1 = min(i0 + (int64_t)a.segsize, a.n);
        for (int64_t j0 = i0; j0 < i1; j0 += CLS_TILE) classify_tile<R, NF, false>(a, j0, i1, sm);
        __syncthreads();
        int *dst = a.seghist + (size_t)seg * GF_FAR_BUCKETS;
        for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += CLS_THR) {
            const int h = sm.hist[b];
            dst[b] = h;
            total[b] += h;
        }
        __syncthreads();
    }
    for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += CLS_THR)
        if (total[b]) atomicAdd(&a.far_count[1 + b], total[b]);
}

// The targets listed by a classification pass.
template <typename R, int NF>
__global__ void __launch_bounds__(32 * NEAR_WARPS) near3d_list(const __grid_constant__ EvalArgs a)
{
    __shared__ __align__(16) NearWarp<R, NF> smem[NEAR_WARPS];
    NearWarp<R, NF> &sm = smem[threadIdx.x >> 5];
    const int nnear = a.far_count[GF_NEAR_SLOT], nfg = a.far_count[GF_FGRID_SLOT];
    const int tiles = ((nnear + 31) >> 5) + ((nfg + 31) >> 5);
    int nq = 0;
    // (neighbouring tiles on different CTAs: a short list still reaches every SM)
    for (int t = blockIdx.x + gridDim.x * (threadIdx.x >> 5); t < tiles; t += gridDim.x * NEAR_WARPS)
        near_list_tile<R, NF>(&a, 0, t, nnear, nfg, sm, nq);
    if (nq) sing_flush<R, NF>(&a, sm, nq);
}

template <typename R, int NF>
__global__ void __launch_bounds__(256) near3d(EvalArgs a)
{
    __shared__ int hist[GF_FAR_BUCKETS];
    for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    near3d_tiles<R, NF>(a, (int64_t)blockIdx.x * blockDim.x, (int64_t)gridDim.x * blockDim.x, hist);
    __syncthreads();
    for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += blockDim.x)
        if (hist[b]) atomicAdd(&a.far_count[1 + b], hist[b]);
}

// Batched classification: persistent CTAs walk the (pair, tile) list, GF_BATCH_TILE targets a tile.
template <typename R, int NF>
__global__ void __launch_bounds__(CLS_THR) classify_batch(const EvalArgs *args, const int *prefix, int np)
{
    __shared__ ClassifySmem sm;
    __shared__ EvalArgs sa;
    const int total = prefix[np];
    int p = -1;
    for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
        if (p < 0 || vb >= prefix[p + 1]) {
            p = p < 0 ? 0 : p;
            while (vb >= prefix[p + 1]) ++p;
            const int *src = reinterpret_cast<const int *>(args + p);
            for (int i = threadIdx.x; i < (int)(sizeof(EvalArgs) / sizeof(int)); i += CLS_THR) reinterpret_cast<int *>(&sa)[i] = src[i];
        }
        for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += CLS_THR) sm.hist[b] = 0;
        __syncthreads();
        const int64_t base = (int64_t)(vb - prefix[p]) * GF_BATCH_TILE, end = min(base + GF_BATCH_TILE, sa.n);
        for (int64_t j0 = base; j0 < end; j0 += CLS_TILE) classify_tile<R, NF, true>(sa, j0, end, sm);
        __syncthreads();
        for (int b = threadIdx.x; b < GF_FAR_BUCKETS; b += CLS_THR)
            if (sm.hist[b]) atomicAdd(&sa.far_count[1 + b], sm.hist[b]);
        __syncthreads();
    }
}

// Batched near targets from the pairs' near lists: the pairs' tiles form one list, pair after pair, dealt out to the
// warps of the grid in turn, so that the warps are in one or two pairs' grids
// at a time and every warp has its share of the whole.
template <typename R, int NF>
__global__ void __launch_bounds__(32 * NEAR_WARPS) near3d_list_batch(const EvalArgs *args, int np)
{
    __shared__ __align__(16) NearWarp<R, NF> smem[NEAR_WARPS];
    NearWarp<R, NF> &sm = smem[threadIdx.x >> 5];
    int t = blockIdx.x * NEAR_WARPS + (threadIdx.x >> 5), nq = 0;
    for (int p = 0; p < np; ++p) {
        const int nnear = args[p].far_count[GF_NEAR_SLOT], nfg = args[p].far_count[GF_FGRID_SLOT];
        const int tiles = ((nnear + 31) >> 5) + ((nfg + 31) >> 5);
        for (; t < tiles; t += gridDim.x * NEAR_WARPS) near_list_tile<R, NF>(args, p, t, nnear, nfg, sm, nq);
        t -= tiles;
    }
    if (nq) sing_flush<R, NF>(args, sm, nq);
}

// ---------------------------------------------------------------------------
// 2D near kernel (Algorithm 1): K = L + f1 - i alpha f2, G = e^{i alpha x1} K,
// f1 = -(1/2pi) ln r Y_eps(r), f2 = t f1 at the reduced point (t, x2).
// NF fields per node: 1 (L), 3 (derivative plans: L, K_1 - h_1, K_2 - h_2) or
// 6 (and T_11 - h_11, T_12 - h_12, T_22 - h_22).  Outputs: G; GF_OUT_GRAD = G,
// dG/dx1, dG/dx2 (Sec. 2.4.1: K_i = (K_i - h_i)_N + h_i, dG/dx_i = e^{i alpha x1}
// K_i); GF_OUT_HESSDIFF = T_11, T_12, T_22 (Sec. 2.4.2, the same with h_pq), the
// singular parts
//   h_1  = -(1/2pi)[-(k^2/2) x1 ln r + x1/r^2 - i alpha x1^2/r^2 - (alpha^2/2) x1^3/r^2] Y
//   h_2  = -(1/2pi)[-(k^2/2) x2 ln r + x2/r^2 - i alpha x1 x2/r^2 - (alpha^2/2) x1^2 x2/r^2] Y
//   h_11 = (dk2/2pi)[ln r/2 - (i alpha/2) x1 ln r + x1^2/(2r^2) - i alpha x1^3/(2r^2)] Y
//   h_12 = (dk2/2pi)[x1 x2/(2r^2) - (i alpha/2) x1^2 x2/r^2] Y
//   h_22 = (dk2/2pi)[ln r/2 - (i alpha/2) x1 ln r + x2^2/(2r^2) - (i alpha/2) x1 x2^2/r^2] Y
// (dk2 = k^2 - k2^2) at (x1, x2) = (t, x2), in double.
// ---------------------------------------------------------------------------
template <typename R, int NF>
__global__ void __launch_bounds__(256) near2d(EvalArgs a)
{
    typedef typename cplx_t<R>::T C;
    const C *G = reinterpret_cast<const C *>(a.grid);
    C *out = reinterpret_cast<C *>(a.out);
    const double ih1 = 1.0 / a.h1, ih2 = 1.0 / a.h2;
    const int ne = n_entries(a.which);
    const int f0 = a.which == GF_OUT_HESSDIFF ? 3 : 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < a.n; base += stride) {
        const int64_t i = base + threadIdx.x;
        bool valid = i < a.n;
        double x1 = 0, x2 = 0;
        if (valid) {
            x1 = a.x[2 * i];
            x2 = a.x[2 * i + 1];
        }
        bool finite = isfinite(x1) && isfinite(x2);
        bool isfar = valid && finite && fabs(x2) > a.c;
        push_far(isfar, (int)i, a.far_idx, a.far_count);
        if (!valid || isfar) continue;
        if (!finite) {
            for (int e = 0; e < ne; ++e) out[i * ne + e] = nan_c<R>();
            continue;
        }
        double t, m;
        reduce_period(x1, t, m);
        double f1, f2;
        int i1 = stencil_origin(t, -GF_PI, a.h1, ih1, a.M1, f1);
        int i2 = stencil_origin(x2, -a.ct, a.h2, ih2, a.M2, f2);
        double w1[4], w2[4];
        lagrange4(f1, w1);
        lagrange4(f2, w2);
        double acc[3][2] = {{0, 0}, {0, 0}, {0, 0}};
#pragma unroll
        for (int d2 = 0; d2 < 4; ++d2) {
            const C *row = G + ((size_t)(i2 + d2) * a.P1 + i1) * NF + f0;
#pragma unroll
            for (int e = 0; e < (NF == 1 ? 1 : 3); ++e) {
                if (e >= ne) break;
                double sr = 0, si = 0;
#pragma unroll
                for (int d1 = 0; d1 < 4; ++d1) {
                    double2 g = ld_grid(row + d1 * NF + e);
                    sr = fma(w1[d1], g.x, sr);
                    si = fma(w1[d1], g.y, si);
                }
                acc[e][0] = fma(w2[d2], sr, acc[e][0]);
                acc[e][1] = fma(w2[d2], si, acc[e][1]);
            }
        }
        double r = sqrt(t * t + x2 * x2);
        if (r < 2.0 * a.eps) {
            const double Y = 1.0 - smooth8((r - a.eps) / a.eps), lr = log(r), ir2 = 1.0 / (r * r);
            const double al = a.a1, kk = a.k * a.k, i2p = 0.5 / GF_PI;
            if (a.which != GF_OUT_HESSDIFF) {
                // K = L + f1 - i alpha f2
                const double fa = -lr * Y * i2p;
                acc[0][0] += fa;
                acc[0][1] -= al * t * fa;
            }
            if (a.which == GF_OUT_GRAD) {
                acc[1][0] += -i2p * (-0.5 * kk * t * lr + t * ir2 - 0.5 * al * al * t * t * t * ir2) * Y;
                acc[1][1] += i2p * al * t * t * ir2 * Y;
                acc[2][0] += -i2p * (-0.5 * kk * x2 * lr + x2 * ir2 - 0.5 * al * al * t * t * x2 * ir2) * Y;
                acc[2][1] += i2p * al * t * x2 * ir2 * Y;
            } else if (a.which == GF_OUT_HESSDIFF) {
                const double s = (kk - a.k2 * a.k2) * i2p * Y;
                acc[0][0] += s * (0.5 * lr + 0.5 * t * t * ir2);
                acc[0][1] += s * (-0.5 * al * t * lr - 0.5 * al * t * t * t * ir2);
                acc[1][0] += s * (0.5 * t * x2 * ir2);
                acc[1][1] += s * (-0.5 * al * t * t * x2 * ir2);
                acc[2][0] += s * (0.5 * lr + 0.5 * x2 * x2 * ir2);
                acc[2][1] += s * (-0.5 * al * t * lr - 0.5 * al * t * x2 * x2 * ir2);
            }
        }
        double sa, ca;
        sincos(a.a1 * t, &sa, &ca);
        const double2 lift = cmul(make_double2(ca, sa), lattice_phase(a.a1, m, 0.0, 0.0));
#pragma unroll
        for (int e = 0; e < 3; ++e)
            if (e < ne) store_out(out + i * ne + e, cmul(lift, make_double2(acc[e][0], acc[e][1])));
    }
}

// ---------------------------------------------------------------------------
// Counting-sort scatter of the far list by |x3| bucket, largest truncation
// radius first (bucket NB-1 first), so that warps see homogeneous lanes and
// the heaviest targets are scheduled first.
// ---------------------------------------------------------------------------
// Start of each bucket's run in the far list, the buckets in descending order
// (nearest the slab first), from the counts a.far_count[1 + b]; called by all
// threads of the block, by one warp: lane l takes the descending positions
// l PER .. l PER + PER - 1.
__device__ void far_bucket_starts(const EvalArgs &a, int *off)
{
    static_assert(GF_FAR_BUCKETS % 32 == 0, "bucket count: a multiple of 32");
    if (threadIdx.x < 32) {
        constexpr int PER = GF_FAR_BUCKETS / 32;
        const int lane = threadIdx.x;
        int c[PER], tot = 0;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            c[i] = a.far_count[1 + (GF_FAR_BUCKETS - 1 - (lane * PER + i))];
            tot += c[i];
        }
        int incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        int s = incl - tot;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            off[GF_FAR_BUCKETS - 1 - (lane * PER + i)] = s;
            s += c[i];
        }
    }
    __syncthreads();
}

// Bucket sort of the appended far list (the batched sweeps): positions within a
// bucket in the order of the cursor atomics.
__device__ void far_scatter_body(const EvalArgs &a, int blk, int nblk, int *off)
{
    far_bucket_starts(a, off);
    const int count = a.far_count[0];
    int *cursor = a.far_count + 1 + GF_FAR_BUCKETS;
    for (int i = blk * blockDim.x + threadIdx.x; i < count; i += nblk * blockDim.x) {
        int idx = a.far_idx[i];
        double z = fabs(a.x[3 * (size_t)idx + 2]);
        int b = far_bucket(z, a.c);
        int pos = off[b] + atomicAdd(&cursor[b], 1);
        a.far_sorted[pos] = idx;
    }
}

// Stable counting sort of the far targets (single-plan evaluations), from the
// bucket codes the classification pass left in a.far_idx: the far kernels' warps
// take 32 consecutive list entries and set their truncation and precision bands
// from them, so a list that is the same from call to call makes the sums the same
// bit for bit.  Over segments of a.segsize targets: counts per segment and bucket (by the
// classification), their exclusive scan over the segments (per
// bucket, from the bucket's start), and the scatter in index order, one warp a segment.
constexpr int SEG_WARPS = 4;

// One block per 32 buckets (a lane each), 32 warps over contiguous ranges of
// segments: each warp's sum, the warps' exclusive prefix, then the running
// position written back over the counts.
__global__ void __launch_bounds__(1024) far_seg_scan(EvalArgs a)
{
    __shared__ int start[GF_FAR_BUCKETS];
    __shared__ int part[32][32];
    if (a.far_count[0] == 0) return;
    far_bucket_starts(a, start);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x * 32 + lane;
    const int per = (a.nseg + 31) / 32;
    const int s0 = min(w * per, a.nseg), s1 = min(s0 + per, a.nseg);
    int *col = a.seghist + b;
    int sum = 0;
#pragma unroll 8
    for (int sg = s0; sg < s1; ++sg) sum += col[(size_t)sg * GF_FAR_BUCKETS];
    part[w][lane] = sum;
    __syncthreads();
    int run = start[b];
    for (int v = 0; v < w; ++v) run += part[v][lane];
#pragma unroll 8
    for (int sg = s0; sg < s1; ++sg) {
        const int c = col[(size_t)sg * GF_FAR_BUCKETS];
        col[(size_t)sg * GF_FAR_BUCKETS] = run;
        run += c;
    }
}

// Each warp walks its segment in index order, 32 targets a step: the lanes with
// the same bucket take consecutive positions from the segment's running start.
__global__ void __launch_bounds__(32 * SEG_WARPS) far_seg_scatter(EvalArgs a)
{
    __shared__ int pos0[SEG_WARPS][GF_FAR_BUCKETS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int seg = blockIdx.x * SEG_WARPS + w;
    if (seg >= a.nseg || a.far_count[0] == 0) return;
    const int *src = a.seghist + (size_t)seg * GF_FAR_BUCKETS;
    for (int b = lane; b < GF_FAR_BUCKETS; b += 32) pos0[w][b] = src[b];
    __syncwarp();
    const unsigned below = (1u << lane) - 1u;
    const int64_t i0 = (int64_t)seg * a.segsize, i1 = min(i0 + (int64_t)a.segsize, a.n);
    // eight steps' codes are loaded at once
    for (int64_t j0 = i0; j0 < i1; j0 += 256) {
        int code[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t i = j0 + 32 * u + lane;
            code[u] = i < i1 ? a.far_idx[i] : -1;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int c = code[u];
            if (__ballot_sync(0xffffffffu, c >= 0) == 0u) continue;
            const unsigned peers = __match_any_sync(0xffffffffu, c);
            const int before = __popc(peers & below);
            const int pos = c >= 0 ? pos0[w][c] + before : 0;
            __syncwarp();
            if (c >= 0) {
                a.far_sorted[pos] = (int)(j0 + 32 * u + lane);
                if (before == 0) pos0[w][c] += __popc(peers);
            }
            __syncwarp();
        }
    }
}

__global__ void __launch_bounds__(256) far_scatter(EvalArgs a)
{
    __shared__ int off[GF_FAR_BUCKETS];
    far_scatter_body(a, blockIdx.x, gridDim.x, off);
}

// batched: `per` CTAs per pair, persistent over the np * per work list
__global__ void __launch_bounds__(256) far_scatter_batch(const EvalArgs *args, int np, int per)
{
    __shared__ int off[GF_FAR_BUCKETS];
    __shared__ EvalArgs sa;
    for (int vb = blockIdx.x; vb < np * per; vb += gridDim.x) {
        if (threadIdx.x == 0) sa = args[vb / per];
        __syncthreads();
        far_scatter_body(sa, vb % per, per, off);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Far-series tables: |beta_n|, ln|beta_n| and 1/|beta_n| for evanescent n
// (beta_n = i |beta_n|); zeros for propagating n, whose terms are summed from
// the short list PropEntry instead.
// ---------------------------------------------------------------------------
// Propagating n (b = 0) get bl2 = +inf, so that the float sums' ex2(-bl2 z) is 0
// for them without a test.
__device__ __forceinline__ void set_entry(BetaEntry &e, double b, double ib)
{
    e.b = b;
    e.lnb = b > 0.0 ? log(b) : 0.0;
    e.bf = (float)b;
    e.blo = (float)(b - (double)e.bf);
    e.lnbf = (float)e.lnb;
    e.lnblo = (float)(e.lnb - (double)e.lnbf);
}
__device__ __forceinline__ void set_entry(BetaEntryF &e, double b, double ib)
{
    e.bl2 = b > 0.0 ? (float)(b * 1.4426950408889634) : CUDART_INF_F;  // b log2(e)
    e.ib = (float)ib;
    e.b = (float)b;
    e.pad = 0.f;
}

// Split plans: the Helmholtz sums' rows (series_tables) behind the b table.
__device__ __forceinline__ const float *far_rows_f32(const EvalArgs &a)
{
    const size_t ne = (size_t)(a.n1hi - a.n1lo + 1) * (a.n2hi - a.n2lo + 1);
    return reinterpret_cast<const float *>(reinterpret_cast<const BetaEntryF *>(a.btab) + ((ne + 1) & ~(size_t)1));  // 32-byte loads
}

// Series tables of a 3D plan, built on the device: the b table over the index
// box, the exponential table e^{-(j - j0)/GF_EXPTAB_STEPS}, and (block 0, warp 0) the list
// of propagating indices in row-major order of the sub-box pbox = [n1lo, n1hi,
// n2lo, n2hi] (ballot compaction keeps the order fixed).
template <typename E>
__global__ void series_tables(EvalArgs a, E *tab, double2 *exptab, longlong2 *trig, PropEntry *prop, int *nprop, int4 pbox)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < GF_TRIG_STEPS; j += gridDim.x * blockDim.x) {
        double sn, cn;
        sincospi(2.0 * j / GF_TRIG_STEPS, &sn, &cn);
        trig[j] = longlong2{__double2ll_rn(cn * 0x1p61), __double2ll_rn(sn * 0x1p61)};
    }
    const int W2 = a.n2hi - a.n2lo + 1;
    const int tot = (a.n1hi - a.n1lo + 1) * W2;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += gridDim.x * blockDim.x) {
        int n1 = a.n1lo + i / W2, n2 = a.n2lo + i % W2;
        double c1 = a.a1 + n1, c2 = a.a2 + n2;
        double aa = sqrt(c1 * c1 + c2 * c2);
        E e;
        if (aa <= a.k) {
            set_entry(e, 0.0, 0.0);
        } else {
            double b = sqrt((aa - a.k) * (aa + a.k));
            set_entry(e, b, 1.0 / b);
        }
        tab[i] = e;
    }
    if (sizeof(E) == sizeof(BetaEntryF)) {
        // the Helmholtz sums' rows behind it: by groups of four, -b log2(e) and then -log2 b, padded
        // with weight 0
        float *fb = const_cast<float *>(far_rows_f32(a));
        const int W4 = (W2 + 3) & ~3, rows = a.n1hi - a.n1lo + 1;
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows * W4; i += gridDim.x * blockDim.x) {
            const int r = i / W4, q = i - r * W4;
            const double c1 = a.a1 + (a.n1lo + r), c2 = a.a2 + (a.n2lo + q);
            const double aa = sqrt(c1 * c1 + c2 * c2);
            const bool ev = q < W2 && aa > a.k;
            const double b = ev ? sqrt((aa - a.k) * (aa + a.k)) : 1.0;
            float *f = fb + ((size_t)r * W4 + (q & ~3)) * 2 + (q & 3);
            f[0] = ev ? (float)(-b * 1.4426950408889634) : -CUDART_INF_F;
            f[4] = ev ? (float)-log2(b) : 0.f;
        }
    }
    if (exptab)
        for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < a.exptab_n; j += gridDim.x * blockDim.x)
        {
            const double off = (double)(j - a.exptab_j0) * (1.0 / GF_EXPTAB_STEPS);
            const double ev = exp(-off);
            exptab[j] = make_double2(ev, off);
            // the float-float copy after it: (hi, lo) of e^{-y_j} and y_j (exact in float)
            const float hi = (float)ev;
            reinterpret_cast<float4 *>(exptab + a.exptab_n)[j] = make_float4(hi, (float)(ev - (double)hi), (float)off, 0.f);
        }
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        const int pw = pbox.w - pbox.z + 1, ptot = (pbox.y - pbox.x + 1) * pw;
        const int N0 = (int)rint(-a.a2);
        int cnt = 0;
        for (int base = 0; base < ptot; base += 32) {
            const int i = base + (int)threadIdx.x;
            bool in = false;
            double c1 = 0, c2 = 0, aa = 0;
            if (i < ptot) {
                c1 = a.a1 + (pbox.x + i / pw);
                c2 = a.a2 + (pbox.z + i % pw);
                aa = sqrt(c1 * c1 + c2 * c2);
                in = aa <= a.k;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, in);
            if (in) {
                const double br = sqrt((a.k - aa) * (a.k + aa));
                prop[cnt + __popc(bal & ((1u << threadIdx.x) - 1u))] =
                    PropEntry{c1, c2, br, 1.0 / br, (double)(pbox.z + i % pw - N0), 1, pbox.x + i / pw,
                              (float)c1, (float)c2, (float)br, (float)(1.0 / br)};
            }
            cnt += __popc(bal);
        }
        __syncwarp();
        // row starts: first = 0 where the previous entry is (n1, n2 - 1) (reads n1
        // and m2, writes only first)
        for (int q = (int)threadIdx.x; q < cnt; q += 32)
            prop[q].first = (q > 0 && prop[q - 1].n1 == prop[q].n1 && prop[q - 1].m2 + 1.0 == prop[q].m2) ? 0 : 1;
        if (threadIdx.x == 0) *nprop = cnt;
    }
}

// Warp maximum / minimum of non-negative doubles, compared as 64-bit integers
// (for x >= 0 the IEEE bit pattern orders like the value), which keeps the
// comparisons off the FP64 pipe; the result is one of the lanes' values.
__device__ __forceinline__ double warp_max(double v)
{
    long long b = __double_as_longlong(v);
    for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
    return __longlong_as_double(b);
}

__device__ __forceinline__ double warp_min(double v)
{
    long long b = __double_as_longlong(v);
    for (int o = 16; o > 0; o >>= 1) b = min(b, __shfl_xor_sync(0xffffffffu, b, o));
    return __longlong_as_double(b);
}

// A float as a double by integer operations (no conversion instruction, which
// would occupy the FP64 pipe): exact for zero and normal floats; denormal floats
// (below 1.2e-38) read as zero.  Not for infinities or NaN.
__device__ __forceinline__ double f2d_exact(float f)
{
    const unsigned u = __float_as_uint(f);
    const bool nz = (u & 0x7F800000u) != 0u;
    const unsigned hi = (u & 0x80000000u) | (nz ? ((u & 0x7FFFFFFFu) >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, nz ? (int)(u << 29) : 0);
}

// e^{-y} by Tang's table-driven method (ACM TOMS 15, 1989): y = y_j + r with
// y_j = (j - j0)/S, S = GF_EXPTAB_STEPS, |r| <= (1/2 + 4e-2)/S; e^{-y} = T[j] e^{-r},
// the plan table holding (e^{-y_j}, y_j).  The index is rint(S yf) + j0 for a
// float evaluation yf of y (|yf - y| < 6e-8 (2 b|x3| + 2 |ln b| + |y|), so that
// |S (yf - y)| < 4e-2 for the core terms, b|x3| < 20, and S <= 4096; rounding
// by the 1.5 * 2^23 shift), clamped to the table (callers discard the
// terms whose y lies beyond it).  Returns e^{-r} by its Taylor polynomial of
// degree DEG and T[j].x.  The truncation relative to e^{-y} is at most
// |r|^{DEG+1}/(DEG+1)! e^{|r|}; the far kernel takes three degrees (EXP_DEG_A >
// B > C), switching where a term lies e^{EXP_GAP_B} and e^{EXP_GAP_C} below the
// largest term of its series, so that every term's truncation stays below
// about 1e-17 of that largest term (bounds at |r| = 0.51/S, 0.52/S for S = 2048,
// 0.54/S for S = 4096):
//   S = 128: degrees 5/4/3 (5.6e-18, 8.4e-15, 1.1e-11), gaps 7 and 14;
//   S = 256: degrees 5/4/3 (8.7e-20, 2.6e-16, 6.6e-13), gaps 4 and 12;
//   S = 512: degrees 4/3/2 (8.2e-18, 4.1e-14, 1.7e-10), gaps 9 and 17.5;
//   S = 1024: degrees 4/3/2 (2.6e-19, 2.6e-15, 2.1e-11), gaps 6.25 and 15.25;
//   S = 2048: degrees 4/3/2 (8.8e-21, 1.7e-16, 2.7e-12), gaps 3.5 and 13.25;
//   S = 4096: degrees 3/2/1 (1.3e-17, 3.8e-13, 8.7e-9), gaps 10.75 and 20.75.
constexpr int EXP_DEG_A = GF_EXPTAB_STEPS >= 4096 ? 3 : GF_EXPTAB_STEPS >= 512 ? 4 : 5;
constexpr int EXP_DEG_B = EXP_DEG_A - 1, EXP_DEG_C = EXP_DEG_A - 2;
constexpr double EXP_GAP_B = GF_EXPTAB_STEPS >= 4096 ? 10.75 : GF_EXPTAB_STEPS >= 2048 ? 3.5
                           : GF_EXPTAB_STEPS >= 1024 ? 6.25 : GF_EXPTAB_STEPS >= 512 ? 9.0
                           : GF_EXPTAB_STEPS >= 256  ? 4.0 : 7.0;
constexpr double EXP_GAP_C = GF_EXPTAB_STEPS >= 4096 ? 20.75 : GF_EXPTAB_STEPS >= 2048 ? 13.25
                           : GF_EXPTAB_STEPS >= 1024 ? 15.25 : GF_EXPTAB_STEPS >= 512 ? 17.5
                           : GF_EXPTAB_STEPS >= 256  ? 12.0 : 14.0;

// (-1)^i / i!
__host__ __device__ constexpr double exp_taylor_coef(int i) { return i == 0 ? 1.0 : -exp_taylor_coef(i - 1) / i; }

template <int DEG>
__device__ __forceinline__ double exp_neg_split(double y, float yf, const double2 *__restrict__ T, int j0, int jmax,
                                                double &Tj)
{
    const float jm = fmaf((float)GF_EXPTAB_STEPS, yf, 12582912.0f);
    const int idx = min(max(__float_as_int(jm) - 0x4B400000 + j0, 0), jmax);
    const double2 t = __ldg(T + idx);
    const double r = y - t.y;
    Tj = t.x;
    if (DEG <= 1) return 1.0 - r;
    constexpr double c5 = exp_taylor_coef(5), c4 = exp_taylor_coef(4), c3 = exp_taylor_coef(3),
                     c2 = exp_taylor_coef(2);
    double p;
    if (DEG >= 5) {
        p = fma(r, c5, c4);
        p = fma(p, r, c3);
    } else if (DEG == 4) {
        p = fma(r, c4, c3);
    } else {
        p = c3;
    }
    if (DEG >= 3)
        p = fma(p, r, c2);
    else
        p = c2;
    p = fma(p, r, -1.0);
    return fma(p, r, 1.0);
}

// x with its sign bit flipped where m = 0x80000000 (an integer operation).
__device__ __forceinline__ double flip_sign(double x, int m)
{
    return __hiloint2double(__double2hiint(x) ^ m, __double2loint(x));
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Per-lane set-up of a far target (double): reduced t, lattice index m, z, sign.
struct FarLane {
    double t1, m1, t2, m2, z, iz, sg, R2;
    int idx;
    bool valid;
};

__device__ __forceinline__ FarLane far_lane(const EvalArgs &a, int slot, int count)
{
    FarLane L;
    L.valid = slot < count;
    L.idx = L.valid ? a.far_sorted[slot] : 0;
    double x1 = 0, x2 = 0, x3 = 1;
    if (L.valid) {
        x1 = a.x[3 * (size_t)L.idx];
        x2 = a.x[3 * (size_t)L.idx + 1];
        x3 = a.x[3 * (size_t)L.idx + 2];
    }
    // cell reduction by a multiply and a floor: the series does not depend on
    // the decomposition x = 2 pi m + t, so the near branch's exact cell decision
    // is not needed here
    L.m1 = floor(fma(x1, INV_TWO_PI, 0.5));
    L.m2 = floor(fma(x2, INV_TWO_PI, 0.5));
    L.t1 = fma(-TWO_PI, L.m1, x1);
    L.t2 = fma(-TWO_PI, L.m2, x2);
    L.z = fabs(x3);
    L.sg = x3 >= 0.0 ? 1.0 : -1.0;
    // explicitly rounded (no contraction): R2 decides the row split, which the
    // double-precision and float-tail kernels must reproduce exactly
    L.iz = __ddiv_rn(1.0, L.z);
    const double Tz = __dmul_rn(a.T, L.iz);
    L.R2 = L.valid ? __dadd_rn(__dmul_rn(a.k, a.k), __dmul_rn(Tz, Tz)) : 0.0;
    return L;
}

// Per-lane constants of Reinsch's form of the Clenshaw recurrence for the row
// sums sum_{k>=0} w_k e^{ik theta}, theta = t2, real weights w_k:
//   s = sign(cos theta), lambda = 2 cos theta - 2 s (-4 sin^2(theta/2) or 4 cos^2(theta/2)),
//   d_k = w_k + lambda b_{k+1} + s d_{k+1},  b_k = d_k + s b_{k+1},
//   sum = d_0 - (lambda/2) b_1 + i b_1 sin theta,  b_1 = s (b_0 - d_0).
// Unlike the plain three-term recurrence it keeps its accuracy for theta near
// 0 and pi (C. Reinsch, 1967; error analysis by Gentleman, Comput. J. 12, 1969).
struct Reinsch {
    double lam, hlam, sv;
    int m;  // sign bit of s
};

__device__ __forceinline__ Reinsch reinsch_lane(double sv, double cv)
{
    // 2 - 2 cos = 2 sin^2/(1 + cos) and 2 + 2 cos = 2 sin^2/(1 - cos), free of
    // cancellation on the side where each is used
    Reinsch R;
    const double s2 = 2.0 * sv * sv;
    R.m = cv >= 0.0 ? 0 : (int)0x80000000;
    R.lam = cv >= 0.0 ? -s2 / (1.0 + cv) : s2 / (1.0 - cv);
    R.hlam = 0.5 * R.lam;
    R.sv = sv;
    return R;
}

// Double-precision Reinsch state of NH row sums.  NH = 1 (G_d): w = e^{-bz}/b.
// NH = 6 (Maxwell partial sums): A = sum w, B = sum c2 w, C = sum c2^2 w,
// D = sum b^2 w, E = sum b w, F = sum c2 b w.
template <int NH>
struct RState {
    double d[NH], b[NH];
};

// ---------------------------------------------------------------------------
// Float-float arithmetic: a value is an unevaluated sum h + l of two floats
// (about 48 significant bits).  Error-free sum by Knuth's TwoSum, product by
// an fma (Dekker, Numer. Math. 18, 1971).  Every operation is explicitly
// rounded, so no contraction can break the error-free steps.
// ---------------------------------------------------------------------------
struct FF {
    float h, l;
};

__device__ __forceinline__ FF two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    return FF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v))};
}

// a double as a float pair
__device__ __forceinline__ FF ff_split(double x)
{
    const float h = (float)x;
    return FF{h, (float)(x - (double)h)};
}

// Float-float Reinsch state of one sum (Helmholtz far series).
struct RStateFF {
    float dh, dl, bh, bl;
};

// The terms of the float-float band: n2, n2 + dir, ... (count of them), each
// at least e^{-FF_GAP} below the largest term of the series.  Float-float
// rounding perturbs y by about 1.3e-14 max(|y|, 1) (emulated over random b,
// |x3|), so a term at y = y_max + 8 is off by about 1.4e-13 e^{-8} < 5e-17 of
// the largest term: below half a double rounding of that term.  Per term: y = b z + ln b and e^{-y} =
// T[j] e^{-r} (the float-float table of the same step, r = y - y_j, |r| <=
// 0.54/S, e^{-r} to r^3 with r^2/2 - r^3/6 in float), then one Reinsch step:
// d' = w + lambda b + s d, b' = d' + s b.
constexpr float FF_GAP = 8.0f;

// One float-float Reinsch step with the term n2 (weight 0 outside the lane's
// truncation set).  Lazy form: the high words follow the recurrence in plain
// float, d' = (lambda b + w) + s d, b' = d' + s b; their rounding errors, exact
// by TwoProd and TwoSum, go into the low words, which follow the same
// recurrence.  The caller renormalizes the pairs every second step, so a low
// word stays within a few units of the high word's last place, while the high
// words' dependency chain is four float operations per term (a normalized
// float-float step chains about a dozen).
__device__ __forceinline__ void ff_step(RStateFF &st, const BetaEntry *__restrict__ row, int n2, float c2f,
                                        float c1sq, float R2f, FF z, FF lam, float sf, const float4 *__restrict__ T,
                                        int j0, int jmax)
{
    const float4 q = *reinterpret_cast<const float4 *>(&row[n2].bf);  // b hi, lo; ln b hi, lo
    const bool ok = fmaf(c2f, c2f, c1sq) <= R2f && q.x != 0.f;
    const float p = __fmul_rn(q.x, z.h);
    float pe = __fmaf_rn(q.x, z.h, -p);
    pe = __fmaf_rn(q.x, z.l, __fmaf_rn(q.y, z.h, pe));
    const FF y0 = two_sum(p, q.z);
    const FF y = two_sum(y0.h, __fadd_rn(__fadd_rn(y0.l, pe), q.w));
    const float jm = __fmaf_rn((float)GF_EXPTAB_STEPS, y.h, 12582912.0f);
    const int idx = min(max(__float_as_int(jm) - 0x4B400000 + j0, 0), jmax);
    const float4 t = __ldg(T + idx);
    const float rh = __fsub_rn(y.h, t.z);
    const float rs = __fadd_rn(rh, y.l);
    const float qq = __fmul_rn(__fmul_rn(rs, rs), __fmaf_rn(rs, -1.0f / 6.0f, 0.5f));
    const FF a = two_sum(1.0f, -rh);
    const float al = __fadd_rn(__fsub_rn(a.l, y.l), qq);
    float wh = __fmul_rn(t.x, a.h);
    float wl = __fmaf_rn(t.x, a.h, -wh);
    wl = __fmaf_rn(t.x, al, __fmaf_rn(t.y, a.h, wl));
    wh = ok ? wh : 0.f;
    wl = ok ? wl : 0.f;
    // high words
    const float m = __fmul_rn(lam.h, st.bh);
    const float me = __fmaf_rn(lam.h, st.bh, -m);
    const FF u = two_sum(m, wh);
    const FF dn = two_sum(u.h, __fmul_rn(sf, st.dh));
    // low words: the errors, then lambda b and s d on the low parts
    const float dl = __fadd_rn(__fadd_rn(__fadd_rn(me, u.l), __fadd_rn(dn.l, wl)),
                               __fmaf_rn(lam.h, st.bl, __fmaf_rn(lam.l, st.bh, __fmul_rn(sf, st.dl))));
    const FF bn = two_sum(dn.h, __fmul_rn(sf, st.bh));
    st.bl = __fadd_rn(__fadd_rn(bn.l, dl), __fmul_rn(sf, st.bl));
    st.dh = dn.h;
    st.dl = dl;
    st.bh = bn.h;
}

// Renormalized pair (Fast2Sum of the high and the low word).
__device__ __forceinline__ void ff_renorm(float &h, float &l)
{
    const float s = __fadd_rn(h, l);
    l = __fsub_rn(l, __fsub_rn(s, h));
    h = s;
}

__device__ __forceinline__ void reinsch_seg_ff(RStateFF &st, const BetaEntry *__restrict__ row, int &n2, int count,
                                               int dir, float &c2f, float c1sq, float R2f, FF z, FF lam, float sf,
                                               const float4 *__restrict__ T, int j0, int jmax)
{
    const float df = (float)dir;
    int i = 0;
    for (; i + 1 < count; i += 2, n2 += 2 * dir, c2f += 2.0f * df) {
        ff_step(st, row, n2, c2f, c1sq, R2f, z, lam, sf, T, j0, jmax);
        ff_step(st, row, n2 + dir, c2f + df, c1sq, R2f, z, lam, sf, T, j0, jmax);
        ff_renorm(st.dh, st.dl);
        ff_renorm(st.bh, st.bl);
    }
    if (i < count) {
        ff_step(st, row, n2, c2f, c1sq, R2f, z, lam, sf, T, j0, jmax);
        ff_renorm(st.dh, st.dl);
        ff_renorm(st.bh, st.bl);
        n2 += dir;
        c2f += df;
    }
}

// Feed `count` terms n2, n2 + dir, ... into the state (the first has the
// highest recurrence index), advancing n2 and c2; weights on the lane's own
// truncation set, exponential of degree DEG.  Per term and sum the recurrence
// costs three FP64 operations; for NH = 1 the product T[j] e^{-r} is folded
// into the first.
template <int NH, int DEG>
__device__ __forceinline__ void reinsch_seg(RState<NH> &st, const BetaEntry *__restrict__ row, int &n2, int count,
                                            int dir, float &c2f, double &c2, float c1sq, float R2f, double z,
                                            const Reinsch &RS, const double2 *__restrict__ T, int j0, int jmax)
{
    const float zf = (float)z;
    const float df = (float)dir;
    const double dd = (double)dir;
#pragma unroll 2
    for (int i = 0; i < count; ++i, n2 += dir, c2f += df) {
        const BetaEntry be = row[n2];
        const bool ok = fmaf(c2f, c2f, c1sq) <= R2f && be.bf != 0.f;
        double Tj;
        double p = exp_neg_split<DEG>(fma(be.b, z, be.lnb), fmaf(be.bf, zf, be.lnbf), T, j0, jmax, Tj);
        p = ok ? p : 0.0;
        if (NH == 1) {
            const double dn = fma(RS.lam, st.b[0], fma(Tj, p, flip_sign(st.d[0], RS.m)));
            st.b[0] = dn + flip_sign(st.b[0], RS.m);
            st.d[0] = dn;
        } else {
            double wv[NH];
            wv[0] = Tj * p;
            wv[1] = c2 * wv[0];
            wv[2] = c2 * wv[1];
            wv[4] = be.b * wv[0];
            wv[3] = be.b * wv[4];
            wv[5] = c2 * wv[4];
            c2 += dd;
#pragma unroll
            for (int e = 0; e < NH; ++e) {
                const double dn = fma(RS.lam, st.b[e], wv[e] + flip_sign(st.d[e], RS.m));
                st.b[e] = dn + flip_sign(st.b[e], RS.m);
                st.d[e] = dn;
            }
        }
    }
}

// The terms n2 = start, start + dir, ... (nc + nb + na of them, from the outer
// end of the row towards the anchor): the first nc with the degree-EXP_DEG_C
// exponential, the next nb with degree EXP_DEG_B, the rest with EXP_DEG_A.
template <int NH>
__device__ __forceinline__ void reinsch_run(RState<NH> &st, const BetaEntry *__restrict__ row, int start, int dir,
                                            int nc, int nb, int na, double a2, float c1sq, float a2f, float R2f,
                                            double z, const Reinsch &RS, const double2 *__restrict__ T, int j0, int jmax)
{
    int n2 = start;
    float c2f = a2f + (float)start;
    double c2 = a2 + start;
    reinsch_seg<NH, EXP_DEG_C>(st, row, n2, nc, dir, c2f, c2, c1sq, R2f, z, RS, T, j0, jmax);
    reinsch_seg<NH, EXP_DEG_B>(st, row, n2, nb, dir, c2f, c2, c1sq, R2f, z, RS, T, j0, jmax);
    reinsch_seg<NH, EXP_DEG_A>(st, row, n2, na, dir, c2f, c2, c1sq, R2f, z, RS, T, j0, jmax);
}

// Helmholtz rows: the first nff terms (the outer ones, all in the float-float
// band) in float-float, the state then carried over to double for the
// remaining nd terms (all within e^{-FF_GAP} of the largest term, where the
// degree-EXP_DEG_A exponential is exact to double precision).
__device__ __forceinline__ void reinsch_run_ff(RState<1> &st, const BetaEntry *__restrict__ row, int start, int dir,
                                               int nff, int nd, float c1sq, float a2f, float R2f, double z, FF zff,
                                               const Reinsch &RS, FF lamff, float sf, const double2 *__restrict__ T,
                                               int j0, int jmax)
{
    int n2 = start;
    float c2f = a2f + (float)start;
    double c2 = 0.0;  // not used by single sums
    if (nff > 0) {
        RStateFF f{0.f, 0.f, 0.f, 0.f};
        reinsch_seg_ff(f, row, n2, nff, dir, c2f, c1sq, R2f, zff, lamff, sf,
                       reinterpret_cast<const float4 *>(T + (jmax + 1)), j0, jmax);
        st.d[0] = f2d_exact(f.dh) + f2d_exact(f.dl);
        st.b[0] = f2d_exact(f.bh) + f2d_exact(f.bl);
    }
    reinsch_seg<1, EXP_DEG_A>(st, row, n2, nd, dir, c2f, c2, c1sq, R2f, z, RS, T, j0, jmax);
}

// One recurrence step with zero weight (recurrence index 0 of a sum whose
// index-0 term belongs to another sum).
template <int NH>
__device__ __forceinline__ void reinsch_zero(RState<NH> &st, const Reinsch &RS)
{
#pragma unroll
    for (int e = 0; e < NH; ++e) {
        const double dn = fma(RS.lam, st.b[e], flip_sign(st.d[e], RS.m));
        st.b[e] = dn + flip_sign(st.b[e], RS.m);
        st.d[e] = dn;
    }
}

// sin x and cos x in float for |x| < 6000, by Cody and Waite's reduction
// (Software Manual for the Elementary Functions, 1980): r = x - q pi/2 with
// pi/2 in three parts (the first two of 12 significant bits, so q times each
// is exact for |q| <= 4096), |r| <= pi/4, then the Taylor polynomials of sin
// (to r^9, truncation < 2e-9) and cos (to r^10, < 2e-10) at 0 and the quadrant
// q mod 4.  Error about 1.5 ulp; float arithmetic only (no FP64-pipe
// conversion, no MUFU).
__device__ __forceinline__ void sincos_cw(float x, float &s, float &c)
{
    const float qm = fmaf(x, 0.636619772f, 12582912.0f);  // rint(2x/pi) + 1.5 * 2^23
    const int q = __float_as_int(qm) - 0x4B400000;
    const float qf = qm - 12582912.0f;
    float r = fmaf(-qf, 1.5703125f, x);
    r = fmaf(-qf, 4.837512969970703e-4f, r);
    r = fmaf(-qf, 7.549790126404332e-8f, r);
    const float r2 = r * r;
    float ps = fmaf(r2, 1.0f / 362880.0f, -1.0f / 5040.0f);
    ps = fmaf(ps, r2, 1.0f / 120.0f);
    ps = fmaf(ps, r2, -1.0f / 6.0f);
    const float sr = fmaf(ps * r2, r, r);
    float pc = fmaf(r2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
    pc = fmaf(pc, r2, -1.0f / 720.0f);
    pc = fmaf(pc, r2, 1.0f / 24.0f);
    pc = fmaf(pc, r2, -0.5f);
    const float cr = fmaf(pc, r2, 1.0f);
    const bool odd = (q & 1) != 0;
    const float ss = odd ? cr : sr, cc = odd ? sr : cr;
    s = (q & 2) ? -ss : ss;
    c = ((q + 1) & 2) ? -cc : cc;
}

// e^{i m t2} in float for an integer |m| < 2^11, with no double arithmetic:
// t2 = th + tl with th of 12 significant bits (m th exact in float), the
// product reduced by 2 pi = C1 + C2 + C3 (C1 of 8 bits, so k C1 is exact).
struct PhaseF {
    float th, tl;
};

__device__ __forceinline__ PhaseF phase_split(double t2)
{
    PhaseF P;
    P.th = __int_as_float(__float_as_int((float)t2) & (int)0xFFFFF800);
    P.tl = (float)(t2 - (double)P.th);
    return P;
}

__device__ __forceinline__ void phase_m(const PhaseF &P, int m, float &s, float &c)
{
    const float mf = (float)m;
    const float x = mf * P.th;
    const float kq = rintf(x * 0.15915494f);
    float r = fmaf(-kq, 6.28125f, x);
    r = fmaf(-kq, 1.9353071693331003e-3f, r);
    r = fmaf(-kq, 1.0253131677018246e-11f, r);
    r = fmaf(mf, P.tl, r);
    sincos_cw(r, s, c);
}

// Row sums combined into the outputs with the row's real factors (c1 fixed):
// G: A; xx: (1 - c1^2/k^2) A; yy: A - C/k^2; zz: A + D/k^2; xy: -(c1/k^2) B;
// xz: -(c1/k^2) E (real factor); yz: -(1/k^2) F (real factor).
template <int NH, typename F>
__device__ __forceinline__ void add_row(F S[][2], const F rr[][2], F c1, F ik2)
{
    if (NH == 1) {
        S[0][0] += rr[0][0];
        S[0][1] += rr[0][1];
    } else {
        const F fxx = (F)1 - c1 * c1 * ik2;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            S[0][q] += rr[0][q];
            S[1][q] += fxx * rr[0][q];
            S[2][q] += rr[0][q] - ik2 * rr[2][q];
            S[3][q] += rr[0][q] + ik2 * rr[3][q];
            S[4][q] += -c1 * ik2 * rr[1][q];
            S[5][q] += -c1 * ik2 * rr[4][q];
            S[6][q] += -ik2 * rr[5][q];
        }
    }
}

// The same segment sums in float (hardware ex2 and rsqrt), for the
// exponentially small tail of a double-precision plan:
// sum_{n2=lo}^{hi} w(n2) v^{n2-lo}, v = e^{i t2}.  b and 1/b come from the
// lattice index itself (b^2 = c1^2 + c2^2 - k^2, one rsqrt), so the loop loads
// nothing; in float b is good to ~1e-7 relative, e^{-b|x3|} to ~4e-6 for
// b|x3| <= 40, well inside the tail's error budget.  The terms go in groups of
// four aligned at lo, by Horner's rule in v^4 from the top group down: each
// group adds w0 + w1 v + w2 v^2 + w3 v^3 (powers formed once per target), so
// the dependent chain is one complex multiply-add per four terms and the four
// weights are independent work.
__device__ __forceinline__ float rsqrt_approx(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// weights of one index: q0 = c1^2 - k^2, zl2 = |x3| log2(e); propagating n
// (b^2 <= 0) get weight 0.  No per-lane truncation test: the terms of the
// warp's disk beyond the lane's own set are below e^{-T} of its largest term
// (they add accuracy).
template <int NH>
__device__ __forceinline__ void tail_weights(float c2, float q0, float zl2, float wv[NH])
{
    const float x = fmaf(c2, c2, q0);
    const bool ev = x > 0.f;
    const float ib = rsqrt_approx(ev ? x : 1.f);
    const float b = x * ib;
    const float e = ev ? ex2_approx(-b * zl2) : 0.f;
    wv[0] = e * ib;
    if (NH > 1) {
        wv[1] = c2 * wv[0];
        wv[2] = c2 * wv[1];
        wv[3] = b * e;
        wv[4] = e;
        wv[5] = c2 * e;
    }
}

// Powers v, v^2, v^3, v^4 of v = (cv, sv).
struct VPow {
    float x[4], y[4];
};

__device__ __forceinline__ VPow vpowers(float cv, float sv)
{
    VPow P;
    P.x[0] = cv;
    P.y[0] = sv;
#pragma unroll
    for (int k = 1; k < 4; ++k) {
        P.x[k] = P.x[k - 1] * cv - P.y[k - 1] * sv;
        P.y[k] = P.x[k - 1] * sv + P.y[k - 1] * cv;
    }
    return P;
}

// One group n0 .. n0+3 (GUARD: indices above hi weigh zero): acc = acc v^4 +
// sum_t w(n0 + t) v^t.
template <int NH, bool GUARD>
__device__ __forceinline__ void horner_group_f32(int n0, int hi, float a2f, float q0, float zl2, const VPow &V,
                                                 float acc[NH][2])
{
    float w[4][NH];
    const float cb = a2f + (float)n0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        tail_weights<NH>(cb + (float)t, q0, zl2, w[t]);
        if (GUARD && n0 + t > hi) {
#pragma unroll
            for (int e = 0; e < NH; ++e) w[t][e] = 0.f;
        }
    }
#pragma unroll
    for (int e = 0; e < NH; ++e) {
        const float cx = fmaf(w[3][e], V.x[2], fmaf(w[2][e], V.x[1], fmaf(w[1][e], V.x[0], w[0][e])));
        const float cy = fmaf(w[3][e], V.y[2], fmaf(w[2][e], V.y[1], w[1][e] * V.y[0]));
        const float nx = fmaf(acc[e][0], V.x[3], fmaf(-acc[e][1], V.y[3], cx));
        const float ny = fmaf(acc[e][0], V.y[3], fmaf(acc[e][1], V.x[3], cy));
        acc[e][0] = nx;
        acc[e][1] = ny;
    }
}

template <int NH>
__device__ __forceinline__ void seg_horner_f32(int lo, int hi, float a2f, float q0, float zl2, const VPow &V,
                                               float acc[NH][2])
{
#pragma unroll
    for (int e = 0; e < NH; ++e) acc[e][0] = acc[e][1] = 0.f;
    const int g = (hi - lo + 4) >> 2;  // groups; the top one may pass hi
    if (g <= 0) return;
    horner_group_f32<NH, true>(lo + 4 * (g - 1), hi, a2f, q0, zl2, V, acc);
    for (int j = g - 2; j >= 0; --j) horner_group_f32<NH, false>(lo + 4 * j, hi, a2f, q0, zl2, V, acc);
}

// ---------------------------------------------------------------------------
// 3D far kernel for double-precision plans.  Series (he), and for Maxwell the
// second derivatives (each term times delta_pq - c^p c^q/k^2, c = (alpha_n,
// beta sgn x3)):
//   S = sum_n beta_n^{-1} e^{i beta_n |x3|} e^{i alpha_n . t},  G_d = e^{i2pi<alpha.m>} (i/8pi^2) S.
// Propagating n (|alpha_n| < k, a handful) are summed from a list.  For the
// evanescent n, beta = i b and 1/beta = -i/b; with w = e^{-bz}/b (real) the row
// n1 contributes -i sum_{n2} w e^{i(c1 t1 + c2 t2)}.  Every row is summed
// relative to the fixed anchor n2 = N0: the core outwards from N0 by two
// Reinsch recurrences, the float tails by Horner's rule in v = e^{i t2} from
// their first index, moved to N0 by a float phase.  The row phase e^{i c1 t1}
// follows a recurrence over the rows and e^{i(alpha_2 + N0) t2} is applied once
// per target.  Each lane keeps only its own truncation set
// |alpha_n|^2 <= k^2 + (T/z)^2.
//
// Precision, by term size (every term is at most e^{-(b - bmin) z} of the
// largest): the warp's core disk |alpha_n|^2 <= k^2 + (Y0/z_min)^2 (b z_min <=
// Y0 = 18, z_min the warp's smallest |x3|) is summed by the recurrences, its
// outer band (b >= bmin + FF_GAP/z_min, Helmholtz) in float-float and its inner
// terms in double with the table-driven exponential; the remaining terms, each
// below e^{-18} = 1.5e-8 of the leading ones and all together below
// 2 pi e^{-18}/z of the series scale, are summed in float (by far3d_tail, or
// here when TAILS): their float rounding (< 1e-5 relative) contributes < 2e-12
// of the series scale.
// ---------------------------------------------------------------------------
constexpr double FAR_CORE_Y0 = 18.0;

// Row slab `slab` of `nslab` of the rows of a chunk: the warp's core rows
// (|c1| <= sqrt(Rc2)) split evenly, the tail-only rows below and above the core
// joined to the first and the last slab.  Every row falls in exactly one slab.
__device__ __forceinline__ void slab_rows(int n1a, int n1b, float Rc2f, float a1f, int slab, int nslab, int &lo, int &hi)
{
    lo = n1a;
    hi = n1b;
    if (nslab <= 1) return;
    const float rcf = sqrtf(fmaxf(Rc2f, 0.f));
    const int k0 = max(n1a, (int)ceilf(-a1f - rcf)), k1 = min(n1b, (int)floorf(-a1f + rcf));
    const int Lc = max(k1 - k0 + 1, 0);
    if (slab > 0) lo = k0 + (slab * Lc) / nslab;
    if (slab < nslab - 1) hi = k0 + ((slab + 1) * Lc) / nslab - 1;
}

// The rows of a warp's far sums and their core segments.  The double-precision
// kernel and the float-tail kernel must split every row identically, so every
// operation here (and in far_lane) is explicitly rounded: no contraction can
// make the two kernels disagree on a term.
struct FarWarp {
    double izmax;      // 1/z_min over the warp's lanes
    float R2mf, Rc2f;  // truncation disk |alpha_n|^2 <= R2m (warp maximum) and core disk Rc2
    float a1f, a2f;
    float k2f, bff;    // k^2; the float-float band edge b >= bff = bmin + FF_GAP/z_min (Helmholtz)
    int n1a, n1b;      // rows of the truncation disk (one index of margin)
    int N0;            // anchor n2 = rint(-alpha_2)
};

__device__ __forceinline__ FarWarp far_warp(const EvalArgs &a, const FarLane &L)
{
    FarWarp W;
    const double R2m = warp_max(L.R2);
    W.izmax = warp_max(L.valid ? L.iz : 0.0);
    // core disk of the warp: b z_min <= Y0
    const double Rc2 = fmin(__dadd_rn(__dmul_rn(a.k, a.k), __dmul_rn(__dmul_rn(FAR_CORE_Y0 * FAR_CORE_Y0, W.izmax), W.izmax)), R2m);
    W.R2mf = __double2float_rn(R2m);
    W.Rc2f = __double2float_rn(Rc2);
    W.a1f = __double2float_rn(a.a1);
    W.a2f = __double2float_rn(a.a2);
    const float Rmf = __fsqrt_rn(W.R2mf);
    W.n1a = max(a.n1lo, (int)floorf(__fsub_rn(-W.a1f, Rmf)) - 1);
    W.n1b = min(a.n1hi, (int)ceilf(__fadd_rn(-W.a1f, Rmf)) + 1);
    W.N0 = (int)rint(-a.a2);
    W.k2f = __double2float_rn(__dmul_rn(a.k, a.k));
    W.bff = __double2float_rn(__fma_rn((double)FF_GAP, W.izmax, a.bmin));
    return W;
}

// Row n1 of the float-float band edge (Helmholtz): q^2 = bff^2 + k^2 - c1^2 raised
// by more than the float roundings of its parts (1e-5 of their sizes, and 1e-3),
// so that every term with |c2| >= sqrt(q^2) has b >= bff (below zero: the whole
// row lies in the band).
__device__ __forceinline__ float far_ff_q2(const FarWarp &W, float c1sq)
{
    const float qq = __fmaf_rn(W.bff, W.bff, W.k2f);
    return __fadd_rn(__fmaf_rn(1e-5f, __fadd_rn(qq, c1sq), 1e-3f), __fsub_rn(qq, c1sq));
}

// Row n1 of the warp's truncation disk: its index range [n2a, n2b] (false when
// the row is empty) and core segment [ca, cb] (ca > cb: no core), the core
// widened to contain N0.  Bounds are formed in float with a one-index margin:
// every lane still keeps exactly its own truncation set in the double sums, and
// the core/tail split only moves terms of size ~e^-18 between double and float.
__device__ __forceinline__ bool far_row(const FarWarp &W, const EvalArgs &a, int n1, float &c1f, float &c1sq, int &n2a,
                                        int &n2b, int &ca, int &cb)
{
    c1f = __fadd_rn(W.a1f, (float)n1);
    c1sq = __fmul_rn(c1f, c1f);
    const float remf = __fsub_rn(W.R2mf, c1sq);
    if (remf < -1.0f) return false;
    const float srf = __fsqrt_rn(fmaxf(remf, 0.f));
    n2a = max(a.n2lo, (int)floorf(__fsub_rn(-W.a2f, srf)) - 1);
    n2b = min(a.n2hi, (int)ceilf(__fadd_rn(-W.a2f, srf)) + 1);
    if (n2a > n2b) return false;
    ca = n2b + 1;
    cb = n2b;
    const float remc = __fsub_rn(W.Rc2f, c1sq);
    if (remc >= 0.f) {
        const float src = __fsqrt_rn(remc);
        ca = max(n2a, (int)ceilf(__fsub_rn(-W.a2f, src)));
        cb = min(n2b, (int)floorf(__fadd_rn(-W.a2f, src)));
        if (ca > cb) {
            ca = n2b + 1;
            cb = n2b;
        } else {
            ca = min(ca, W.N0);
            cb = max(cb, W.N0);
        }
    }
    return true;
}

// The float tails of row n1 (the segments outside its core, or the whole row
// when it has none), each by Horner's rule from its first index and moved to the
// anchor N0, rotated by the row phase A = e^{i c1 t1} and added into Sf.
template <int NH, int NS>
__device__ __forceinline__ void far_row_tails(int n2a, int n2b, int ca, int cb, int N0, float a2f, float c1f,
                                              float c1sq, float k2f, float zf, const VPow &V, const PhaseF &PF,
                                              float Ax, float Ay, float ik2f, float Sf[NS][2])
{
    const float q0 = c1sq - k2f, zl2 = zf * 1.44269504f;
    const int tl_hi = (ca <= cb) ? ca - 1 : n2b;
    const int th_lo = (ca <= cb) ? cb + 1 : n2b + 1;
    if (n2a > tl_hi && th_lo > n2b) return;
    float tf[NH][2];
#pragma unroll
    for (int e = 0; e < NH; ++e) tf[e][0] = tf[e][1] = 0.f;
    if (n2a <= tl_hi) {
        float acc[NH][2], ps, pc;
        seg_horner_f32<NH>(n2a, tl_hi, a2f, q0, zl2, V, acc);
        phase_m(PF, n2a - N0, ps, pc);
#pragma unroll
        for (int e = 0; e < NH; ++e) {
            tf[e][0] += pc * acc[e][0] - ps * acc[e][1];
            tf[e][1] += pc * acc[e][1] + ps * acc[e][0];
        }
    }
    if (th_lo <= n2b) {
        float acc[NH][2], ps, pc;
        seg_horner_f32<NH>(th_lo, n2b, a2f, q0, zl2, V, acc);
        phase_m(PF, th_lo - N0, ps, pc);
#pragma unroll
        for (int e = 0; e < NH; ++e) {
            tf[e][0] += pc * acc[e][0] - ps * acc[e][1];
            tf[e][1] += pc * acc[e][1] + ps * acc[e][0];
        }
    }
#pragma unroll
    for (int e = 0; e < NH; ++e) {
        const float x = tf[e][0], y = tf[e][1];
        tf[e][0] = Ax * x - Ay * y;
        tf[e][1] = Ax * y + Ay * x;
    }
    add_row<NH, float>(Sf, tf, c1f, ik2f);
}

// One warp, row slab `slab` of `nslab` of chunk w (32 consecutive entries of
// the sorted far list).  The slab's share of the series is added into the
// output entries, which the near pass set to zero; the propagating terms go
// with slab 0.  TAILS: the float tails are summed here too; otherwise the
// float-tail kernel (far3d_tail) adds them.
template <int NF, bool TAILS>
__device__ void far3d_f64_chunk(const EvalArgs &a, int w, int count, int slab, int nslab)
{
    constexpr int NH = NF == 1 ? 1 : 6;
    constexpr int NS = NF == 1 ? 1 : 7;
    const BetaEntry *tab = reinterpret_cast<const BetaEntry *>(a.btab);
    double2 *out = reinterpret_cast<double2 *>(a.out);
    const int ne = n_entries(a.which);
    const int W2 = a.n2hi - a.n2lo + 1;
    const int lane = threadIdx.x & 31;
    const double k2 = a.k * a.k, ik2 = 1.0 / k2;
    const float ik2f = (float)ik2;
    const double2 *T = a.exptab;
    const int jmax = a.exptab_n - 1, j0 = a.exptab_j0;
    const float a2f = (float)a.a2;
    {
        FarLane L = far_lane(a, w * 32 + lane, count);
        const FarWarp W = far_warp(a, L);
        const float R2f = (float)L.R2;
        const double izmax = W.izmax;
        // every row is summed from the anchor n2 = N0 outwards (the centre of all
        // rows' truncation intervals); e^{i(alpha_2 + N0) t2} multiplies the total
        const int N0 = W.N0;
        double sv, cv, s1, c1v;
        sincos(L.t2, &sv, &cv);
        sincos(L.t1, &s1, &c1v);
        const double2 E1 = make_double2(c1v, s1);
        const Reinsch RS = reinsch_lane(sv, cv);
        const PhaseF PF = phase_split(L.t2);
        // every term is at most e^{-(b - bmin) z_min} of the largest one (e^{-bz}/b
        // decreases in b): degree B from b >= bmin + EXP_GAP_B/z_min, C from
        // bmin + EXP_GAP_C/z_min
        const float b4 = (float)(a.bmin + EXP_GAP_B * izmax), b3 = (float)(a.bmin + EXP_GAP_C * izmax);
        // Helmholtz: the float-float band from b >= W.bff = bmin + FF_GAP/z_min
        const FF zff = ff_split(L.z), lamff = ff_split(RS.lam);
        const float sgn = RS.m ? -1.0f : 1.0f;
        const float k2f = (float)k2;
        const float svf = (float)sv, cvf = (float)cv, zf = (float)L.z;
        const VPow VP = vpowers(cvf, svf);
        double P[NF][2];
        double S[NS][2];
        float Sf[NS][2];
#pragma unroll
        for (int e = 0; e < NF; ++e) P[e][0] = P[e][1] = 0.0;
#pragma unroll
        for (int e = 0; e < NS; ++e) S[e][0] = S[e][1] = 0.0, Sf[e][0] = Sf[e][1] = 0.f;
        // propagating terms, in the anchor frame: e^{i(c1 t1 + (c2 - alpha_2 - N0) t2)};
        // the list is in row-major order, so within a row the phase steps by e^{i t2}.
        // e^{i beta z} = e^{i beta z_w} e^{i beta (z - z_w)}, z_w the warp's smallest
        // |x3|: the lanes share a narrow |x3| bucket, so the first factor is one sincos
        // per entry per warp (lane q mod 32 forms it, shuffles hand it out) and the
        // second a Taylor polynomial while |beta (z - z_w)| <= 0.02 (cos to theta^6,
        // sin to theta^7: truncation below 1e-17); a warp whose spread is wider takes
        // a sincos per lane.
        double2 ph = make_double2(1.0, 0.0);
        const int nq = slab == 0 ? *a.nprop : 0;
        const double zw = warp_min(L.valid ? L.z : 1e300);
        const double dz = L.z - zw;
        const bool taylor = nq > 0 && warp_max(L.valid ? dz : 0.0) * a.k <= 0.02;
        double ewx = 1.0, ewy = 0.0;  // e^{i beta_{q0 + lane} z_w} / beta_{q0 + lane}
        for (int q = 0; q < nq; ++q) {
            if (taylor && (q & 31) == 0) {
                if (q + lane < nq) {
                    const PropEntry &pl = a.prop[q + lane];
                    sincos(pl.br * zw, &ewy, &ewx);
                    ewx *= pl.ibr;
                    ewy *= pl.ibr;
                }
            }
            const PropEntry &pe = a.prop[q];
            if (pe.first) {
                double sp, cp;
                sincos(fma(pe.c1, L.t1, pe.m2 * L.t2), &sp, &cp);
                ph = make_double2(cp, sp);
            } else {
                ph = cmul(ph, make_double2(cv, sv));
            }
            // u = e^{i beta z} / beta
            double ux, uy;
            if (taylor) {
                const double Ex = __shfl_sync(0xffffffffu, ewx, q & 31), Ey = __shfl_sync(0xffffffffu, ewy, q & 31);
                const double th = pe.br * dz, th2 = th * th;
                const double ct = fma(fma(fma(th2, -1.0 / 720.0, 1.0 / 24.0), th2, -0.5), th2, 1.0);
                const double st = th * fma(fma(fma(th2, -1.0 / 5040.0, 1.0 / 120.0), th2, -1.0 / 6.0), th2, 1.0);
                ux = Ex * ct - Ey * st;
                uy = Ex * st + Ey * ct;
            } else {
                double sz, cz;
                sincos(pe.br * L.z, &sz, &cz);
                ux = pe.ibr * cz;
                uy = pe.ibr * sz;
            }
            const double cp = ph.x, sp = ph.y;
            if (NF == 1) {
                P[0][0] = fma(ux, cp, fma(-uy, sp, P[0][0]));
                P[0][1] = fma(ux, sp, fma(uy, cp, P[0][1]));
            }
            if (NF > 1) {
                const double tx = ux * cp - uy * sp, ty = ux * sp + uy * cp;
                P[0][0] += tx;
                P[0][1] += ty;
                double b3 = pe.br * L.sg;
                double f[6] = {1.0 - pe.c1 * pe.c1 * ik2, 1.0 - pe.c2 * pe.c2 * ik2, 1.0 - b3 * b3 * ik2,
                               -pe.c1 * pe.c2 * ik2, -pe.c1 * b3 * ik2, -pe.c2 * b3 * ik2};
#pragma unroll
                for (int e = 0; e < 6; ++e) {
                    P[1 + e][0] += f[e] * tx;
                    P[1 + e][1] += f[e] * ty;
                }
            }
        }
        int r_lo, r_hi;
        slab_rows(W.n1a, W.n1b, W.Rc2f, W.a1f, slab, nslab, r_lo, r_hi);
        if (!TAILS) {
            // only rows with a core segment: |c1| <= sqrt(Rc2), one row of margin
            const float rcf = sqrtf(fmaxf(W.Rc2f, 0.f));
            r_lo = max(r_lo, (int)ceilf(-W.a1f - rcf) - 1);
            r_hi = min(r_hi, (int)floorf(-W.a1f + rcf) + 1);
        }
        double2 A = make_double2(1.0, 0.0);  // e^{i c1 t1}
        // Helmholtz: Reinsch's closing step is linear in the state (d, b), so the
        // rows' final states, times the row phase A, are summed first and closed
        // once: DR, BR from the right sums (index n2 - N0 >= 0), DL, BL from the
        // left ones (index N0 - n2 >= 1, before their zero step)
        double2 DR = make_double2(0.0, 0.0), BR = DR, DL = DR, BL = DR;
        for (int n1 = r_lo; n1 <= r_hi; ++n1) {
            // row phase by recurrence, re-anchored every 16 rows
            if (((n1 - r_lo) & 15) == 0) {
                double sa, ca_;
                sincos((a.a1 + n1) * L.t1, &sa, &ca_);
                A = make_double2(ca_, sa);
            } else {
                A = cmul(A, E1);
            }
            // float tails fold into the double sums every 8 rows
            if (TAILS && ((n1 - r_lo) & 7) == 7) {
#pragma unroll
                for (int e = 0; e < NS; ++e) {
                    S[e][0] += f2d_exact(Sf[e][0]);
                    S[e][1] += f2d_exact(Sf[e][1]);
                    Sf[e][0] = Sf[e][1] = 0.f;
                }
            }
            float c1f, c1sq;
            int n2a, n2b, ca, cb;
            if (!far_row(W, a, n1, c1f, c1sq, n2a, n2b, ca, cb)) continue;
            const BetaEntry *row = tab + (size_t)(n1 - a.n1lo) * W2 - a.n2lo;
            if (ca <= cb) {
                // right: n2 = cb .. N0 (index n2 - N0); left: n2 = ca .. N0-1 (index
                // N0 - n2, e^{-i theta}) and a zero step for index 0
                RState<NH> R, Lt;
#pragma unroll
                for (int e = 0; e < NH; ++e) R.d[e] = R.b[e] = Lt.d[e] = Lt.b[e] = 0.0;
                // degree bands (Maxwell): |c2| >= q3 (degree C), >= q4 (degree B),
                // one index of margin; Helmholtz: |c2| >= qff (float-float, from
                // far_ff_q2: no term with b < bff leaves the double band, no margin)
                const float q3 = sqrtf(fmaxf(b3 * b3 + k2f - c1sq, 0.f)), q4 = sqrtf(fmaxf(b4 * b4 + k2f - c1sq, 0.f));
                const float qff = sqrtf(fmaxf(far_ff_q2(W, c1sq), 0.f));
                if (NH == 1) {
                    const int tot = cb - N0 + 1;
                    const int mff = max(0, cb - max((int)ceilf(qff - a2f), N0) + 1);
                    reinsch_run_ff(*reinterpret_cast<RState<1> *>(&R), row, cb, -1, mff, tot - mff, c1sq, a2f, R2f, L.z,
                                   zff, RS, lamff, sgn, T, j0, jmax);
                    DR.x = fma(A.x, R.d[0], DR.x);
                    DR.y = fma(A.y, R.d[0], DR.y);
                    BR.x = fma(A.x, R.b[0], BR.x);
                    BR.y = fma(A.y, R.b[0], BR.y);
                    if (ca < N0) {
                        const int mffl = max(0, min((int)floorf(-qff - a2f), N0 - 1) - ca + 1);
                        reinsch_run_ff(*reinterpret_cast<RState<1> *>(&Lt), row, ca, 1, mffl, N0 - ca - mffl, c1sq, a2f,
                                       R2f, L.z, zff, RS, lamff, sgn, T, j0, jmax);
                        DL.x = fma(A.x, Lt.d[0], DL.x);
                        DL.y = fma(A.y, Lt.d[0], DL.y);
                        BL.x = fma(A.x, Lt.b[0], BL.x);
                        BL.y = fma(A.y, Lt.b[0], BL.y);
                    }
                } else {
                    const int tot = cb - N0 + 1;
                    const int r3 = (int)ceilf(q3 - a2f) + 1, r4 = (int)ceilf(q4 - a2f) + 1;
                    const int m3 = max(0, cb - max(r3, N0) + 1);
                    const int m4 = max(0, min(cb - m3, cb) - max(r4, N0) + 1);
                    reinsch_run<NH>(R, row, cb, -1, m3, m4, tot - m3 - m4, a.a2, c1sq, a2f, R2f, L.z, RS, T, j0, jmax);
                    // Maxwell: each row closed and combined with its own factors in c1
                    double rr[NH][2];
#pragma unroll
                    for (int e = 0; e < NH; ++e) {
                        const double b1 = flip_sign(R.b[e] - R.d[e], RS.m);
                        rr[e][0] = fma(-RS.hlam, b1, R.d[e]);
                        rr[e][1] = b1 * RS.sv;
                    }
                    if (ca < N0) {
                        const int totl = N0 - ca;
                        const int l3 = (int)floorf(-q3 - a2f) - 1, l4 = (int)floorf(-q4 - a2f) - 1;
                        const int m3l = max(0, min(l3, N0 - 1) - ca + 1);
                        const int m4l = max(0, min(l4, N0 - 1) - (ca + m3l) + 1);
                        reinsch_run<NH>(Lt, row, ca, 1, m3l, m4l, totl - m3l - m4l, a.a2, c1sq, a2f, R2f, L.z, RS, T, j0,
                                        jmax);
                        reinsch_zero<NH>(Lt, RS);
#pragma unroll
                        for (int e = 0; e < NH; ++e) {
                            const double b1 = flip_sign(Lt.b[e] - Lt.d[e], RS.m);
                            rr[e][0] += fma(-RS.hlam, b1, Lt.d[e]);
                            rr[e][1] -= b1 * RS.sv;
                        }
                    }
#pragma unroll
                    for (int e = 0; e < NH; ++e) {
                        const double x = rr[e][0], y = rr[e][1];
                        rr[e][0] = A.x * x - A.y * y;
                        rr[e][1] = A.x * y + A.y * x;
                    }
                    add_row<NH, double>(S, rr, a.a1 + n1, ik2);
                }
            }
            // float tails [n2a, ca-1] and [cb+1, n2b] (the whole row when there is
            // no core)
            if (TAILS)
                far_row_tails<NH, NS>(n2a, n2b, ca, cb, N0, a2f, c1f, c1sq, k2f, zf, VP, PF, (float)A.x, (float)A.y,
                                      ik2f, Sf);
        }
        if (NH == 1) {
            // right: sum = D + U (-lambda/2 + i sin theta), U = s (B - D);
            // left, after the zero step: sum = s D + B (lambda/2 - i sin theta)
            const double ux = flip_sign(BR.x - DR.x, RS.m), uy = flip_sign(BR.y - DR.y, RS.m);
            S[0][0] += fma(-RS.hlam, ux, fma(-RS.sv, uy, DR.x));
            S[0][1] += fma(-RS.hlam, uy, fma(RS.sv, ux, DR.y));
            S[0][0] += fma(RS.hlam, BL.x, fma(RS.sv, BL.y, flip_sign(DL.x, RS.m)));
            S[0][1] += fma(RS.hlam, BL.y, fma(-RS.sv, BL.x, flip_sign(DL.y, RS.m)));
        }
        if (TAILS) {
#pragma unroll
            for (int e = 0; e < NS; ++e) {
                S[e][0] += f2d_exact(Sf[e][0]);
                S[e][1] += f2d_exact(Sf[e][1]);
            }
        }
        // back from the anchor frame with the lattice phase: one factor
        // e^{i(2 pi <alpha.m> + (alpha_2 + N0) t2)} (i/8pi^2)
        double ph2 = a.a1 * L.m1 + a.a2 * L.m2;
        ph2 -= rint(ph2);
        double sN, cN;
        sincos(fma(2.0 * GF_PI, ph2, (a.a2 + N0) * L.t2), &sN, &cN);
        const double2 pre = make_double2(-sN / (8.0 * GF_PI * GF_PI), cN / (8.0 * GF_PI * GF_PI));
        // evanescent sums carry the factor -i (from 1/beta = -i/b), except the
        // xz, yz entries whose factor (-i)(-i sgn) = -sgn is real
        constexpr int NE = NF == 1 ? 1 : 7;
        double2 vals[NE];
        if (NF == 1) {
            vals[0] = cmul(pre, make_double2(P[0][0] + S[0][1], P[0][1] - S[0][0]));
        } else {
#pragma unroll
            for (int e = 0; e < 6; ++e) {
                const double *s = S[1 + e];
                double2 v;
                if (e < 4)
                    v = make_double2(P[1 + e][0] + s[1], P[1 + e][1] - s[0]);
                else
                    v = make_double2(P[1 + e][0] + L.sg * s[0], P[1 + e][1] + L.sg * s[1]);
                vals[e] = cmul(pre, v);
            }
            vals[NE - 1] = cmul(pre, make_double2(P[0][0] + S[0][1], P[0][1] - S[0][0]));
        }
        far_deposit(a, 0, w, slab, nslab, ((count + 31) >> 5) * 32, L.valid, L.idx, ne, vals);
        (void)out;
    }
}

// Far work items (a row slab of a chunk of 32 consecutive entries of the
// sorted list) are handed out one at a time from a counter, the most expensive
// chunks first: the list is in ascending bucket order and the bucket
// GF_FAR_BUCKETS c/|x3| grows as the target nears the slab, where the truncation
// disk (radius ~ T/|x3|) is largest, so the t-th item taken is slab t % S of
// chunk nch-1-t/S.  S (row slabs per chunk) is chosen so that there are about
// per_warp items per resident warp, which keeps the end of the launch short; the
// double-precision kernel asks for four, so that long lists keep one slab per
// chunk and its per-target set-up (double sines, divisions) is not repeated.
__device__ __forceinline__ int far_slabs(int nch, int smax, int per_warp = 8)
{
    const int nwarps = (int)(gridDim.x * blockDim.x) >> 5;
    if (nch <= 0) return 1;
    const int s = (per_warp * nwarps + nch - 1) / nch;
    return s < 1 ? 1 : s > smax ? smax : s;
}

__device__ __forceinline__ int far_take(int *counter, int nitems)
{
    int t = 0;
    if ((threadIdx.x & 31) == 0) t = atomicAdd(counter, 1);
    t = __shfl_sync(0xffffffffu, t, 0);
    return t < nitems ? t : -1;
}

// Row slabs per chunk at most.  A short list leaves the GPU empty unless its chunks are cut
// into single rows (1017 targets: far3d_f64 378 us with 8 slabs, 90 us with 32); from about
// 300 chunks on the slabs' repeated set-up costs more (13000 far targets: 559 us for
// the evaluation with 8 slabs, 681 us with 32).  Up to some 24 chunks even single rows pay (whole
// evaluations with 32 / 64 / 128 slabs: 1017 targets 146 / 132 / 131 us, 3000 targets 153 / 159 / 177).
// The float sums' set-up is cheap, their rows short: half as many.  These figures are for c = 0.6, 133 rows a
// target.  With fewer rows (larger c) a slab has two of them at least and a list is long sooner (25000 targets, a quarter
// of them far: c = 3, 27 rows 226 us with 32 slabs, 171 with 8; c = 1.2, 67 rows 246 and 190).
constexpr int FAR_SLABS_SHORT = 64, FAR_SLABS_MAX = 32, FAR_SLABS_LONG = 8, FAR_SHORT = 24, FAR_LONG = 300, FAR_HALF_ROWS = 66;

// Row slabs per chunk of a far launch over `count` targets (a.nfar: the far list, or what the
// products left of it, a list of its own: a look-up of the left chunks in the kernels cost far3d_f64 registers
// and shared memory that kept the tails from running beside it, a million targets with k = 7.3 7.65 -> 8.95 ms,
// |x3| <= 3 4.70 -> 8.80).
__device__ __forceinline__ int far_chunk_slabs(const EvalArgs &a, int kind, bool fp64, int nch)
{
    const float Tc = (float)a.T / (float)a.c, kf = (float)a.k;
    const int half_rows = (int)fminf(sqrtf(fmaf(Tc, Tc, kf * kf)), 1e6f);  // at |x3| = c
    const int longer = FAR_LONG * min(half_rows, FAR_HALF_ROWS) / FAR_HALF_ROWS;
    const int s = nch <= FAR_SHORT ? FAR_SLABS_SHORT : nch <= longer || !fp64 ? FAR_SLABS_MAX : FAR_SLABS_LONG;
    return far_slabs_capped(a, kind, nch, far_slabs(nch, max(FAR_SLABS_LONG, min(fp64 ? s : s / 2, half_rows))));
}

template <int NF, bool TAILS>
__global__ void __launch_bounds__(128, NF == 1 ? 5 : 1) far3d_f64(EvalArgs a)
{
    const int count = *a.nfar;
    const int nch = (count + 31) >> 5, S = far_chunk_slabs(a, 0, true, nch);
    int *ctr = a.far_count + GF_WORK_SLOT;
    for (int t = far_take(ctr, nch * S); t >= 0; t = far_take(ctr, nch * S))
        far3d_f64_chunk<NF, TAILS>(a, nch - 1 - t / S, count, t % S, S);
}

// ---------------------------------------------------------------------------
// Float tails of a double-precision plan's far series, as a kernel of their
// own: the terms of each warp's truncation disk outside its core disk (the
// same chunks of the sorted far list and the same row split as far3d_f64, from
// far_warp and far_row), summed in float with the hardware ex2 and added into
// the double outputs.  Kept apart from the double sums so that the FP64 pipe is
// fed only by warps with double work, while these warps run on the FP32 and
// transcendental pipes.  The per-target set-up and the lattice phase are in
// double; the row phase e^{i c1 t1} = e^{i alpha_1 t1} e^{i n1 t1} in float.
// ---------------------------------------------------------------------------

template <int NF>
__device__ void far3d_tail_chunk(const EvalArgs &a, int w, int count, int slab, int nslab)
{
    constexpr int NH = NF == 1 ? 1 : 6;
    constexpr int NS = NF == 1 ? 1 : 7;
    double2 *out = reinterpret_cast<double2 *>(a.out);
    const int ne = n_entries(a.which);
    const int lane = threadIdx.x & 31;
    const float ik2f = (float)(1.0 / (a.k * a.k)), k2f = (float)(a.k * a.k);
    const FarLane L = far_lane(a, w * 32 + lane, count);
    const FarWarp W = far_warp(a, L);
    const int N0 = W.N0;
    const float zf = (float)L.z;
    float svf, cvf;
    sincos_cw((float)L.t2, svf, cvf);
    const VPow VP = vpowers(cvf, svf);
    const PhaseF P1 = phase_split(L.t1), P2 = phase_split(L.t2);
    // e^{i alpha_1 t1} in float (the tails are summed in float; this kernel
    // leaves the FP64 pipe to the double sums running beside it)
    float A0x, A0y;
    sincos_cw(W.a1f * (float)L.t1, A0y, A0x);
    double S[NS][2];
    float Sf[NS][2];
#pragma unroll
    for (int e = 0; e < NS; ++e) S[e][0] = S[e][1] = 0.0, Sf[e][0] = Sf[e][1] = 0.f;
    // the rows split evenly over the slabs
    const int nr = W.n1b - W.n1a + 1;
    const int r_lo = W.n1a + (slab * nr) / nslab, r_hi = W.n1a + ((slab + 1) * nr) / nslab - 1;
    for (int n1 = r_lo; n1 <= r_hi; ++n1) {
        if (((n1 - r_lo) & 7) == 7) {
#pragma unroll
            for (int e = 0; e < NS; ++e) {
                S[e][0] += f2d_exact(Sf[e][0]);
                S[e][1] += f2d_exact(Sf[e][1]);
                Sf[e][0] = Sf[e][1] = 0.f;
            }
        }
        float c1f, c1sq;
        int n2a, n2b, ca, cb;
        if (!far_row(W, a, n1, c1f, c1sq, n2a, n2b, ca, cb)) continue;
        float sn, cn;
        phase_m(P1, n1, sn, cn);
        far_row_tails<NH, NS>(n2a, n2b, ca, cb, N0, W.a2f, c1f, c1sq, k2f, zf, VP, P2, A0x * cn - A0y * sn,
                              A0x * sn + A0y * cn, ik2f, Sf);
    }
#pragma unroll
    for (int e = 0; e < NS; ++e) {
        S[e][0] += f2d_exact(Sf[e][0]);
        S[e][1] += f2d_exact(Sf[e][1]);
    }
    // the same lattice phase and factors as far3d_f64_chunk (no propagating
    // terms); the fractional part of <alpha.m> in double, its sine and cosine in
    // float
    double ph2 = a.a1 * L.m1 + a.a2 * L.m2;
    ph2 -= rint(ph2);
    float sNf, cNf;
    sincos_cw((float)fma(2.0 * GF_PI, ph2, (a.a2 + N0) * L.t2), sNf, cNf);
    constexpr double i8pi2 = 1.0 / (8.0 * GF_PI * GF_PI);
    const double2 pre = make_double2(-f2d_exact(sNf) * i8pi2, f2d_exact(cNf) * i8pi2);
    constexpr int NE = NF == 1 ? 1 : 7;
    double2 vals[NE];
    if (NF == 1) {
        vals[0] = cmul(pre, make_double2(S[0][1], -S[0][0]));
    } else {
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            const double *s = S[1 + e];
            const double2 v = e < 4 ? make_double2(s[1], -s[0]) : make_double2(L.sg * s[0], L.sg * s[1]);
            vals[e] = cmul(pre, v);
        }
        vals[NE - 1] = cmul(pre, make_double2(S[0][1], -S[0][0]));
    }
    far_deposit(a, 1, w, slab, nslab, ((count + 31) >> 5) * 32, L.valid, L.idx, ne, vals);
    (void)out;
}

template <int NF>
__global__ void __launch_bounds__(128) far3d_tail(EvalArgs a)
{
    const int count = *a.nfar;
    const int nch = (count + 31) >> 5, S = far_chunk_slabs(a, 1, true, nch);
    int *ctr = a.far_count + GF_TAIL_SLOT;
    for (int t = far_take(ctr, nch * S); t >= 0; t = far_take(ctr, nch * S))
        far3d_tail_chunk<NF>(a, nch - 1 - t / S, count, t % S, S);
}

// ---------------------------------------------------------------------------
// 3D far kernel, split precision: the same sums in float with the hardware
// ex2; the per-target cell reduction and the lattice phase's fractional part in
// double, everything else in float.
// ---------------------------------------------------------------------------
// Pairs of floats in a 64-bit register: the packed multiply-add issues once for two.
__device__ __forceinline__ uint64_t pack2(float x, float y)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    return v;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t ex2x2(uint64_t a)
{
    float x, y;
    unpack2(a, x, y);
    return pack2(ex2_approx(x), ex2_approx(y));
}

// Helmholtz sums of H = 1 or 2 chunks of 32 targets (chunk indices w, -1: none), a target of
// each per lane.
//
// A row's evanescent terms: weights e^{-b|x3|}/b = 2^(-b log2(e) |x3| - log2 b) by one multiply-add and ex2 from
// the rows behind the b table, summed by Horner's rule in v^4, v = e^{i t2}, the even and the odd terms
// in the halves of packed multiply-adds (eight, four ex2 and one load for four terms).  Issue bounds
// it, so the loads, the row bounds (formed by one lane per row, 32 rows at a time) and the loops
// are shared by two targets where the list is long enough.  64 pairs with 2.2 million far targets:
// term by term with 1/b from the table 2.61 ms, groups 2.21, two targets a lane 1.68 (at 80 registers:
// with 102 and 16 warps an SM 2.44).  A million targets of one plan (series kernels alone) 605 -> 556 us.
__device__ __forceinline__ void load_rows(const float *p, uint64_t &b0, uint64_t &b1, uint64_t &l0, uint64_t &l1)
{
    const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2 *>(p)), l = __ldg(reinterpret_cast<const ulonglong2 *>(p + 4));
    b0 = b.x;
    b1 = b.y;
    l0 = l.x;
    l1 = l.y;
}

template <int H>
__device__ void far3d_f32_helm(const EvalArgs &a, const int (&w)[H], int count, int slab, int nslab)
{
    const int W2 = a.n2hi - a.n2lo + 1, W4 = (W2 + 3) & ~3;
    const float *frows = far_rows_f32(a);
    const int lane = threadIdx.x & 31;
    const float a1f = (float)a.a1, a2f = (float)a.a2, k2f = (float)(a.k * a.k);
    int idx[H];
    bool valid[H];
    double m1[H], m2[H];
    float z[H], t1[H], t2[H], sv[H], cv[H], Px[H], Py[H], Sx[H], Sy[H];
    float R2mf = 0.f;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int slot = w[h] * 32 + lane;
        valid[h] = w[h] >= 0 && slot < count;
        idx[h] = valid[h] ? a.far_sorted[slot] : 0;
        double x1 = 0, x2 = 0, x3 = 1;
        if (valid[h]) {
            x1 = a.x[3 * (size_t)idx[h]];
            x2 = a.x[3 * (size_t)idx[h] + 1];
            x3 = a.x[3 * (size_t)idx[h] + 2];
        }
        // cell reduction by a multiply and a floor: the series is the same for any
        // decomposition x = 2 pi m + t (e^{i alpha_n . x} = e^{i alpha_n . t}
        // e^{i 2 pi alpha . m}), so the exact cell decision of the near branch
        // is not needed here
        m1[h] = floor(fma(x1, INV_TWO_PI, 0.5));
        m2[h] = floor(fma(x2, INV_TWO_PI, 0.5));
        t1[h] = (float)fma(-TWO_PI, m1[h], x1);
        t2[h] = (float)fma(-TWO_PI, m2[h], x2);
        z[h] = fabsf((float)x3);
        const float Tz = (float)a.T / z[h];
        if (valid[h]) R2mf = fmaxf(R2mf, k2f + Tz * Tz);
        sincos_cw(t2[h], sv[h], cv[h]);
        Px[h] = Py[h] = Sx[h] = Sy[h] = 0.f;
    }
    for (int o = 16; o > 0; o >>= 1) R2mf = fmaxf(R2mf, __shfl_xor_sync(0xffffffffu, R2mf, o));
    for (int q = 0, nq = slab == 0 ? *a.nprop : 0; q < nq; ++q) {
        const PropEntry &pe = a.prop[q];
        const float br = pe.brf, ibr = pe.ibrf, c1 = pe.c1f, c2 = pe.c2f;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            float sz, cz, sp, cp;
            sincos_cw(br * z[h], sz, cz);
            sincos_cw(c1 * t1[h] + c2 * t2[h], sp, cp);
            Px[h] += ibr * (cz * cp - sz * sp);
            Py[h] += ibr * (cz * sp + sz * cp);
        }
    }
    uint64_t zz[H], v2x[H], v2y[H], v4x[H], v4y[H], nv4y[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        // v^2 and v^4 from their own angles: v^4 carries one rounding to the power n/4 where products of v would carry
        // four
        float q2x, q2y, q4x, q4y;
        sincos_cw(2.f * t2[h], q2y, q2x);
        sincos_cw(4.f * t2[h], q4y, q4x);
        zz[h] = pack2(z[h], z[h]);
        v2x[h] = pack2(q2x, q2x);
        v2y[h] = pack2(q2y, q2y);
        v4x[h] = pack2(q4x, q4x);
        v4y[h] = pack2(q4y, q4y);
        nv4y[h] = pack2(-q4y, -q4y);
    }
    // row bounds in float with a one-index margin; row slab: the rows split evenly
    const float Rmf = sqrtf(R2mf);
    const int n1a = max(a.n1lo, (int)floorf(-a1f - Rmf) - 1), n1b = min(a.n1hi, (int)ceilf(-a1f + Rmf) + 1);
    const int nr = n1b - n1a + 1;
    const int r_lo = n1a + (slab * nr) / nslab, r_hi = n1a + ((slab + 1) * nr) / nslab - 1;
    for (int r0 = r_lo; r0 <= r_hi; r0 += 32) {
        // groups of four from n2lo on, first and number, of row r0 + lane (the groups at the ends may pass
        // the truncation: the terms are there and below e^{-T})
        int gfirst = 0, gnum = 0;
        {
            const float c1 = a1f + (float)(r0 + lane), remf = R2mf - c1 * c1, srf = sqrtf(fmaxf(remf, 0.f));
            const int n2a = max(a.n2lo, (int)floorf(-a2f - srf) - 1), n2b = min(a.n2hi, (int)ceilf(-a2f + srf) + 1);
            if (remf >= -1.0f && n2a <= n2b && r0 + lane <= r_hi) {
                gfirst = (n2a - a.n2lo) & ~3;
                gnum = (((n2b - a.n2lo) & ~3) - gfirst) / 4 + 1;
            }
        }
        for (int r = 0; r < min(32, r_hi - r0 + 1); ++r) {
            const int g0 = __shfl_sync(0xffffffffu, gfirst, r), ng = __shfl_sync(0xffffffffu, gnum, r);
            if (ng == 0) continue;
            const float *rb = frows + (size_t)(r0 + r - a.n1lo) * 2 * W4 + 2 * (g0 + 4 * (ng - 1));
            uint64_t X[H], Y[H];  // (even, odd) terms' sums
#pragma unroll
            for (int h = 0; h < H; ++h) X[h] = Y[h] = 0;
            auto group = [&](uint64_t B0, uint64_t B1, uint64_t L0, uint64_t L1) {
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    // propagating n (summed separately) have -inf, so weight 0
                    const uint64_t w01 = ex2x2(fma2(B0, zz[h], L0)), w23 = ex2x2(fma2(B1, zz[h], L1));
                    const uint64_t x = fma2(w23, v2x[h], w01), y = mul2(w23, v2y[h]);
                    const uint64_t nX = fma2(X[h], v4x[h], fma2(Y[h], nv4y[h], x));
                    Y[h] = fma2(X[h], v4y[h], fma2(Y[h], v4x[h], y));
                    X[h] = nX;
                }
            };
            // two groups a turn, both loads first
            uint64_t A0, A1, A2, A3, B0, B1, B2, B3;
            if (ng & 1) {
                load_rows(rb, A0, A1, A2, A3);
                group(A0, A1, A2, A3);
                rb -= 8;
            }
#pragma unroll 1
            for (int g = ng >> 1; g > 0; --g, rb -= 16) {
                load_rows(rb, A0, A1, A2, A3);
                load_rows(rb - 8, B0, B1, B2, B3);
                group(A0, A1, A2, A3);
                group(B0, B1, B2, B3);
            }
            const float c1 = a1f + (float)(r0 + r), c2 = a2f + (float)(a.n2lo + g0);
#pragma unroll
            for (int h = 0; h < H; ++h) {
                float xe, xo, ye, yo, sp, cp;
                unpack2(X[h], xe, xo);
                unpack2(Y[h], ye, yo);
                const float hx = fmaf(cv[h], xo, fmaf(-sv[h], yo, xe)), hy = fmaf(cv[h], yo, fmaf(sv[h], xo, ye));
                // the row's phase with the roundings of its argument (up to 200) put back: they were most of the
                // sum's error (split evaluations against 64 bits: 1.2e-6 where term by term had 1.0e-6; with this and
                // the powers above 0.52e-6 against 0.86e-6)
                const float p1 = c1 * t1[h], p2 = c2 * t2[h], ps = p1 + p2, pb = ps - p1;
                const float lo = ((p1 - (ps - pb)) + (p2 - pb)) + fmaf(c1, t1[h], -p1) + fmaf(c2, t2[h], -p2);
                sincos_cw(ps, sp, cp);
                const float sq = fmaf(cp, lo, sp), cq = fmaf(-sp, lo, cp);
                Sx[h] += cq * hx - sq * hy;
                Sy[h] += cq * hy + sq * hx;
            }
        }
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
        if (w[h] < 0) continue;
        // e^{i 2pi <alpha.m>} (i/8pi^2): the fractional part in double, the phase in float
        double ph = a.a1 * m1[h] + a.a2 * m2[h];
        ph -= rint(ph);
        float sl, cl;
        sincospif(2.0f * (float)ph, &sl, &cl);
        const float sc = (float)(1.0 / (8.0 * GF_PI * GF_PI));
        float2 vals[1];
        vals[0] = cmulf(make_float2(-sl * sc, cl * sc), make_float2(Px[h] + Sy[h], Py[h] - Sx[h]));
        far_deposit(a, 0, w[h], slab, nslab, ((count + 31) >> 5) * 32, valid[h], idx[h], 1, vals);
    }
}

// Maxwell sums of one chunk of 32 targets.
__device__ void far3d_f32_maxwell(const EvalArgs &a, int w, int count, int slab, int nslab)
{
    const BetaEntryF *tab = reinterpret_cast<const BetaEntryF *>(a.btab);
    const int ne = n_entries(a.which);
    const int W2 = a.n2hi - a.n2lo + 1;
    const int lane = threadIdx.x & 31;
    const float ik2 = (float)(1.0 / (a.k * a.k));
    const float a2f = (float)a.a2;
    {
        // per-target set-up: the cell reduction in double, the rest in float
        const int slot = w * 32 + lane;
        const bool valid = slot < count;
        const int idx = valid ? a.far_sorted[slot] : 0;
        double x1 = 0, x2 = 0, x3 = 1;
        if (valid) {
            x1 = a.x[3 * (size_t)idx];
            x2 = a.x[3 * (size_t)idx + 1];
            x3 = a.x[3 * (size_t)idx + 2];
        }
        // cell reduction by a multiply and a floor: the series is the same for any
        // decomposition x = 2 pi m + t (e^{i alpha_n . x} = e^{i alpha_n . t}
        // e^{i 2 pi alpha . m}), so the exact cell decision of the near branch
        // is not needed here
        const double m1 = floor(fma(x1, INV_TWO_PI, 0.5)), m2 = floor(fma(x2, INV_TWO_PI, 0.5));
        const double t1d = fma(-TWO_PI, m1, x1), t2d = fma(-TWO_PI, m2, x2);
        const float z = fabsf((float)x3), t1 = (float)t1d, t2 = (float)t2d, sg = x3 >= 0.0 ? 1.f : -1.f;
        const float Tz = (float)a.T / z;
        const float R2f = valid ? (float)(a.k * a.k) + Tz * Tz : 0.f;
        float R2mf = R2f;
        for (int o = 16; o > 0; o >>= 1) R2mf = fmaxf(R2mf, __shfl_xor_sync(0xffffffffu, R2mf, o));
        float sv, cv;
        sincos_cw(t2, sv, cv);
        float P[7][2], S[7][2];
#pragma unroll
        for (int e = 0; e < 7; ++e) P[e][0] = P[e][1] = S[e][0] = S[e][1] = 0.f;
        for (int q = 0, nq = slab == 0 ? *a.nprop : 0; q < nq; ++q) {
            const PropEntry &pe = a.prop[q];
            const float br = pe.brf, ibr = pe.ibrf, c1 = pe.c1f, c2 = pe.c2f;
            float sz, cz, sp, cp;
            sincos_cw(br * z, sz, cz);
            sincos_cw(c1 * t1 + c2 * t2, sp, cp);
            float tx = ibr * (cz * cp - sz * sp), ty = ibr * (cz * sp + sz * cp);
            P[0][0] += tx;
            P[0][1] += ty;
            float b3 = br * sg;
            float f[6] = {1.f - c1 * c1 * ik2, 1.f - c2 * c2 * ik2, 1.f - b3 * b3 * ik2,
                          -c1 * c2 * ik2, -c1 * b3 * ik2, -c2 * b3 * ik2};
#pragma unroll
            for (int e = 0; e < 6; ++e) {
                P[1 + e][0] += f[e] * tx;
                P[1 + e][1] += f[e] * ty;
            }
        }
        // row bounds in float with a one-index margin
        const float a1f = (float)a.a1;
        const float Rmf = sqrtf(R2mf);
        const int n1a = max(a.n1lo, (int)floorf(-a1f - Rmf) - 1), n1b = min(a.n1hi, (int)ceilf(-a1f + Rmf) + 1);
        // row slab: the rows split evenly
        const int nr = n1b - n1a + 1;
        const int r_lo = n1a + (slab * nr) / nslab, r_hi = n1a + ((slab + 1) * nr) / nslab - 1;
        for (int n1 = r_lo; n1 <= r_hi; ++n1) {
            const float c1 = a1f + (float)n1;
            const float c1sq = c1 * c1;
            const float remf = R2mf - c1sq;
            if (remf < -1.0f) continue;
            const float srf = sqrtf(fmaxf(remf, 0.f));
            const int n2a = max(a.n2lo, (int)floorf(-a2f - srf) - 1), n2b = min(a.n2hi, (int)ceilf(-a2f + srf) + 1);
            if (n2a > n2b) continue;
            const BetaEntryF *row = tab + (size_t)(n1 - a.n1lo) * W2 - a.n2lo;
            float c2 = a2f + (float)n2b;
            float h[6][2];
#pragma unroll
            for (int e = 0; e < 6; ++e) h[e][0] = h[e][1] = 0.f;
            for (int n2 = n2b; n2 >= n2a; --n2, c2 -= 1.0f) {
                const BetaEntryF be = row[n2];
                // propagating n (summed separately) have bl2 = +inf, so e = 0; no
                // per-lane truncation test (terms beyond the lane's set are below e^{-T})
                const float e = ex2_approx(-be.bl2 * z);
                float wv[6];
                wv[0] = e * be.ib;
                wv[1] = c2 * wv[0];
                wv[2] = c2 * wv[1];
                wv[3] = be.b * e;
                wv[4] = e;
                wv[5] = c2 * e;
#pragma unroll
                for (int e2 = 0; e2 < 6; ++e2) {
                    const float nx = fmaf(h[e2][0], cv, fmaf(-h[e2][1], sv, wv[e2]));
                    const float ny = fmaf(h[e2][0], sv, h[e2][1] * cv);
                    h[e2][0] = nx;
                    h[e2][1] = ny;
                }
            }
            float sp, cp;
            sincos_cw(c1 * t1 + (a2f + (float)n2a) * t2, sp, cp);
            float r[6][2];
#pragma unroll
            for (int e2 = 0; e2 < 6; ++e2) {
                r[e2][0] = cp * h[e2][0] - sp * h[e2][1];
                r[e2][1] = cp * h[e2][1] + sp * h[e2][0];
            }
            const float fxx = 1.f - c1 * c1 * ik2;
            S[0][0] += r[0][0];
            S[0][1] += r[0][1];
            S[1][0] += fxx * r[0][0];
            S[1][1] += fxx * r[0][1];
            S[2][0] += r[0][0] - ik2 * r[2][0];
            S[2][1] += r[0][1] - ik2 * r[2][1];
            S[3][0] += r[0][0] + ik2 * r[3][0];
            S[3][1] += r[0][1] + ik2 * r[3][1];
            S[4][0] += -c1 * ik2 * r[1][0];
            S[4][1] += -c1 * ik2 * r[1][1];
            S[5][0] += -c1 * ik2 * r[4][0];
            S[5][1] += -c1 * ik2 * r[4][1];
            S[6][0] += -ik2 * r[5][0];
            S[6][1] += -ik2 * r[5][1];
        }
        // e^{i 2pi <alpha.m>} (i/8pi^2): the fractional part in double, the phase in float
        double ph = a.a1 * m1 + a.a2 * m2;
        ph -= rint(ph);
        float sl, cl;
        sincospif(2.0f * (float)ph, &sl, &cl);
        const float sc = (float)(1.0 / (8.0 * GF_PI * GF_PI));
        const float2 pre = make_float2(-sl * sc, cl * sc);
        float2 vals[7];
#pragma unroll
        for (int e = 0; e < 6; ++e) {
            const float *s = S[1 + e];
            float2 v;
            if (e < 4)
                v = make_float2(P[1 + e][0] + s[1], P[1 + e][1] - s[0]);
            else
                v = make_float2(P[1 + e][0] + sg * s[0], P[1 + e][1] + sg * s[1]);
            vals[e] = cmulf(pre, v);
        }
        vals[6] = cmulf(pre, make_float2(P[0][0] + S[0][1], P[0][1] - S[0][0]));
        far_deposit(a, 0, w, slab, nslab, ((count + 31) >> 5) * 32, valid, idx, ne, vals);
    }
}

// Chunks per warp of the grid from which a lane takes two targets.
constexpr int FAR_PAIRS = 1;

template <int NF>
__global__ void __launch_bounds__(128, NF == 1 ? 6 : 1) far3d_f32(const __grid_constant__ EvalArgs a)
{
    const int count = *a.nfar, nch = (count + 31) >> 5;
    int *ctr = a.far_count + GF_WORK_SLOT;
    if (NF == 1 && nch >= FAR_PAIRS * (int)(gridDim.x * blockDim.x >> 5)) {
        const int np = (nch + 1) >> 1, S = far_slabs_capped(a, 0, nch, far_slabs(np, FAR_SLABS_MAX / 2, 2));
        for (int t = far_take(ctr, np * S); t >= 0; t = far_take(ctr, np * S)) {
            const int u = 2 * (t / S);
            far3d_f32_helm<2>(a, {nch - 1 - u, nch - 2 - u}, count, t % S, S);
        }
        return;
    }
    const int S = far_chunk_slabs(a, 0, false, nch);
    for (int t = far_take(ctr, nch * S); t >= 0; t = far_take(ctr, nch * S)) {
        const int w = nch - 1 - t / S;
        if constexpr (NF > 1)
            far3d_f32_maxwell(a, w, count, t % S, S);
        else
            far3d_f32_helm<1>(a, {w}, count, t % S, S);
    }
}

// Batched far kernel: one persistent launch for all pairs.  The work items of
// all pairs form one global list (pair after pair, each pair's chunks most
// expensive first, S row slabs per chunk with S from the total chunk count)
// handed out from pair 0's work counter, so no pair waits for another and the
// load stays balanced across pair boundaries.  The taken index only grows, so
// each warp walks the pair list forward.
template <typename R, int NF>
__global__ void __launch_bounds__(256, sizeof(R) == 4 && NF == 1 ? 3 : 1) far3d_batch(const EvalArgs *args, int np)
{
    if (np <= 0) return;
    int tot = 0;
    for (int q = 0; q < np; ++q) tot += (args[q].far_count[0] + 31) >> 5;
    // split Helmholtz sweeps of some length: items of two chunks
    const bool pairs = sizeof(R) == 4 && NF == 1 && tot >= FAR_PAIRS * (int)(gridDim.x * blockDim.x >> 5);
    const int S = pairs ? far_slabs(tot / 2, 4, 2) : far_slabs(tot, sizeof(R) == 8 ? 8 : 4);
    int *ctr = args[0].far_count + GF_WORK_SLOT;
    auto items = [&](int n) { return (pairs ? (n + 63) >> 6 : (n + 31) >> 5) * S; };
    int p = 0, base = 0;
    int count = args[0].far_count[0];
    int nit = items(count);
    for (;;) {
        int t = 0;
        if ((threadIdx.x & 31) == 0) t = atomicAdd(ctr, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        while (p < np && t >= base + nit) {
            base += nit;
            if (++p < np) {
                count = args[p].far_count[0];
                nit = items(count);
            }
        }
        if (p >= np) return;
        const int u = t - base, nch = (count + 31) >> 5;
        if constexpr (sizeof(R) == 8)
            far3d_f64_chunk<NF, true>(args[p], nch - 1 - u / S, count, u % S, S);
        else if constexpr (NF > 1)
            far3d_f32_maxwell(args[p], nch - 1 - u / S, count, u % S, S);
        else if (pairs)
            far3d_f32_helm<2>(args[p], {nch - 1 - 2 * (u / S), nch - 2 - 2 * (u / S)}, count, u % S, S);
        else
            far3d_f32_helm<1>(args[p], {nch - 1 - u / S}, count, u % S, S);
    }
}

// ---------------------------------------------------------------------------
// 2D far branch (|x2| > c): G = e^{i2pi alpha m} (i/4pi) sum_n beta_n^{-1} e^{i alpha_n t + i beta_n |x2|}
// (ei), terms and sums in double for both precisions.
// GF_OUT_GRAD adds the term-by-term derivatives (i alpha_n/beta_n) E_n and
// i sgn(x2) E_n; GF_OUT_HESSDIFF sums, over the indices of both wave numbers'
// truncation sets, -alpha_n^2 (E_n/beta_n - E'_n/beta'_n), -alpha_n sgn (E_n - E'_n)
// and -(beta_n E_n - beta'_n E'_n) (primes: k2).
// OUT: the output kind (GF_OUT_G, GF_OUT_GRAD or GF_OUT_HESSDIFF), one kernel
// instance each so that the plain G sum carries none of the others' registers.
//
// The double pipe bounds it.  A CTA keeps b_n = |beta_n|, 1/b_n and alpha_n of the index
// range of |x2| = c in shared memory, and e^{-j/64}.  The
// evanescent indices' weights are real, so their sums sum_n w_n v^n, v = e^{it}, go by Horner's rule
// in v^4, four terms to a group; e^{-b|x2|} is the table's entry and a degree-6 polynomial.
// About 15, 21 and 38 double operations a term for G, GRAD and HESSDIFF against 60,
// 65 and 120 with a square root, a quotient, exp and a phase step in every term.  The
// propagating indices are summed apart.  A target is shared by as many
// lanes (1 .. 32, a run of indices each) as give an SM up to four warps, more only where the
// runs are long (lgmin): they would cost more than they hide (two sines and the powers of v per
// lane).  A CTA orders its targets by |x2|, so that the lanes of a warp have runs of about the
// same length.  Short lists and some long index ranges go to far2d_warps.  10,000 targets, G
// 111 -> 49 us; 100,000: GRAD 998 -> 256, HESSDIFF 1597 -> 455 us (without the ordering and the even
// shares of the CTAs 479 and 861).
// ---------------------------------------------------------------------------
constexpr int F2_THR = 512;
constexpr int F2_TAB = 1024;            // indices kept (the middle of the range)
constexpr int F2_Y = 48;                // the exponential's table, y < F2_Y
constexpr int F2_S = 64;                // steps per unit of y
// Indices of a lane's run to either side of the middle at |x2| = c: with a small c the targets nearest the slab have
// thousands, and a warp of them would outlast all others (c = 0.01, 4000 indices, 50,000 targets with |x2| <= 0.3: 11.1 ms with
// a lane a target).  Default plans have 67.
constexpr int F2_RUN = 512;

// (|beta_n|, 1/|beta_n|), the first negative for a propagating n.
__device__ __forceinline__ double2 ei_beta(double kk, double c1)
{
    const double aa = fabs(c1), b = sqrt(fabs(aa - kk) * (aa + kk));
    return make_double2(aa > kk ? b : -b, 1.0 / b);
}

// e^{-y}, y >= 0: y = j/64 + r, |r| <= 1/128, T[j] = e^{-j/64}; truncation r^7/5040 < 4e-19.
// Propagating indices come with y = -|beta||x2| and discard the result; from 2^25 on the
// low word of their j has wrapped to any value, so the index is bounded on both sides.
__device__ __forceinline__ double exp_neg_tab(double y, const double *T)
{
    const double w = fma(y, (double)F2_S, 6755399441055744.0);
    const int j = __double2loint(w);
    if (y >= (double)F2_Y) return exp(-y);
    const double r = fma(w - 6755399441055744.0, -1.0 / F2_S, y);
    double p = fma(r, 1.0 / 720.0, -1.0 / 120.0);
    p = fma(p, r, 1.0 / 24.0);
    p = fma(p, r, -1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p, r, -1.0);
    const double t = T[min(max(j, 0), F2_Y * F2_S)];
    return fma(t, p * r, t);
}

template <typename R, int OUT>
__global__ void __launch_bounds__(F2_THR) far2d(const __grid_constant__ EvalArgs a, int lgmin)
{
    typedef typename cplx_t<R>::T C;
    constexpr bool hess = OUT == GF_OUT_HESSDIFF, grad = OUT == GF_OUT_GRAD;
    constexpr int ne = OUT == GF_OUT_G ? 1 : 3;
    extern __shared__ double f2s[];
    __shared__ double hi[F2_Y + 1], lo[F2_S];
    __shared__ int bins[32], order[F2_THR];
    double *T = f2s, *tc = T + F2_Y * F2_S + 1;
    double2 *tb = reinterpret_cast<double2 *>(f2s + ((F2_Y * F2_S + 1 + F2_TAB + 1) & ~1)), *tb2 = tb + F2_TAB;
    C *out = reinterpret_cast<C *>(a.out);
    const int count = *a.far_count;
    if (count == 0) return;
    const double kmax = (hess && a.k2 > a.k) ? a.k2 : a.k;
    // the kept indices: the range at |x2| = c, or its middle
    const double Tc = a.T / a.c, Rc = sqrt(kmax * kmax + Tc * Tc);
    const int mid = (int)rint(-a.a1), hw = (int)fmin(ceil(Rc) + 5.0, (double)(F2_TAB / 2));
    const int tlo = mid - hw, tn = 2 * hw;
    for (int i = threadIdx.x; i <= F2_Y; i += blockDim.x) hi[i] = exp(-(double)i);
    for (int i = threadIdx.x; i < F2_S; i += blockDim.x) lo[i] = exp(-(double)i / F2_S);
    for (int i = threadIdx.x; i < tn; i += blockDim.x) {
        const double c1 = a.a1 + (tlo + i);
        tc[i] = c1;
        tb[i] = ei_beta(a.k, c1);
        if (hess) tb2[i] = ei_beta(a.k2, c1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= F2_Y * F2_S; i += blockDim.x) T[i] = hi[i / F2_S] * lo[i % F2_S];
    __syncthreads();
    // propagating indices: at most one past either end is not (skipped there)
    int plo[2], phi[2];
#pragma unroll
    for (int q = 0; q < (hess ? 2 : 1); ++q) {
        const double kk = q ? a.k2 : a.k;
        plo[q] = (int)ceil(-a.a1 - kk - 1e-9 * kk);
        phi[q] = (int)floor(-a.a1 + kk + 1e-9 * kk);
    }
    // the CTA's share of the targets; lanes per target
    const int share = (count + gridDim.x - 1) / gridDim.x, c0 = blockIdx.x * share, c1e = min(count, c0 + share);
    int lgl = lgmin;
    while (lgl < 5 && (share << (lgl + 1)) <= 128) ++lgl;
    const int lpt = 1 << lgl, sub = threadIdx.x & (lpt - 1), chunk = F2_THR >> lgl;
    for (int base = c0; base < c1e; base += chunk) {
        // order by the length of the sums, R ~ 1/|x2|: 32 bins
        const int nt = min(chunk, c1e - base);
        __syncthreads();
        if (threadIdx.x < 32) bins[threadIdx.x] = 0;
        __syncthreads();
        int bin = 0, pos = 0, mine = 0;
        if ((int)threadIdx.x < nt) {
            mine = a.far_idx[base + threadIdx.x];
            bin = min(31, (int)(32.f * (float)a.c / fabsf((float)a.x[2 * (size_t)mine + 1])));
            pos = atomicAdd(&bins[bin], 1);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            const int v = bins[threadIdx.x];
            int sum = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, sum, o);
                if ((int)threadIdx.x >= o) sum += u;
            }
            bins[threadIdx.x] = sum - v;
        }
        __syncthreads();
        if ((int)threadIdx.x < nt) order[bins[bin] + pos] = mine;
        __syncthreads();
        const int slot = threadIdx.x >> lgl;
        if (__ballot_sync(0xffffffffu, slot < nt) == 0u) continue;
        const int idx = order[slot < nt ? slot : nt - 1];
        const double x1 = a.x[2 * (size_t)idx], x2 = a.x[2 * (size_t)idx + 1];
        double t, m;
        reduce_period(x1, t, m);
        const double z = fabs(x2), sg = x2 >= 0.0 ? 1.0 : -1.0;
        const double Tz = a.T * (1.0 / z);
        const double Rr = sqrt(kmax * kmax + Tz * Tz);
        const int na = (int)floor(-a.a1 - Rr), nb = (int)ceil(-a.a1 + Rr);
        // runs of `per` indices outwards from mid, n = mid + k and n = mid - 1 - k: even lanes up, odd
        // lanes down, one lane alone both; anchored at their inner ends, so that the
        // large terms have small powers of v (groups of four: the outermost run may pass the
        // truncation, which only adds accuracy)
        const int lgr = lgl ? lgl - 1 : 0, kmx = max(nb - mid + 1, mid - na);
        const int per = ((kmx + (1 << lgr) - 1) >> lgr) + 3 & ~3, k0 = (sub >> 1) * per;
        double sv, cv;
        sincos(t, &sv, &cv);
        const double v2x = cv * cv - sv * sv, v2y = 2.0 * cv * sv;
        const double v3x = v2x * cv - v2y * sv, v3y = v2x * sv + v2y * cv;
        const double v4x = v2x * v2x - v2y * v2y, v4y = 2.0 * v2x * v2y;
        double acc[ne][2];
#pragma unroll
        for (int e = 0; e < ne; ++e) acc[e][0] = acc[e][1] = 0.0;
        for (int q = 0; q < (lgl ? 1 : 2); ++q) {
            const bool down = lgl ? sub & 1 : q;
            const int n0 = down ? mid - 1 - k0 : mid + k0, d = down ? -1 : 1;
            if (k0 >= kmx) continue;
            const double dsv = down ? -sv : sv, w2y = down ? -v2y : v2y, w3y = down ? -v3y : v3y, w4y = down ? -v4y : v4y;
            double h[ne][2];
#pragma unroll
            for (int e = 0; e < ne; ++e) h[e][0] = h[e][1] = 0.0;
            for (int g = per - 4; g >= 0; g -= 4) {
                double w[ne][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int n = n0 + d * (g + u), i = n - tlo;
                    double c1;
                    double2 q1, q2 = make_double2(0.0, 0.0);
                    if ((unsigned)i < (unsigned)tn) {
                        q1 = tb[i];
                        c1 = ne > 1 ? tc[i] : 0.0;
                        if (hess) q2 = tb2[i];
                    } else {
                        c1 = a.a1 + n;
                        q1 = ei_beta(a.k, c1);
                        if (hess) q2 = ei_beta(a.k2, c1);
                    }
                    // propagating indices weigh zero (the sign tested on the high word, off the double pipe)
                    const double ex = exp_neg_tab(q1.x * z, T), e = __double2hiint(q1.x) > 0 ? ex : 0.0;
                    if constexpr (!hess) {
                        w[0][u] = e * q1.y;
                        if constexpr (grad) {
                            w[1][u] = c1 * w[0][u];
                            w[2][u] = e;
                        }
                    } else {
                        const double ex2 = exp_neg_tab(q2.x * z, T), e2 = __double2hiint(q2.x) > 0 ? ex2 : 0.0;
                        w[0][u] = c1 * c1 * fma(e, q1.y, -(e2 * q2.y));
                        w[1][u] = c1 * (e - e2);
                        w[2][u] = fma(q1.x, e, -(q2.x * e2));
                    }
                }
#pragma unroll
                for (int e = 0; e < ne; ++e) {
                    const double x = fma(w[e][3], v3x, fma(w[e][2], v2x, fma(w[e][1], cv, w[e][0])));
                    const double y = fma(w[e][3], w3y, fma(w[e][2], w2y, w[e][1] * dsv));
                    const double nx = fma(h[e][0], v4x, fma(-h[e][1], w4y, x));
                    h[e][1] = fma(h[e][0], w4y, fma(h[e][1], v4x, y));
                    h[e][0] = nx;
                }
            }
            // the run's phase e^{i alpha_{n0} t} and the factors of E_n = e^{-b|x2|} e^{i alpha_n t}, 1/beta_n = -i/b:
            // G: -i; GRAD: 1, i sgn; HESSDIFF: i, -sgn, -i
            double sp, cp;
            sincos((a.a1 + n0) * t, &sp, &cp);
#pragma unroll
            for (int e = 0; e < ne; ++e) {
                const double x = h[e][0] * cp - h[e][1] * sp, y = h[e][0] * sp + h[e][1] * cp;
                if constexpr (!hess) {
                    acc[e][0] += e == 0 ? y : e == 1 ? x : -sg * y;
                    acc[e][1] += e == 0 ? -x : e == 1 ? y : sg * x;
                } else {
                    acc[e][0] += e == 0 ? -y : e == 1 ? -sg * x : y;
                    acc[e][1] += e == 0 ? x : e == 1 ? -sg * y : -x;
                }
            }
        }
        // propagating indices of k (and, with the opposite sign, of k2)
#pragma unroll
        for (int q = 0; q < (hess ? 2 : 1); ++q) {
            const double kk = q ? a.k2 : a.k, s = q ? -1.0 : 1.0;
            for (int n = plo[q] + sub; n <= phi[q]; n += lpt) {
                const double c1 = a.a1 + n;
                const int i = n - tlo;
                const double2 bq = (unsigned)i < (unsigned)tn ? (q ? tb2 : tb)[i] : ei_beta(kk, c1);
                if (__double2hiint(bq.x) > 0) continue;
                const double b = -bq.x, ib = bq.y;
                double sz, cz;
                sincos(fma(b, z, c1 * t), &sz, &cz);
                if constexpr (!hess) {
                    acc[0][0] = fma(cz, ib, acc[0][0]);
                    acc[0][1] = fma(sz, ib, acc[0][1]);
                    if constexpr (grad) {
                        const double ci = c1 * ib;
                        acc[1][0] = fma(-ci, sz, acc[1][0]);
                        acc[1][1] = fma(ci, cz, acc[1][1]);
                        acc[2][0] = fma(-sg, sz, acc[2][0]);
                        acc[2][1] = fma(sg, cz, acc[2][1]);
                    }
                } else {
                    const double f0 = -s * c1 * c1 * ib, f1 = -s * c1 * sg, f2 = -s * b;
                    acc[0][0] = fma(f0, cz, acc[0][0]);
                    acc[0][1] = fma(f0, sz, acc[0][1]);
                    acc[1][0] = fma(f1, cz, acc[1][0]);
                    acc[1][1] = fma(f1, sz, acc[1][1]);
                    acc[2][0] = fma(f2, cz, acc[2][0]);
                    acc[2][1] = fma(f2, sz, acc[2][1]);
                }
            }
        }
        for (int o = 1; o < lpt; o <<= 1)
#pragma unroll
            for (int e = 0; e < ne; ++e) {
                acc[e][0] += __shfl_xor_sync(0xffffffffu, acc[e][0], o);
                acc[e][1] += __shfl_xor_sync(0xffffffffu, acc[e][1], o);
            }
        if (sub == 0 && slot < nt) {
            const double2 lat = lattice_phase(a.a1, m, 0.0, 0.0);
            const double2 pre = cmul(lat, make_double2(0.0, 0.25 / GF_PI));
            for (int e = 0; e < ne; ++e)
                store_out(out + (size_t)idx * ne + e, cmul(pre, make_double2(acc[e][0], acc[e][1])));
        }
    }
}

// Lists by a warp per target, lanes over the indices, every term by itself.  Short lists: no tables to fill and no
// order to make, which is most of far2d's time there: whole evaluations of 1 / 1000 / 3000 targets (40% far) G 48 / 70 / 95
// us against far2d's 59 / 81 / 99, GRAD 50 / 80 / 108 against 64 / 91 / 110, HESSDIFF 59 / 92 / 137 against 66 / 97 / 131.
// And lists whose targets near |x2| = c have more indices R than far2d's table, up to 16 R targets or where most of the
// indices propagate (far2d passes them twice): 50,000 targets |x2| <= 0.3, c = 0.01 (R = 4000) 5.6 ms against 6.8, c = 0.002 9.6
// against 14.7, c = 0.03 3.7 against 3.2; |x2| <= 1, c = 0.6, k = 900 4.4 against 6.1, k = 300 1.74 against 1.53.
constexpr int64_t F2_SHORT = 2048;      // targets

// -1: by a warp per target; else far2d's least number of lanes a target (its logarithm).
inline int far2d_route(const EvalArgs &a)
{
    const double kmax = a.which == GF_OUT_HESSDIFF ? fmax(a.k, a.k2) : a.k, Tc = a.T / a.c, R = sqrt(kmax * kmax + Tc * Tc);
    if (a.n <= F2_SHORT || (R > F2_TAB / 2 - 5 && ((double)a.n <= 16.0 * R || kmax > F2_TAB / 2 - 5))) return -1;
    int lg = 0;
    while (lg < 5 && R > (double)(F2_RUN << std::max(lg - 1, 0))) ++lg;
    return lg;
}

template <typename R, int OUT>
__global__ void __launch_bounds__(128) far2d_warps(const __grid_constant__ EvalArgs a)
{
    typedef typename cplx_t<R>::T C;
    constexpr int ne = OUT == GF_OUT_G ? 1 : 3;
    constexpr bool hess = OUT == GF_OUT_HESSDIFF, grad = OUT == GF_OUT_GRAD;
    C *out = reinterpret_cast<C *>(a.out);
    const int count = *a.far_count, lane = threadIdx.x & 31;
    const double kmax = (hess && a.k2 > a.k) ? a.k2 : a.k;
    for (int slot = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; slot < count; slot += (gridDim.x * blockDim.x) >> 5) {
        const int idx = a.far_idx[slot];
        const double x1 = a.x[2 * (size_t)idx], x2 = a.x[2 * (size_t)idx + 1];
        double t, m;
        reduce_period(x1, t, m);
        const double z = fabs(x2), sg = x2 >= 0.0 ? 1.0 : -1.0, Tz = a.T * (1.0 / z), Rr = sqrt(kmax * kmax + Tz * Tz);
        const int na = (int)floor(-a.a1 - Rr) - 1, nb = (int)ceil(-a.a1 + Rr) + 1;
        // e^{i alpha_n t} by steps of 32 indices
        double2 p, step;
        sincos((a.a1 + (na + lane)) * t, &p.y, &p.x);
        sincos(32.0 * t, &step.y, &step.x);
        double acc[ne][2];
#pragma unroll
        for (int e = 0; e < ne; ++e) acc[e][0] = acc[e][1] = 0.0;
        // s E_n/beta_n, s E_n and s beta_n E_n of one wave number, E_n = e^{i beta_n |x2|} e^{i alpha_n t},
        // times what the output has of each
        auto add = [&](double kk, double c1, double s) {
            const double2 q = ei_beta(kk, c1);
            const bool prop = q.x < 0.0;  // beta_n = -q.x, else i q.x
            double2 f;
            if (prop)
                sincos(-q.x * z, &f.y, &f.x);
            else
                f = make_double2(exp(-q.x * z), 0.0);
            const double2 E = cscale(cmul(f, p), s);
            const double2 Eb = prop ? cscale(E, q.y) : make_double2(E.y * q.y, -E.x * q.y);
            if constexpr (!hess) {
                acc[0][0] += Eb.x;
                acc[0][1] += Eb.y;
                if constexpr (grad) {
                    acc[1][0] -= c1 * Eb.y;  // i alpha_n E_n/beta_n
                    acc[1][1] += c1 * Eb.x;
                    acc[2][0] -= sg * E.y;   // i sgn E_n
                    acc[2][1] += sg * E.x;
                }
            } else {
                acc[0][0] -= c1 * c1 * Eb.x;
                acc[0][1] -= c1 * c1 * Eb.y;
                acc[1][0] -= c1 * sg * E.x;
                acc[1][1] -= c1 * sg * E.y;
                acc[2][0] += prop ? q.x * E.x : q.x * E.y;  // -beta_n E_n
                acc[2][1] += prop ? q.x * E.y : -q.x * E.x;
            }
        };
        for (int n = na + lane; n <= nb; n += 32, p = cmul(p, step)) {
            const double c1 = a.a1 + n;
            if (fabs(c1) > Rr) continue;
            add(a.k, c1, 1.0);
            if constexpr (hess) add(a.k2, c1, -1.0);
        }
#pragma unroll
        for (int e = 0; e < ne; ++e)
            for (int o = 16; o > 0; o >>= 1) {
                acc[e][0] += __shfl_xor_sync(0xffffffffu, acc[e][0], o);
                acc[e][1] += __shfl_xor_sync(0xffffffffu, acc[e][1], o);
            }
        if (lane == 0) {
            const double2 pre = cmul(lattice_phase(a.a1, m, 0.0, 0.0), make_double2(0.0, 0.25 / GF_PI));
            for (int e = 0; e < ne; ++e) store_out(out + (size_t)idx * ne + e, cmul(pre, make_double2(acc[e][0], acc[e][1])));
        }
    }
}

template <typename R, int OUT>
cudaError_t launch_far2d(const EvalArgs &a, int nsm, cudaStream_t s)
{
    const int lgmin = far2d_route(a);
    if (lgmin < 0) {
        far2d_warps<R, OUT><<<(int)std::min<int64_t>((a.n + 3) / 4, (int64_t)nsm * 16), 128, 0, s>>>(a);
        return cudaSuccess;
    }
    const size_t sm = sizeof(double) * ((F2_Y * F2_S + 1 + F2_TAB + 1) & ~1) + sizeof(double2) * F2_TAB * (OUT == GF_OUT_HESSDIFF ? 2 : 1);
    cudaError_t e = cudaFuncSetAttribute(far2d<R, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    far2d<R, OUT><<<nsm, F2_THR, sm, s>>>(a, lgmin);
    return cudaSuccess;
}

// Persistent far grid: as many 128-thread CTAs as are resident at once (a
// grid beyond that would leave the extra CTAs waiting for a second wave).
template <void (*K)(EvalArgs)>
int resident_grid(int nsm)
{
    static const int per = [] {
        int v = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, K, 128, 0) != cudaSuccess || v < 1) {
            cudaGetLastError();
            v = 1;
        }
        return v;
    }();
    return per * nsm;
}

// The same for the near list: no more CTAs than the targets have tiles (100,000 targets: 62 -> 56 us with the
// tiles dealt out over the CTAs first).
template <void (*K)(const EvalArgs)>
int near_grid(int64_t n, int nsm)
{
    const int64_t want = n / 32 + 2;
    return (int)std::min<int64_t>(want, resident_grid<K>(nsm));
}

// Concurrent far kernels of a Helmholtz double-precision plan: the double
// kernel gives up FAR_F64_DROP of its resident CTAs per SM, and the float-tail
// kernel (64-thread CTAs) fills the registers left free, so that both run at
// once on every SM.
constexpr int FAR_F64_DROP = 1;

struct FarShare {
    int f64, tail;  // resident CTAs per SM of each kernel
};

FarShare far_share()
{
    FarShare sh{1, 1};
    int dev = 0, regs_sm = 65536, per = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
    cudaFuncAttributes fa, ta;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, far3d_f64<1, false>, 128, 0) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, far3d_f64<1, false>) != cudaSuccess ||
        cudaFuncGetAttributes(&ta, far3d_tail<1>) != cudaSuccess) {
        cudaGetLastError();
        return sh;
    }
    // registers are allocated per warp in units of 8 per thread
    auto cta_regs = [](int regs, int threads) { return (regs + 7) / 8 * 8 * 32 * ((threads + 31) / 32); };
    sh.f64 = per > FAR_F64_DROP ? per - FAR_F64_DROP : 1;
    sh.tail = (regs_sm - sh.f64 * cta_regs(fa.numRegs, 128)) / cta_regs(ta.numRegs, 64);
    if (sh.tail < 1) sh.tail = 1;
    return sh;
}

// The double sums and float tails of a double-precision plan's far series.
// With a fork (Helmholtz only), the tails run on the side stream alongside the
// double kernel, with the resident CTAs split by far_share; otherwise (and for
// Maxwell plans, whose double kernel leaves too few registers) after it, at full
// occupancy.
template <int NF>
cudaError_t launch_far_f64(const EvalArgs &a, int nsm, cudaStream_t s, const EvalFork *fork)
{
    if (NF != 1) fork = nullptr;
    if (!fork) {
        far3d_f64<NF, false><<<resident_grid<far3d_f64<NF, false>>(nsm), 128, 0, s>>>(a);
        far3d_tail<NF><<<resident_grid<far3d_tail<NF>>(nsm), 128, 0, s>>>(a);
        return cudaSuccess;
    }
    static const FarShare sh = far_share();
    cudaError_t e;
    if ((e = cudaEventRecord(fork->fork, s)) != cudaSuccess || (e = cudaStreamWaitEvent(fork->aux, fork->fork, 0)) != cudaSuccess)
        return e;
    far3d_f64<NF, false><<<sh.f64 * nsm, 128, 0, s>>>(a);
    far3d_tail<NF><<<sh.tail * nsm, 64, 0, fork->aux>>>(a);
    if ((e = cudaEventRecord(fork->join, fork->aux)) != cudaSuccess) return e;
    return cudaStreamWaitEvent(s, fork->join, 0);
}

// The far list, bucket-sorted: stable when the evaluation brought segment
// scratch, else from the appended list.
void launch_far_list(const EvalArgs &a, int nsm, cudaStream_t s)
{
    if (a.seghist) {
        const int blocks = (a.nseg + SEG_WARPS - 1) / SEG_WARPS;
        far_seg_scan<<<GF_FAR_BUCKETS / 32, 1024, 0, s>>>(a);
        far_seg_scatter<<<blocks, 32 * SEG_WARPS, 0, s>>>(a);
    } else {
        far_scatter<<<nsm * 2, 256, 0, s>>>(a);
    }
}

template <typename R>
cudaError_t launch_eval_t(const EvalArgs &a0, cudaStream_t s, cudaEvent_t ev_mid, const EvalFork *fork)
{
    EvalArgs a = a0;
    a.nfar = a.far_count;
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = (a.n + 255) / 256;
    if (blocks > (int64_t)nsm * 16) blocks = (int64_t)nsm * 16;
    if (blocks < 1) blocks = 1;
    if (a.dim == 2) {
        if (a.nf == 1)
            near2d<R, 1><<<(int)blocks, 256, 0, s>>>(a);
        else if (a.nf == 3)
            near2d<R, 3><<<(int)blocks, 256, 0, s>>>(a);
        else
            near2d<R, 6><<<(int)blocks, 256, 0, s>>>(a);
        if (ev_mid) cudaEventRecord(ev_mid, s);
        cudaError_t e = a.which == GF_OUT_GRAD       ? launch_far2d<R, GF_OUT_GRAD>(a, nsm, s)
                        : a.which == GF_OUT_HESSDIFF ? launch_far2d<R, GF_OUT_HESSDIFF>(a, nsm, s)
                                                     : launch_far2d<R, GF_OUT_G>(a, nsm, s);
        if (e != cudaSuccess) return e;
    } else if (a.nf == 1) {
        // with a near list: classify, then the near targets in full warps
        if (a.near_idx) {
            classify_segs<R, 1><<<std::min(a.nseg, 4 * nsm), CLS_THR, 0, s>>>(a);
            near3d_list<R, 1><<<near_grid<near3d_list<R, 1>>(a.n, nsm), 32 * NEAR_WARPS, 0, s>>>(a);
        } else {
            near3d<R, 1><<<(int)blocks, 256, 0, s>>>(a);
        }
        if (ev_mid) cudaEventRecord(ev_mid, s);
        launch_far_list(a, nsm, s);
        if (a.mma) {
            cudaError_t e = gf_launch_far_product(a, sizeof(R) == 8 ? GF_FP64 : GF_FP32_SPLIT, nsm, s);
            if (e != cudaSuccess) return e;
        }
        if (sizeof(R) == 8) {
            cudaError_t e = launch_far_f64<1>(a, nsm, s, fork);
            if (e != cudaSuccess) return e;
        } else
            far3d_f32<1><<<resident_grid<far3d_f32<1>>(nsm), 128, 0, s>>>(a);
    } else {
        if (a.near_idx) {
            classify_segs<R, 7><<<std::min(a.nseg, 4 * nsm), CLS_THR, 0, s>>>(a);
            near3d_list<R, 7><<<near_grid<near3d_list<R, 7>>(a.n, nsm), 32 * NEAR_WARPS, 0, s>>>(a);
        } else {
            near3d<R, 7><<<(int)blocks, 256, 0, s>>>(a);
        }
        if (ev_mid) cudaEventRecord(ev_mid, s);
        launch_far_list(a, nsm, s);
        if (a.mma) {
            cudaError_t e = gf_launch_far_product(a, sizeof(R) == 8 ? GF_FP64 : GF_FP32_SPLIT, nsm, s);
            if (e != cudaSuccess) return e;
        }
        if (sizeof(R) == 8) {
            cudaError_t e = launch_far_f64<7>(a, nsm, s, fork);
            if (e != cudaSuccess) return e;
        } else
            far3d_f32<7><<<resident_grid<far3d_f32<7>>(nsm), 128, 0, s>>>(a);
    }
    gf_count_launch(a.dim == 2 ? 2 : (sizeof(R) == 8 ? 4 : 3) + (a.near_idx ? 2 : 0));
    return cudaGetLastError();
}

template <typename R, int NF>
cudaError_t launch_eval_batch_nf(const EvalBatch &b, cudaStream_t s)
{
    // classification, then the near targets in full warps
    int dev = 0, per = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, near3d_list_batch<R, NF>, 32 * NEAR_WARPS, 0) != cudaSuccess || per < 1) {
        cudaGetLastError();
        per = 1;
    }
    classify_batch<R, NF><<<b.grid_near, CLS_THR, 0, s>>>(b.args, b.prefix, b.np);
    near3d_list_batch<R, NF><<<per * nsm, 32 * NEAR_WARPS, 0, s>>>(b.args, b.np);
    far_scatter_batch<<<b.grid_scatter, 256, 0, s>>>(b.args, b.np, b.scatter_per_pair);
    far3d_batch<R, NF><<<b.grid_far, b.block_far, 0, s>>>(b.args, b.np);
    gf_count_launch(4);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_eval_batch_t(const EvalBatch &b, cudaStream_t s)
{
    return b.nf == 1 ? launch_eval_batch_nf<R, 1>(b, s) : launch_eval_batch_nf<R, 7>(b, s);
}

}  // namespace

cudaError_t gf_launch_eval_batch(const EvalBatch &b, int precision, cudaStream_t s)
{
    return precision == GF_FP64 ? launch_eval_batch_t<double>(b, s) : launch_eval_batch_t<float>(b, s);
}

cudaError_t gf_launch_series_tables(const EvalArgs &a, int precision, double2 *exptab, longlong2 *trig, PropEntry *prop, int *nprop,
                                    const int pbox[4], cudaStream_t s)
{
    const int4 pb = make_int4(pbox[0], pbox[1], pbox[2], pbox[3]);
    if (precision == GF_FP64)
        series_tables<BetaEntry><<<256, 256, 0, s>>>(a, (BetaEntry *)const_cast<void *>(a.btab), exptab, trig, prop, nprop, pb);
    else
        series_tables<BetaEntryF><<<256, 256, 0, s>>>(a, (BetaEntryF *)const_cast<void *>(a.btab), exptab, trig, prop, nprop, pb);
    gf_count_launch(1);
    return cudaGetLastError();
}

cudaError_t gf_launch_eval(const EvalArgs &a, int precision, cudaStream_t s, cudaEvent_t ev_mid, const EvalFork *fork)
{
    return precision == GF_FP64 ? launch_eval_t<double>(a, s, ev_mid, fork) : launch_eval_t<float>(a, s, ev_mid, fork);
}
