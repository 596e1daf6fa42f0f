// Tables of the coefficients' radial transforms (3D h(s); 2D Hankel transforms) by
// Taylor sums: each panel's polynomial from the derivatives at its centre, instead
// of transforming the quadrature at fifteen points of every panel.
//
// At s = cen + x, |x| <= 1, a transform sum_m w_m f(s r_m) has the Taylor coefficients
//   a_p = (1/p!) sum_m w_m r_m^p f^(p)(cen r_m),
// and f^(p) is a sine or cosine, or a combination of Bessel functions J_n(cen r_m) of
// nearby orders (2 J_n' = J_{n-1} - J_{n+1}).  One sincos, or one J0, J1 and a recurrence,
// per panel and node thus replace fifteen evaluations (sixty with the derivative plans'
// J2 and J3).  For r_m <= 1 the terms beyond p = 18 are below 1e-17; powers 15 .. 18 are
// folded into the lower ones by Chebyshev economization (x^p -> x^p - 2^{1-p} T_p, at
// most 1e-16 here), so that the stored degree stays GF_HDEG.  Plans with 2 eps > 1 keep the
// interpolation at Chebyshev points (synth.cu).
//
// Before, the double pipe was the limit (15 points a panel); now the chains are: J0 or J1, the
// recurrence, the sums.  Cold, per plan: 3D 128 x 128 x 64 (71 panels, 64 nodes) 44 -> 21 us;
// 2D 64 x 64 (57 panels) 68 -> 32 us; 2D derivatives 256 x 256 (161 panels, 240 nodes) 953 -> 108 us.
#include "gf_internal.cuh"

namespace {

constexpr int PT = 18;        // highest Taylor power
constexpr int P0MAX = 26;     // highest power of the 3D panel at s = 0
constexpr int NJ = PT + 4;    // Bessel orders 0 .. 21 (J3 differentiated 18 times)
constexpr int NQ = PT + 3;    // node powers 0 .. 20 (weights r^2)

// T_k by powers of x, and x^15 .. x^26 folded into degree 14.
struct Economy {
    double e[P0MAX - GF_HDEG][GF_HDEG + 1];
};
constexpr Economy economy()
{
    double T[P0MAX + 1][P0MAX + 1] = {};
    T[0][0] = 1.0;
    T[1][1] = 1.0;
    for (int k = 2; k <= P0MAX; ++k)
        for (int t = 0; t <= k; ++t) T[k][t] = (t ? 2.0 * T[k - 1][t - 1] : 0.0) - T[k - 2][t];
    Economy E{};
    for (int P = GF_HDEG + 1; P <= P0MAX; ++P) {
        double v[P0MAX + 1] = {};
        v[P] = 1.0;
        for (int p = P; p > GF_HDEG; --p) {
            const double c = v[p] / T[p][p];
            for (int t = 0; t <= p; ++t) v[t] -= c * T[p][t];
        }
        for (int t = 0; t <= GF_HDEG; ++t) E.e[P - GF_HDEG - 1][t] = v[t];
    }
    return E;
}
__device__ const Economy c_econ = economy();

// C(p, j) for p <= 26 (exact), 1/p!.
struct Binomials {
    double c[P0MAX + 1][P0MAX + 1], ifact[P0MAX + 2];
};
constexpr Binomials binomials()
{
    Binomials B{};
    for (int p = 0; p <= P0MAX; ++p) {
        B.c[p][0] = 1.0;
        for (int j = 1; j <= p; ++j) B.c[p][j] = B.c[p - 1][j - 1] + (j < p ? B.c[p - 1][j] : 0.0);
    }
    double f = 1.0;
    for (int p = 0; p <= P0MAX + 1; ++p) {
        if (p) f *= p;
        B.ifact[p] = 1.0 / f;
    }
    return B;
}
__device__ const Binomials c_bin = binomials();

// The sums over the nodes of one 2D panel, (set, order n, power q): set 0 the J0
// transform (n <= q, n + q even), set 1 the J1 transform (n <= q + 1, n + q odd), set 2 the
// derivative plans' five (n + q odd).
struct Combos {
    int n01, n;
    unsigned char set[448], ord[448], pw[448];
};
constexpr Combos combos()
{
    Combos C{};
    for (int s = 0; s < 3; ++s) {
        if (s == 2) C.n01 = C.n;
        for (int n = 0; n < NJ; ++n)
            for (int q = 0; q < (s == 2 ? NQ : PT + 1); ++q) {
                if (((n + q + (s ? 1 : 0)) & 1) || (s == 0 && n > q) || (s == 1 && n > q + 1)) continue;
                C.set[C.n] = (unsigned char)s;
                C.ord[C.n] = (unsigned char)n;
                C.pw[C.n] = (unsigned char)q;
                ++C.n;
            }
    }
    return C;
}
constexpr Combos COMBOS = combos();
static_assert(COMBOS.n <= 448 && COMBOS.n01 <= 256, "one thread per sum");
__device__ const Combos c_combos = combos();

// Last-axis phases E[b][m] = e^{i q_b t_m}, q_b = j qs (qs = pi / c~) with j = b for b <
// Mlast/2, else b - Mlast (the last-axis frequencies of Eq. (fck-coef)), t_m the Gauss nodes
// of the X' integrals; and the nodes' powers that the panels' sums share:
//   3D: Bp[p][m] = B_m r_m^p / p!, p <= 27;
//   2D: W[p][m] = P0_m r_m^p and then P1_m r_m^p, p <= 18, [2][19][nodes], over Q nodes, or (derivative
//   plans) 2 Q of which the first Q weigh zero, followed by wy_m r_m^q, [21][2 Q].
__global__ void node_tables(NodeTables a)
{
    const int stride = gridDim.x * blockDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (int i = i0; i < a.Mlast * a.Q; i += stride) {
        const int b = i / a.Q, m = i - b * a.Q;
        const int jl = b < a.Mlast / 2 ? b : b - a.Mlast;
        const double q = (double)jl * a.qs;
        double sv, cv;
        sincos(q * a.tt[m], &sv, &cv);
        a.E[i] = make_double2(cv, sv);
        // float copy by node, [m][b] for b <= Mlast/2 (the coefficients formed)
        if (a.Ef && b <= a.Mlast / 2) a.Ef[(size_t)m * GF_EF_ROW(a.Mlast) + b] = make_float2((float)cv, (float)sv);
    }
    if (a.Bp)
        for (int i = i0; i < (P0MAX + 2) * a.Q; i += stride) {
            const int p = i / a.Q, m = i - p * a.Q;
            const double r = a.rr[m];
            double f = c_bin.ifact[p];
            for (int j = 0; j < p; ++j) f *= r;
            a.Bp[i] = make_double2(a.B[m].x * f, a.B[m].y * f);
        }
    if (a.W) {
        const int NM = a.rrd ? 2 * a.Q : a.Q, rows = 2 * (PT + 1) + (a.rrd ? NQ : 0);
        for (int i = i0; i < rows * NM; i += stride) {
            const int row = i / NM, m = i - row * NM, set = row / (PT + 1);
            const double r = a.rrd ? a.rrd[m] : a.rr[m];
            double w;
            int p = row - (set < 2 ? set : 2) * (PT + 1);
            if (set < 2)
                w = m < NM - a.Q ? 0.0 : (set ? a.P1 : a.P0)[m - (NM - a.Q)];
            else
                w = a.wyd[m];
            for (int j = 0; j < p; ++j) w *= r;
            a.W[i] = w;
        }
    }
}

// 3D panels of h(s) = sum_m B_m sin(s r_m)/s: with H(s) = s h(s),
// H_p = sum_m (B_m r_m^p/p!) sin(cen r_m + p pi/2), and h = H/(cen + x) by h_p = (H_p - h_{p-1})/cen;
// the panel at s = 0 from the odd moments, h(1 + x) = sum_j (-1)^j M_j (1 + x)^{2j}.
__global__ void __launch_bounds__(256) panels_3d(const double *rr, const double2 *Bp, int Q, double2 *out, float2 *outf)
{
    extern __shared__ double2 trig[];  // [Q] (cos, sin)(cen r_m)
    __shared__ double2 H[P0MAX + 1];
    const int panel = blockIdx.x, t = threadIdx.x;
    const double cen = 2.0 * panel + 1.0;
    const int np = panel ? PT + 1 : 14, part = t & 7;
    if (panel)
        for (int m = t; m < Q; m += blockDim.x) {
            double s, c;
            sincos(cen * rr[m], &s, &c);
            trig[m] = make_double2(c, s);
        }
    __syncthreads();
    for (int p0 = 0; p0 < np; p0 += 32) {
        // eight lanes a sum
        const int p = p0 + (t >> 3);
        double ax = 0.0, ay = 0.0;
        if (p < np) {
            const double2 *b = Bp + (size_t)(panel ? p : 2 * p + 1) * Q;
#pragma unroll 8
            for (int m = part; m < Q; m += 8) {
                const double2 v = b[m];
                double f = 1.0;
                if (panel) f = (p & 1) ? trig[m].x : trig[m].y;
                ax = fma(v.x, f, ax);
                ay = fma(v.y, f, ay);
            }
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            ax += __shfl_xor_sync(0xffffffffu, ax, o);
            ay += __shfl_xor_sync(0xffffffffu, ay, o);
        }
        // derivatives of sin: sin, cos, -sin, -cos; the moments' signs alternate
        if (p < np && part == 0) {
            const bool neg = panel ? (p & 2) : (p & 1);
            H[p] = neg ? make_double2(-ax, -ay) : make_double2(ax, ay);
        }
    }
    __syncthreads();
    int top = PT;
    if (panel) {
        if (t < 2) {
            double *h = reinterpret_cast<double *>(H) + t;
            const double ic = 1.0 / cen;
            double prev = 0.0;
            for (int p = 0; p <= PT; ++p) {
                prev = (h[2 * p] - prev) * ic;
                h[2 * p] = prev;
            }
        }
        __syncthreads();
    } else {
        // powers of 1 + x to powers of x
        top = P0MAX;
        double vx = 0.0, vy = 0.0;
        if (t <= top)
            for (int j = 13; 2 * j >= t; --j) {
                vx = fma(c_bin.c[2 * j][t], H[j].x, vx);
                vy = fma(c_bin.c[2 * j][t], H[j].y, vy);
            }
        __syncthreads();
        if (t <= top) H[t] = make_double2(vx, vy);
        __syncthreads();
    }
    if (t <= GF_HDEG) {
        double vx = 0.0, vy = 0.0;
        for (int p = top; p > GF_HDEG; --p) {
            vx = fma(c_econ.e[p - GF_HDEG - 1][t], H[p].x, vx);
            vy = fma(c_econ.e[p - GF_HDEG - 1][t], H[p].y, vy);
        }
        vx += H[t].x;
        vy += H[t].y;
        out[(size_t)panel * (GF_HDEG + 1) + t] = make_double2(vx, vy);
        if (outf) outf[(size_t)t * gridDim.x + panel] = make_float2((float)vx, (float)vy);
    }
}

// J_0 .. J_{NJ-1} at u >= 0 into out[n stride]; J0 and J1 are there already for u >= 22: J0, J1 and the upward recurrence
// (stable for n <= u).  Below: the downward one (J. C. P. Miller's algorithm) from an order whose J is
// below 1e-22 of J_{NJ-1}, normalized by J_0 + 2 J_2 + 2 J_4 + ... = 1.  u < 1e-3: the first
// terms of the power series (the downward recurrence could overflow).
__device__ void bessel_orders(double u, double *out, int stride)
{
    if (u >= 22.0) {
        const double iu2 = 2.0 / u;
        double a = out[0], b = out[stride];
        for (int n = 1; n < NJ - 1; ++n) {
            const double c = fma(iu2 * n, b, -a);
            a = b;
            b = c;
            out[(n + 1) * stride] = c;
        }
    } else if (u >= 1e-3) {
        const double iu2 = 2.0 / u;
        double a = 0.0, b = 1e-200, sum = 0.0;  // orders n + 1, n
        for (int n = u < 2.0 ? 36 : 64; n >= 1; --n) {
            if (n < NJ) out[n * stride] = b;
            if (!(n & 1)) sum += b;
            const double c = fma(iu2 * n, b, -a);
            a = b;
            b = c;
        }
        const double nrm = 1.0 / fma(2.0, sum, b);
        out[0] = b * nrm;
        for (int n = 1; n < NJ; ++n) out[n * stride] *= nrm;
    } else {
        const double z = 0.25 * u * u;
        double f = 1.0;
        for (int n = 0; n < NJ; ++n) {
            out[n * stride] = f * (1.0 - z / (n + 1) * (1.0 - z / (2 * (n + 2))));
            f *= 0.5 * u / (n + 1);
        }
    }
}

// X' sums s1, s3 = sum_m W_m e^{-g t_m} (cos, sin)(q_b t_m) of evanescent columns on panels in g: with
// x = g - cen, e^{-g t} = e^{-x tc} e^{-cen t} e^{-x (t - tc)}, tc the middle of the nodes, and the last factor's
// Taylor sum to power 11: |x (t - tc)| <= 0.2, remainder below 1e-17.
constexpr int XB = 16;
__global__ void __launch_bounds__(XB * GF_XDEG1) xprime_panels(NodeTables a, const double *tW, double w, double tc, double2 *out)
{
    extern __shared__ double U[];  // [GF_XDEG1][Q]
    const double cen = (blockIdx.x + 0.5) * w;
    const int Q = a.Q, nh = (a.Mlast >> 1) + 1;
    for (int m = threadIdx.x; m < Q; m += blockDim.x) {
        const double t = a.tt[m], d = tc - t;
        double f = tW[m] * exp(-cen * t);
#pragma unroll
        for (int k = 0; k < GF_XDEG1; ++k) {
            U[k * Q + m] = f * c_bin.ifact[k];
            f *= d;
        }
    }
    __syncthreads();
    const int k = threadIdx.x / XB, b = blockIdx.y * XB + threadIdx.x % XB;
    if (b >= nh) return;
    const double2 *E = a.E + (size_t)b * Q;
    const double *u = U + k * Q;
    double s1[2] = {0.0, 0.0}, s3[2] = {0.0, 0.0};
#pragma unroll 8
    for (int m = 0; m < Q; ++m) {
        const double2 e = __ldg(E + m);
        s1[m & 1] = fma(u[m], e.x, s1[m & 1]);
        s3[m & 1] = fma(u[m], e.y, s3[m & 1]);
    }
    out[((size_t)blockIdx.x * GF_XDEG1 + k) * nh + b] = make_double2(s1[0] + s1[1], s3[0] + s3[1]);
}

constexpr int NC = 128;       // nodes per chunk
constexpr int LD = NC + 1;    // row length in shared memory (conflict-free columns)

// 2D panels.  S_{set,n,q} = sum_m W_{set,q,m} J_n(cen r_m), one thread a sum, then
//   a_p = (2^-p/p!) sum_j (-1)^j C(p,j) S_{nu-p+2j, p+e}
// for the transform of order nu with weight r^e, J_{-n} = (-1)^n J_n:
// (S0, S1) of gf_internal.cuh's hcheb, and with DERIV the tables
//   0: (Q1, R0) = (sum wy J1(s r), sum wy J0(s r) r)
//   1: (R2, S1) = (sum wy J2(s r) r, sum wy J1(s r) r^2)
//   2: (S3, 0)  = (sum wy J3(s r) r^2, 0)
// over the nodes of [0, eps] and [eps, 2 eps] (the latter are hcheb's), wy = w Y.
template <bool DERIV>
__global__ void __launch_bounds__(DERIV ? 448 : 256, 1) panels_2d(const double *r, const double *W, int NM, double2 *out, double2 *dout)
{
    constexpr int ROWS = 2 * (PT + 1) + (DERIV ? NQ : 0), NF = DERIV ? 7 : 2;
    extern __shared__ double sm[];
    double *J = sm, *w = J + NJ * LD, *S = w + ROWS * LD, *A = S + 3 * NJ * NQ;
    const int panel = blockIdx.x, t = threadIdx.x;
    const double cen = 2.0 * panel + 1.0;
    const int nsum = DERIV ? c_combos.n : c_combos.n01;
    const int set = t < nsum ? c_combos.set[t] : 0, ord = t < nsum ? c_combos.ord[t] : 0, pw = t < nsum ? c_combos.pw[t] : 0;
    const double *Jr = J + ord * LD, *wr = w + (set * (PT + 1) + pw) * LD;
    double acc = 0.0;
    for (int m0 = 0; m0 < NM; m0 += NC) {
        const int nc = min(NC, NM - m0);
        __syncthreads();
        for (int i = t; i < ROWS * NC; i += blockDim.x) {
            const int row = i / NC, m = i - row * NC;
            if (m < nc) w[row * LD + m] = W[(size_t)row * NM + m0 + m];
        }
        // J0 and J1 by different warps, then the other orders by one thread a node
        for (int i = t; i < 2 * NC; i += blockDim.x) {
            const int m = i & (NC - 1);
            if (m >= nc) continue;
            const double u = cen * r[m0 + m];
            if (u >= 22.0) J[(i / NC) * LD + m] = i < NC ? j0(u) : j1(u);
        }
        __syncthreads();
        for (int m = t; m < nc; m += blockDim.x) bessel_orders(cen * r[m0 + m], J + m, LD);
        __syncthreads();
        if (t < nsum) {
            double a1 = 0.0, a2 = 0.0, a3 = 0.0;
            int m = 0;
            for (; m + 4 <= nc; m += 4) {
                acc = fma(wr[m], Jr[m], acc);
                a1 = fma(wr[m + 1], Jr[m + 1], a1);
                a2 = fma(wr[m + 2], Jr[m + 2], a2);
                a3 = fma(wr[m + 3], Jr[m + 3], a3);
            }
            for (; m < nc; ++m) acc = fma(wr[m], Jr[m], acc);
            acc += a1 + (a2 + a3);
        }
    }
    if (t < nsum) S[(set * NJ + ord) * NQ + pw] = acc;
    __syncthreads();
    // transforms: set, order, power of r: S0, S1, Q1, R0, R2, S1, S3
    const int fset[7] = {0, 1, 2, 2, 2, 2, 2}, fnu[7] = {0, 1, 1, 0, 2, 1, 3}, fe[7] = {0, 0, 0, 1, 1, 2, 2};
    for (int i = t; i < NF * (PT + 1); i += blockDim.x) {
        const int f = i / (PT + 1), p = i - f * (PT + 1);
        int s0 = 0, nu = 0, e = 0;
#pragma unroll
        for (int g = 0; g < NF; ++g)
            if (f == g) {
                s0 = fset[g];
                nu = fnu[g];
                e = fe[g];
            }
        double v = 0.0;
        for (int j = 0; j <= p; ++j) {
            const int n = nu - p + 2 * j, an = abs(n);
            const double c = c_bin.c[p][j] * S[(s0 * NJ + an) * NQ + p + e];
            v += ((j & 1) ^ (n < 0 && (n & 1))) ? -c : c;
        }
        A[f * (PT + 1) + p] = v * c_bin.ifact[p] * __hiloint2double((1023 - p) << 20, 0);  // 2^-p
    }
    __syncthreads();
    const int tab = gridDim.x * (GF_HDEG + 1);
    for (int i = t; i < (DERIV ? 4 : 1) * (GF_HDEG + 1); i += blockDim.x) {
        const int pair = i / (GF_HDEG + 1), k = i - pair * (GF_HDEG + 1);
        double v[2] = {0.0, 0.0};
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int f = 2 * pair + q;
            if (f >= NF) continue;
            const double *a = A + f * (PT + 1);
            for (int p = PT; p > GF_HDEG; --p) v[q] = fma(c_econ.e[p - GF_HDEG - 1][k], a[p], v[q]);
            v[q] += a[k];
        }
        const size_t o = (size_t)panel * (GF_HDEG + 1) + k;
        if (pair == 0)
            out[o] = make_double2(v[0], v[1]);
        else
            dout[(size_t)(pair - 1) * tab + o] = make_double2(v[0], v[1]);
    }
}

template <bool DERIV>
size_t smem_2d()
{
    return sizeof(double) * (NJ * LD + (2 * (PT + 1) + (DERIV ? NQ : 0)) * LD + 3 * NJ * NQ + 7 * (PT + 1));
}

}  // namespace

// Doubles of the node power tables of a plan (0: its panels come from synth.cu).
size_t gf_node_powers(int dim, int Q, bool deriv, double eps)
{
    if (2.0 * eps > 1.0) return 0;
    if (dim == 3) return 2 * (size_t)(P0MAX + 2) * Q;
    return (size_t)(2 * (PT + 1) + (deriv ? NQ : 0)) * (deriv ? 2 * Q : Q);
}

cudaError_t gf_launch_node_tables(const NodeTables &a, cudaStream_t s)
{
    int blocks = (a.Mlast * a.Q + 127) / 128;
    if (blocks > 1024) blocks = 1024;
    node_tables<<<blocks, 128, 0, s>>>(a);
    gf_count_launch(1);
    return cudaGetLastError();
}

cudaError_t gf_launch_xprime_panels(const NodeTables &a, const double *tW, int npan, double w, double tc, double2 *out, cudaStream_t s)
{
    const size_t sm = sizeof(double) * GF_XDEG1 * a.Q;
    cudaError_t e = cudaFuncSetAttribute(xprime_panels, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const int nh = (a.Mlast >> 1) + 1;
    xprime_panels<<<dim3(npan, (nh + XB - 1) / XB), XB * GF_XDEG1, sm, s>>>(a, tW, w, tc, out);
    gf_count_launch(1);
    return cudaGetLastError();
}

cudaError_t gf_launch_panels(const NodeTables &a, int dim, int npan, double2 *out, float2 *outf, double2 *dout, cudaStream_t s)
{
    cudaError_t e;
    if (dim == 3) {
        panels_3d<<<npan, 256, sizeof(double2) * a.Q, s>>>(a.rr, a.Bp, a.Q, out, outf);
    } else if (a.rrd) {
        if ((e = cudaFuncSetAttribute(panels_2d<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_2d<true>())) != cudaSuccess)
            return e;
        panels_2d<true><<<npan, 448, smem_2d<true>(), s>>>(a.rrd, a.W, 2 * a.Q, out, dout);
    } else {
        if ((e = cudaFuncSetAttribute(panels_2d<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_2d<false>())) != cudaSuccess)
            return e;
        panels_2d<false><<<npan, 256, smem_2d<false>(), s>>>(a.rr, a.W, a.Q, out, dout);
    }
    gf_count_launch(1);
    return cudaGetLastError();
}
