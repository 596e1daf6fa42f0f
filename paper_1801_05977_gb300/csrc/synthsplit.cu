// First synthesis pass of the split plans in 3D: the Fourier coefficients of
// Eqs. (kdj1), (fj) (Maxwell: the multipliers of Sec. 4) along x3, their
// inverse transform along x3, and the store of the x3 planes that are kept.
//
// Two kinds of CTA in one launch:
// - a unit forms one column (n1, n2) in double: the columns that propagate or
//   lie within gfloat of a Wood anomaly, a box around |alpha_n| <= k;
// - a tile forms TJ adjacent columns in float, and leaves the units' columns out.
//
// A tile keeps its columns in the lanes: element j of column t lies at [j TJ + t], so
// the shared-memory accesses and the stores are contiguous (TJ = 32: 256 bytes
// a store), the X' nodes' phases E are the same address for a whole warp, and
// neighbouring columns read neighbouring panels of the h(s) table.  A thread
// keeps the X' sums of eight b: per node one load of A and four of E (two b
// each) against sixteen FMAs.
//
// What bounds it: issue (the X' sums, 15 multiply-adds on a table entry each for h(s), the
// transforms), about a third of the slots used; the store is 0.3 GB of the 1.1 ms below.
// Before, a CTA held 8 columns by [column][b]: half its threads had no item, each lane read its
// own line of E, the double set-up ran on 8 lanes of a warp and the double columns held
// their CTA up.  Batched, 64 pairs with 0.5 <= k <= 5 on 32^2 x 64 to 256^2 x 64: 5.86 -> 1.14 ms.
// One plan (cold): 128 x 128 x 64 85 -> 32 us, Maxwell 256 x 256 x 64 319 -> 125 us.
#include <stdint.h>

#include "gf_internal.cuh"
#include "synth_fft.cuh"

namespace {

constexpr int THR = 128;

__device__ __forceinline__ int freq_of(int b, int M) { return b < (M >> 1) ? b : b - M; }

// |alpha|^2 and |alpha|^2 - k^2 of a column; the same rounding in tiles and units, which
// share the columns out by it.
__device__ __forceinline__ double column_d(const SynthArgs &a, int jx, int jy, double &A2)
{
    const double x1 = a.a1 + jx, x2 = a.a2 + jy;
    A2 = __fma_rn(x1, x1, __dmul_rn(x2, x2));
    return __fma_rn(-a.k, a.k, A2);
}

// Shared memory of a tile and of a unit (byte offsets).
struct TileLay {
    size_t X, base, Y, tw, qq, A2mk, qf, A2f, g, flag, tW, tt, end;
};
__host__ __device__ inline TileLay tile_lay(int n, int nf, int T, int Q)
{
    TileLay l;
    const size_t nh = (n >> 1) + 1, line = sizeof(float2) * (size_t)T, a = sizeof(float) * (size_t)Q * T;
    l.X = 0;  // the transforms' first buffer; before them A_m [Q][T]
    l.base = n * line > a ? n * line : a;
    l.Y = nf == 1 ? l.base : l.base + nh * line;  // one field: the coefficients are dead by then
    l.tw = l.Y + n * line;
    l.qq = l.tw + sizeof(float2) * (n >> 1);
    l.A2mk = l.qq + sizeof(float2) * nh;
    l.qf = l.A2mk + sizeof(float2) * T;
    l.A2f = l.qf + sizeof(float) * nh;
    l.g = l.A2f + sizeof(float) * T;
    l.flag = l.g + sizeof(float) * T;
    l.tW = l.flag + sizeof(int) * T;
    l.tt = l.tW + sizeof(float) * Q;
    l.end = l.tt + sizeof(float) * Q;
    return l;
}
struct UnitLay {
    size_t A, S, base, X, Y, tw, end;
};
__host__ __device__ inline UnitLay unit_lay(int n, int Q)
{
    UnitLay l;
    const size_t nh = (n >> 1) + 1;
    l.A = 0;                                // double2 [Q]
    l.S = l.A + sizeof(double2) * (size_t)Q;  // double2 [nh][2]: the X' sums, then C_j
    l.base = l.S + 2 * sizeof(double2) * nh;
    l.X = l.base + sizeof(float2) * (nh + 1);
    l.Y = l.X + sizeof(float2) * n;
    l.tw = l.Y + sizeof(float2) * n;
    l.end = l.tw + sizeof(float2) * (n >> 1);
    return l;
}

__device__ void load_tw(float2 *tw, int n)
{
    for (int i = threadIdx.x; i < (n >> 1); i += blockDim.x) {
        float s, c;
        sincospif(2.0f * (float)i / (float)n, &s, &c);
        tw[i] = make_float2(c, s);
    }
}

__device__ void tile_body(const SynthArgs &a, int blk, unsigned char *smem)
{
    const int n = a.Mlast, lg = a.lgMlast, T = a.TJ, Q = a.Q, nf = a.nf, half = n >> 1, nh = half + 1;
    const int lgT = 31 - __clz(T);
    const TileLay L = tile_lay(n, nf, T, Q);
    float2 *X = reinterpret_cast<float2 *>(smem + L.X), *base = reinterpret_cast<float2 *>(smem + L.base);
    float2 *Y = reinterpret_cast<float2 *>(smem + L.Y), *tw = reinterpret_cast<float2 *>(smem + L.tw);
    float2 *qq = reinterpret_cast<float2 *>(smem + L.qq), *A2mks = reinterpret_cast<float2 *>(smem + L.A2mk);
    float *qfs = reinterpret_cast<float *>(smem + L.qf), *A2fs = reinterpret_cast<float *>(smem + L.A2f);
    float *gs = reinterpret_cast<float *>(smem + L.g);
    int *flags = reinterpret_cast<int *>(smem + L.flag);
    float *tWs = reinterpret_cast<float *>(smem + L.tW), *tts = reinterpret_cast<float *>(smem + L.tt);
    float *Av = reinterpret_cast<float *>(X);
    const int ncols = a.M1 * a.M2, ntiles = ncols >> lgT;
    // tiles alternately from both ends of the column range: the low frequencies
    // (whose X' integrals are formed, the expensive tiles) sit at both ends
    const int col0 = ((blk & 1) ? ntiles - 1 - (blk >> 1) : (blk >> 1)) << lgT;

    load_tw(tw, n);
    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        const int col = col0 + t;
        double A2;
        const double d = column_d(a, freq_of(col % a.M1, a.M1), freq_of(col / a.M1, a.M2), A2);
        const float h = (float)d;
        A2fs[t] = (float)A2;
        A2mks[t] = make_float2(h, (float)(d - (double)h));
        gs[t] = sqrtf(fmaxf(h, 0.f));
        // bit 0: X' integrals skipped (below rounding); bit 1: a unit's column
        flags[t] = (d > a.gskip * a.gskip ? 1 : 0) | (d >= a.gfloat * a.gfloat ? 0 : 2);
    }
    // q_b = b q_s and q_b^2 as float pairs from q_s's pair (qsh, qsl), with no double
    // operation: b q_sh by TwoProd, then the square of the pair (its l^2 term dropped),
    // about 2^-46 relative.  (b = n/2 stands for j = -n/2, the Nyquist index.)
    for (int b = threadIdx.x; b < nh; b += blockDim.x) {
        const float jf = b < half ? (float)b : -(float)half;
        const float ph = jf * a.qsh;
        const float pl = __fmaf_rn(jf, a.qsh, -ph) + jf * a.qsl;
        const float h = ph * ph;
        const float l = __fmaf_rn(ph, ph, -h) + 2.0f * ph * pl;
        const float s = h + l;
        qq[b] = make_float2(s, l - (s - h));
        qfs[b] = ph + pl;
    }
    for (int m = threadIdx.x; m < Q; m += blockDim.x) {
        tWs[m] = (float)a.tW[m];
        tts[m] = (float)a.tt[m];
    }
    __syncthreads();
    // THR is a multiple of T: a thread's items all lie in one column
    const int t = threadIdx.x & (T - 1), flag = flags[t];
    const float g = gs[t], A2f = A2fs[t];
    const float2 Ad = A2mks[t];
    if (!flag)
        for (int i = threadIdx.x; i < Q << lgT; i += blockDim.x) {
            const int m = i >> lgT;
            Av[i] = tWs[m] * expf(-g * tts[m]);
        }
    __syncthreads();

    const float ihpanf = (float)a.ihpan, hpanf = (float)a.hpan, invVf = (float)a.invV, hmaxf = (float)(a.hnpan - 1);
    const float x2h = 2.0f / hpanf;
    // One coefficient from its X' sums, with no double operation.  D = |xi|^2 - k^2
    // (small near the resonance sphere) is the sum of two float pairs, exact
    // to ~2^-46 relative to its terms (Knuth's TwoSum), then rounded: since
    // |D| >= 1e-6 k^2 (the resonance rule), this is below float rounding of D.
    // Every other factor is O(1) in relative terms.
    auto coef = [&](int b, float s1, float s3) {
        const float qf = qfs[b];
        const float T12f = flag ? 0.f : (g * s1 - qf * s3) * __frcp_rn(g * fmaf(g, g, qf * qf));
        const float2 Qd = qq[b];
        const float dh = __fadd_rn(Ad.x, Qd.x), dv = __fsub_rn(dh, Ad.x);
        const float de = __fadd_rn(__fsub_rn(Ad.x, __fsub_rn(dh, dv)), __fsub_rn(Qd.x, dv));
        const float iD = __frcp_rn(__fadd_rn(dh, __fadd_rn(de, __fadd_rn(Ad.y, Qd.y))));
        // |xi| by the hardware reciprocal square root (its ~2^-23 relative error moves
        // the point of the panel by less than the float rounding of h)
        const float s2 = fmaf(qf, qf, A2f);
        const float sf = s2 > 0.f ? s2 * rsqrtf(s2) : 0.f;
        const float pf = fminf(floorf(sf * ihpanf), hmaxf);
        const float x = (sf - (pf + 0.5f) * hpanf) * x2h;
        const float2 *cc = a.hchebf + (int)pf;  // [degree][panel]: the lanes' panels are neighbours
        float2 h = __ldg(cc + GF_HDEG * a.hnpan);
#pragma unroll
        for (int kk = GF_HDEG - 1; kk >= 0; --kk) {
            const float2 ck = __ldg(cc + kk * a.hnpan);
            h.x = fmaf(h.x, x, ck.x);
            h.y = fmaf(h.y, x, ck.y);
        }
        return make_float2(fmaf(h.x, iD, T12f) * invVf, h.y * iD * invVf);
    };
    // The coefficients are even in the last-axis index j (they depend on q_j
    // through q_j^2, and the two X' terms of Eqs. (fck-coef)/(kdj1) trade places
    // under q -> -q), except the Maxwell xz and yz fields, whose factor c^3 = q_j
    // makes them odd (Sec. 4).  Only b = 0 .. n/2 are formed; the transform reads
    // b > n/2 (j = b - n) from b' = n - b (j' = -j).
    const int EP = GF_EF_ROW(n), ng = (half + 7) >> 3;
    for (int i = threadIdx.x; i < (ng + 1) << lgT; i += blockDim.x) {
        const int gr = i >> lgT;
        if (flag & 2) continue;
        if (gr == ng) {
            float s1 = 0.f, s3 = 0.f;
            if (!flag) {
                const float2 *E = a.Ef + half;
#pragma unroll 8
                for (int m = 0; m < Q; ++m) {
                    const float A = Av[(m << lgT) + t];
                    const float2 e = __ldg(E + m * EP);
                    s1 = fmaf(A, e.x, s1);
                    s3 = fmaf(A, e.y, s3);
                }
            }
            base[(half << lgT) + t] = coef(half, s1, s3);
            continue;
        }
        float s1[8] = {0.f}, s3[8] = {0.f};
        if (!flag) {
            const float4 *E = reinterpret_cast<const float4 *>(a.Ef + gr * 8);
#pragma unroll 4
            for (int m = 0; m < Q; ++m) {
                const float A = Av[(m << lgT) + t];
                const float4 *Em = E + m * (EP >> 1);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float4 e = __ldg(Em + u);
                    s1[2 * u] = fmaf(A, e.x, s1[2 * u]);
                    s3[2 * u] = fmaf(A, e.y, s3[2 * u]);
                    s1[2 * u + 1] = fmaf(A, e.z, s1[2 * u + 1]);
                    s3[2 * u + 1] = fmaf(A, e.w, s3[2 * u + 1]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int b = gr * 8 + u;
            if (b < half) base[(b << lgT) + t] = coef(b, s1[u], s3[u]);
        }
    }
    __syncthreads();

    float2 *W = reinterpret_cast<float2 *>(a.work);
    const int planes = a.L3count + a.nyq;  // work planes per field
    const int col = col0 + t;
    const float ik2f = (float)(1.0 / (a.k * a.k));
    const float cv0 = (float)(a.a1 + freq_of(col % a.M1, a.M1)), cv1 = (float)(a.a2 + freq_of(col / a.M1, a.M2));
    const bool mine = !(flag & 2);
    for (int f = 0; f < nf; ++f) {
        // Maxwell (Sec. 4): combined fields (delta_pq - c^p c^q / k^2) C, c = (alpha1+j1, alpha2+j2, q),
        // order xx, yy, zz, xy, xz, yz, then the plain field C (for G_d): factor pf, pf q or 1 - q^2/k^2
        const bool odd = (a.oddmask >> f) & 1;
        const float pf = nf == 1 || f == 6 ? 1.f
                         : f == 0          ? 1.f - cv0 * cv0 * ik2f
                         : f == 1          ? 1.f - cv1 * cv1 * ik2f
                         : f == 3          ? -cv0 * cv1 * ik2f
                                           : -(f == 4 ? cv0 : cv1) * ik2f;
        auto ld = [&](int b, int) {
            const int bb = b <= half ? b : n - b;
            const float2 v = base[(bb << lgT) + t];
            if (nf == 1) return v;
            const float q = qfs[bb];
            float m = odd ? pf * q : f == 2 ? 1.f - q * q * ik2f : pf;
            if (odd && b > half) m = -m;
            return make_float2(m * v.x, m * v.y);
        };
        if (a.nyq && odd && threadIdx.x < T && mine)
            W[((size_t)f * planes + a.L3count) * ncols + col] = ld(half, t);
        float2 *Wf = W + (size_t)f * planes * ncols + col;
        // only the x3 nodes the last two passes transform (a3first .. a3first +
        // L3count - 1), compact: work plane y holds node a3first + y, whose output
        // index is l = (a3first + y + n/2) mod n
        fft_cols(X, Y, n, lg, lgT, tw, ld, [&](int l, int, float2 v) {
            const int y = (l - half - a.a3first) & (n - 1);
            if (y < a.L3count && mine) Wf[(size_t)y * ncols] = v;
        });
    }
}

__device__ void unit_body(const SynthArgs &a, int u, unsigned char *smem)
{
    const int n = a.Mlast, lg = a.lgMlast, Q = a.Q, nf = a.nf, half = n >> 1, nh = half + 1;
    const int jx = a.dbx0 + u % a.dbw, jy = a.dby0 + u / a.dbw;
    double A2;
    if (column_d(a, jx, jy, A2) >= a.gfloat * a.gfloat) return;  // a tile's column (the same for all threads)
    const UnitLay L = unit_lay(n, Q);
    double2 *Am = reinterpret_cast<double2 *>(smem + L.A), *S = reinterpret_cast<double2 *>(smem + L.S);
    float2 *base = reinterpret_cast<float2 *>(smem + L.base), *X = reinterpret_cast<float2 *>(smem + L.X);
    float2 *Y = reinterpret_cast<float2 *>(smem + L.Y), *tw = reinterpret_cast<float2 *>(smem + L.tw);
    // beta (Sec. 1): sqrt(k^2 - |alpha|^2), k^2 - |alpha|^2 formed as (k - |alpha|)(k + |alpha|)
    const double ra = sqrt(A2);
    const bool prop = ra <= a.k;
    const double bt = prop ? sqrt((a.k - ra) * (a.k + ra)) : sqrt((ra - a.k) * (ra + a.k));
    const bool skip = !prop && bt > a.gskip;
    load_tw(tw, n);
    if (!skip)
        for (int m = threadIdx.x; m < Q; m += blockDim.x) {
            const double tm = a.tt[m], w = a.tW[m];
            double sn = 0.0, cs;
            if (prop)
                sincos(bt * tm, &sn, &cs);
            else
                cs = exp(-bt * tm);
            Am[m] = make_double2(cs * w, sn * w);
        }
    __syncthreads();
    // X' sums: four lanes per b, a quarter of the nodes each
    const int part = threadIdx.x & 3;
    for (int b0 = 0; b0 < nh; b0 += THR / 4) {
        const int b = b0 + (threadIdx.x >> 2);
        double s1 = 0.0, s2 = 0.0, s3 = 0.0, s4 = 0.0;
        if (b < nh && !skip) {
            const double2 *E = a.E + (size_t)b * Q;
            for (int m = part; m < Q; m += 4) {
                const double2 A = Am[m], e = E[m];
                s1 = fma(A.x, e.x, s1);
                s3 = fma(A.x, e.y, s3);
                if (prop) {
                    s2 = fma(A.y, e.y, s2);
                    s4 = fma(A.y, e.x, s4);
                }
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            s3 += __shfl_xor_sync(0xffffffffu, s3, o);
            s4 += __shfl_xor_sync(0xffffffffu, s4, o);
        }
        if (b < nh && part == 0) {
            S[2 * b] = make_double2(s1, s2);
            S[2 * b + 1] = make_double2(s3, s4);
        }
    }
    __syncthreads();
    const double k2 = a.k * a.k;
    for (int b = threadIdx.x; b < nh; b += blockDim.x) {
        const double q = (double)(b < half ? b : -half) * a.qs;
        const double2 sa = S[2 * b], sb = S[2 * b + 1];
        double2 T12 = make_double2(0.0, 0.0);
        if (prop) {
            // T1 - T2 = I1/(2 beta (q - beta)) - I2/(2 beta (q + beta))
            const double2 I1 = make_double2(sa.x + sa.y, sb.y - sb.x), I2 = make_double2(sa.x - sa.y, sb.x + sb.y);
            const double i1 = 1.0 / (2.0 * bt * (q - bt)), i2 = 1.0 / (2.0 * bt * (q + bt));
            T12 = make_double2(I1.x * i1 - I2.x * i2, I1.y * i1 - I2.y * i2);
        } else if (!skip) {
            T12.x = (bt * sa.x - q * sb.x) / (bt * (bt * bt + q * q));
        }
        const double D = A2 + q * q - k2, s = sqrt(A2 + q * q);
        const int pnl = min((int)(s * a.ihpan), a.hnpan - 1);
        const double2 h = poly_eval(a.hcheb + (size_t)pnl * (GF_HDEG + 1), GF_HDEG, (s - (pnl + 0.5) * a.hpan) * (2.0 / a.hpan));
        const double iD = 1.0 / D;
        S[2 * b] = make_double2(fma(h.x, iD, T12.x) * a.invV, fma(h.y, iD, T12.y) * a.invV);
    }
    __syncthreads();
    float2 *W = reinterpret_cast<float2 *>(a.work);
    const int planes = a.L3count + a.nyq, ncols = a.M1 * a.M2;
    const int col = (jy & (a.M2 - 1)) * a.M1 + (jx & (a.M1 - 1));
    const double ik2 = 1.0 / k2, cv0 = a.a1 + jx, cv1 = a.a2 + jy;
    for (int f = 0; f < nf; ++f) {
        const bool odd = (a.oddmask >> f) & 1;
        for (int b = threadIdx.x; b < nh; b += blockDim.x) {
            const double q = (double)(b < half ? b : -half) * a.qs;
            const double m = nf == 1 || f == 6 ? 1.0
                             : f == 0          ? 1.0 - cv0 * cv0 * ik2
                             : f == 1          ? 1.0 - cv1 * cv1 * ik2
                             : f == 2          ? 1.0 - q * q * ik2
                             : f == 3          ? -cv0 * cv1 * ik2
                                               : -(f == 4 ? cv0 : cv1) * q * ik2;
            const double2 C = S[2 * b];
            base[b] = make_float2((float)(m * C.x), (float)(m * C.y));
        }
        __syncthreads();
        if (a.nyq && odd && threadIdx.x == 0) W[((size_t)f * planes + a.L3count) * ncols + col] = base[half];
        float2 *Wf = W + (size_t)f * planes * ncols + col;
        auto ld = [&](int b, int) {
            const float2 v = base[b <= half ? b : n - b];
            return odd && b > half ? make_float2(-v.x, -v.y) : v;
        };
        fft_rows(X, Y, n, lg, 1, tw, ld, [&](int l, int, float2 v) {
            const int y = (l - half - a.a3first) & (n - 1);
            if (y < a.L3count) Wf[(size_t)y * ncols] = v;
        });
    }
}

__device__ __forceinline__ void first_split_body(const SynthArgs &a, int blk, unsigned char *smem)
{
    // the units first: one of them is the longest CTA
    if (blk < a.ndbl)
        unit_body(a, blk, smem);
    else
        tile_body(a, blk - a.ndbl, smem);
}

__global__ void __launch_bounds__(THR, 6) first_split(const __grid_constant__ SynthArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    first_split_body(a, blockIdx.x, smem);
}

__global__ void __launch_bounds__(THR, 6) first_split_batch(const SynthArgs *args, const int *prefix, int np)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ SynthArgs sa;
    const int total = prefix[np];
    int p = -1;
    for (int vb = blockIdx.x; vb < total; vb += gridDim.x) {
        if (p < 0 || vb >= prefix[p + 1]) {
            p = p < 0 ? 0 : p;
            while (vb >= prefix[p + 1]) ++p;
            const int *src = reinterpret_cast<const int *>(args + p);
            for (int i = threadIdx.x; i < (int)(sizeof(SynthArgs) / sizeof(int)); i += blockDim.x)
                reinterpret_cast<int *>(&sa)[i] = src[i];
            __syncthreads();
        }
        first_split_body(sa, vb - prefix[p], smem);
        __syncthreads();
    }
}

}  // namespace

// Columns per tile (at most tj_max, a power of two in [8, 32]: fewer while the tile's
// shared memory would leave less than about four CTAs on an SM) and the CTA's shared
// memory; sets a.TJ.
size_t gf_first_split_config(SynthArgs &a, int tj_max)
{
    int T = tj_max > 32 ? 32 : tj_max < 8 ? 8 : tj_max;
    while (T > 8 && tile_lay(a.Mlast, a.nf, T, a.Q).end > 56 * 1024) T >>= 1;
    a.TJ = T;
    const size_t t = tile_lay(a.Mlast, a.nf, T, a.Q).end, u = unit_lay(a.Mlast, a.Q).end;
    return t > u ? t : u;
}

cudaError_t gf_launch_first_split(const SynthArgs &a, size_t smem, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(first_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    first_split<<<a.ndbl + a.M1 * a.M2 / a.TJ, THR, smem, s>>>(a);
    gf_count_launch(1);
    return cudaGetLastError();
}

cudaError_t gf_launch_first_split_batch(const SynthBatch &b, int nsm, cudaStream_t s)
{
    cudaError_t e =
        cudaFuncSetAttribute(first_split_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b.smem[0]);
    if (e != cudaSuccess) return e;
    int per = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, first_split_batch, THR, b.smem[0])) != cudaSuccess) return e;
    const int want = per * nsm;
    first_split_batch<<<b.total0 < want ? b.total0 : want, THR, b.smem[0], s>>>(b.args, b.prefix[0], b.np);
    gf_count_launch(1);
    return cudaGetLastError();
}
