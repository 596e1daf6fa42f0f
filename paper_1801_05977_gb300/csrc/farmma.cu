// Far series of 3D plans on the tensor cores.
//
// After the sort by |x3|, 128 consecutive far targets (a tile) share nearly one
// |x3|, and a run of tiles (a cell) is expanded about one z_w:
//   e^{-b z}/b = sum_p ((z - z_w)/delta)^p  (-b delta)^p/p! e^{-b z_w}/b,
// delta the cell's half width.  With the in-plane index taken from the anchors
// N_i = rint(-alpha_i), n_i = N_i + m_i, and the weights of m2 and -m2 joined
// (W+- = w(m1, m2) +- w(m1, -m2)), the series of a target is
//   sum_{m1} e^{i m1 t1} [ sum_{p, m2 >= 0} W+_p cos_p(m2 t2) + i W-_p sin_p(m2 t2) ],
// cos_p = ((z - z_w)/delta)^p cos: the bracket is a matrix product of the tile's
// cos_p, sin_p [128 x K] with the cell's weights [K x rows], the outer sum one
// polynomial per target.  (The terms are those of the eigen-series (he); Maxwell
// entries take their factors delta_pq - c_p c_q/k^2 into the weights.)
//
// Precision.  Both factors are fixed-point numbers, cut into L signed 10-bit digits
// (exact in f16): v = sum_i d_i 2^{-10 i - 9}, |d_i| <= 512.  The product of digit i
// of a weight with digit j of a phase factor goes to the accumulator of level
// i + j, a sum of integers, exact in the tensor cores' FP32 accumulation up to 2^24 in size.
// No bound in the layout keeps the sums below that (a level adds hundreds of products of up to
// 2^18): digits other than a number's leading ones are as good as random, so the sums are those of a
// random walk.  Emulated in integers for k = 0.4 .. 6.8, |x3| = 0.6 .. 2.5 and targets at and
// off multiples of pi/6: levels 0 .. 3 at most 2^17.3, 2^20.2, 2^21.2 and 2^21.7, root mean square 2^19 at
// most (2^24 is 30 of those away); one that passed it would be rounded in its last bit.  Levels 4 and 5, up
// to 2^22.8, are rounded in the end anyway.  Levels 0 .. L-1 are kept: L = 6 for
// double-precision plans (2^-60 of the cell's largest weight, where the
// recurrences of far3d_f64 round at 2^-53 of their state), L = 3 (2^-30) for split
// plans.  A weight 2^-10 below the largest has no digit 0, and so on, so the
// tails of the series take part with the few digits that they need: the
// rows, columns and digits of each product follow from the decay of the weights.
// The outer sum is in 64-bit fixed point (L = 6) or float (L = 3).
//
// Why: the FP64 pipe of this GPU retires one warp instruction in 16 cycles per SM,
// and the recurrences took 5450 of them per far target; here no per-term work is
// left on it.
#include <cuda_fp16.h>
#include <math_constants.h>

#include "gf_internal.cuh"
#include "umma_gemm.cuh"

namespace {

constexpr int TILE = 128;                 // targets per tile (MMA rows)
constexpr int KB = 16;                    // m2 per block (MMA K)
constexpr int NKB = 4;                    // blocks: m2 < 64
constexpr int PMAX = 12;                  // orders in z - z_w
constexpr int MAXST = 32;                 // stages of a cell (also the lanes of a warp)
constexpr int RBLK = 16;                  // rows (m1) per block of rows (MMA N): 8 of either sign
constexpr int MAXRB = 8;                  // blocks of rows: |m1| <= 64
constexpr int NGW = 16;                   // warps that make phase digits and finish the sums
constexpr int NMW = 3;                    // warps that issue MMAs (each for its own accumulator levels)
constexpr int THREADS = (NGW + 1 + NMW) * 32;  // one more issues the copies
constexpr int USLICES = 12;               // digit slices (4 KiB) of a unit's A buffer
constexpr int UBYTES = 32 << 10;          // weight images of a unit

// One product stage of a cell: columns 16 kb .. + 15 at order p, weight digits
// i0 .. L-1 with rows[i] blocks of rows each; the propagating part of the other
// phase quadrature ("prop", 16 rows m1 = r - 8) from digit pi0 (L: none).
// An image holds, per digit, blocks of 8 rows m1 = 8 m + r and 8 rows m1 = -1 - (8 m
// + r); in a merged cell the 16 propagating rows come before them, otherwise they
// have images of their own.  The cos images of all stages follow each other, then
// the sin images, then those of the propagating part.
struct Stage {
    unsigned char kb, p, i0, pi0;
    unsigned char rows[8];
    int off, img;    // byte offset among the cos (sin) images, bytes of one
    int poff, pimg;  // the same for the propagating part (cells not merged)
};

// Stages are made and multiplied in units, as many as fit the A and B buffers: one
// hand-over each.
struct Cell {
    double zw, delta, idelta, scale;
    int ex;                         // scale = 2^ex
    int ok, nst, npst;              // accepted; stages, those among them with a prop part
    int merged;                     // the propagating rows share the full passes' accumulators
    int timg, tpimg;                // bytes of all cos images, of all prop cos images
    int nu, npu;                    // units of a full pass, of one phase factor of the propagating pass (L = 6)
    unsigned char width[8];         // blocks of rows per level
    unsigned char col[8];           // first column of a level, in blocks of 16
    int cols;                       // columns of one accumulator set
    unsigned char pwidth[8];        // levels of the prop set (0 or 1)
    unsigned char ust[MAXST + 4];   // first stage of each unit, then nst
    unsigned char pust[PMAX + 4];   // the same for the propagating pass, then npst
    Stage st[MAXST];
};

template <int L> struct Cap;
// bytes of images per cell and output entry; a cell that needs more is left to the series kernels
template <> struct Cap<6> { static constexpr int BYTES = 400 << 10; };
template <> struct Cap<3> { static constexpr int BYTES = 64 << 10; };

// Largest b at which the bound of |weight| at order p still reaches digit i, or -1 where it does
// nowhere:
//   F(b) = ln(2 m(b) e^{-b z} (b delta)^p / (p! b S)) >= -10 (i + 1) ln 2 (a little less
// is asked, so that no carry reaches a digit that is left out), m(b) = 1 or 2 + b^2/k^2 the
// bound of the entry's factor.  F rises up to its peak, which lies between (p - 1)/z and
// (p + 1)/z (F's derivative is -z + (p - 1)/b plus at most 2/b), and falls beyond it; at the
// left end of the indices, b = bmin, it may be past the peak.
__device__ float digit_radius(float z, int p, int i, float ldelta, float lfact, float lS, float bmin, bool maxwell, float ik2)
{
    const float thr = -6.9314718f * (float)(i + 1) - 0.05f;
    auto F = [&](float b) {
        const float lm = maxwell ? logf(2.f + b * b * ik2) : 0.f;
        return 0.6931472f + lm - b * z + (float)(p - 1) * logf(b) + (float)p * ldelta - lfact - lS;
    };
    const float b0 = fmaxf(bmin, (float)(p + 1) / z);
    // Helmholtz: the peak itself; Maxwell: the sum of the bounds' peaks (2 at (p - 1)/z, b^2/k^2 at
    // (p + 1)/z) is above it
    const float bp = fmaxf(bmin, (float)(p - 1) / z);
    float peak = F(bp);
    if (maxwell) {
        auto G = [&](float b, float m) { return 0.6931472f + m - b * z + (float)(p - 1) * logf(b) + (float)p * ldelta - lfact - lS; };
        peak = fmaxf(G(bp, 0.6931472f), G(b0, logf(b0 * b0 * ik2))) + 0.6931472f;
    }
    if (peak < thr) return -1.f;
    if (F(b0) < thr) return b0;
    float lo = b0, hi = 400.f;
    if (F(hi) >= thr) return hi;
    for (int it = 0; it < 24; ++it) {
        const float m = 0.5f * (lo + hi);
        if (F(m) >= thr) lo = m; else hi = m;
    }
    return hi;
}

// One block per cell: the |x3| range of its targets, the expansion's orders, the
// rows of every digit and the layout of its images.  Cells that the product kernel
// cannot take (too wide in |x3|, too many rows, columns or bytes) are flagged for the
// series kernels: rej[0] the number of their targets, rej[1] tiles per cell, rej[2 + cell] 1.
template <int L>
__global__ void __launch_bounds__(128) far_cells(EvalArgs a, Cell *cells, int *rej, int maxcells, int out_e)
{
    __shared__ float rad[PMAX * 8];
    __shared__ unsigned char rws[NKB * PMAX * 8];
    __shared__ double zr[2][4];
    __shared__ Cell C;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x;
    const int count = a.far_count[0], ntiles = (count + TILE - 1) / TILE;
    const int T = max(1, (ntiles + maxcells - 1) / maxcells);
    if (threadIdx.x == 0 && c == 0) rej[1] = T;
    if (c * T >= ntiles) return;
    const int s0 = c * T * TILE, s1 = min(count, s0 + T * TILE);
    double zmin = 1e300, zmax = 0.0;
#pragma unroll 4
    for (int s = s0 + threadIdx.x; s < s1; s += 128) {
        const double z = fabs(a.x[3 * (size_t)a.far_sorted[s] + 2]);
        zmin = fmin(zmin, z);
        zmax = fmax(zmax, z);
    }
    for (int o = 16; o > 0; o >>= 1) {
        zmin = fmin(zmin, __shfl_xor_sync(0xffffffffu, zmin, o));
        zmax = fmax(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
    }
    if (lane == 0) {
        zr[0][w] = zmin;
        zr[1][w] = zmax;
    }
    __syncthreads();
    zmin = fmin(fmin(zr[0][0], zr[0][1]), fmin(zr[0][2], zr[0][3]));
    zmax = fmax(fmax(zr[1][0], zr[1][1]), fmax(zr[1][2], zr[1][3]));
    const bool maxwell = a.nf > 1 && out_e < 6;
    const float z = (float)zmin, k = (float)a.k, ik2 = (float)(1.0 / (a.k * a.k));
    const double zw = 0.5 * (zmin + zmax);
    const double delta = fmax(0.5 * (zmax - zmin) * 1.0000001, 1e-12 * zw);
    // scale: at least twice every weight at order 0 (weights of m2 and -m2 are joined)
    const float bm = (float)a.bmin, bs = fmaxf(bm, 1.f / z);
    float top = expf(-bm * z) / bm * (maxwell ? 2.f : 1.f);
    if (maxwell) top += expf(-bs * z) * bs * ik2;
    if (a.bprop > 0.0) top = fmaxf(top, (maxwell ? 2.f : 1.f) / (float)a.bprop + (maxwell ? (float)(1.0 / a.k) : 0.f));
    int ex;
    frexpf(2.02f * top, &ex);
    const float lS = (float)ex * 0.6931472f, ld = logf((float)delta);
    // propagating weights at order p: at most (k delta)^p/p! 1/beta_min (times the factor's bound)
    auto prop_digit = [&](int p, int i) {
        if (!(a.bprop > 0.0)) return false;
        float v = logf((maxwell ? 2.f : 1.f) / (float)a.bprop + (maxwell ? 1.f / k : 0.f)) + 0.6931472f - lS;
        for (int t = 1; t <= p; ++t) v += logf(k * (float)delta / (float)t);
        return v >= -6.9314718f * (float)(i + 1) - 0.05f;
    };
    // radii of digit i at order p, then the blocks of rows (bit 7: with a propagating part)
    for (int q = threadIdx.x; q < PMAX * L; q += 128) {
        const int p = q / L, i = q % L;
        float lf = 0.f;
        for (int t = 2; t <= p; ++t) lf += logf((float)t);
        rad[p * 8 + i] = digit_radius(z, p, i, ld, lf, lS, bm, maxwell, ik2);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < NKB * PMAX * L; q += 128) {
        const int st = q / L, i = q % L, kb = st / PMAX, p = st % PMAX;
        const float c2 = fmaxf(0.f, (float)(KB * kb) - 0.5f), b = rad[p * 8 + i];
        int rows = 0, pr = 0;
        if (b > 0.f) {
            const float v = b * b + k * k - c2 * c2;
            if (v >= 0.f) rows = (int)fminf(floorf(sqrtf(v) + 0.502f), 1000.f) + 1;
        }
        if (kb == 0 && prop_digit(p, i)) {
            rows = max(rows, (int)ceilf(k + 0.5f) + 1);
            pr = 128;
        }
        int rb = (rows + RBLK / 2 - 1) / (RBLK / 2);
        // the last digit of rows |m1| > 64 may be left out while it is below 2^-53 of the scale
        if (i == L - 1 && L == 6 && rb == MAXRB + 1) rb = MAXRB;
        rws[st * 8 + i] = (unsigned char)(min(100, rb) | pr);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    C.zw = zw;
    C.delta = delta;
    C.idelta = 1.0 / delta;
    C.scale = exp2((double)ex);
    C.ex = ex;
    bool ok = isfinite(zw) && (float)delta * 64.f < 0.5f && ex > -200 && ex < 200;
    int nst = 0, npst = 0;
    for (int l = 0; l < 8; ++l) C.width[l] = C.pwidth[l] = 0;
    for (int kb = 0; kb < NKB && ok; ++kb) {
        for (int p = 0; p < PMAX && ok; ++p) {
            Stage S;
            S.kb = (unsigned char)kb;
            S.p = (unsigned char)p;
            S.i0 = S.pi0 = L;
#pragma unroll
            for (int i = 0; i < L; ++i) {
                const int rw = rws[(kb * PMAX + p) * 8 + i], rb = rw & 127;
                if ((rw & 128) && S.pi0 == L) S.pi0 = (unsigned char)i;
                if (rb > MAXRB) ok = false;
                S.rows[i] = (unsigned char)rb;
                if (rb > 0 && S.i0 == L) S.i0 = (unsigned char)i;
                if (kb == 0 && p == 0) {
                    C.width[i] = (unsigned char)rb;
                    C.pwidth[i] = (unsigned char)(S.pi0 < L ? 1 : 0);
                }
                if (rb > C.width[i]) ok = false;  // (a higher order or block never needs more rows)
            }
            if (S.i0 == L) break;
            if (p == PMAX - 1 || nst == MAXST) {  // the expansion would need more orders
                ok = false;
                break;
            }
            if (S.pi0 < L) npst = nst + 1;
            C.st[nst++] = S;
        }
    }
    {
        // nothing may be left beyond the last block
        const float c2n = (float)(KB * NKB) - 0.5f, b = rad[L - 1];
        if (L == 3 && b * b + k * k - c2n * c2n >= 0.f) ok = false;
        if (L == 6 && b >= c2n + 8.f) ok = false;  // (as for the rows: a last digit below 2^-53)
    }
    int cols = 0;
    for (int l = 0; l < L; ++l) cols += C.width[l] * RBLK;
    // accumulator columns: cos, then sin for L = 6, both at once for L = 3; with the propagating
    // rows where they fit (always for L = 3)
    const int room = L == 6 ? 512 : 256;
    if (cols > room) ok = false;
    C.merged = npst > 0 && cols + L * RBLK <= room ? 1 : 0;
    if (L == 3 && npst > 0 && !C.merged) ok = false;
    cols = 0;
    for (int l = 0; l < L; ++l) {
        C.col[l] = (unsigned char)(cols / 16);
        cols += (C.width[l] + C.merged) * RBLK;
    }
    C.cols = cols;
    int off = 0, poff = 0;
    for (int t = 0; t < nst && ok; ++t) {
        Stage &S = C.st[t];
        int blocks = 0;
        for (int i = 0; i < L; ++i) blocks += S.rows[i];
        const int pblocks = L - S.pi0;
        if (C.merged) blocks += pblocks;
        S.off = off;
        S.img = blocks * RBLK * KB * 2;
        S.poff = poff;
        S.pimg = C.merged ? 0 : pblocks * RBLK * KB * 2;
        off += S.img;
        poff += S.pimg;
    }
    if (2 * (off + poff) > Cap<L>::BYTES || nst == 0 || npst > 12) ok = false;
    C.nst = nst;
    C.npst = npst;
    C.timg = off;
    C.tpimg = poff;
    // units: L = 6 one phase factor's digits and images at a time; L = 3 both and the propagating part
    int nu = 0, slices = 0, bytes = 0;
    for (int t = 0; t < nst; ++t) {
        const Stage &S = C.st[t];
        const int sl = (L == 6 ? 1 : 2) * (L - (C.merged ? min(S.i0, S.pi0) : S.i0)), by = (L == 6 ? 1 : 2) * S.img;
        if (t == 0 || slices + sl > USLICES || bytes + by > UBYTES) {
            C.ust[nu++] = (unsigned char)t;
            slices = bytes = 0;
        }
        slices += sl;
        bytes += by;
        if (by > UBYTES) ok = false;
    }
    C.ust[nu] = (unsigned char)nst;
    C.nu = nu;
    int npu = 0;
    slices = 0;
    for (int t = 0; t < npst && !C.merged; ++t) {
        const int sl = L - C.st[t].pi0;
        if (t == 0 || slices + sl > USLICES) {
            C.pust[npu++] = (unsigned char)t;
            slices = 0;
        }
        slices += sl;
    }
    C.pust[npu] = (unsigned char)(C.merged ? 0 : npst);
    C.npu = npu;
    C.ok = ok ? 1 : 0;
    rej[2 + c] = ok ? 0 : 1;
    if (!ok) atomicAdd(rej, s1 - s0);
    cells[c] = C;
}

// ---------------------------------------------------------------------------
// Digits
// ---------------------------------------------------------------------------
// biased digits of a fixed-point number with 2^B for 1 (B = 59 or 61 for L = 6): digit i is
// ((x + bias) >> (B - 9 - 10 i) & 1023) - 512 (the first one unmasked: it may be 512)
template <int B>
__device__ __forceinline__ long long with_bias(long long x)
{
    constexpr long long one = 1ll << (B - 9);
    constexpr long long bias = 512ll * (one + (one >> 10) + (one >> 20) + (one >> 30) + (one >> 40) + (one >> 50)) +
                               (B > 59 ? 1ll << (B - 60) : 0ll);
    return x + bias;
}

// digit i of two biased numbers as a pair of f16 (a in the low half)
template <int B, int I>
__device__ __forceinline__ uint32_t digit_pair(long long a, long long b)
{
    constexpr int s = B - 9 - 10 * I;
    const uint32_t al = (uint32_t)a, ah = (uint32_t)((unsigned long long)a >> 32);
    const uint32_t bl = (uint32_t)b, bh = (uint32_t)((unsigned long long)b >> 32);
    const uint32_t lo = s >= 32 ? ah >> (s - 32) : __funnelshift_r(al, ah, s);
    constexpr int t = s - 16;
    const uint32_t hi = t >= 32 ? bh >> (t - 32) : t > 0 ? __funnelshift_r(bl, bh, t) : bl << (-t);
    uint32_t u;
    if (I == 0)  // 0 .. 1024
        u = ((lo & 0x7FFu) | (hi & 0x07FF0000u)) + 0x64006400u;
    else
        u = ((lo & 0x3FFu) | (hi & 0x03FF0000u)) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&u), __halves2half2(__ushort_as_half(0x6600), __ushort_as_half(0x6600)));
    return *reinterpret_cast<const uint32_t *>(&h);
}

// ---------------------------------------------------------------------------
// 64-bit fixed point: 2^61 for 1 in the phase factors.  Products by 31-bit limbs
// (x = h 2^31 + l, 0 <= l < 2^31), the l l part left out (below 2 units).
// ---------------------------------------------------------------------------
struct C64 {
    long long x, y;
};
__device__ __forceinline__ int lim_h(long long v) { return (int)(v >> 31); }
__device__ __forceinline__ int lim_l(long long v) { return (int)((uint32_t)v & 0x7FFFFFFFu); }

// a * v / 2^61
__device__ __forceinline__ long long mulq(long long a, int vh, int vl)
{
    const int ah = lim_h(a), al = lim_l(a);
    const long long hi = (long long)ah * vh;
    const long long mid = (long long)ah * vl + (long long)al * vh + (1ll << 29);
    return 2 * hi + (mid >> 30);
}

// the same with the l l part: rounded without bias, for the weights (their errors all add up
// where t is near a lattice point)
__device__ __forceinline__ long long mulq_unbiased(long long a, int vh, int vl)
{
    const int ah = lim_h(a), al = lim_l(a);
    const long long hi = (long long)ah * vh;
    const long long mid = (long long)ah * vl + (long long)al * vh + (((long long)al * vl) >> 31) + (1ll << 29);
    return 2 * hi + (mid >> 30);
}

struct Lim {
    int ch, cl, sh, sl;  // limbs of a phase factor (c, s)
};
__device__ __forceinline__ Lim limbs(const C64 &v) { return Lim{lim_h(v.x), lim_l(v.x), lim_h(v.y), lim_l(v.y)}; }

// the real and the imaginary part of a v / 2^61
__device__ __forceinline__ long long mulq_re(const C64 &a, const Lim &v)
{
    const int xh = lim_h(a.x), xl = lim_l(a.x), yh = lim_h(a.y), yl = lim_l(a.y);
    const long long h = (long long)xh * v.ch - (long long)yh * v.sh;
    const long long m = (long long)xh * v.cl + (long long)xl * v.ch - (long long)yh * v.sl - (long long)yl * v.sh + (1ll << 29);
    return 2 * h + (m >> 30);
}
__device__ __forceinline__ long long mulq_im(const C64 &a, const Lim &v)
{
    const int xh = lim_h(a.x), xl = lim_l(a.x), yh = lim_h(a.y), yl = lim_l(a.y);
    const long long h = (long long)xh * v.sh + (long long)yh * v.ch;
    const long long m = (long long)xh * v.sl + (long long)xl * v.sh + (long long)yh * v.cl + (long long)yl * v.ch + (1ll << 29);
    return 2 * h + (m >> 30);
}
__device__ __forceinline__ C64 cmulq(const C64 &a, const Lim &v) { return C64{mulq_re(a, v), mulq_im(a, v)}; }

// 32-bit fixed point, 2^30 for 1 in the phase factors
struct C32 {
    int x, y;
};
__device__ __forceinline__ C32 to_c32(const C64 &v) { return C32{(int)(v.x >> 31), (int)(v.y >> 31)}; }
__device__ __forceinline__ int mul30(int a, int b) { return (int)(((long long)a * b + (1 << 29)) >> 30); }
__device__ __forceinline__ int mul30_re(const C32 &a, const C32 &v) { return (int)(((long long)a.x * v.x - (long long)a.y * v.y + (1 << 29)) >> 30); }
__device__ __forceinline__ int mul30_im(const C32 &a, const C32 &v) { return (int)(((long long)a.x * v.y + (long long)a.y * v.x + (1 << 29)) >> 30); }
__device__ __forceinline__ C32 cmul30(const C32 &a, const C32 &v) { return C32{mul30_re(a, v), mul30_im(a, v)}; }

// ---------------------------------------------------------------------------
// Weights: images of the cells' weight digits, one CTA per (cell, part): part kb <
// NKB the columns 16 kb .. + 15 of all rows, part NKB the propagating block (cells
// not merged).  All output entries of a plan come from one exponential per index.
// What bounds it: the FP64 pipe (seven operations per index at order 0), so the
// conversion to fixed point, the scaling and the higher orders are integer work.
// ---------------------------------------------------------------------------
// One index n: evanescent: v = e^{-b z_w}/b, g = -b delta; propagating: (v + i vi) =
// e^{i beta z_w}, g = beta delta, b = beta.
struct WIndex {
    double v, vi, b, g;
    bool prop;
};

// x 2^{B - ex} rounded to an integer, |x| <= 2^ex (integer operations; denormals are zero)
template <int B>
__device__ __forceinline__ long long to_fixed(double x, int ex)
{
    const long long u = __double_as_longlong(x);
    const int e = (int)((u >> 52) & 0x7FF);              // biased exponent
    const unsigned long long m = ((unsigned long long)u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = e - 1023 - 52 + B - ex;               // left shift of the mantissa
    unsigned long long r;
    if (sh >= 0)
        r = m << min(sh, 10);
    else
        r = sh > -54 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0ull;
    return u < 0 ? -(long long)r : (long long)r;
}

template <int L>
__device__ __forceinline__ WIndex weight_index(const EvalArgs &a, const Cell &C, int n1, int n2, bool full)
{
    WIndex w;
    w.v = w.vi = w.b = w.g = 0.0;
    w.prop = false;
    if (n1 < a.n1lo || n1 > a.n1hi || n2 < a.n2lo || n2 > a.n2hi) return w;
    const size_t at = (size_t)(n1 - a.n1lo) * (a.n2hi - a.n2lo + 1) + (n2 - a.n2lo);
    bool ev;
    if (L == 6) {
        const BetaEntry be = reinterpret_cast<const BetaEntry *>(a.btab)[at];
        ev = be.bf > 0.f;
        if (ev && full) {
            // Tang's table-driven exponential (as in the series kernels), degree 3
            const double y = fma(be.b, C.zw, be.lnb);
            const float jm = fmaf((float)GF_EXPTAB_STEPS, fmaf(be.bf, (float)C.zw, be.lnbf), 12582912.0f);
            const int idx = __float_as_int(jm) - 0x4B400000 + a.exptab_j0;
            if (idx >= 0 && idx < a.exptab_n) {
                const double2 t = a.exptab[idx];
                const double r = y - t.y;
                w.v = t.x * fma(fma(fma(r, -1.0 / 6.0, 0.5), r, -1.0), r, 1.0);
            }
            w.b = be.b;
            w.g = -be.b * C.delta;
        }
    } else {
        const BetaEntryF be = reinterpret_cast<const BetaEntryF *>(a.btab)[at];
        ev = isfinite(be.bl2);
        if (ev && full) {
            w.v = (double)(exp2f(-be.bl2 * (float)C.zw) * be.ib);
            w.b = (double)be.b;
            w.g = (double)(-be.b * (float)C.delta);
        }
    }
    if (ev) return w;
    const double c1 = a.a1 + n1, c2 = a.a2 + n2;
    const double aa = sqrt(c1 * c1 + c2 * c2);
    w.b = sqrt((a.k - aa) * (a.k + aa));
    sincos(w.b * C.zw, &w.vi, &w.v);
    w.g = w.b * C.delta;
    w.prop = true;
    return w;
}

// Value of entry e at an index: factor delta_pq - c_p c_q/k^2 (c_3^2 = beta^2 = -b^2 or
// beta^2) times -v (evanescent: Im of the weight) or (v + i vi)/beta; xz and yz (e = 4, 5), whose
// c_3 cancels 1/beta, -c/k^2 times b v (Re of the weight) or (v + i vi).
__device__ __forceinline__ double2 entry_value(const WIndex &w, int e, double c1, double c2, double ik2)
{
    double f = 1.0;
    if (e != 6) {
        const double b2 = w.prop ? w.b * w.b : -w.b * w.b;
        f = e == 0 ? 1.0 - c1 * c1 * ik2 : e == 1 ? 1.0 - c2 * c2 * ik2 : e == 2 ? 1.0 - b2 * ik2 : e == 3 ? -c1 * c2 * ik2 : e == 4 ? -c1 * ik2 : -c2 * ik2;
    }
    const bool mixed = e == 4 || e == 5;
    if (!w.prop) return make_double2(e == 6 ? -w.v : mixed ? f * w.b * w.v : -f * w.v, 0.0);
    if (!mixed) f /= w.b;
    return make_double2(f * w.v, f * w.vi);
}

__device__ __forceinline__ uint32_t pair_at(int i, long long a, long long b)
{
    switch (i) {
    case 0: return digit_pair<59, 0>(a, b);
    case 1: return digit_pair<59, 1>(a, b);
    case 2: return digit_pair<59, 2>(a, b);
    case 3: return digit_pair<59, 3>(a, b);
    case 4: return digit_pair<59, 4>(a, b);
    default: return digit_pair<59, 5>(a, b);
    }
}

// 2^61/p
__device__ __forceinline__ long long recip61(int p) { return (1ll << 61) / p; }

template <int L>
__global__ void __launch_bounds__(256) far_weights(EvalArgs a, const Cell *cells, int *rej, unsigned char *images, int maxcells, int nent)
{
    __shared__ Cell C;
    __shared__ long long rcp[PMAX + 1];
    const int c = blockIdx.x, kb = blockIdx.y;
    const int ntiles = (a.far_count[0] + TILE - 1) / TILE, T = rej[1];
    if (c * T >= ntiles) return;
    {
        const int *src = reinterpret_cast<const int *>(cells + c);
        for (int i = threadIdx.x; i < (int)(sizeof(Cell) / 4); i += blockDim.x) reinterpret_cast<int *>(&C)[i] = src[i];
    }
    if (threadIdx.x >= 1 && threadIdx.x <= PMAX) rcp[threadIdx.x] = recip61(threadIdx.x);
    __syncthreads();
    if (!C.ok) {
        // left over: its targets go to the series kernels' list, after those of the flagged cells before it (only the
        // last cell is shorter than T tiles, so the list's chunks are the far list's)
        if (kb != NKB) return;
        static_assert(GF_FAR_CELLS <= 256, "a thread per cell");
        const int before = __syncthreads_count(threadIdx.x < c && rej[2 + threadIdx.x] != 0);
        const int per = T * TILE, count = a.far_count[0];
        for (int i = threadIdx.x; i < per && c * per + i < count; i += blockDim.x) rej[2 + maxcells + before * per + i] = a.far_sorted[c * per + i];
        return;
    }
    if (kb == NKB && C.merged) return;
    const int kcol = kb == NKB ? 0 : kb;
    const int N1 = (int)rint(-a.a1), N2 = (int)rint(-a.a2);
    const double ik2 = 1.0 / (a.k * a.k);
    const float iscale = exp2f(-(float)C.ex);
    int st0 = 0;
    while (st0 < C.nst && C.st[st0].kb != kcol) ++st0;
    if (st0 == C.nst || (kb == NKB && C.st[st0].pi0 >= L)) return;
    // full rows: groups of 8, m1 = 8 m + r (even groups) and -1 - (8 m + r) (odd ones), then the
    // propagating ones
    const int frows = kb == NKB ? 0 : C.st[st0].rows[L - 1] * RBLK;
    const int rows = frows + (kb == NKB || (C.merged && kb == 0) ? RBLK : 0);
    for (int item = threadIdx.x; item < rows * (KB / 2); item += blockDim.x) {
        const int irow = item / (KB / 2), cp = item % (KB / 2);
        const bool prop = irow >= frows;
        const int row = prop ? irow - frows : irow;
        const int grp = row >> 3, r = row & 7;
        const int m1 = prop ? row - 8 : (grp & 1) ? -1 - (8 * (grp >> 1) + r) : 8 * (grp >> 1) + r;
        const bool first = kcol == 0 && cp == 0;  // its first column is m2 = 0: no partner, no sine
        const int m2 = kcol * KB + 2 * cp;
        WIndex w[4];                               // +m2, -m2 of the two columns
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q == 1 && first) {
                w[1].v = w[1].vi = w[1].b = w[1].g = 0.0;
                w[1].prop = false;
            } else {
                w[q] = weight_index<L>(a, C, N1 + m1, (q & 1) ? N2 - m2 - (q >> 1) : N2 + m2 + (q >> 1), !prop);
            }
        }
        const double c1 = a.a1 + (N1 + m1);
        for (int eo = 0; eo < nent; ++eo) {
            const int e = nent == 1 ? 6 : eo;
            // the full rows sum Im of the weights, for xz and yz Re (real for evanescent indices)
            const bool take_re = (e == 4 || e == 5) != prop;
            unsigned char *base = images + ((size_t)eo * maxcells + c) * Cap<L>::BYTES;
            long long X[4], Y[4], G[4];
            int x[4], y[4];
            float fr[4], fi[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const double2 v = entry_value(w[q], e, c1, a.a2 + ((q & 1) ? N2 - m2 - (q >> 1) : N2 + m2 + (q >> 1)), ik2);
                if (L == 6) {
                    X[q] = to_fixed<59>(v.x, C.ex);
                    Y[q] = w[q].prop ? to_fixed<59>(v.y, C.ex) : 0;
                    G[q] = to_fixed<61>(w[q].g, 0);
                } else {
                    fr[q] = (float)v.x * iscale;
                    fi[q] = (float)v.y * iscale;
                }
            }
            bool small = false;  // L = 6: below 2^-30 of the scale, carried in 32 bits
            for (int s = st0; s < C.nst && C.st[s].kb == kcol; ++s) {
                const Stage &S = C.st[s];
                const int p = S.p, i0 = prop ? S.pi0 : S.i0;
                if (i0 >= L) break;
                long long xc[2], xs[2];
                if (L == 6) {
                    if (p > 0) {
                        const long long rp = rcp[p];
                        if (small) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int g30 = mul30((int)(G[q] >> 31), (int)(rp >> 31)), t = mul30(x[q], g30);
                                x[q] = w[q].prop ? -mul30(y[q], g30) : t;
                                y[q] = t;
                            }
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const long long gp = p == 1 ? G[q] : mulq_unbiased(G[q], lim_h(rp), lim_l(rp));
                                const int gh = lim_h(gp), gl = lim_l(gp);
                                const long long t = mulq_unbiased(X[q], gh, gl);
                                if (w[q].prop) {
                                    X[q] = -mulq_unbiased(Y[q], gh, gl);
                                    Y[q] = t;
                                } else {
                                    X[q] = t;
                                }
                            }
                        }
                    }
                    if (!small && i0 >= 3) {
                        small = true;
#pragma unroll
                        for (int q = 0; q < 4; ++q) x[q] = (int)X[q], y[q] = (int)Y[q];
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const bool ru = !w[2 * q].prop || take_re, rv = !w[2 * q + 1].prop || take_re;
                        long long u, v;
                        if (small) {
                            u = ru ? x[2 * q] : y[2 * q];
                            v = rv ? x[2 * q + 1] : y[2 * q + 1];
                        } else {
                            u = ru ? X[2 * q] : Y[2 * q];
                            v = rv ? X[2 * q + 1] : Y[2 * q + 1];
                        }
                        xc[q] = u + v;
                        xs[q] = u - v;
                    }
                } else {
                    if (p > 0) {
                        const float ip = 1.0f / (float)p;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float gq = (float)w[q].g * ip, t = fr[q] * gq;
                            fr[q] = w[q].prop ? -fi[q] * gq : t;
                            fi[q] = t;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float u = !w[2 * q].prop || take_re ? fr[2 * q] : fi[2 * q],
                                    v = !w[2 * q + 1].prop || take_re ? fr[2 * q + 1] : fi[2 * q + 1];
                        xc[q] = (long long)__float2int_rn((u + v) * 0x1p29f) << 30;
                        xs[q] = (long long)__float2int_rn((u - v) * 0x1p29f) << 30;
                    }
                }
                if (first) xs[0] = 0;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    xc[q] = with_bias<59>(xc[q]);
                    xs[q] = with_bias<59>(xs[q]);
                }
                const bool own = prop && !C.merged;  // an image of its own
                unsigned char *img = base + (own ? 2 * C.timg + S.poff : S.off);
                const int step = own ? C.tpimg : C.timg;
                for (int i = C.merged ? min(S.i0, S.pi0) : i0; i < L; ++i) {
                    const int lead = C.merged && i >= S.pi0 ? RBLK : 0;  // propagating rows first
                    const int N = own ? RBLK : S.rows[i] * RBLK + lead;
                    const int at = prop ? row : row + lead;
                    if (at < N && i >= i0) {
                        const int o = (cp >> 2) * (N * 16) + (at >> 3) * 128 + (at & 7) * 16 + (cp & 3) * 4;
                        *reinterpret_cast<uint32_t *>(img + o) = pair_at(i, xc[0], xc[1]);
                        *reinterpret_cast<uint32_t *>(img + step + o) = pair_at(i, xs[0], xs[1]);
                    }
                    img += N * KB * 2;
                }
            }
        }
    }
}

// e^{2 pi i f}, 2^61 for 1, in integers: f = j/1024 + d, the plan's table of e^{2 pi i j/1024} and the
// Taylor polynomials of theta = 2 pi d (|theta| <= 3.1e-3: truncations below 2^-59).  An FP64 sine
// and cosine would hold the tile's warps for 16 cycles an operation.
__device__ __forceinline__ long long mulc(long long a, long long c) { return mulq(a, lim_h(c), lim_l(c)); }
__device__ __forceinline__ C64 phase64(const longlong2 *tab, double f)
{
    const long long F = __double2ll_rn((f - rint(f)) * 0x1p63);                // turns, 2^63 for 1
    const long long j = (F + (1ll << 52)) >> 53, rem = F - (j << 53);
    const longlong2 T = __ldg(tab + ((int)j & (GF_TRIG_STEPS - 1)));
    const long long th = mulc(rem << 9, 0x1921FB54442D1847ll);                 // theta 2^69: times pi/4
    const long long t2 = mulq(th, lim_h(th), lim_l(th));                      // theta^2 2^77
    const long long t4 = mulq(t2, lim_h(t2), lim_l(t2)) >> 16;                // theta^4 2^77
    const long long c6 = mulc(t2, (1ll << 61) / 6) - mulc(t4, (1ll << 61) / 120);
    const long long sn = (th - mulc(th, c6 >> 16)) >> 8;                      // sin theta 2^61
    const long long cm = (mulc(t4, (1ll << 61) / 24) - (t2 >> 1)) >> 16;      // (cos theta - 1) 2^61
    const C64 d = cmulq(C64{T.x, T.y}, limbs(C64{cm, sn}));
    return C64{T.x + d.x, T.y + d.y};
}

// x / (2 pi) as m + f, |f| <= 1/2
__device__ __forceinline__ double turns(double x, double &m)
{
    constexpr double i2p = 0.15915494309189535, i2p_lo = -9.839338337591243e-18;
    m = rint(x * i2p);
    return fma(x, i2p_lo, fma(x, i2p, -m));
}

// per target: v1^{1, 4, 8}, v2^{1, 2, 3, 4, 8, 12, 16}, (z - z_w)/delta, the lift
enum { V1 = 0, V1_4, V1_8, V2, V2_2, V2_3, V2_4, V2_8, V2_12, V2_16, VD, VLIFT, NVEC };

template <int L>
struct Smem {
    static constexpr int A_SLICE = TILE * KB * 2;                // 4 KiB
    static constexpr int A_BYTES = USLICES * A_SLICE;
    static constexpr int NBUF = 2;                               // units in flight
    static constexpr int SUMS = L == 6 ? 0 : TILE * 4 * 16;      // the four partial sums per target (L = 6: over the A buffers)
    static constexpr int VECS = TILE * NVEC * 16;                // powers, (z - z_w)/delta, the lift per target
    // MMA commands of a cell's stages, a list per issuing warp (at most 7 per image for L = 6,
    // 3 for L = 3), and where each stage's begin
    static constexpr int NCMD = L == 6 ? (MAXST + 24) * 7 : MAXST * 6;
    static constexpr int CMDS = NMW * (NCMD * 16 + (2 * MAXST + 4) * 4);
    static constexpr int CELL = ((int)sizeof(Cell) + 15) / 16 * 16;
    static constexpr int TOTAL = NBUF * (A_BYTES + UBYTES) + SUMS + VECS + CMDS + CELL + 256;
    static_assert(TOTAL <= 232448, "shared memory of one CTA");
};

__device__ __forceinline__ void arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(umma::smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(umma::smem_u32(bar)));
}
__device__ __forceinline__ void gen_sync() { asm volatile("bar.sync 1, %0;" ::"r"(NGW * 32) : "memory"); }

// One MMA: A slice (16-byte units from the stage's A buffer), B slice (from its B buffer; the
// stride of its row groups in the upper half), accumulator column with bit 31 =
// accumulate, instruction descriptor (f16 operands, fp32 accumulator, both K-major).
__device__ __forceinline__ uint4 mma_cmd(int aoff, int boff, int N, int col, bool acc)
{
    return make_uint4((uint32_t)aoff >> 4, ((uint32_t)boff >> 4) | ((uint32_t)N << 16), (uint32_t)col | (acc ? 0x80000000u : 0u),
                      (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TILE >> 4) << 24));
}
__device__ __forceinline__ void mma_issue(const uint4 &c, uint32_t tmem, uint32_t a16, uint32_t b16)
{
    // descriptors: no swizzle, 128 bytes between row groups of 8 (bits 32-45), version 1 (bit 46);
    // between the two K groups TILE * 16 bytes (A), N * 16 (B)
    constexpr uint32_t HI = (128u >> 4) | (1u << 14);
    const uint64_t ad = ((uint64_t)HI << 32) | (c.x + a16 + ((uint32_t)TILE << 16));
    const uint64_t bd = ((uint64_t)HI << 32) | (c.y + b16);
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                     tmem + (c.z & 0x7FFFFFFFu)),
                 "l"(ad), "l"(bd), "r"(c.w), "r"(c.z >> 31));
}

// Accumulator level l belongs to issuing warp owner(l): MMAs of different warps are not ordered
// against each other, those of one level are.  (L = 6: levels 0 and 5, 1 and 4, 2 and 3: seven
// products each.)
template <int L>
__device__ __forceinline__ int level_owner(int l) { return L == 6 ? min(l, 5 - l) : l; }

// The MMAs of one image with one phase factor's digits: weight digit i (of the stage's full
// rows, of its propagating rows or, merged, of both) times digit j into level i + j, those of
// issuing warp w.  `first`: the set's first stage, whose (i, 0) products start the levels.
// Written to out (null: counted only).
template <int L>
__device__ int image_cmds(uint4 *out, int w, int tset, const Cell &c, const Stage &S, int aoff, int boff, bool own, bool first)
{
    int n = 0;
    const int i0 = own ? S.pi0 : c.merged ? min(S.i0, S.pi0) : S.i0;
    for (int pass = first ? 0 : 1; pass < 2; ++pass) {
        int b = boff;
        for (int i = i0; i < L; ++i) {
            const bool lead = c.merged && i >= S.pi0;
            const int N = (own ? 1 : S.rows[i] + (lead ? 1 : 0)) * RBLK;
            const int j1 = pass == 0 ? 1 : L - i;
            for (int j = (pass == 1 && first) ? 1 : 0; j < j1; ++j) {
                if (level_owner<L>(i + j) != w) continue;
                const int col = own ? (i + j) * RBLK : c.col[i + j] * 16 + (c.merged && !lead ? RBLK : 0);
                if (out) out[n] = mma_cmd(aoff + j * Smem<L>::A_SLICE, b, N, tset + col, pass == 1);
                ++n;
            }
            b += N * KB * 2;
        }
    }
    return n;
}

// Unit of stage t: its first stage.
__device__ __forceinline__ int unit_begin(const unsigned char *ust, int nu, int t)
{
    int u = 0;
    while (u + 1 < nu && ust[u + 1] <= t) ++u;
    return ust[u];
}

// Digits of a stage's phase factor.
template <int L>
__device__ __forceinline__ int stage_digits(const Cell &c, const Stage &S, bool own)
{
    return L - (own ? S.pi0 : c.merged ? min(S.i0, S.pi0) : S.i0);
}

// The commands of issuing warp w for stage s: of a full pass (cos or sin; L = 3: both), or of the
// pass of the propagating part (L = 6, not merged; its stages are all cos, then all sin).
template <int L>
__device__ int stage_cmds(uint4 *out, int w, const Cell &c, int s, bool own)
{
    constexpr int AS = Smem<L>::A_SLICE;
    const int q = own && s >= c.npst, t = s - q * c.npst;
    const int t0 = own ? unit_begin(c.pust, c.npu, t) : unit_begin(c.ust, c.nu, t);
    const Stage &S = c.st[t];
    int sl = 0;
    for (int k = t0; k < t; ++k) sl += stage_digits<L>(c, c.st[k], own);
    if (L == 6)
        return image_cmds<L>(out, w, q * L * RBLK, c, S, sl * AS, own ? S.poff - c.st[t0].poff : S.off - c.st[t0].off, own, t == 0);
    // L = 3: a unit's B buffer holds its cos images, then its sin images; a stage's digits: cos, sin
    int t1 = c.nst;
    for (int u = c.nu; u > 0 && c.ust[u] > t; --u) t1 = c.ust[u];
    const int ub = c.st[t1 - 1].off + c.st[t1 - 1].img - c.st[t0].off;
    int n = 0;
    for (int h = 0; h < 2; ++h)
        n += image_cmds<L>(out ? out + n : nullptr, w, h * c.cols, c, S, (2 * sl + h * stage_digits<L>(c, S, false)) * AS,
                           h * ub + S.off - c.st[t0].off, false, t == 0);
    return n;
}

// accumulator columns c .. c + 3 of this thread's row (the load is not waited for)
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr));
}

// digits 0 .. J-1 of four columns (2^61 for 1) into the A slices of one phase factor
template <int J>
__device__ __forceinline__ void put_digits(uint32_t dst, const long long (&x)[4])
{
    const long long b0 = with_bias<61>(x[0]), b1 = with_bias<61>(x[1]), b2 = with_bias<61>(x[2]), b3 = with_bias<61>(x[3]);
#define GF_PUT(I)                                                                                                       \
    if (J > I)                                                                                                          \
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + I * (TILE * KB * 2)), "r"(digit_pair<61, I>(b0, b1)), \
                     "r"(digit_pair<61, I>(b2, b3))                                                                      \
                     : "memory");
    GF_PUT(0) GF_PUT(1) GF_PUT(2) GF_PUT(3) GF_PUT(4) GF_PUT(5)
#undef GF_PUT
}

// the same for at most three digits of 32-bit numbers (2^30 for 1)
template <int I>
__device__ __forceinline__ uint32_t digit_pair32(uint32_t a, uint32_t b)
{
    constexpr int s = 21 - 10 * I, t = s - 16;
    const uint32_t lo = a >> s, hi = t > 0 ? b >> t : b << (-t);
    uint32_t u;
    if (I == 0)
        u = ((lo & 0x7FFu) | (hi & 0x07FF0000u)) + 0x64006400u;
    else
        u = ((lo & 0x3FFu) | (hi & 0x03FF0000u)) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&u), __halves2half2(__ushort_as_half(0x6600), __ushort_as_half(0x6600)));
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ void put_digits32(int J, uint32_t dst, const int (&x)[4])
{
    constexpr uint32_t bias = (512u << 21) + (512u << 11) + (512u << 1) + 1u;
    const uint32_t b0 = (uint32_t)x[0] + bias, b1 = (uint32_t)x[1] + bias, b2 = (uint32_t)x[2] + bias, b3 = (uint32_t)x[3] + bias;
#define GF_PUT(I)                                                                                                      \
    if (J > I)                                                                                                         \
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + I * (TILE * KB * 2)), "r"(digit_pair32<I>(b0, b1)), \
                     "r"(digit_pair32<I>(b2, b3))                                                                       \
                     : "memory");
    GF_PUT(0) GF_PUT(1) GF_PUT(2)
#undef GF_PUT
}

// One accumulator block of this thread: its four rows at every level, combined.  64-bit:
// 2^56 for 1; levels 0 .. 3 are exact integers, 4 and 5 are rounded below the last unit.
// col: a level's first column in blocks of 16 (null: levels 16 columns apart).
__device__ __forceinline__ void block64(uint32_t t, const unsigned char *col, const unsigned char *width, int m, long long (&R)[4])
{
    constexpr int L = 6;
    uint32_t d[L][4];
#pragma unroll
    for (int l = 0; l < L; ++l) {
        if (width[l] > m)
            tmem_ld4(t + (col ? col[l] : l) * 16, d[l]);
        else
            d[l][0] = d[l][1] = d[l][2] = d[l][3] = 0u;
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const float low = fmaf(__uint_as_float(d[5][s]), 0x1p-12f, __uint_as_float(d[4][s]) * 0x1p-2f);
        R[s] = (long long)__float2int_rn(low) + ((long long)__float2int_rn(__uint_as_float(d[3][s])) << 8) +
               ((long long)__float2int_rn(__uint_as_float(d[2][s])) << 18) + ((long long)__float2int_rn(__uint_as_float(d[1][s])) << 28) +
               ((long long)__float2int_rn(__uint_as_float(d[0][s])) << 38);
    }
}
// rows that have no digit at levels 0 .. 2 (below 2^-30 of the scale each): 32 bits, 2^53 for 1
__device__ __forceinline__ void block32(uint32_t t, const unsigned char *col, const unsigned char *width, int m, int (&R)[4])
{
    uint32_t d[3][4];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        if (width[l + 3] > m)
            tmem_ld4(t + col[l + 3] * 16, d[l]);
        else
            d[l][0] = d[l][1] = d[l][2] = d[l][3] = 0u;
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int s = 0; s < 4; ++s)
        R[s] = __float2int_rn(fmaf(__uint_as_float(d[2][s]), 0x1p-15f, __uint_as_float(d[1][s]) * 0x1p-5f)) +
               (__float2int_rn(__uint_as_float(d[0][s])) << 5);
}
__device__ __forceinline__ void blockf(uint32_t t, const unsigned char *col, const unsigned char *width, int m, float (&R)[4])
{
    constexpr int L = 3;
    uint32_t d[L][4];
#pragma unroll
    for (int l = 0; l < L; ++l) {
        if (width[l] > m)
            tmem_ld4(t + (col ? col[l] : l) * 16, d[l]);
        else
            d[l][0] = d[l][1] = d[l][2] = d[l][3] = 0u;
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int s = 0; s < 4; ++s)
        R[s] = fmaf(__uint_as_float(d[0][s]), 0x1p-18f, fmaf(__uint_as_float(d[1][s]), 0x1p-28f, __uint_as_float(d[2][s]) * 0x1p-38f));
}

__device__ __forceinline__ float2 cmf(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 to_f2(const C64 &v) { return make_float2((float)v.x * 0x1p-61f, (float)v.y * 0x1p-61f); }
// t v + r
__device__ __forceinline__ float2 horner(float2 t, float2 v, float rx, float ry)
{
    return make_float2(fmaf(t.x, v.x, fmaf(-t.y, v.y, rx)), fmaf(t.x, v.y, fmaf(t.y, v.x, ry)));
}

// What bounds it: integer issue.  Per tile and thread about 3000 instructions make the digits
// and 2500 finish the sums; the products themselves keep the tensor pipe busy for a fifth of
// the time.  Hence: cos and sin in passes of their own (each digit is made once, and both halves of
// the rows share it: 512 accumulator columns are what one phase factor needs), 32-bit arithmetic
// for every stage and row block that needs at most 30 bits, real parts only where a pass needs no
// others, MMA commands written once per cell.
template <typename R, int L>
__global__ void __launch_bounds__(THREADS, 1) far_product(EvalArgs a, const Cell *cells, const int *rej, const unsigned char *images, int maxcells,
                                                          int nent, int *err)
{
    typedef Smem<L> SM;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sA = smem, *sB = smem + SM::NBUF * SM::A_BYTES;
    // L = 6: the partial sums lie over the A buffers, whose MMAs are done by then
    longlong2 *sums = reinterpret_cast<longlong2 *>(L == 6 ? sA : sB + SM::NBUF * UBYTES);
    longlong2 *vecs = reinterpret_cast<longlong2 *>(sB + SM::NBUF * UBYTES + SM::SUMS);
    uint4 *cmds = reinterpret_cast<uint4 *>(vecs + TILE * NVEC);
    int *cmd0 = reinterpret_cast<int *>(cmds + NMW * SM::NCMD);  // per issuing warp: [MAXST + 1] full stages, [MAXST + 1] propagating
    Cell *cell = reinterpret_cast<Cell *>(cmd0 + NMW * (2 * MAXST + 4));
    uint64_t *bars = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(cell) + SM::CELL);
    // A unit written; B unit landed; A, B unit multiplied (an arrival per issuing warp); pass done; accumulators read
    // and, after a wait that ran out, an issuing warp's MMAs
    uint64_t *afull = bars, *bfull = bars + 2, *afree = bars + 4, *bfree = bars + 6, *accf = bars + 8, *tfree = bars + 9, *mdone = bars + 10;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 10 + NMW);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int count = a.far_count[0], ntiles = (count + TILE - 1) / TILE, T = rej[1];
    if ((int)blockIdx.x >= ntiles) return;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(umma::smem_u32(tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        for (int q = 0; q < 10 + NMW; ++q) {
            const int n = (q < 2 || q == 9) ? NGW : (q < 4 || q > 9 ? 1 : NMW);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(umma::smem_u32(&bars[q])), "r"(n));
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tslot;
    constexpr int NPASS = L == 6 ? 3 : 1;  // L = 6: cos, sin, propagating (cells not merged); L = 3: cos and sin at once
    int ga = 0, gu = 0, gp = 0;            // A units, B units and passes so far (barrier phases)
    int cur = -1;                          // cell held in shared memory
    bool ok = true;
    // self-test: the unit (copies, MMAs) or the pass (a warp that finishes sums) whose wait counts as run out
    const int drop = blockIdx.x == 0 && warp == (a.drop_warp < 4 ? NGW + a.drop_warp : 0) ? a.drop_unit - 1 : -1;
    // After a wait that ran out every warp still takes part in the barriers of its tile;
    // the whole CTA leaves at the next tile.
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int ci = tile / T;
        ok = __syncthreads_and(ok ? 1 : 0) != 0;
        if (!ok) break;
        if (ci != cur) {
            const int *src = reinterpret_cast<const int *>(cells + ci);
            for (int i = threadIdx.x; i < (int)(sizeof(Cell) / 4); i += blockDim.x) reinterpret_cast<int *>(cell)[i] = src[i];
            __syncthreads();
            cur = ci;
            if (warp > NGW && cell->ok) {
                // this warp's MMA commands for the cell, a lane per stage
                const int w = warp - NGW - 1;
                uint4 *cw = cmds + w * SM::NCMD;
                int *c0 = cmd0 + w * (2 * MAXST + 4);
                int at = 0;
                for (int q = 0; q < (L == 6 ? 2 : 1); ++q) {
                    const int ns = q ? (cell->merged ? 0 : 2 * cell->npst) : cell->nst;
                    const int mine = lane < ns ? stage_cmds<L>(nullptr, w, *cell, lane, q == 1) : 0;
                    int incl = mine;
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += v;
                    }
                    if (lane < ns) {
                        c0[q * (MAXST + 1) + lane] = at + incl - mine;
                        stage_cmds<L>(cw + at + incl - mine, w, *cell, lane, q == 1);
                    }
                    at += __shfl_sync(0xffffffffu, incl, 31);
                    if (lane == 0) c0[q * (MAXST + 1) + ns] = at;
                }
                __syncwarp();
            }
        }
        if (!cell->ok) continue;
        // L = 3 with several entries: digits that fit the buffers are made once
        const bool resident = L == 3 && cell->nu <= SM::NBUF;
        if (warp >= NGW) {
            if (lane == 0) {
                const int w = warp - NGW - 1;  // -1: copies
                const int ga0 = ga;
                for (int eo = 0; ok && eo < nent; ++eo) {
                  const unsigned char *img = images + ((size_t)eo * maxcells + ci) * Cap<L>::BYTES;
                  for (int pass = 0; ok && pass < NPASS; ++pass) {
                    const int npu = cell->npu, nu = pass == 2 ? 2 * npu : cell->nu;
                    if (nu == 0) continue;
                    // the previous pass's accumulators have been read
                    if (w >= 0 && gp > 0) ok = umma::mbar_wait_sleep(umma::smem_u32(tfree), (gp - 1) & 1) && !*abort_flag;
                    for (int u = 0; ok && u < nu; ++u, ++gu) {
                        const int buf = gu % SM::NBUF, ph = (gu / SM::NBUF) & 1;
                        const bool again = resident && eo > 0;  // the digits are there already
                        const int au = again ? ga0 + u : ga, abuf = au % SM::NBUF;
                        if (!again) ++ga;
                        const int q = pass == 2 && u >= npu;
                        const int t0 = pass == 2 ? cell->pust[u - q * npu] : cell->ust[u];
                        const int t1 = pass == 2 ? cell->pust[u - q * npu + 1] : cell->ust[u + 1];
                        if (w < 0) {
                            if (gu >= SM::NBUF) ok = umma::mbar_wait_sleep(umma::smem_u32(&bfree[buf]), ph ^ 1) && !*abort_flag;
                            if (!ok || gu == drop) {
                                ok = false;
                                break;
                            }
                            const Stage &S0 = cell->st[t0], &S1 = cell->st[t1 - 1];
                            const int ub = S1.off + S1.img - S0.off, up = S1.poff + S1.pimg - S0.poff;
                            const int bytes = L == 3 ? 2 * ub : pass == 2 ? up : ub;
                            const uint32_t bar = umma::smem_u32(&bfull[buf]);
                            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
                            auto copy = [&](int dst, int src, int n) {
                                if (n > 0)
                                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                                     umma::smem_u32(sB + buf * UBYTES) + dst),
                                                 "l"(img + src), "r"(n), "r"(bar)
                                                 : "memory");
                            };
                            if (L == 3) {
                                copy(0, S0.off, ub);
                                copy(ub, cell->timg + S0.off, ub);
                            } else if (pass == 2) {
                                copy(0, 2 * cell->timg + q * cell->tpimg + S0.poff, up);
                            } else {
                                copy(0, pass * cell->timg + S0.off, ub);
                            }
                        } else {
                            ok = (again || umma::mbar_wait_sleep(umma::smem_u32(&afull[abuf]), (au / SM::NBUF) & 1)) &&
                                 umma::mbar_wait_sleep(umma::smem_u32(&bfull[buf]), ph) && !*abort_flag && gu != drop;
                            if (!ok) break;
                            asm volatile("tcgen05.fence::after_thread_sync;");
                            const uint32_t a16 = umma::smem_u32(sA + abuf * SM::A_BYTES) >> 4, b16 = umma::smem_u32(sB + buf * UBYTES) >> 4;
                            const int *c0 = cmd0 + w * (2 * MAXST + 4) + (pass == 2 ? MAXST + 1 + q * cell->npst : 0);
                            const uint4 *cp = cmds + w * SM::NCMD + c0[t0], *ce = cmds + w * SM::NCMD + c0[t1];
#pragma unroll 4
                            for (; cp < ce; ++cp) mma_issue(*cp, tmem, a16, b16);
                            if (!resident || eo == nent - 1) commit(&afree[abuf]);
                            commit(&bfree[buf]);
                        }
                    }
                    if (ok && w >= 0) commit(accf);
                    ++gp;
                  }
                }
                if (!ok) {
                    *abort_flag = 1;
                    if (err) atomicExch(err, 1);
                }
            }
            __syncwarp();
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            // (lane 0 keeps the phase counters; the other lanes only follow the cells)
        } else {
            const int quarter = warp & 3, g = warp >> 2, r = quarter * 32 + lane;
            const int slot = tile * TILE + r;
            const bool valid = slot < count;
            const int idx = valid ? a.far_sorted[slot] : 0;
            if (g == 2) {
                // the lift e^{i alpha.x} e^{i N.t}
                C64 li{0, 0};
                if (valid) {
                    double m1, m2;
                    const double f1 = turns(a.x[3 * (size_t)idx], m1), f2 = turns(a.x[3 * (size_t)idx + 1], m2);
                    double ph = a.a1 * m1 + a.a2 * m2;
                    ph -= rint(ph);
                    ph += (a.a1 + rint(-a.a1)) * f1 + (a.a2 + rint(-a.a2)) * f2;
                    li = phase64(a.trig, ph);
                }
                reinterpret_cast<double2 *>(vecs)[TILE * VLIFT + r] = make_double2((double)li.x * 0x1p-61, (double)li.y * 0x1p-61);
            } else if (g < 2) {
                // the powers of v_1 = e^{i t1} (g = 0), of v_2 = e^{i t2}, and (z - z_w)/delta (g = 1)
                double m;
                const double f = valid ? turns(a.x[3 * (size_t)idx + g], m) : 0.0;
                auto put = [&](int i, const C64 &v) { vecs[TILE * i + r] = longlong2{v.x, v.y}; };
                const C64 v = phase64(a.trig, f);
                const Lim l = limbs(v);
                const C64 u2 = cmulq(v, l);
                const Lim l2 = limbs(u2);
                const C64 u4 = cmulq(u2, l2);
                const Lim l4 = limbs(u4);
                const C64 u8 = cmulq(u4, l4);
                if (g == 0) {
                    put(V1, v);
                    put(V1_4, u4);
                    put(V1_8, u8);
                } else {
                    put(V2, v);
                    put(V2_2, u2);
                    put(V2_3, cmulq(v, l2));
                    put(V2_4, u4);
                    put(V2_8, u8);
                    put(V2_12, cmulq(u8, l4));
                    put(V2_16, cmulq(u8, limbs(u8)));
                    const double z = valid ? fabs(a.x[3 * (size_t)idx + 2]) : cell->zw;
                    vecs[TILE * VD + r].x = __double2ll_rn((z - cell->zw) * cell->idelta * 0x1p61);
                }
            }
            gen_sync();
            const uint32_t adst = umma::smem_u32(sA) + (g >> 1) * (TILE * 16) + (r >> 3) * 128 + (r & 7) * 16 + (g & 1) * 8;
            auto vec = [&](int i) { return C64{vecs[TILE * i + r].x, vecs[TILE * i + r].y}; };
            auto unit_start = [&]() {
                if (ga >= SM::NBUF)
                    ok = __all_sync(0xffffffffu,
                                    umma::mbar_wait_sleep(umma::smem_u32(&afree[ga % SM::NBUF]), (ga / SM::NBUF - 1) & 1) && !*abort_flag);
                return adst + (ga % SM::NBUF) * SM::A_BYTES;
            };
            auto unit_end = [&]() {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive(&afull[ga % SM::NBUF]);
                ++ga;
            };
            auto pass_begin = [&]() {
                if (ok) ok = __all_sync(0xffffffffu, umma::mbar_wait_sleep(umma::smem_u32(accf), gp & 1) && !*abort_flag) && gp != drop;
                asm volatile("tcgen05.fence::after_thread_sync;");
            };
            auto pass_end = [&]() {
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0) arrive(tfree);
                ++gp;
            };
            const uint32_t tw = tmem + ((uint32_t)(quarter * 32) << 16);
            for (int eo = 0; eo < nent; ++eo) {
            const int e = nent == 1 ? 6 : eo;
            C64 full{0, 0}, pr{0, 0};  // this thread's share of the sums
            float2 fullf = make_float2(0.f, 0.f), prf = fullf;
            if (L == 6) {
                for (int pass = 0; pass < NPASS; ++pass) {
                    const int nu = pass == 2 ? 2 * cell->npu : cell->nu;
                    if (nu == 0) continue;
                    {
                        // powers of v2: this thread's columns are 16 kb + 4 g + q, q < 4
                        const long long D = vecs[TILE * VD + r].x;
                        const int Dh = lim_h(D), Dl = lim_l(D), D30 = (int)(D >> 31);
                        const Lim l1 = limbs(vec(V2)), l2 = limbs(vec(V2_2)), l3 = limbs(vec(V2_3));
                        const C64 base0 = g == 0 ? C64{1ll << 61, 0} : vec(V2_3 + g);
                        C64 base = base0;
                        long long x[4];
                        int y[4];
                        bool small = false;  // carried in 32 bits
                        for (int u = 0; ok && u < nu; ++u) {
                          const int q1 = pass == 2 && u >= cell->npu, pu = u - q1 * cell->npu;
                          const int t0 = pass == 2 ? cell->pust[pu] : cell->ust[u], t1 = pass == 2 ? cell->pust[pu + 1] : cell->ust[u + 1];
                          uint32_t dst = unit_start();
                          if (!ok) break;
                          for (int s = t0; s < t1; ++s) {
                            const Stage &S = cell->st[s];
                            const bool sine = pass == 1 || q1;
                            const int J = stage_digits<L>(*cell, S, pass == 2);
                            if (S.p == 0) {
                                if (S.kb > 0)
                                    base = cmulq(base, limbs(vec(V2_16)));
                                else
                                    base = base0;
                                small = J <= 3;
                                if (small) {
                                    const C32 b3 = to_c32(base);
                                    const C32 w1{l1.ch, l1.sh}, w2{l2.ch, l2.sh}, w3{l3.ch, l3.sh};
                                    y[0] = sine ? b3.y : b3.x;
                                    y[1] = sine ? mul30_im(b3, w1) : mul30_re(b3, w1);
                                    y[2] = sine ? mul30_im(b3, w2) : mul30_re(b3, w2);
                                    y[3] = sine ? mul30_im(b3, w3) : mul30_re(b3, w3);
                                } else {
                                    x[0] = sine ? base.y : base.x;
                                    x[1] = sine ? mulq_im(base, l1) : mulq_re(base, l1);
                                    x[2] = sine ? mulq_im(base, l2) : mulq_re(base, l2);
                                    x[3] = sine ? mulq_im(base, l3) : mulq_re(base, l3);
                                }
                            } else {
                                if (!small && J <= 3) {
                                    small = true;
#pragma unroll
                                    for (int q = 0; q < 4; ++q) y[q] = (int)(x[q] >> 31);
                                }
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    if (small)
                                        y[q] = mul30(y[q], D30);
                                    else
                                        x[q] = mulq(x[q], Dh, Dl);
                                }
                            }
                            if (small)
                                put_digits32(J, dst, y);
                            else if (J == 6)
                                put_digits<6>(dst, x);
                            else if (J == 5)
                                put_digits<5>(dst, x);
                            else
                                put_digits<4>(dst, x);
                            dst += J * SM::A_SLICE;
                          }
                          unit_end();
                        }
                    }
                    pass_begin();
                    if (ok) {
                        auto conj64 = [](C64 v) { return C64{v.x, -v.y}; };
                        if (pass < 2) {
                            // this thread's rows: 8 m + 4 (g & 1) + s, s < 4, of the blocks' half g >> 1
                            // (half 1: powers of the conjugate); R is real
                            const bool h = g >= 2;
                            const uint32_t t0 = tw + (cell->merged ? RBLK : 0) + 4 * g;
                            const Lim lv = limbs(h ? conj64(vec(V1)) : vec(V1));
                            const C64 p8 = h ? conj64(vec(V1_8)) : vec(V1_8);
                            const int w5 = cell->width[L - 1], w2 = min(w5, (int)cell->width[2]);
                            C64 Z{0, 0};
                            {
                                // blocks without a digit at levels 0 .. 2 take 32 bits
                                const C32 s1{lv.ch, lv.sh}, s8 = to_c32(p8);
                                C32 Y{0, 0};
                                for (int m = w5 - 1; m >= w2; --m) {
                                    int Rv[4];
                                    block32(t0 + m * RBLK, cell->col, cell->width, m, Rv);
                                    C32 t{Rv[3], 0};
#pragma unroll
                                    for (int s = 2; s >= 0; --s) {
                                        t = cmul30(t, s1);
                                        t.x += Rv[s];
                                    }
                                    Y = cmul30(Y, s8);
                                    Y.x += t.x;
                                    Y.y += t.y;
                                }
                                Z = C64{(long long)Y.x << 3, (long long)Y.y << 3};
                            }
                            const Lim l8 = limbs(p8);
                            for (int m = w2 - 1; m >= 0; --m) {
                                long long Rv[4];
                                block64(t0 + m * RBLK, cell->col, cell->width, m, Rv);
                                C64 t{Rv[3], 0};
#pragma unroll
                                for (int s = 2; s >= 0; --s) {
                                    t = cmulq(t, lv);
                                    t.x += Rv[s];
                                }
                                Z = cmulq(Z, l8);
                                Z.x += t.x;
                                Z.y += t.y;
                            }
                            if (g & 1) Z = cmulq(Z, limbs(h ? conj64(vec(V1_4)) : vec(V1_4)));
                            if (h) Z = cmulq(Z, lv);
                            if (pass == 0) {
                                full.x += Z.x;
                                full.y += Z.y;
                            } else {  // times i
                                full.x -= Z.y;
                                full.y += Z.x;
                            }
                        }
                        if (pass == 2 || cell->merged) {
                            // propagating rows m1 = 4 g + s - 8
                            const Lim lv = limbs(vec(V1));
                            long long Rc[4], Rs[4] = {0, 0, 0, 0};
                            block64(tw + 4 * g, pass == 2 ? nullptr : cell->col, cell->pwidth, 0, Rc);
                            if (pass == 2) block64(tw + L * RBLK + 4 * g, nullptr, cell->pwidth, 0, Rs);
                            C64 t{Rc[3], Rs[3]};
#pragma unroll
                            for (int s = 2; s >= 0; --s) {
                                t = cmulq(t, lv);
                                t.x += Rc[s];
                                t.y += Rs[s];
                            }
                            if (g != 2) t = cmulq(t, limbs(g == 0 ? conj64(vec(V1_8)) : g == 1 ? conj64(vec(V1_4)) : vec(V1_4)));
                            if (pass == 1) {
                                pr.x -= t.y;
                                pr.y += t.x;
                            } else {
                                pr.x += t.x;
                                pr.y += t.y;
                            }
                        }
                    }
                    pass_end();
                }
            } else {
                if (!(resident && eo > 0)) {
                    const int D30 = (int)(vecs[TILE * VD + r].x >> 31);
                    const C32 w1 = to_c32(vec(V2)), w16 = to_c32(vec(V2_16));
                    C32 b3 = g == 0 ? C32{1 << 30, 0} : to_c32(vec(V2_3 + g));
                    int yc[4], ys[4];
                    for (int u = 0; ok && u < cell->nu; ++u) {
                      uint32_t dst = unit_start();
                      if (!ok) break;
                      for (int s = cell->ust[u]; s < cell->ust[u + 1]; ++s) {
                        const Stage &S = cell->st[s];
                        const int J = stage_digits<L>(*cell, S, false);
                        if (S.p == 0) {
                            if (S.kb > 0) b3 = cmul30(b3, w16);
                            C32 t = b3;
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                yc[q] = t.x;
                                ys[q] = t.y;
                                if (q < 3) t = cmul30(t, w1);
                            }
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                yc[q] = mul30(yc[q], D30);
                                ys[q] = mul30(ys[q], D30);
                            }
                        }
                        put_digits32(J, dst, yc);
                        put_digits32(J, dst + J * SM::A_SLICE, ys);
                        dst += 2 * J * SM::A_SLICE;
                      }
                      unit_end();
                    }
                }
                pass_begin();
                if (ok) {
                    const float2 v1 = to_f2(vec(V1)), v4 = to_f2(vec(V1_4)), v8 = to_f2(vec(V1_8));
                    auto cj = [](float2 v, bool h) { return make_float2(v.x, h ? -v.y : v.y); };
                    const int cs = cell->cols;
                    {
                        const bool h = g >= 2;  // rows as for L = 6
                        const uint32_t t0 = tw + (cell->merged ? RBLK : 0) + 4 * g;
                        const float2 v = cj(v1, h), p8 = cj(v8, h);
                        float2 Z = make_float2(0.f, 0.f);
                        for (int m = cell->width[L - 1] - 1; m >= 0; --m) {
                            float Rc[4], Rs[4];
                            blockf(t0 + m * RBLK, cell->col, cell->width, m, Rc);
                            blockf(t0 + cs + m * RBLK, cell->col, cell->width, m, Rs);
                            float2 t = make_float2(Rc[3], Rs[3]);
#pragma unroll
                            for (int s = 2; s >= 0; --s) t = horner(t, v, Rc[s], Rs[s]);
                            Z = horner(Z, p8, t.x, t.y);
                        }
                        if (g & 1) Z = cmf(Z, cj(v4, h));
                        if (h) Z = cmf(Z, v);
                        fullf = Z;
                    }
                    if (cell->merged) {
                        float Rc[4], Rs[4];
                        blockf(tw + 4 * g, cell->col, cell->pwidth, 0, Rc);
                        blockf(tw + cs + 4 * g, cell->col, cell->pwidth, 0, Rs);
                        float2 t = make_float2(Rc[3], Rs[3]);
#pragma unroll
                        for (int s = 2; s >= 0; --s) t = horner(t, v1, Rc[s], Rs[s]);
                        if (g != 2) t = cmf(t, g == 0 ? cj(v8, true) : cj(v4, g == 1));
                        prf = t;
                    }
                }
                pass_end();
            }
            // the four threads of a target add up
            if (L == 6) {
                sums[g * TILE + r] = longlong2{full.x, full.y};
                sums[(4 + g) * TILE + r] = longlong2{pr.x, pr.y};
            } else {
                reinterpret_cast<float4 *>(sums)[g * TILE + r] = make_float4(fullf.x, fullf.y, prf.x, prf.y);
            }
            gen_sync();
            if (ok && g == 0 && valid) {
                // S = prop + i full (xz, yz: full + i prop, times the sign of x3), lifted by
                // e^{i alpha.x} e^{i N.t} (i/8pi^2)
                const double2 li = reinterpret_cast<const double2 *>(vecs)[TILE * VLIFT + r];
                const int ne = gf_out_entries(a.which);
                const bool re_full = e == 4 || e == 5;
                const double sg = re_full && a.x[3 * (size_t)idx + 2] < 0.0 ? -1.0 : 1.0;
                if (L == 6) {
                    for (int q = 1; q < 4; ++q) {
                        const longlong2 t = sums[q * TILE + r], u = sums[(4 + q) * TILE + r];
                        full.x += t.x;
                        full.y += t.y;
                        pr.x += u.x;
                        pr.y += u.y;
                    }
                    const double sc = sg * cell->scale * 0x1p-56 * (1.0 / (8.0 * GF_PI * GF_PI));
                    const long long ix = re_full ? full.x - pr.y : pr.x - full.y, iy = re_full ? full.y + pr.x : pr.y + full.x;
                    reinterpret_cast<double2 *>(a.out)[(size_t)idx * ne + eo] =
                        cmul(make_double2(-li.y, li.x), make_double2((double)ix * sc, (double)iy * sc));
                } else {
                    for (int q = 1; q < 4; ++q) {
                        const float4 t = reinterpret_cast<const float4 *>(sums)[q * TILE + r];
                        fullf.x += t.x;
                        fullf.y += t.y;
                        prf.x += t.z;
                        prf.y += t.w;
                    }
                    const float sc = (float)(sg * cell->scale * (1.0 / (8.0 * GF_PI * GF_PI)));
                    const float fx = fullf.x * sc, fy = fullf.y * sc, px = prf.x * sc, py = prf.y * sc;
                    const float2 S = re_full ? make_float2(fx - py, fy + px) : make_float2(px - fy, py + fx);
                    reinterpret_cast<float2 *>(a.out)[(size_t)idx * ne + eo] = cmul(make_float2(-(float)li.y, (float)li.x), S);
                }
            }
            if (eo + 1 < nent) gen_sync();  // (the sums' memory is free again)
            }
            if (!ok) {
                *abort_flag = 1;
                if (err) atomicExch(err, 1);
            }
        }
    }
    // After a wait that ran out anywhere: before the CTA exits, copies in flight (of the last NBUF units
    // issued, gu of them) land and issued MMAs are done.  (Otherwise the last pass's accumulators, which every
    // copy and MMA precedes, have been read.)
    if (!__syncthreads_and(ok ? 1 : 0)) {
        if (warp == NGW && lane == 0)
            for (int g = max(0, gu - SM::NBUF); g < gu; ++g) umma::mbar_wait_sleep(umma::smem_u32(&bfull[g % SM::NBUF]), (g / SM::NBUF) & 1);
        if (warp > NGW && lane == 0) {
            commit(&mdone[warp - NGW - 1]);
            umma::mbar_wait_sleep(umma::smem_u32(&mdone[warp - NGW - 1]), 0);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

}  // namespace

// Cells' flags and the targets left over (at most all), before the images.
static size_t rej_bytes(int nc, int64_t n) { return (sizeof(int) * (nc + 2 + n) + 255) / 256 * 256; }

// Bytes of scratch for n targets (cells, list of targets left over, images) and the
// number of cells; 0 bytes: no product path for so few targets.
size_t gf_far_product_bytes(int precision, int64_t n, int nent, int *maxcells)
{
    const int64_t tiles = (n + TILE - 1) / TILE;
    const int nc = (int)(tiles < GF_FAR_CELLS ? tiles : GF_FAR_CELLS);
    *maxcells = nc;
    const size_t img = precision == GF_FP64 ? (size_t)Cap<6>::BYTES : (size_t)Cap<3>::BYTES;
    return (sizeof(Cell) * nc + 255) / 256 * 256 + rej_bytes(nc, n) + img * nc * nent;
}

template <typename R, int L>
static cudaError_t launch_product(EvalArgs &a, int nsm, cudaStream_t s)
{
    const int nc = a.mma_cells;
    unsigned char *p = reinterpret_cast<unsigned char *>(a.mma);
    Cell *cells = reinterpret_cast<Cell *>(p);
    int *rej = reinterpret_cast<int *>(p + (sizeof(Cell) * nc + 255) / 256 * 256);
    unsigned char *img = reinterpret_cast<unsigned char *>(rej) + rej_bytes(nc, a.n);
    cudaError_t e = cudaFuncSetAttribute(far_product<R, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<L>::TOTAL);
    if (e != cudaSuccess) return e;
    const int ne = a.nf == 1 ? 1 : gf_out_entries(a.which);
    // one layout for all Maxwell entries (their bound covers G_d's)
    far_cells<L><<<nc, 128, 0, s>>>(a, cells, rej, nc, a.nf == 1 ? 6 : 0);
    far_weights<L><<<dim3(nc, NKB + 1), 256, 0, s>>>(a, cells, rej, img, nc, ne);
    far_product<R, L><<<nsm, THREADS, Smem<L>::TOTAL, s>>>(a, cells, rej, img, nc, ne, a.err);
    gf_count_launch(3);
    a.nfar = rej;
    a.far_sorted = rej + 2 + nc;
    return cudaGetLastError();
}

// The far targets' series by matrix products; a.far_sorted and a.nfar are then the list of
// those left to the series kernels.
cudaError_t gf_launch_far_product(EvalArgs &a, int precision, int nsm, cudaStream_t s)
{
    unsigned char *p = reinterpret_cast<unsigned char *>(a.mma);
    int *rej = reinterpret_cast<int *>(p + (sizeof(Cell) * a.mma_cells + 255) / 256 * 256);
    cudaError_t e = cudaMemsetAsync(rej, 0, 2 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    return precision == GF_FP64 ? launch_product<double, 6>(a, nsm, s) : launch_product<float, 3>(a, nsm, s);
}
