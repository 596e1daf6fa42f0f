// Inverse transforms of lines held by a CTA (+ sign, unnormalised), Stockham autosort: radix-4
// stages after one radix-2 stage when lg is odd (n = 2^lg >= 8).  A stage that combines
// sub-transforms of length Ns takes, for j < n/4 and k = j mod Ns, v_r = x[j + r n/4]
// e^{2 pi i r k/(4 Ns)} and writes the 4-point inverse DFT of (v_0..v_3) to 4(j - k) + k + m Ns,
// m = 0 .. 3.  The first stage reads element j of line t by ld(j, t), the last one
// hands output l of line t to st(l, t, v): neither has a pass over shared memory of its
// own; the stages between go through x and y.  tw[m] = e^{2 pi i m/n}, m < n/2.  All threads
// of the CTA call it; what the last stage reads may be written again after the next
// barrier.
//
// fft_cols: T = 2^lgT lines, element j of line t at [j T + t], consecutive threads take
// consecutive lines.  fft_rows: nlines lines, element j of line t at [t n + j],
// consecutive threads take consecutive elements.
#pragma once
#include "gf_internal.cuh"

template <bool ROWS, typename C, class Ld, class St>
__device__ __forceinline__ void fft_stages(C *x, C *y, int n, int lg, int lgT, int nlines, const C *tw, Ld ld, St st)
{
    const int half = n >> 1, q = n >> 2;
    const int es = ROWS ? 1 : 1 << lgT, ls = ROWS ? n : 1;  // strides of an element and of a line
    int Ns, lns;
    if (lg & 1) {
        for (int it = threadIdx.x; it < half * nlines; it += blockDim.x) {
            const int t = ROWS ? it >> (lg - 1) : it & ((1 << lgT) - 1), j = ROWS ? it & (half - 1) : it >> lgT;
            const C v0 = ld(j, t), v1 = ld(j + half, t);
            C *o = x + t * ls + 2 * j * es;
            o[0] = cadd(v0, v1);
            o[es] = csub(v0, v1);
        }
        Ns = 2;
        lns = 1;
    } else {
        for (int it = threadIdx.x; it < q * nlines; it += blockDim.x) {
            const int t = ROWS ? it >> (lg - 2) : it & ((1 << lgT) - 1), j = ROWS ? it & (q - 1) : it >> lgT;
            const C a = ld(j, t), b = ld(j + q, t), c = ld(j + 2 * q, t), d = ld(j + 3 * q, t);
            const C apc = cadd(a, c), amc = csub(a, c), bpd = cadd(b, d), bmd = csub(b, d);
            C *o = x + t * ls + 4 * j * es;
            o[0] = cadd(apc, bpd);
            o[es] = cmk(amc.x - bmd.y, amc.y + bmd.x);
            o[2 * es] = csub(apc, bpd);
            o[3 * es] = cmk(amc.x + bmd.y, amc.y - bmd.x);
        }
        Ns = 4;
        lns = 2;
    }
    __syncthreads();
    for (;; Ns <<= 2, lns += 2) {
        const bool last = Ns == q;
        const int sh = lg - 2 - lns;
        for (int it = threadIdx.x; it < q * nlines; it += blockDim.x) {
            const int t = ROWS ? it >> (lg - 2) : it & ((1 << lgT) - 1), j = ROWS ? it & (q - 1) : it >> lgT;
            const int k = j & (Ns - 1), k3 = (3 * k) << sh;
            const C *xl = x + t * ls + j * es;
            C w3 = tw[k3 & (half - 1)];
            if (k3 >= half) w3 = cmk(-w3.x, -w3.y);
            const C a = xl[0];
            const C b = cmul(xl[q * es], tw[k << sh]);
            const C c = cmul(xl[2 * q * es], tw[(2 * k) << sh]);
            const C d = cmul(xl[3 * q * es], w3);
            const C apc = cadd(a, c), amc = csub(a, c), bpd = cadd(b, d), bmd = csub(b, d);
            const C o0 = cadd(apc, bpd), o1 = cmk(amc.x - bmd.y, amc.y + bmd.x), o2 = csub(apc, bpd),
                    o3 = cmk(amc.x + bmd.y, amc.y - bmd.x);
            const int o = ((j - k) << 2) + k;
            if (last) {
                st(o, t, o0);
                st(o + Ns, t, o1);
                st(o + 2 * Ns, t, o2);
                st(o + 3 * Ns, t, o3);
            } else {
                C *yl = y + t * ls + o * es;
                yl[0] = o0;
                yl[Ns * es] = o1;
                yl[2 * Ns * es] = o2;
                yl[3 * Ns * es] = o3;
            }
        }
        __syncthreads();
        if (last) return;
        C *z = x;
        x = y;
        y = z;
    }
}

template <typename C, class Ld, class St>
__device__ __forceinline__ void fft_cols(C *x, C *y, int n, int lg, int lgT, const C *tw, Ld ld, St st)
{
    fft_stages<false>(x, y, n, lg, lgT, 1 << lgT, tw, ld, st);
}

template <typename C, class Ld, class St>
__device__ __forceinline__ void fft_rows(C *x, C *y, int n, int lg, int nlines, const C *tw, Ld ld, St st)
{
    fft_stages<true>(x, y, n, lg, 0, nlines, tw, ld, st);
}
