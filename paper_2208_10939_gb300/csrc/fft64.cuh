// FP64 FFTs of length L = 2^a 3^b (L <= 1024) over columns held in shared
// memory, for the complex128 range-Doppler map (rdm.cu).
//
// The FP64 pipe (a 64th of the FP32 rate) bounds these transforms: 12 x 128 x
// 384 samples take 2 x 0.6 M points x ~25 FP64 operations, and everything that
// is not a butterfly is kept off it.  So
//  - the passes are Stockham autosort passes of radix 8, 4, 6, 2 and 3 with the
//    DFT in registers: 29 (L = 384) and 21 (L = 128) FP64 operations a point,
//    against 35 and 28 with radix 2 and 3;
//  - the last pass (all twiddles 1) multiplies by none;
//  - a block forms the twiddles and the window once, in shared memory, for all
//    the columns it transforms, and a twiddle table of L % 8 == 0 entries from
//    one octant (an eighth of the sincospi).
// Small maps wait for chains of dependent operations, so a block has at least 192
// threads, and both tables come from one loop, a warp of either kind (the four
// launches of the map's adjoint, 12 x 32 x 128: 47.4 us, 62.6 with 64 threads and
// a loop for each; 4 x 27 x 288: 49.0 and 69.2; radix 2 and 3 in blocks of 8 rows
// took 51.5 and 57.7).
#pragma once

#include <cuda_runtime.h>

#include "fft_stockham.cuh"

namespace bart {
namespace fft64 {

__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 mul(double2 a, double2 w)
{
    return make_double2(fma(a.x, w.x, -a.y * w.y), fma(a.x, w.y, a.y * w.x));
}
// a (-i)
__device__ __forceinline__ double2 mnj(double2 a) { return make_double2(a.y, -a.x); }

template <int R> __device__ __forceinline__ void dft(double2 *a);

template <> __device__ __forceinline__ void dft<2>(double2 *a)
{
    const double2 t = a[0];
    a[0] = add(t, a[1]);
    a[1] = sub(t, a[1]);
}

template <> __device__ __forceinline__ void dft<3>(double2 *a)
{
    const double h = 0.86602540378443864676;          // sin(2 pi / 3)
    const double2 t = add(a[1], a[2]), u = sub(a[1], a[2]);
    const double2 m = make_double2(fma(-0.5, t.x, a[0].x), fma(-0.5, t.y, a[0].y));
    a[0] = add(a[0], t);
    a[1] = make_double2(fma(h, u.y, m.x), fma(-h, u.x, m.y));
    a[2] = make_double2(fma(-h, u.y, m.x), fma(h, u.x, m.y));
}

template <> __device__ __forceinline__ void dft<4>(double2 *a)
{
    const double2 t0 = add(a[0], a[2]), t1 = sub(a[0], a[2]);
    const double2 t2 = add(a[1], a[3]), t3 = mnj(sub(a[1], a[3]));
    a[0] = add(t0, t2);
    a[1] = add(t1, t3);
    a[2] = sub(t0, t2);
    a[3] = sub(t1, t3);
}

// 6 = 2 x 3, prime factors: n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6), no twiddles
template <> __device__ __forceinline__ void dft<6>(double2 *a)
{
    double2 e[3] = {a[0], a[2], a[4]}, o[3] = {a[3], a[5], a[1]};
    dft<3>(e);
    dft<3>(o);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) {
        a[(4 * k2) % 6] = add(e[k2], o[k2]);
        a[(3 + 4 * k2) % 6] = sub(e[k2], o[k2]);
    }
}

template <> __device__ __forceinline__ void dft<8>(double2 *a)
{
    const double r = 0.70710678118654752440;
    double2 e[4] = {a[0], a[2], a[4], a[6]}, o[4] = {a[1], a[3], a[5], a[7]};
    dft<4>(e);
    dft<4>(o);
    o[1] = make_double2(r * (o[1].x + o[1].y), r * (o[1].y - o[1].x));
    o[2] = mnj(o[2]);
    o[3] = make_double2(r * (o[3].y - o[3].x), -r * (o[3].x + o[3].y));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a[k] = add(e[k], o[k]);
        a[k + 4] = sub(e[k], o[k]);
    }
}

// Twiddles exp(-2 pi i t / L), t < L, from one octant where 8 divides L, and the
// window of window_val, its mirror image copied: one loop over both, since the
// chain of a sine is what a small transform's block waits for.
__device__ inline void fill_tables(double2 *tw, double *win, int L, int kind)
{
    const bool oct = (L & 7) == 0;
    const int h = L / 2, q = L / 4, nt = oct ? L / 8 + 1 : L;
    const int w0 = (nt + 31) & ~31;                  // the window from a warp of its own on
    for (int i = threadIdx.x; i < w0 + (L + 1) / 2; i += blockDim.x) {
        if (i >= w0) {
            const int k = i - w0;
            win[k] = win[L - 1 - k] = window_val<double>(k, L, kind);
            continue;
        }
        if (i >= nt) continue;
        double s, c;
        sincospi((double)(2 * i) / (double)L, &s, &c);
        if (!oct) {
            tw[i] = make_double2(c, -s);
            continue;
        }
        tw[i] = make_double2(c, -s);
        tw[q - i] = make_double2(s, -c);
        tw[q + i] = make_double2(-s, -c);
        tw[h - i] = make_double2(-c, -s);
        tw[h + i] = make_double2(-c, s);
        tw[h + q - i] = make_double2(-s, c);
        tw[h + q + i] = make_double2(s, c);
        if (i > 0) tw[L - i] = make_double2(c, s);
    }
}

// One Stockham pass of radix R over `cols` columns (element idx of column c at
// c (L + 1) + idx; the odd stride keeps a warp that walks across the columns on
// different banks): current length n, stride s = L / n, m = n / R, butterfly
// b = q + s j:  y[q + s (R j + k')] = w_n^{j k'} sum_k x[b + (L / R) k] w_R^{k k'}.
// win: the first pass's window (s == 1, so that element k of a butterfly is
// sample b + (L / R) k) or null.
template <int R>
__device__ __forceinline__ void pass(const double2 *x, double2 *y, const double2 *tw,
                                     const double *win, int L, int n, int s, int cols)
{
    const int per = L / R;
    const bool last = n == R;
    for (int t = threadIdx.x; t < per * cols; t += blockDim.x) {
        const int col = t / per, b = t - col * per;
        const int j = b / s, q = b - j * s;
        const double2 *xc = x + col * (L + 1) + b;
        double2 *yc = y + col * (L + 1) + q + s * R * j;
        double2 a[R];
#pragma unroll
        for (int k = 0; k < R; ++k) a[k] = xc[per * k];
        if (win) {
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const double w = win[b + per * k];
                a[k].x *= w;
                a[k].y *= w;
            }
        }
        dft<R>(a);
        if (!last && j > 0) {
#pragma unroll
            for (int k = 1; k < R; ++k) a[k] = mul(a[k], tw[s * j * k]);   // s j k < L
        }
#pragma unroll
        for (int k = 0; k < R; ++k) yc[s * k] = a[k];
    }
}

// the radix of the next pass of length n = 2^a 3^b
__device__ __forceinline__ int radix(int n)
{
    if (n == 16) return 4;
    return n % 8 == 0 ? 8 : n % 4 == 0 ? 4 : n % 6 == 0 ? 6 : n % 2 == 0 ? 2 : 3;
}

// Forward transforms of `cols` columns, in x; returns the buffer that holds
// the results (x or y).  The block's threads call it together; it ends on a
// block barrier.
__device__ inline double2 *transform(double2 *x, double2 *y, const double2 *tw, const double *win,
                                     int L, int cols)
{
    for (int n = L, s = 1; n > 1;) {
        const int R = radix(n);
        switch (R) {
        case 8: pass<8>(x, y, tw, win, L, n, s, cols); break;
        case 6: pass<6>(x, y, tw, win, L, n, s, cols); break;
        case 4: pass<4>(x, y, tw, win, L, n, s, cols); break;
        case 3: pass<3>(x, y, tw, win, L, n, s, cols); break;
        default: pass<2>(x, y, tw, win, L, n, s, cols); break;
        }
        __syncthreads();
        double2 *t = x;
        x = y;
        y = t;
        win = nullptr;
        n /= R;
        s *= R;
    }
    return x;
}

}  // namespace fft64
}  // namespace bart
