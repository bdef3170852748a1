// Bounds of a rigid instance's residual phase, for the plans of the
// band-limited evaluations (band.cu, band64.cu).
#pragma once

#include <cuda_runtime.h>

#include "bart_internal.cuh"
#include "mixed_record.cuh"

namespace bart {

// floats as unsigned integers of the same order, and back
__device__ __forceinline__ unsigned int ord_u(float f)
{
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float ord_f(unsigned int u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// range of p / sqrt(p^2 + q^2) over p in [p0, p1], q in [q0, q1], q0 >= 0:
// it grows with p, and its size falls with q
__device__ __forceinline__ void cos_range(float p0, float p1, float q0, float q1, float &lo,
                                          float &hi)
{
    const float qh = p1 > 0.f ? q0 : q1, ql = p0 > 0.f ? q1 : q0;
    const float rh = sqrtf(p1 * p1 + qh * qh), rl = sqrtf(p0 * p0 + ql * ql);
    hi = rh > 0.f ? p1 / rh : 1.f;
    lo = rl > 0.f ? p0 / rl : -1.f;
}

// Bounds of an instance's residual phase after the reference of its box
// centre: the largest offsets of path and path rate from the centre's, over
// its box and the frame.
struct BandBounds {
    float c[3];      // box centre at t0
    float rf;        // largest facet radius
    float speed;
    float beta;      // beat-frequency offset, cycles per sample
    float turn;      // phase turn over half the frame, radians
    float p2;        // quadratic phase, cycles per sample^2
    bool ok;         // the bounds hold
};

// of box bi, moving with instance i, by one warp, a lane per antenna; the
// result in lane 0
__device__ __forceinline__ BandBounds band_bounds(const unsigned int *__restrict__ box, int bi, int i,
                                                  const RadarDev &rd, const MixConsts &K,
                                                  const float *__restrict__ vel32)
{
    const int a = threadIdx.x & 31;
    float c[3], h[3];
    for (int r = 0; r < 3; ++r) {
        const float lo = ord_f(~box[8 * bi + r]), hi = ord_f(box[8 * bi + 3 + r]);
        c[r] = 0.5f * (lo + hi);
        h[r] = fmaxf(hi - c[r], c[r] - lo);
    }
    const float rf = sqrtf(ord_f(box[8 * bi + 6]));          // largest facet radius
    const float v[3] = {vel32[4 * i], vel32[4 * i + 1], vel32[4 * i + 2]};
    const float speed = sqrtf(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    const float diag = sqrtf(h[0] * h[0] + h[1] * h[1] + h[2] * h[2]);
    const float T = (float)((rd.N - 1) * rd.slots + rd.slots - 1) * K.tc;
    // the box in the velocity's frame: half-extents along and across it
    float ep = 0.f, eq = 0.f;
    float vh[3] = {0.f, 0.f, 0.f};
    if (speed > 0.f) {
        for (int r = 0; r < 3; ++r) {
            vh[r] = v[r] / speed;
            ep += fabsf(vh[r]) * h[r];
        }
        for (int k = 0; k < 4; ++k) {
            const float s1 = k & 1 ? -h[1] : h[1], s2 = k & 2 ? -h[2] : h[2];
            const float al = vh[0] * h[0] + vh[1] * s1 + vh[2] * s2;
            const float x = h[0] - al * vh[0], y = s1 - al * vh[1], z = s2 - al * vh[2];
            eq = fmaxf(eq, x * x + y * y + z * z);
        }
        eq = sqrtf(eq);
    }
    float dL = 0.f, dV = 0.f, dA = 0.f, near = 0.f;           // this antenna's offsets
    if (a < rd.A) {
        for (int k = 0; k < 3; ++k) {                          // frame start, middle, end
            const float t = 0.5f * (float)k * T;
            float y[3];
            for (int r = 0; r < 3; ++r) y[r] = (c[r] - K.ant[a][r]) + v[r] * t;
            const float R = sqrtf(y[0] * y[0] + y[1] * y[1] + y[2] * y[2]);
            if (R < 1.5f * diag + speed * T) near = 1.f;
            // R is convex, so its largest offset over the box is at a corner
            // and the smallest above the tangent's, which is less
            float far2 = 0.f;
            for (int q = 0; q < 8; ++q) {
                const float x0 = y[0] + (q & 1 ? -h[0] : h[0]), x1 = y[1] + (q & 2 ? -h[1] : h[1]),
                            x2 = y[2] + (q & 4 ? -h[2] : h[2]);
                far2 = fmaxf(far2, x0 * x0 + x1 * x1 + x2 * x2);
            }
            // a facet's phases are linear about its centroid: a little beyond the box
            const float bend = R > 0.f ? 2.f * rf * diag / R : 0.f;
            dL = fmaxf(dL, sqrtf(far2) - R + bend);
            if (speed > 0.f && R > 0.f) {
                const float p = y[0] * vh[0] + y[1] * vh[1] + y[2] * vh[2];
                const float q = sqrtf(fmaxf(R * R - p * p, 0.f));
                float lo, hi;
                cos_range(p - ep, p + ep, fmaxf(q - eq, 0.f), q + eq, lo, hi);
                dV = fmaxf(dV, speed * (fmaxf(hi - p / R, p / R - lo) + bend / R));
                dA = fmaxf(dA, 2.f * speed * speed * diag / (R * R));
            }
        }
        if (!rd.intra) dA = 0.f;
    }
    // largest over the TX and over the RX antennas
    const bool is_tx = a < rd.P;
    float tL = is_tx ? dL : 0.f, tV = is_tx ? dV : 0.f, rL = is_tx ? 0.f : dL, rV = is_tx ? 0.f : dV;
    for (int off = 16; off > 0; off >>= 1) {
        tL = fmaxf(tL, __shfl_xor_sync(0xffffffffu, tL, off));
        tV = fmaxf(tV, __shfl_xor_sync(0xffffffffu, tV, off));
        rL = fmaxf(rL, __shfl_xor_sync(0xffffffffu, rL, off));
        rV = fmaxf(rV, __shfl_xor_sync(0xffffffffu, rV, off));
        dA = fmaxf(dA, __shfl_xor_sync(0xffffffffu, dA, off));
        near = fmaxf(near, __shfl_xor_sync(0xffffffffu, near, off));
    }
    const float L = 1.02f * (tL + rL), V = 1.05f * (tV + rV), Vi = rd.intra ? V : 0.f;
    const float p2 = K.mu_c_fs2 * Vi + 2.f * K.half_f0c_fs2 * dA;
    const float kmax_c = K.kmax;                               // 2 pi f_max / c
    // beat-frequency offset: range, Doppler within the chirp, its change
    const float beta = K.muc * L + kmax_c / 6.2831853f * Vi / (float)rd.fs + 2.f * p2 * (float)rd.M;
    const float turn = kmax_c * V * 0.5f * T;
    BandBounds q;
    for (int r = 0; r < 3; ++r) q.c[r] = c[r];
    q.rf = rf;
    q.speed = speed;
    q.beta = beta;
    q.turn = turn;
    q.p2 = p2;
    q.ok = near == 0.f && isfinite(beta) && isfinite(turn);
    return q;
}

// first entry of an ascending list at or beyond key, a warp together: 32
// probes a round (4 rounds for a million entries, where one thread's binary
// search chains 20 dependent loads)
__device__ __forceinline__ int warp_lower_bound(const int32_t *list, int n, int64_t key, int lane)
{
    int lo = 0, hi = n;                           // answer in [lo, hi]
    while (lo < hi) {
        const int step = (hi - lo + 31) / 32;
        const int at = lo + lane * step;
        const bool less = at < hi && list[at] < key;
        const int c = __popc(__ballot_sync(0xffffffffu, less));
        if (c == 0) return lo;
        const int base = lo + (c - 1) * step;     // the last probe below key
        hi = min(hi, base + step);
        lo = base + 1;
    }
    return lo;
}

}  // namespace bart
