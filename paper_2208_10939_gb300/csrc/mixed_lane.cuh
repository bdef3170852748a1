// What a lane of the mixed echo synthesis does with one record (RecM) over
// its S consecutive samples: the vertex form's phasor recurrence, the series
// and edge forms sample by sample, and the compensated accumulation.  Shared
// by the direct kernel (synth.cu) and the band-limited one (band.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mixed_record.cuh"

namespace bart {

// Packed FP32 pairs (sm_100+ f32x2 arithmetic): two floats in one 64-bit
// register pair, one instruction for both lanes of a pair.  The mixed
// kernel keeps two consecutive samples of a lane in one pair.
__device__ __forceinline__ uint64_t pk2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t r, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fadd2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fsub2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Vertex form: the lane's samples start at fm0 (in samples; fm0sq its square,
// less the constant that centres the chord's error where the caller wants
// it); eps_lane p2 is the angle that the within-chirp quadratic phase adds to
// each step.
// PAIR: the pair form, whose first phasor has the amplitude kappa sinc(kappa x)
// at each sample; over a lane that is linear to 1e-7 (kappa changes by less
// than 1e-3 there).
template <int S, bool PAIR = false>
__device__ __forceinline__ void vertex_form_lane(const float *rec, float fm0, float fm0sq,
                                                 float eps_lane, uint64_t (&PR)[(S + 1) / 2],
                                                 uint64_t (&PI)[(S + 1) / 2], float kap_step = 0.f,
                                                 float d = 1.f)
{
    constexpr int S2 = (S + 1) / 2;
    // e^{j(phi + (s+2) a)} = 2 cos(a) e^{j(phi + (s+1) a)} - e^{j(phi + s a)}:
    // on sample pairs (2k, 2k+1) with the two-sample angle, one FMA
    // per pair and component.  Pair k is held times sg(k) = +1 for
    // k mod 4 in {0, 1}, else -1, so that the recurrence needs no
    // negated addend: held(k) = sg(k) sg(k-1) c2 held(k-1) + held(k-2).
    // 128-bit broadcast loads of the record
    const float4 *R4 = reinterpret_cast<const float4 *>(rec);
    const float4 q0 = R4[0], q1 = R4[1], q2v = R4[2], q3 = R4[3], q4 = R4[4],
                 q5 = R4[5];
    const float ph0[3] = {q0.x, q0.y, q0.z};
    const float lo[3] = {q0.w, q1.x, q1.y};
    const float wv[3] = {q1.z, q1.w, q2v.x};
    const float sre[3] = {q2v.y, q2v.z, q2v.w};
    const float sim[3] = {q3.x, q3.y, q3.z};
    const float c2x2[3] = {q4.y, q4.z, q4.w};     // 2 cos(2 step)
    const float s2x4[3] = {q5.x, q5.y, q5.z};     // 4 sin(2 step)
    const float hi = q3.w, p2 = q4.x;
    // the vertices' common phase at the lane's first sample
    const float tq = red1(hi * fm0) + p2 * fm0sq;
    const float eps = p2 * eps_lane;
#pragma unroll
    for (int v = 0; v < 3; ++v) {
        const float thv = red1(fmaf(lo[v], fm0, ph0[v] + tq));
        float zs, zc;
        __sincosf(6.283185307179586f * thv, &zs, &zc);
        zc *= wv[v];
        zs *= wv[v];
        // the lane's step (angle + eps) and its doubled cosines
        const float stc = fmaf(-eps, sim[v], sre[v]);
        const float sts = fmaf(eps, sre[v], sim[v]);
        const float a1 = 2.f * stc;
        const float a2 = fmaf(-eps, s2x4[v], c2x2[v]);
        // samples m0 + 1 (rotation), m0 + 2 and m0 + 3 (recurrence)
        const float zc1 = fmaf(zc, stc, -zs * sts), zs1 = fmaf(zc, sts, zs * stc);
        const float zc2 = fmaf(a1, zc1, -zc), zs2 = fmaf(a1, zs1, -zs);
        const float zc3 = fmaf(a1, zc2, -zc1), zs3 = fmaf(a1, zs2, -zs1);
        uint64_t XC = pk2(zc, zc1), XS = pk2(zs, zs1);       // held(k - 1)
        uint64_t YC = pk2(zc2, zc3), YS = pk2(zs2, zs3);     // held(k)
        const uint64_t A2 = pk2(a2, a2), NA2 = pk2(-a2, -a2);
        if (PAIR && v == 0) {
            const float kc = fmaf(kap_step, fmaf(0.5f * (S - 1), d, fm0), 1.f);
            const float q = q5.w * kc * kc;
            const float amp = kc * fmaf(q, fmaf(q, 1.f / 120.f, -1.f / 6.f), 1.f);
            const float slope = kap_step * d * fmaf(q, fmaf(q, 1.f / 24.f, -0.5f), 1.f);
            const float a0 = fmaf(-0.5f * (S - 1), slope, amp);
            const uint64_t inc = pk2(2.f * slope, 2.f * slope);
            uint64_t am = pk2(a0, a0 + slope);
#pragma unroll
            for (int k = 0; k < S2; ++k) {
                const bool neg = (k & 2) != 0;
                uint64_t zc2p, zs2p;
                if (k == 0) {
                    zc2p = XC;
                    zs2p = XS;
                } else if (k == 1) {
                    zc2p = YC;
                    zs2p = YS;
                } else {
                    const uint64_t A = (((k - 1) & 2) != 0) != neg ? NA2 : A2;
                    const uint64_t NC = ffma2(A, YC, XC), NS = ffma2(A, YS, XS);
                    XC = YC;
                    XS = YS;
                    YC = zc2p = NC;
                    YS = zs2p = NS;
                }
                const uint64_t ak = neg ? fsub2(pk2(0.f, 0.f), am) : am;
                PR[k] = ffma2(ak, zc2p, PR[k]);
                PI[k] = ffma2(ak, zs2p, PI[k]);
                am = fadd2(am, inc);
            }
            continue;
        }
        PR[0] = fadd2(PR[0], XC);
        PI[0] = fadd2(PI[0], XS);
        if (S2 > 1) {
            PR[1] = fadd2(PR[1], YC);
            PI[1] = fadd2(PI[1], YS);
        }
#pragma unroll
        for (int k = 2; k < S2; ++k) {
            const bool neg = (k & 2) != 0;                   // sg(k) = -1
            const uint64_t A = (((k - 1) & 2) != 0) != neg ? NA2 : A2;
            const uint64_t NC = ffma2(A, YC, XC), NS = ffma2(A, YS, XS);
            XC = YC;
            XS = YS;
            YC = NC;
            YS = NS;
            if (neg) {
                PR[k] = fsub2(PR[k], YC);
                PI[k] = fsub2(PI[k], YS);
            } else {
                PR[k] = fadd2(PR[k], YC);
                PI[k] = fadd2(PI[k], YS);
            }
        }
    }
}

// Series and edge forms: sample j of the lane is at fm0 + j d and turned by
// j turn cycles.
template <int S>
__device__ __forceinline__ void series_edge_lane(const float *rec, bool series, float fm0, float d,
                                                 float turn, const MixConsts &K, uint64_t (&PR)[(S + 1) / 2],
                                                 uint64_t (&PI)[(S + 1) / 2])
{
#pragma unroll
    for (int j = 0; j < S; ++j) {
        float dr, di;
        series_edge_term(rec, series, fmaf((float)j, d, fm0), K, dr, di, (float)j * turn);
        // into sample j's half of its pair
        const uint64_t DR = (j & 1) ? pk2(0.f, dr) : pk2(dr, 0.f);
        const uint64_t DI = (j & 1) ? pk2(0.f, di) : pk2(di, 0.f);
        PR[j >> 1] = fadd2(PR[j >> 1], DR);
        PI[j >> 1] = fadd2(PI[j >> 1], DI);
    }
}

// Kahan-compensated accumulation of the pair v into (sum, comp)
__device__ __forceinline__ void kahan_pair(uint64_t &sum, uint64_t &comp, uint64_t v)
{
    const uint64_t s = sum, y = fsub2(v, comp), t = fadd2(s, y);
    comp = fsub2(fsub2(t, s), y);
    sum = t;
}

}  // namespace bart
