// BART single-bounce visibility (Sec. 2.2): the forward ray from a TX and the
// backward ray from an RX "meet" on a facet when the facet is lit from the
// TX and seen from the RX.  Each (antenna, facet) pair gets a state from the
// facet-centroid -> antenna segment cast through the LBVH:
//   BACK  (facing away), LIT, GRAZE (within margins: excluded, counted),
//   OCCL  (a robust hit on another facet), LIT_REV (a two-sided facet lit on
//   its reverse side).
// In far-field mode the segment ends at p_a + (c_k - r), r the instance
// origin at the frame start: every facet of an instance looks along the same
// plane-wave direction, over the origin's range.
// The segment/triangle decision is Moller-Trumbore (1997) in FP64 with one
// IEEE rounding per operation in a fixed order (explicit __d*_rn intrinsics:
// no FMA contraction), so states are reproducible bit for bit by any
// IEEE-754 implementation of the same steps.  The BVH boxes are FP32,
// rounded outward and padded, so box culling never drops a candidate.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "bart_internal.cuh"
#include "geom64.cuh"

namespace bart {

// a four-wide node leaves up to three children waiting a level, and the
// hierarchy of 30-bit codes with 31-bit index tie-breaks is at most 62 deep
constexpr int kWideStack = 96;

// Antennas in groups whose segments from a facet are traced as one bundle:
// group g holds antennas first[g] .. first[g] + n[g] - 1 (at most 16, all TX
// or all RX), centred on mid[g] with half-extents half[g].
struct AntGroups {
    int n_groups;
    int first[kMaxAnt], n[kMaxAnt];
    float mid[kMaxAnt][3], mid_lo[kMaxAnt][3];   // float pairs
    float half[kMaxAnt][3];
    float ant[kMaxAnt][3], ant_lo[kMaxAnt][3];
};

// A block takes up to kVisPairs (facet, antenna group) pairs: first the facing
// decisions, whose back-facing half is done, then the others go down the
// hierarchy four lanes a ray.  A visit tests a node's four boxes, one a lane;
// leaves wait in a queue until there are four, which are tested one a lane;
// quads that finish take the block's next ray.  (A lane a ray left 6 to 7 of
// 32 lanes active, or 17 with rays packed and nodes and leaves in separate
// phases, and a chain of 130 instructions a visit: 92 us on the sedan, 20k
// facets and 7 antennas, either way.)
//
// BUNDLE: the segments of a group start at the same centroid and end within
// centimetres of each other, so they go down the hierarchy once, as a bundle:
// a box is visited if any direction of the group's box of directions reaches
// it, and a candidate facet is decided for the whole bundle where the
// relative pre-test's bounds allow it, else antenna by antenna (FP32, then
// FP64).  States are per antenna and the same as from single segments: the
// boxes only over-report, and a bundle's decision holds for each segment.
//
// What bounds it: instruction issue, and the chain of node loads of the
// longest rays.  A frame's visibility and lists, against single segments over
// binary nodes with the absolute pre-test: sedan 0.143 -> 0.085 ms, eight
// dataset scenes 0.34 -> 0.16, intersection (345k facets, 28 antennas)
// 12.0 -> 1.75.
constexpr int kVisThreads = 128, kVisPairs = kVisThreads;    // at most, a block
constexpr int kVisQuads = kVisThreads / 4;

struct VisArgs {
    const double *tri64;
    const float4 *trel;
    const double *c64;
    const FacetRec *fac;
    const float *fac_lo;
    const double *ref64;
    const WideNode *nodes;
    const int32_t *order;
    int64_t F;
    RadarDev rd;
    AntGroups ag;
    SceneSplit sc;
    int pairs;
    uint8_t *state;
    unsigned long long *n_graze;
    int *status;
};

template <bool BUNDLE, bool FAR>
__device__ __forceinline__ void visibility_pairs(const VisArgs &v)
{
    constexpr float u24 = 5.9604645e-8f;
    const double *__restrict__ tri64 = v.tri64, *__restrict__ c64 = v.c64, *__restrict__ ref64 = v.ref64;
    const float4 *__restrict__ trel = v.trel;
    const FacetRec *__restrict__ fac = v.fac;
    const float *__restrict__ fac_lo = v.fac_lo;
    const WideNode *__restrict__ nodes = v.nodes;
    const int32_t *__restrict__ order = v.order;
    uint8_t *__restrict__ state = v.state;
    const int64_t F = v.F;
    const RadarDev &rd = v.rd;
    const AntGroups &ag = v.ag;
    const SceneSplit &sc = v.sc;
    const int pairs = v.pairs;
    int *status = v.status;
    __shared__ int s_k[kVisPairs];
    __shared__ uint16_t s_live[kVisPairs], s_rev[kVisPairs], s_graze[kVisPairs];
    __shared__ int s_cnt[kVisThreads / 32], s_next;
    __shared__ int s_stack[kVisQuads][kWideStack], s_leaf[kVisQuads][8];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int g = blockIdx.y;
    const int a0 = ag.first[g], na = BUNDLE ? ag.n[g] : 1;
    // the FP64 segment of antenna a from c (far field: to p_a + (c - r), r the
    // instance origin), each step rounded once
    auto segment = [&](int a, const double *c, const double *r0, double *D) {
        double pa[3] = {rd.ant[a][0], rd.ant[a][1], rd.ant[a][2]};
        if (FAR)
            for (int r = 0; r < 3; ++r) pa[r] = __dadd_rn(pa[r], __dsub_rn(c[r], r0[r]));
        sub3(pa, c, D);
    };
    auto origin = [&](int64_t k, const double *s64, float *h, float *l) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            if (FAR) {
                h[r] = (float)s64[r];
                l[r] = (float)(s64[r] - (double)h[r]);
            } else {
                h[r] = fac[k].c[r];
                l[r] = fac_lo[12 * k + r];
            }
        }
    };
    // ---- facing ----
    int nq = 0;
    {
        const int64_t gid = (int64_t)blockIdx.x * pairs + t;
        unsigned int live = 0, rev = 0, graze = 0;
        int64_t k = 0;
        if (t < pairs && gid < F) {
            // facets in Morton order, so that a warp's segments start close
            // together and traverse similar paths
            k = order ? (int64_t)order[gid] : gid;
            // the segments' start (far field: the instance origin that D is
            // taken from) as a float pair; the facet record's centroid and its
            // residue, since a conversion from FP64 holds an SM's FP64 pipe for
            // 16 cycles a warp
            const FacetRec *fr = fac + k;
            const double *s64 = FAR ? ref64 + 3 * fr->inst : c64 + 3 * k;
            float sh[3], sl[3];
            origin(k, s64, sh, sl);
            // FP32 pre-test of the facing test below.  n is the unit normal
            // formed in FP64 and rounded (error < 2e-7), Df the segment
            // (relative error 2^-23 per component); with the dot product's and
            // rsqrt's rounding, |cos32 - cos| < 7e-7, so beyond +-(eps_face +
            // 2e-6) the FP64 decision is certain.  Slivers (2A below 1e-6 of
            // the squared edge scale), whose FP64 normal direction is
            // ill-conditioned, always take the FP64 test.
            const bool two = fr->two_sided != 0;
            const float n0 = fr->n[0], n1 = fr->n[1], n2 = fr->n[2];
            float L2 = 0.f;
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                const float x = fr->dv[3 * v], y = fr->dv[3 * v + 1], z = fr->dv[3 * v + 2];
                L2 = fmaxf(L2, fmaf(x, x, fmaf(y, y, z * z)));
            }
            const bool sound = 2.f * fr->area >= 4e-6f * L2;
            const float thr = (float)rd.eps_face + 2e-6f;
            for (int q = 0; q < na; ++q) {
                const int a = a0 + q;
                int face = 1;                // 0 back, 2 front, 3 reverse (two-sided), 1 undecided
                float Df[3];
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    Df[r] = (ag.ant[a][r] - sh[r]) + (ag.ant_lo[a][r] - sl[r]);
                const float dd = fmaf(Df[0], Df[0], fmaf(Df[1], Df[1], Df[2] * Df[2]));
                const float cos32 = fmaf(n0, Df[0], fmaf(n1, Df[1], n2 * Df[2])) * rsqrtf(dd);
                if (sound && dd > 0.f) {
                    if (cos32 >= thr) face = 2;
                    else if (cos32 <= -thr) face = two ? 3 : 0;
                }
                if (face == 1) {
                    double D[3], tri[9], e1[3], e2[3], n[3];
                    const double c[3] = {c64[3 * k], c64[3 * k + 1], c64[3 * k + 2]};
                    segment(a, c, s64, D);
                    for (int i = 0; i < 9; ++i) tri[i] = tri64[9 * k + i];
                    sub3(tri + 3, tri, e1);
                    sub3(tri + 6, tri, e2);
                    cross3(e1, e2, n);
                    const double cosang = __ddiv_rn(
                        dot3(n, D), __dmul_rn(__dsqrt_rn(dot3(n, n)), __dsqrt_rn(dot3(D, D))));
                    if (dot3(n, n) == 0.0) face = 0;          // zero area: no normal
                    else if (cosang <= -rd.eps_face) face = two ? 3 : 0;
                    else if (fabs(cosang) < rd.eps_face) graze |= 1u << q;
                }
                if (face == 0) {
                    state[(int64_t)a * F + k] = BART_VIS_BACK;
                } else {
                    live |= 1u << q;
                    if (face == 3) rev |= 1u << q;
                }
            }
        }
        const unsigned int m = __ballot_sync(0xffffffffu, live != 0);
        if (lane == 0) s_cnt[warp] = __popc(m);
        __syncthreads();
        int at = __popc(m & ((1u << lane) - 1u));
        for (int w = 0; w < kVisThreads / 32; ++w) {
            if (w < warp) at += s_cnt[w];
            nq += s_cnt[w];
        }
        if (live) {
            s_k[at] = (int)k;
            s_live[at] = (uint16_t)live;
            s_rev[at] = (uint16_t)rev;
            s_graze[at] = (uint16_t)graze;
        }
        __syncthreads();
    }
    // ---- occlusion, four lanes a ray ----
    if (t == 0) s_next = kVisQuads;
    __syncthreads();
    const int quad = t >> 2, ql = t & 3, qsh = lane & 28;    // quad's first lane in the warp
    int *const stack = s_stack[quad];
    int *const leaves = s_leaf[quad];
    int ray = quad;                          // < nq: the quad has a ray
    int n_graze_q = 0;
    bool fresh = true;                       // its data are still to be loaded
    int64_t k = 0;
    unsigned int live = 0, graze = 0, hit = 0;
    int sp = 0, nl = 0;
    float o[3], ol[3], sh[3], sl[3], Dc[3], inv[3], inl[3], oi[3];
    float wd = 0.f, Dm = 0.f, Om = 0.f;
    // does a segment of the bundle reach the box within its length?  The
    // boxes' pad (1e-4 + 4e-6 of the coordinates) covers the rounding of o
    // and of o / D: both move a plane by at most 2^-23 of a coordinate.
    auto reach = [&](const float4 lo, const float4 hi) -> bool {
        float tn = -1e-3f, tf = 1.0f + 1e-3f;
        const float bl[3] = {lo.x, lo.y, lo.z}, bh[3] = {hi.x, hi.y, hi.z};
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            if (!BUNDLE) {
                const float x = fmaf(bl[r], inv[r], oi[r]), y = fmaf(bh[r], inv[r], oi[r]);
                tn = fmaxf(tn, fminf(x, y));
                tf = fminf(tf, fmaxf(x, y));
            } else {
                const float l = bl[r] - o[r], h = bh[r] - o[r];
                const bool neg = inv[r] < 0.f, span = inl[r] < 0.f && !neg;
                // all slopes of one sign: in at the near plane by the
                // steepest, out at the far one by the flattest; slopes on
                // both sides of 0 enter from below or above and need not leave
                const float nr = neg ? h : l, fr_ = neg ? l : h;
                const float in1 = span ? fmaxf(l * inv[r], h * inl[r])
                                       : fminf(nr * inl[r], nr * inv[r]);
                const float out1 = span ? 2.f : fmaxf(fr_ * inl[r], fr_ * inv[r]);
                tn = fmaxf(tn, in1);
                tf = fminf(tf, out1);
            }
        }
        return tn <= tf;
    };
    for (;;) {
        const unsigned int bf = __ballot_sync(0xffffffffu, ray < nq && fresh);
        const unsigned int ba = __ballot_sync(0xffffffffu, ray < nq && !fresh);
        if (!(bf | ba)) break;
        // new rays, when they are at least as many as the ones under way
        if (ray < nq && fresh && __popc(bf) >= __popc(ba)) {
            fresh = false;
            k = s_k[ray];
            live = s_live[ray];
            graze = s_graze[ray];
            hit = 0;
            sp = nl = 0;
            const double *s64 = FAR ? ref64 + 3 * fac[k].inst : c64 + 3 * k;
            // directions Dc +- wd; for each axis the slopes that enter a slab
            // first and leave it last
            wd = 0.f;
            origin(k, s64, sh, sl);
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                o[r] = fac[k].c[r];
                ol[r] = fac_lo[12 * k + r];
                Dc[r] = (ag.mid[g][r] - sh[r]) + (ag.mid_lo[g][r] - sl[r]);
                if (BUNDLE) {
                    const float wr = ag.half[g][r] + 4.f * u24 * fabsf(Dc[r]);
                    wd = fmaxf(wd, wr);
                    const float dl = Dc[r] - wr, dh = Dc[r] + wr;
                    inl[r] = __frcp_rn(fabsf(dl) < 1e-30f ? -1e-30f : dl);
                    inv[r] = __frcp_rn(fabsf(dh) < 1e-30f ? 1e-30f : dh);
                } else {
                    const float d = fabsf(Dc[r]) < 1e-30f ? copysignf(1e-30f, Dc[r]) : Dc[r];
                    inv[r] = __frcp_rn(d);
                    oi[r] = -o[r] * inv[r];
                }
            }
            Dm = (fmaxf(fmaxf(fabsf(Dc[0]), fabsf(Dc[1])), fabsf(Dc[2])) + wd) * 1.000001f;
            Om = fmaxf(fmaxf(fabsf(o[0]), fabsf(o[1])), fabsf(o[2]));
            // traversal root: the whole tree, or the subtree of the facet's
            // scene (< 0: a one-facet scene, nothing to meet)
            int root = F >= 2 ? 0 : -1;
            if (sc.B > 1) {
                int lo = 0, hi = sc.B - 1;          // last scene with foff <= k
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (sc.foff[mid] <= k) lo = mid;
                    else hi = mid - 1;
                }
                root = sc.root[lo];
            }
            if (root >= 0) {
                if (ql == 0) stack[0] = root;
                sp = 1;
            }
        }
        __syncwarp();
        // a visit, while the quad has nodes and fewer than four leaves wait
        const bool visit = ray < nq && !fresh && sp > 0 && nl < 4;
        if (__any_sync(0xffffffffu, visit)) {
            bool in = false;
            int child = 0;
            if (visit) {
                const WideNode *nd = nodes + stack[sp - 1];
                const float4 lo = nd->lo[ql], hi = nd->hi[ql];
                child = __float_as_int(lo.w);
                in = reach(lo, hi) && child != ~(int)k;
            }
            const unsigned int below = (1u << ql) - 1u;
            const unsigned int bn = (__ballot_sync(0xffffffffu, in && child >= 0) >> qsh) & 15u;
            const unsigned int bl = (__ballot_sync(0xffffffffu, in && child < 0) >> qsh) & 15u;
            if (visit) {
                --sp;
                const int nn = __popc(bn);
                if (sp + nn <= kWideStack) {
                    if (in && child >= 0) stack[sp + __popc(bn & below)] = child;
                    sp += nn;
                } else {
                    if (ql == 0) atomicOr(status, kStatusStackOverflow);
                    graze |= live;
                }
                if (in && child < 0) leaves[nl + __popc(bl & below)] = ~child;
                nl += __popc(bl);
            }
            __syncwarp();
        }
        // four waiting leaves, or the last ones, a lane each
        // (when half of the warp's rays wait for it, or none can do without)
        const bool test = ray < nq && !fresh && (nl >= 4 || (sp == 0 && nl > 0));
        const unsigned int bt = __ballot_sync(0xffffffffu, test);
        const unsigned int bv = __ballot_sync(0xffffffffu, ray < nq && !fresh && sp > 0 && nl < 4);
        if (bt && __popc(bt) >= __popc(bv)) {
            if (test) {
                const int n = min(nl, 4);
                nl -= n;
                unsigned int h_add = 0, g_add = 0;
                if (ql < n) {
                    const int64_t j = leaves[nl + ql];
                    const float4 q0 = trel[3 * j], q1 = trel[3 * j + 1], q2 = trel[3 * j + 2];
                    int res = mt_rel_classify(q0, q1, q2, o, ol, Dc, Dm, wd + 4.f * u24 * Dm, Om);
                    unsigned int todo = live & ~hit;
                    if (res == 2) h_add = todo;     // every segment certainly occluded
                    if (res != 1) todo = 0;
                    while (todo) {
                        const int b = __ffs((int)todo) - 1;
                        todo &= todo - 1;
                        const int a = a0 + b;
                        if (BUNDLE) {
                            float Df[3];
#pragma unroll
                            for (int r = 0; r < 3; ++r)
                                Df[r] = (ag.ant[a][r] - sh[r]) + (ag.ant_lo[a][r] - sl[r]);
                            const float dm = fmaxf(fmaxf(fabsf(Df[0]), fabsf(Df[1])), fabsf(Df[2])) *
                                             1.000001f;
                            res = mt_rel_classify(q0, q1, q2, o, ol, Df, dm, 3.f * u24 * dm, Om);
                        }
                        if (res == 1) {             // undecided: FP64
                            const double *s64 = FAR ? ref64 + 3 * fac[k].inst : c64 + 3 * k;
                            const double c[3] = {c64[3 * k], c64[3 * k + 1], c64[3 * k + 2]};
                            double D[3], tj[9];
                            segment(a, c, s64, D);
                            for (int i = 0; i < 9; ++i) tj[i] = tri64[9 * j + i];
                            const int x = mt_segment(c, D, tj);
                            if (x == 1) g_add |= 1u << b;
                            res = x == 2 ? 2 : 0;
                        }
                        if (res == 2) h_add |= 1u << b;
                    }
                }
#pragma unroll
                for (int m = 1; m <= 2; m <<= 1) {
                    h_add |= __shfl_xor_sync(15u << qsh, h_add, m);
                    g_add |= __shfl_xor_sync(15u << qsh, g_add, m);
                }
                hit |= h_add;
                graze |= g_add;
                if (hit == live) sp = nl = 0;
            }
            __syncwarp();
        }
        // a finished ray: its states, then the block's next one
        if (ray < nq && !fresh && sp == 0 && nl == 0) {
            graze &= live & ~hit;
            const unsigned int rev = s_rev[ray];
            for (int q = ql; q < na; q += 4)
                if ((live >> q) & 1u)
                    state[(int64_t)(a0 + q) * F + k] =
                        (hit >> q) & 1u ? BART_VIS_OCCL
                                        : ((graze >> q) & 1u ? BART_VIS_GRAZE
                                                             : ((rev >> q) & 1u ? BART_VIS_LIT_REV
                                                                                : BART_VIS_LIT));
            if (ql == 0) n_graze_q += __popc(graze);
            int nx = 0;
            if (ql == 0) nx = atomicAdd(&s_next, 1);
            ray = __shfl_sync(15u << qsh, nx, qsh);
            fresh = true;
        }
        __syncwarp();
    }
    const int gz = __reduce_add_sync(0xffffffffu, n_graze_q);
    if (lane == 0 && gz) atomicAdd(v.n_graze, (unsigned long long)gz);
}

__global__ void __launch_bounds__(kVisThreads) visibility_kernel(const __grid_constant__ VisArgs v)
{
    visibility_pairs<true, false>(v);
}
// one antenna a group: plain slabs
__global__ void __launch_bounds__(kVisThreads) visibility_single_kernel(const __grid_constant__ VisArgs v)
{
    visibility_pairs<false, false>(v);
}
__global__ void __launch_bounds__(kVisThreads) visibility_far_kernel(const __grid_constant__ VisArgs v)
{
    visibility_pairs<true, true>(v);
}

// Antennas of a group: all TX or all RX of up to 16 where that leaves 32k
// (facet, group) pairs, fewer for small scenes (sedan, visibility and lists:
// two groups 93 us, four 92, seven single antennas 117), and only neighbours: a
// bundle visits every box between its antennas' directions, so that far-apart
// ones are cheaper alone.  12 x 16 antennas over an intersection of 125k facets,
// bundles of 16 / these / each alone: 0.03 m apart 1.24 / 1.24 / 2.99 ms, 0.1 m
// 2.33 / 1.72 / 3.01, 0.2 m 3.14 / 2.06 / 2.99, 0.3 m 4.1 / 2.9 / 2.9, 5 m
// 31.3 / 2.8 / 2.8; pairs 0.3 m apart over a 100k-facet sedan 1.16, each alone 0.50.
constexpr double kBundleExtent = 0.5;        // metres along an axis
constexpr double kBundleStep = 0.25;         // and for each antenna after the first

static AntGroups ant_groups(const RadarDev &rd, int64_t F)
{
    AntGroups ag;
    const int64_t want = 32 * 1024;
    int size = 16;
    while (size > 1 && F * ((rd.P + size - 1) / size + (rd.Q + size - 1) / size) < want) size /= 2;
    ag.n_groups = 0;
    auto add = [&](int first, int n) {
        for (int s = first; s < first + n;) {
            const int g = ag.n_groups++;
            double lo[3], hi[3];
            for (int r = 0; r < 3; ++r) lo[r] = hi[r] = rd.ant[s][r];
            int e = s + 1;
            for (; e < first + n && e - s < size; ++e) {
                double l[3], h[3], ext = 0.0;
                for (int r = 0; r < 3; ++r) {
                    l[r] = fmin(lo[r], rd.ant[e][r]);
                    h[r] = fmax(hi[r], rd.ant[e][r]);
                    ext = fmax(ext, h[r] - l[r]);
                }
                if (ext > fmin(kBundleExtent, kBundleStep * (e - s))) break;
                for (int r = 0; r < 3; ++r) {
                    lo[r] = l[r];
                    hi[r] = h[r];
                }
            }
            ag.first[g] = s;
            ag.n[g] = e - s;
            for (int r = 0; r < 3; ++r) {
                const double m = 0.5 * (lo[r] + hi[r]);
                ag.mid[g][r] = (float)m;
                ag.mid_lo[g][r] = (float)(m - (double)ag.mid[g][r]);
                ag.half[g][r] = (float)((hi[r] - lo[r]) * 0.50001);
            }
            s = e;
        }
    };
    add(0, rd.P);
    add(rd.P, rd.Q);
    for (int a = 0; a < rd.A; ++a)
        for (int r = 0; r < 3; ++r) {
            ag.ant[a][r] = (float)rd.ant[a][r];
            ag.ant_lo[a][r] = (float)(rd.ant[a][r] - (double)ag.ant[a][r]);
        }
    return ag;
}

void launch_visibility(const double *tri64, const float4 *trel, const double *c64,
                       const FacetRec *fac, const float *fac_lo, const double *ref64,
                       const WideNode *nodes, const int32_t *order, int64_t F, const RadarDev &rd,
                       const SceneSplit &sc, uint8_t *state, unsigned long long *n_graze,
                       int *status, cudaStream_t s)
{
    const AntGroups ag = ant_groups(rd, F);
    // pairs of a block: about one ray per quad while there are too few blocks,
    // more to refill quads from otherwise.  A frame's visibility and lists
    // with 32 / 64 / 128 pairs: 200 facets x 5 antennas 27 / 33 / 41 us, 20k x
    // 7 (four groups) 94 / 82 / 88, eight scenes of 73k x 7 180 / 166 / 157
    const int64_t all = F * ag.n_groups;
    const int pairs = all <= 16 * 1024 ? 32 : all <= 112 * 1024 ? 64 : kVisPairs;
    const dim3 grid((unsigned int)((F + pairs - 1) / pairs), (unsigned int)ag.n_groups);
    const VisArgs v{tri64, trel, c64, fac, fac_lo, ref64, nodes, order, F,
                    rd, ag, sc, pairs, state, n_graze, status};
    if (rd.far_field) visibility_far_kernel<<<grid, kVisThreads, 0, s>>>(v);
    else if (ag.n_groups < rd.A) visibility_kernel<<<grid, kVisThreads, 0, s>>>(v);
    else visibility_single_kernel<<<grid, kVisThreads, 0, s>>>(v);
}

// -------------------------------------------------------------------------
// compaction into ascending facet lists: list l < O holds the facets lit
// from TX p AND RX q of channel l = p Q + q on the same side (both LIT, or
// both LIT_REV); list O + a holds the facets lit from antenna a
// -------------------------------------------------------------------------
constexpr int kCompactBlk = 1024;

int64_t compact_blk_words(int64_t F, int L) { return (int64_t)L * ((F + kCompactBlk - 1) / kCompactBlk); }

// A block holds the states of kCompactBlk facets as bit words per antenna (lit,
// and lit in reverse), so that each of the O + A lists costs two ANDs per 32
// facets instead of two state loads per facet.  192 channels, 345k facets: the
// count took 237 us and the write 335 us with a state load per list and facet.
__device__ __forceinline__ void compact_words(const uint8_t *state, int64_t F, int A, int64_t k,
                                              uint32_t (*lit)[32], uint32_t (*rev)[32])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 4
    for (int a = 0; a < A; ++a) {
        const uint8_t s = k < F ? state[(int64_t)a * F + k] : 0;
        const uint32_t l = __ballot_sync(0xffffffffu, s == BART_VIS_LIT);
        const uint32_t r = __ballot_sync(0xffffffffu, s == BART_VIS_LIT_REV);
        if (lane == 0) {
            lit[a][warp] = l;
            rev[a][warp] = r;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ uint32_t list_word(const uint32_t (*lit)[32], const uint32_t (*rev)[32],
                                              int l, int O, int P, int Q, int w)
{
    if (l >= O) return lit[l - O][w] | rev[l - O][w];
    const int p = l / Q, q = P + l - p * Q;
    return (lit[p][w] & lit[q][w]) | (rev[p][w] & rev[q][w]);
}

__global__ void __launch_bounds__(kCompactBlk)
compact_count_kernel(const uint8_t *__restrict__ state, int64_t F, int O, int P, int Q,
                     int32_t *__restrict__ blk_cnt, int64_t nblk)
{
    __shared__ uint32_t s_lit[kMaxAnt][32], s_rev[kMaxAnt][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, L = O + P + Q;
    compact_words(state, F, P + Q, (int64_t)blockIdx.x * kCompactBlk + threadIdx.x, s_lit, s_rev);
    for (int l = warp; l < L; l += kCompactBlk / 32) {
        const int c = __reduce_add_sync(0xffffffffu, __popc(list_word(s_lit, s_rev, l, O, P, Q, lane)));
        if (lane == 0) blk_cnt[(int64_t)l * nblk + blockIdx.x] = c;
    }
}

// exclusive scan of each channel's block counts (one warp per channel), for
// more than kCompactScan blocks: up to there each block of the write adds the
// counts before it (eight loads a lane at most), which a sedan's 20 blocks do in
// less than the launch (2.9 us and a gap)
constexpr int kCompactScan = 256;

__global__ void compact_scan_kernel(int32_t *__restrict__ blk_cnt, int64_t nblk,
                                    int32_t *__restrict__ vis_cnt)
{
    const int o = blockIdx.x, lane = threadIdx.x;
    int32_t *c = blk_cnt + (int64_t)o * nblk;
    int32_t run = 0;
    for (int64_t b0 = 0; b0 < nblk; b0 += 32) {
        const int64_t b = b0 + lane;
        const int32_t v = b < nblk ? c[b] : 0;
        int32_t x = v;
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (b < nblk) c[b] = run + x - v;
        run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) vis_cnt[o] = run;
}

__global__ void __launch_bounds__(kCompactBlk)
compact_write_kernel(const uint8_t *__restrict__ state, int64_t F, int O, int P, int Q,
                     const int32_t *__restrict__ blk_cnt, int64_t nblk,
                     int32_t *__restrict__ vis_idx, int32_t *__restrict__ vis_cnt)
{
    __shared__ uint32_t s_lit[kMaxAnt][32], s_rev[kMaxAnt][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, L = O + P + Q;
    const int64_t k0 = (int64_t)blockIdx.x * kCompactBlk;
    compact_words(state, F, P + Q, k0 + threadIdx.x, s_lit, s_rev);
    for (int l = warp; l < L; l += kCompactBlk / 32) {
        const uint32_t mine = list_word(s_lit, s_rev, l, O, P, Q, lane);
        const int32_t *cnt = blk_cnt + (int64_t)l * nblk;
        int32_t before = 0;
        if (nblk > kCompactScan) {
            before = cnt[blockIdx.x];                     // scanned
        } else {
            for (int b = lane; b < blockIdx.x; b += 32) before += cnt[b];
            before = __reduce_add_sync(0xffffffffu, before);
            if (blockIdx.x == nblk - 1 && lane == 0) vis_cnt[l] = before + cnt[blockIdx.x];
        }
        // the words' first places, so that the 32 stores do not wait for one another
        int32_t at = __popc(mine);
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, at, off);
            if (lane >= off) at += y;
        }
        at += before - __popc(mine);
        int32_t *out = vis_idx + (int64_t)l * F;
#pragma unroll 8
        for (int w = 0; w < 32; ++w) {
            const uint32_t m = __shfl_sync(0xffffffffu, mine, w);
            const int32_t first = __shfl_sync(0xffffffffu, at, w);
            if ((m >> lane) & 1u)
                out[first + __popc(m & ((1u << lane) - 1u))] = (int32_t)(k0 + 32 * w + lane);
        }
    }
}

int launch_compact(const uint8_t *state, int64_t F, const RadarDev &rd, int32_t *blk_cnt,
                    int32_t *vis_idx, int32_t *vis_cnt, cudaStream_t s)
{
    const int64_t nblk = (F + kCompactBlk - 1) / kCompactBlk;
    const int L = rd.O + rd.A;
    const unsigned int grid = (unsigned int)nblk;
    compact_count_kernel<<<grid, kCompactBlk, 0, s>>>(state, F, rd.O, rd.P, rd.Q, blk_cnt, nblk);
    if (nblk > kCompactScan) compact_scan_kernel<<<L, 32, 0, s>>>(blk_cnt, nblk, vis_cnt);
    compact_write_kernel<<<grid, kCompactBlk, 0, s>>>(state, F, rd.O, rd.P, rd.Q, blk_cnt, nblk,
                                                      vis_idx, vis_cnt);
    return nblk > kCompactScan ? 3 : 2;
}

// lists are ascending in facet index and scenes own consecutive facets, so
// each (scene, channel) part of list o is one contiguous run
__global__ void scene_lists_kernel(const int32_t *__restrict__ vis_idx,
                                   const int32_t *__restrict__ vis_cnt, int64_t F, int O,
                                   const int64_t *__restrict__ foff, int B,
                                   int32_t *__restrict__ vstart, int32_t *__restrict__ vcnt)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= B * O) return;
    const int b = v / O, o = v % O;
    const int32_t *list = vis_idx + (int64_t)o * F;
    const int n = vis_cnt[o];
    int lim[2];
    for (int e = 0; e < 2; ++e) {           // first entry with facet >= foff[b + e]
        const int64_t key = foff[b + e];
        int lo = 0, hi = n;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (list[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        lim[e] = lo;
    }
    vstart[v] = lim[0];
    vcnt[v] = lim[1] - lim[0];
}

void launch_scene_lists(const int32_t *vis_idx, const int32_t *vis_cnt, int64_t F, int O,
                        const int64_t *foff, int B, int32_t *vstart, int32_t *vcnt,
                        cudaStream_t s)
{
    const int T = 128;
    scene_lists_kernel<<<(B * O + T - 1) / T, T, 0, s>>>(vis_idx, vis_cnt, F, O, foff, B, vstart,
                                                         vcnt);
}

}  // namespace bart
