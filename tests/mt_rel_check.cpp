// The cases of mt_pretest_check.cpp, with the relative pre-test of the
// visibility rays (mt_rel_classify, geom64.cuh) in the place of the one over
// absolute coordinates; same counts printed.
#include <cmath>
#include <cstdint>

static inline double rel_dadd(double a, double b) { return a + b; }
static inline double rel_dsub(double a, double b) { return a - b; }
static inline double rel_dmul(double a, double b) { return a * b; }
static inline double rel_ddiv(double a, double b) { return a / b; }
#define __dadd_rn rel_dadd
#define __dsub_rn rel_dsub
#define __dmul_rn rel_dmul
#define __ddiv_rn rel_ddiv
#include "geom64.cuh"
#undef __dadd_rn
#undef __dsub_rn
#undef __dmul_rn
#undef __ddiv_rn

// the inputs as the world-facet and visibility kernels form them
static int rel_classify(const double *tri, const double *O, const float *d, float Dm, float Om)
{
    float h[3], l[3], oh[3], ol[3], e1[3], e2[3];
    for (int r = 0; r < 3; ++r) {
        h[r] = (float)tri[r];
        l[r] = (float)(tri[r] - (double)h[r]);
        oh[r] = (float)O[r];
        ol[r] = (float)(O[r] - (double)oh[r]);
        e1[r] = (float)(tri[3 + r] - tri[r]);
        e2[r] = (float)(tri[6 + r] - tri[r]);
    }
    return bart::mt_rel_classify(make_float4(h[0], h[1], h[2], e1[0]),
                                 make_float4(e1[1], e1[2], e2[0], e2[1]),
                                 make_float4(e2[2], l[0], l[1], l[2]), oh, ol, d, Dm, Dm * 5.9604645e-8f,
                                 Om);
}
#define mt_fp32_classify(t0, t1, t2, o, d, Dm, Om) rel_classify(tri, O, d, Dm, Om)
#include "mt_pretest_check.cpp"
