// Band-limited evaluation of the FP64 echo synthesis and its adjoint
// (band64.cu): the idea of band.cuh at FP64 accuracy.
//   x[n][m] = sum_instances exp(j 2 pi ref(n, m)) sum_j Wn[n][j] sum_s Wm[m][s] C[j][s],
//   C[j][s] = sum_facets exp(-j 2 pi ref) (Eq. 13 term) at chirp n_j, sample m_s.
// Both grids are Chebyshev nodes with polynomial interpolation: a phase that
// turns by at most a radians either way over half the grid's length needs K
// nodes with 4 sum_{k >= K-1} |J_k(a)| < 1e-13 (one node kept for the
// amplitudes' drift), below the direct sum's own rounding (f L / c is some
// 1e4 cycles in FP64: 1e-11 radians).  The reference is a quadratic in fast
// time whose constant is formed in double-double, so that its rounding, which
// the whole instance shares, stays below a facet's.
// An instance of many facets is cut into cells of its box first, each a
// rigid body of its own: half the extent needs half the nodes (see
// band64_cells).
//
// The direct sum is bound by the FP64 pipe (a 64th of the FP32 rate, 86 % busy):
// its time goes with the samples it evaluates.  So it is with the adjoint, whose
// facet sums over samples become sums over nodes once the cube's gradient has
// gone through the interpolation's transpose (a 1.5k-facet car, 8 channels of 32
// x 128: 7.95 ms, now 0.45 and 0.07 for the transpose).  A 5k-facet car on 12 channels
// of 32 x 256 takes 1.9 ms against 33.1.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bart_internal.cuh"

namespace bart {

constexpr int kB64N = 16;           // chirp layouts, at most
constexpr int kB64M = 18;           // sample layouts, at most
constexpr int kB64MaxNodes = 128;   // chirp nodes of a layout that is not every chirp
constexpr int kB64Cells = 4;         // cells of an instance, at most
constexpr int kB64Chunks = 16;      // partial sums of a node, at most

// Layout 0 keeps every chirp / sample; chirp layout 1 is static (one chirp).
struct Band64Shape {
    int N, M, n_n, n_m;
    int kn[kB64N], km[kB64M];       // nodes
    float an[kB64N], am[kB64M];     // largest phase, radians
    int xn[kB64N], xm[kB64M];       // first node in the tables
    int64_t wn[kB64N], wm[kB64M];   // first weight in the tables
};

struct Band64Plan {                 // per body
    int in, im, rotate;
    float c[3];
};

struct Band64Args {
    Band64Shape sh;
    const double *xn, *xm;          // node positions (chirps, samples)
    const double *wn, *wm;          // weights [N][kn], [km][M]
    const double2 *turn;            // [256] exp(j 2 pi i / 256)
    int I, B, O;                    // bodies: instances x cells
    int cells;                      // kB64Cells or 1
    int room;                       // partial sums' room of a body and channel, in cubes
    const unsigned int *box;        // [instances][8] (see launch_build_facets)
    const int32_t *scene_inst;      // [B + 1]
    const int64_t *ioff;            // [instances + 1]
    uint8_t *cell;                  // [F] cell of each facet (cells > 1)
    unsigned int *cbox;             // [I][8] the cells' boxes
    int32_t *list;                  // [O][F] the lists in cell order
    Band64Plan *plan;
    double4 *ref, *refn;            // [I O][N] phase quadratics at the chirps, at the nodes
    int32_t *vstart, *vcnt;         // [I O] list parts
    int32_t *item0;                 // [I O + 1]
    int *ticket;
    double2 *coarse;                // [I O][room N M] partial node sums
};

void band64_shape(int N, int M, Band64Shape &sh);
struct Band64Sizes {
    int64_t xn, xm, wn, wm;         // doubles
};
Band64Sizes band64_sizes(const Band64Shape &sh);
// tables (tab: 512 + the sizes' sum doubles) and their pointers in b
void band64_tables(double *tab, Band64Args &b);
void launch_band64_tables(const Band64Args &b, cudaStream_t s);
// after the world facets: plans and reference phases
void launch_band64_plan(const Band64Args &b, const SynthArgs &a, cudaStream_t s);
// after the lists: items, node sums, expansion
void launch_synth_band64(const Band64Args &b, const SynthArgs &a, cudaStream_t s);
// after the lists: facet gradients gfac [F][10] of the loss whose gradient of the
// cube is grad (the cube's order)
void launch_adjoint_band64(const Band64Args &b, const SynthArgs &a, const void *grad, int grad_c64,
                           double *gfac, cudaStream_t s);
// per-form record counts of the whole frame (stats)
void launch_count_records64(const SynthArgs &a, cudaStream_t s);

}  // namespace bart
