// Band-limited evaluation of the mixed echo synthesis (band.cu).
//
// All facets of one rigid instance move together, so once the phase of a
// point of the instance (the reference: its box centre, with its own exact
// path) is taken off, the sum over its facets varies slowly along the chirps
// and occupies a narrow band of beat frequencies along the samples.  The
// instance's sum is therefore evaluated at a few chirps and on a coarse
// sample grid only, and interpolated:
//   x[n][m] = sum_instances exp(j 2 pi ref(n, m))
//             * sum_j Wn[n][j] sum_s Wm[m][s] C[j][s],
//   C[j][s] = sum_facets exp(-j 2 pi ref) (Eq. 13 term) at chirp n_j (not
//             whole in general) and sample m_s = d s - off.
// Chirps: Chebyshev nodes, polynomial interpolation; a phase that turns by
// at most a radians either way over half the frame needs K nodes with
// 4 sum_{k >= K-1} |J_k(a)| < 2e-7 (the Chebyshev coefficients of
// exp(j a x), one node kept for the amplitudes' drift).  Samples: a uniform
// grid of spacing d with kBandTaps-tap least-squares interpolation over the
// band |f| <= 0.5 / kBandOver of the grid's rate (at most 2e-6 at the band's
// edge, 1e-7 rms).  Static instances have one chirp.  An instance whose
// bounds exceed the tables keeps every chirp and every sample (n_j = n,
// d = 1), which is the direct sum; a moving one lit from both sides keeps every
// chirp, since its facets' obliquity |o| has a kink where they pass edge-on.
//
// What it gives: a 20k-facet sedan on 12 channels of 128 x 256 needs 12
// chirps of 48 samples instead of 128 of 256; its synthesis took 1.19 ms by
// the direct sum (FMA pipe 70 % busy) and takes 0.12 ms, the intersection's
// (300k facets, 192 channels, 64 x 512) 290 ms and 18 ms.  The cube's error
// falls as well, from 8e-6 to 0.8e-6: no lane follows more of the quadratic
// phase than its facet's offset from the reference, and the few records can
// afford double-float projections and the pair form (mixed_record.cuh).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bart_internal.cuh"

namespace bart {

constexpr int kBandS = 16;          // samples per lane
constexpr int kBandTaps = 20;       // taps of the sample interpolation
constexpr int kBandGuard = 4;       // coarse samples beyond either end
constexpr double kBandOver = 1.8;   // grid rate over the band's width
constexpr int kBandMaxM = 12;       // sample layouts
constexpr int kBandMaxN = 16;       // chirp layouts

// Sample layout: Mi = 16 lpr nseg coarse samples of a row, m_s = d s - off,
// lpr lanes per (chirp, segment) row.  Layout 0 keeps every sample.
struct BandM {
    int lpr, nseg, Mi;
    float d, off;
    float beta;          // largest beat-frequency offset, cycles per sample
};
// Chirp layout: nj nodes; layout 0 keeps every chirp, layout 1 is static.
struct BandN {
    int nj;
    float amax;          // largest residual phase over half a frame, radians
    int node0;           // first node position and first weight in the tables
    int64_t w0;
};
struct BandShape {
    int N, M, n_m, n_n;
    BandM m[kBandMaxM];
    BandN n[kBandMaxN];
};
struct BandPlan {        // per instance
    int in, im;          // chirp and sample layout
    int rotate;          // a reference phase is in use
    int exact_u;         // records with double-float projections (see build_mixed_record)
    float c[3];          // reference point at t0
};

// layouts for N chirps of M samples, the sizes of their tables -- node
// positions [sum nj], chirp weights [layout][N][nj] and, per sample layout,
// every sample's first tap [M] and weights [kBandTaps][M] -- and the tables
void band_shape(int N, int M, BandShape &sh);
struct BandSizes {
    int64_t nodes, wn, base, wm;
};
BandSizes band_sizes(const BandShape &sh);
void launch_band_tables(const BandShape &sh, float *nodes, float *wn, int *base, float *wm,
                        cudaStream_t s);

struct BandItem {
    int v;               // instance * O + channel
    int grp;             // row group of the (node, segment) rows
    int rbeg, rend;      // entries of the (instance, channel) list
};

struct BandArgs {
    BandShape sh;
    const float *nodes, *wn;
    const int *base;
    const float *wm;
    int I, B, O;
    const unsigned int *box;     // [I][8] (see launch_build_facets)
    const int32_t *scene_inst;   // [B + 1]
    const int64_t *ioff;         // [I + 1] first facet of each instance
    BandPlan *plan;
    float4 *ref, *refn;          // [I O][N] reference at the chirps, at the nodes
    int32_t *vstart, *vcnt;      // [I O] list parts
    int32_t *item0;              // [I O + 1] first item
    int64_t *coff;               // [I O] first coarse value
    int *item_counter;
    int chunk_target;            // work items to aim for
    int fixed_chunk;             // facets per work item (0: from chunk_target)
    int *chunk;                  // facets per work item, chosen on the device
    BandItem *items;
    float4 *partial;             // [item][8][32] sample pairs
    float2 *coarse;
    int64_t max_items;
};

int64_t band_max_items(const BandShape &sh, int64_t V, int target, int64_t lit_max, int fixed_chunk);
// after the world facets: plan and reference tables
void launch_band_plan(const BandArgs &b, const SynthArgs &a, cudaStream_t s);
// after the lists and the kinematics rows: items, coarse sums, expansion
void launch_synth_band(const BandArgs &b, const SynthArgs &a, cudaStream_t s);
int launch_synth_band_count(const BandArgs &b);      // its launches
// per-form record counts of the whole frame (stats)
void launch_count_records(const SynthArgs &a, cudaStream_t s);

}  // namespace bart
