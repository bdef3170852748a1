// Band-limited mixed echo synthesis (see band.cuh): plan, reference phases,
// work items, coarse sums, interpolation.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "band.cuh"
#include "band_plan.cuh"
#include "mixed_lane.cuh"
#include "mixed_record.cuh"

namespace bart {

// -------------------------------------------------------------------------
// layouts (host)
// -------------------------------------------------------------------------
void band_shape(int N, int M, BandShape &sh)
{
    sh = BandShape{};
    sh.N = N;
    sh.M = M;
    // sample layouts: every sample, then 32, 48, ... coarse samples while
    // they save a fifth of the row
    {
        BandM &f = sh.m[sh.n_m++];
        int lanes = M / kBandS;                   // M is a multiple of 32
        f.nseg = 1;
        while (lanes > 32 || (lanes * f.nseg != M / kBandS)) {
            ++f.nseg;
            lanes = M / kBandS / f.nseg;
        }
        f.lpr = lanes;
        f.Mi = M;
        f.d = 1.f;
        f.off = 0.f;
        f.beta = 1e30f;
    }
    static const int lprs[] = {2, 3, 4, 5, 6, 8, 10, 16};
    // spacing in 1/8 (1/4 beyond 512) samples: the products of a position
    // and a beat frequency's high part stay exact in FP32
    const double q = M <= 512 ? 8.0 : 4.0;
    for (int lpr : lprs) {
        const int Mi = kBandS * lpr;
        if (5 * Mi > 4 * M || sh.n_m == kBandMaxM) break;
        const double d = std::floor((M - 1.0) / (Mi - 1 - 2 * kBandGuard) * q + 1.0) / q;
        BandM &f = sh.m[sh.n_m++];
        f.lpr = lpr;
        f.nseg = 1;
        f.Mi = Mi;
        f.d = (float)d;
        f.off = (float)(d * kBandGuard);
        f.beta = (float)(0.5 / (kBandOver * d));
    }
    // chirp layouts: K nodes carry a phase of up to amax radians
    static const struct { int K; float a; } cheb[] = {
        {8, 0.60f}, {10, 1.27f}, {12, 2.12f}, {14, 3.11f}, {16, 4.22f}, {20, 6.66f}, {24, 9.35f},
        {28, 12.2f}, {32, 15.1f}, {40, 21.3f}, {48, 27.8f}, {64, 41.3f}, {80, 55.2f}, {128, 98.4f}};
    int node0 = 0;
    int64_t w0 = 0;
    sh.n[sh.n_n++] = BandN{N, 1e30f, node0, w0};      // every chirp: nodes 0 .. N - 1
    node0 += N;
    sh.n[sh.n_n++] = BandN{1, 0.f, node0, w0};        // static
    node0 += 1;
    for (auto &c : cheb) {
        if (5 * c.K > 4 * N || sh.n_n == kBandMaxN) break;
        sh.n[sh.n_n++] = BandN{c.K, c.a, node0, w0};
        node0 += c.K;
        w0 += (int64_t)c.K * N;
    }
}

BandSizes band_sizes(const BandShape &sh)
{
    BandSizes z{};
    for (int l = 0; l < sh.n_n; ++l) {
        z.nodes += sh.n[l].nj;
        z.wn += l > 1 ? (int64_t)sh.n[l].nj * sh.N : 0;
    }
    z.base = (int64_t)sh.n_m * sh.M;
    z.wm = z.base * kBandTaps;
    return z;
}

int64_t band_max_items(const BandShape &sh, int64_t V, int target, int64_t lit_max, int fixed_chunk)
{
    int64_t groups = 1;           // row groups of an (instance, channel), at most
    for (int l = 0; l < sh.n_m; ++l) {
        const int rpw = 32 / sh.m[l].lpr;
        groups = std::max<int64_t>(groups, ((int64_t)sh.N * sh.m[l].nseg + rpw - 1) / rpw);
    }
    // ceil(count / chunk) chunks per group: one each, and the target spread
    // over them, a chunk at least 32 facets (a fixed chunk: the whole list's
    // chunks)
    const int64_t more = fixed_chunk > 0 ? groups * (lit_max / fixed_chunk + 1)
                                         : std::min<int64_t>(target, groups * (lit_max / 32 + 1));
    return V * groups + more;
}

// -------------------------------------------------------------------------
// plan: per instance, the largest offsets of path and path rate from its box
// centre, over its box and the frame
// -------------------------------------------------------------------------
namespace {

// Interpolation tables.  Blocks x < n_n fill the chirp layouts (a slice of the
// chirps per y): Chebyshev nodes of [0, N - 1], rounded to 1/1024 chirp (exact
// in FP32 with the slots of time-division MIMO), and the barycentric weights
// of those nodes.  The others fill the sample layouts: least-squares taps,
// the error minimised over |f| <= 0.5 / kBandOver of the coarse rate; the
// normal equations' matrix depends on the taps' spacing alone, so that its
// Cholesky factor, formed once on the host, serves every sample and layout.
struct BandChol {
    double L[kBandTaps * (kBandTaps + 1) / 2];
};

__device__ __host__ __forceinline__ double band_sinc(double x)
{
#ifdef __CUDA_ARCH__
    return x == 0.0 ? 1.0 : sinpi(x) / (kPi * x);
#else
    return x == 0.0 ? 1.0 : sin(kPi * x) / (kPi * x);
#endif
}

// one warp a block: the FP64 work spread over the multiprocessors
constexpr int kTabRows = 32;         // blocks of a layout

__global__ void __launch_bounds__(32)
band_table_kernel(BandShape sh, BandChol ch, float *__restrict__ nodes, float *__restrict__ wn,
                  int *__restrict__ base, float *__restrict__ wm)
{
    constexpr int T = kBandTaps;
    const int N = sh.N, M = sh.M, tid = threadIdx.x;
    __shared__ double x[128], w[128], r[T][32];
    if ((int)blockIdx.x < sh.n_n) {
        const int l = blockIdx.x;
        const BandN lay = sh.n[l];
        if (l < 2) {
            if (blockIdx.y == 0)
                for (int j = tid; j < lay.nj; j += blockDim.x) nodes[lay.node0 + j] = (float)j;
            return;
        }
        const int K = lay.nj;
        for (int j = tid; j < K; j += blockDim.x) {
            const double c = 0.5 * (N - 1) * (1.0 - cospi((j + 0.5) / K));
            x[j] = rint(c * 1024.0) * (1.0 / 1024.0);
            if (blockIdx.y == 0) nodes[lay.node0 + j] = (float)x[j];
        }
        __syncthreads();
        for (int j = tid; j < K; j += blockDim.x) {
            double p[4] = {1.0, 1.0, 1.0, 1.0};                // four chains of products
            const double xj = x[j], sc = 4.0 / (N - 1);
            for (int i = 0; i < K; i += 4)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (i + q != j && i + q < K) p[q] *= (xj - x[i + q]) * sc;
            w[j] = 1.0 / ((p[0] * p[1]) * (p[2] * p[3]));
        }
        __syncthreads();
        const int lane = tid;
        for (int n = blockIdx.y; n < N; n += kTabRows) {
            double sum = 0.0;
            int hit = -1;
            for (int j = lane; j < K; j += 32) {
                if ((double)n == x[j]) hit = j;
                else sum += w[j] / (n - x[j]);
            }
            for (int off = 16; off > 0; off >>= 1) {
                sum += __shfl_xor_sync(0xffffffffu, sum, off);
                hit = max(hit, __shfl_xor_sync(0xffffffffu, hit, off));
            }
            for (int j = lane; j < K; j += 32)
                wn[lay.w0 + (int64_t)n * K + j] =
                    hit >= 0 ? (j == hit ? 1.f : 0.f) : (float)(w[j] / ((n - x[j]) * sum));
        }
        return;
    }
    const int l = blockIdx.x - sh.n_n;
    const BandM lay = sh.m[l];
    for (int m = blockIdx.y * blockDim.x + tid; m < M; m += gridDim.y * blockDim.x) {
        if (l == 0) {
            base[m] = 0;
            continue;
        }
        const double pos = ((double)m + lay.off) / lay.d;
        const int b0 = max(0, min(lay.Mi - T, (int)floor(pos) - T / 2 + 1));
        const double w2 = 1.0 / kBandOver;                // twice the band edge
        // sines of the taps' arguments by turns of w2 (their spacing), then both
        // triangular solves column by column: the updates of a step are
        // independent, where row by row each waited for the last.  Rolled, in
        // shared memory: the table is made once a frame size, so that unrolled
        // code comes from memory (55 us a table, now 43)
        double sn, cs, ds, dc;
        sincospi(w2 * (b0 - pos), &sn, &cs);
        sincospi(w2, &ds, &dc);
#pragma unroll 1
        for (int i = 0; i < T; ++i) {
            const double x = w2 * (b0 + i - pos);
            r[i][tid] = x == 0.0 ? w2 : w2 * sn / (kPi * x);
            const double c2 = cs * dc - sn * ds;
            sn = sn * dc + cs * ds;
            cs = c2;
        }
#pragma unroll 1
        for (int k = 0; k < T; ++k) {
            const double v = r[k][tid] * ch.L[k * (k + 1) / 2 + k];   // the diagonal is stored inverted
            r[k][tid] = v;
#pragma unroll 4
            for (int i = k + 1; i < T; ++i) r[i][tid] -= ch.L[i * (i + 1) / 2 + k] * v;
        }
#pragma unroll 1
        for (int k = T - 1; k >= 0; --k) {
            const double v = r[k][tid] * ch.L[k * (k + 1) / 2 + k];
            r[k][tid] = v;
#pragma unroll 4
            for (int i = 0; i < k; ++i) r[i][tid] -= ch.L[k * (k + 1) / 2 + i] * v;
        }
        base[(int64_t)l * M + m] = b0;
#pragma unroll 4
        for (int i = 0; i < T; ++i) wm[((int64_t)l * T + i) * M + m] = (float)r[i][tid];
    }
}

// one warp per instance
__global__ void band_plan_kernel(BandArgs b, RadarDev rd, MixConsts K, const float *__restrict__ vel32,
                                 const FacetRec *__restrict__ fac)
{
    const int i = blockIdx.x;
    const BandBounds q = band_bounds(b.box, i, i, rd, K, vel32);
    if (threadIdx.x != 0) return;
    BandPlan pl;
    for (int r = 0; r < 3; ++r) pl.c[r] = q.c[r];
    pl.im = pl.in = 0;
    // a static instance keeps every sample: its one chirp costs little
    if (q.ok && q.speed > 0.f)
        for (int l = 1; l < b.sh.n_m; ++l) {
            // a lane follows the residual quadratic phase by its chord
            const float span = 15.f * b.sh.m[l].d;
            if (q.beta <= b.sh.m[l].beta && 6.2831853f * q.p2 * span * span * 0.25f <= 1e-5f) {
                pl.im = l;
                break;
            }
        }
    // a facet lit from both sides has a kink where its obliquity changes sign
    // (interpolated: 1 to 4 % off on a plate that passes edge-on): every chirp is kept
    const bool smooth = b.ioff[i] < b.ioff[i + 1] && !fac[b.ioff[i]].two_sided;
    if (q.speed == 0.f) {
        pl.in = 1;
    } else if (q.ok && smooth) {
        for (int l = 2; l < b.sh.n_n; ++l)
            if (q.turn <= b.sh.n[l].amax) {
                pl.in = l;
                break;
            }
    }
    // a moving instance's reference also takes most of the within-chirp
    // quadratic phase off its lanes' chords, with every sample kept too
    pl.rotate = q.speed > 0.f;
    // double-float u and the pair form for every facet, except on static
    // instances of large facets (the ground): their sums, the same for every
    // chirp, keep the direct kernel's arithmetic
    pl.exact_u = q.speed > 0.f || 2.f * q.rf * K.f0c <= 64.f;
    b.plan[i] = pl;
}

// reference phase of (instance, channel) at chirp n: the box centre's path,
// in FP64; (ph0, hi, lo, p2) as a record's
__device__ __forceinline__ float4 band_ref(const RadarDev &rd, const float *c, const double *v, int p,
                                           int q, double slot)
{
    const double t = slot * rd.Tc;
    double L = 0.0, Ld = 0.0, Ldd = 0.0;
    const double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const double *pa = rd.ant[e == 0 ? p : rd.P + q];
        const double x = ((double)c[0] - pa[0]) + v[0] * t, y = ((double)c[1] - pa[1]) + v[1] * t,
                     z = ((double)c[2] - pa[2]) + v[2] * t;
        const double R2 = x * x + y * y + z * z;
        const double iR = R2 > 0.0 ? rsqrt(R2) : 0.0, R = R2 * iR;
        const double rr = (v[0] * x + v[1] * y + v[2] * z) * iR;
        L += R;
        Ld += rr;
        Ldd += (v2 - rr * rr) * iR;
    }
    if (!rd.intra) Ld = Ldd = 0.0;
    const double ic = 1.0 / kC0, ifs = 1.0 / rd.fs, mc = rd.slope * ic, fc = rd.f0 * ic;
    const double ph = fc * L - 0.5 * mc * ic * L * L;
    double al = (mc * L + fc * Ld - mc * ic * L * Ld) * ifs;
    al -= floor(al);
    const double hi = rint(al * 16384.0) * (1.0 / 16384.0);
    return make_float4((float)(ph - rint(ph)), (float)(hi >= 1.0 ? hi - 1.0 : hi), (float)(al - hi),
                       (float)((0.5 * fc * Ldd + mc * Ld) * ifs * ifs));
}

__global__ void __launch_bounds__(128)
band_ref_kernel(BandArgs b, RadarDev rd, const double *__restrict__ vel64)
{
    const int v = blockIdx.y, i = v / b.O, o = v % b.O;
    const BandPlan pl = b.plan[i];
    const int N = b.sh.N, nj = b.sh.n[pl.in].nj;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const bool node = e >= N;                     // chirps first, then nodes
    const int k = node ? e - N : e;
    if (k >= (node ? nj : N)) return;
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pl.rotate) {
        const int p = o / rd.Q, q = o % rd.Q;
        const double n = node ? (double)b.nodes[b.sh.n[pl.in].node0 + k] : (double)k;
        const double vel[3] = {vel64[3 * i], vel64[3 * i + 1], vel64[3 * i + 2]};
        r = band_ref(rd, pl.c, vel, p, q, n * rd.slots + (rd.tdm ? p : 0));
    }
    (node ? b.refn : b.ref)[(int64_t)v * N + k] = r;
}

// -------------------------------------------------------------------------
// list parts and work items
// -------------------------------------------------------------------------

// warps 2 v, 2 v + 1: the ends of list o's part with instance i's facets
__global__ void band_lists_kernel(BandArgs b, const int32_t *__restrict__ vis_idx,
                                  const int32_t *__restrict__ vis_cnt, int64_t F)
{
    const int lane = threadIdx.x & 31;
    const int v = blockIdx.x * (blockDim.x >> 6) + (threadIdx.x >> 6);
    const int e = (threadIdx.x >> 5) & 1;
    __shared__ int s_lim[8][2];
    const bool ok = v < b.I * b.O;
    if (ok) {
        const int i = v / b.O, o = v % b.O;
        const int at = warp_lower_bound(vis_idx + (int64_t)o * F, vis_cnt[o], b.ioff[i + e], lane);
        if (lane == 0) s_lim[threadIdx.x >> 6][e] = at;
    }
    __syncthreads();
    if (ok && e == 0 && lane == 0) {
        const int lo = s_lim[threadIdx.x >> 6][0];
        b.vstart[v] = lo;
        b.vcnt[v] = s_lim[threadIdx.x >> 6][1] - lo;
    }
}

__device__ __forceinline__ int band_groups(const BandShape &sh, const BandPlan &pl)
{
    const int rpw = 32 / sh.m[pl.im].lpr;
    return (sh.n[pl.in].nj * sh.m[pl.im].nseg + rpw - 1) / rpw;
}

// facets per work item, then the item and coarse-value prefixes (one block)
__device__ __forceinline__ void band_items(const BandArgs &b)
{
    __shared__ long long s_w[32], s_c[32], s_work;
    __shared__ long long s_run, s_crun;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int V = b.I * b.O;
    long long w = 0;
    for (int v = t; v < V; v += 1024) w += (long long)b.vcnt[v] * band_groups(b.sh, b.plan[v / b.O]);
    for (int off = 16; off > 0; off >>= 1) w += __shfl_xor_sync(0xffffffffu, w, off);
    if (lane == 0) s_w[warp] = w;
    __syncthreads();
    if (t == 0) {
        s_work = 0;
        for (int k = 0; k < 32; ++k) s_work += s_w[k];
        s_run = s_crun = 0;
    }
    __syncthreads();
    long long chunk = b.fixed_chunk;
    if (chunk == 0) {
        chunk = (s_work + b.chunk_target - 1) / b.chunk_target;
        if (chunk < 32) chunk = 32;
    }
    if (t == 0) {
        *b.chunk = (int)chunk;
        *b.item_counter = 0;
    }
    for (int v0 = 0; v0 < V; v0 += 1024) {
        const int v = v0 + t;
        long long items = 0, vals = 0;
        if (v < V) {
            const BandPlan &pl = b.plan[v / b.O];
            items = (b.vcnt[v] + chunk - 1) / chunk * band_groups(b.sh, pl);
            vals = b.vcnt[v] > 0 ? (long long)b.sh.n[pl.in].nj * b.sh.m[pl.im].Mi : 0;
        }
        long long x = items, y = vals;
        for (int off = 1; off < 32; off <<= 1) {
            const long long xu = __shfl_up_sync(0xffffffffu, x, off);
            const long long yu = __shfl_up_sync(0xffffffffu, y, off);
            if (lane >= off) {
                x += xu;
                y += yu;
            }
        }
        if (lane == 31) {
            s_w[warp] = x;
            s_c[warp] = y;
        }
        __syncthreads();
        long long bx = s_run, by = s_crun, ax = 0, ay = 0;
        for (int k = 0; k < 32; ++k) {
            if (k < warp) {
                bx += s_w[k];
                by += s_c[k];
            }
            ax += s_w[k];
            ay += s_c[k];
        }
        if (v < V) {
            b.item0[v] = (int)(bx + x - items);
            b.coff[v] = by + y - vals;
        }
        __syncthreads();
        if (t == 0) {
            s_run += ax;
            s_crun += ay;
        }
        __syncthreads();
    }
    if (t == 0) b.item0[V] = (int)s_run;
}

__global__ void __launch_bounds__(1024) band_items_kernel(BandArgs b) { band_items(b); }

// the items of (instance, channel) v, chunk by chunk through the row groups, so
// that a chunk's facet records come from HBM once; by threads first, first + step, ...
__device__ __forceinline__ void band_fill(const BandArgs &b, int v, int first, int step)
{
    const int n = b.item0[v + 1] - b.item0[v];
    const int groups = band_groups(b.sh, b.plan[v / b.O]);
    const int chunk = *b.chunk, cnt = b.vcnt[v];
    for (int k = first; k < n; k += step) {
        const int j = k / groups;
        BandItem it;
        it.v = v;
        it.grp = k - j * groups;
        it.rbeg = j * chunk;
        it.rend = min(cnt, it.rbeg + chunk);
        b.items[b.item0[v] + k] = it;
    }
}

__global__ void band_fill_kernel(BandArgs b) 
{
    band_fill(b, blockIdx.x, threadIdx.x, blockDim.x);
}

// All three in one block for up to kBandSmall (instance, channel) pairs: the
// launches, not their work, are what such a frame spends there (a sedan's 12
// pairs: 14.5 us in three launches and their gaps, 10.8 in one).
constexpr int kBandSmall = 48;

__global__ void __launch_bounds__(1024)
band_small_kernel(BandArgs b, const int32_t *__restrict__ vis_idx,
                  const int32_t *__restrict__ vis_cnt, int64_t F)
{
    __shared__ int s_lim[2 * kBandSmall];
    const int lane = threadIdx.x & 31, V = b.I * b.O;
    for (int w = threadIdx.x >> 5; w < 2 * V; w += 32) {
        const int v = w >> 1, i = v / b.O, o = v % b.O;
        const int at = warp_lower_bound(vis_idx + (int64_t)o * F, vis_cnt[o], b.ioff[i + (w & 1)], lane);
        if (lane == 0) s_lim[w] = at;
    }
    __syncthreads();
    if (threadIdx.x < V) {
        b.vstart[threadIdx.x] = s_lim[2 * threadIdx.x];
        b.vcnt[threadIdx.x] = s_lim[2 * threadIdx.x + 1] - s_lim[2 * threadIdx.x];
    }
    __syncthreads();
    band_items(b);
    __syncthreads();
    for (int v = threadIdx.x >> 5; v < V; v += 32) band_fill(b, v, lane, 32);
}

// -------------------------------------------------------------------------
// coarse sums
// -------------------------------------------------------------------------
constexpr int kBandWarps = 2;
constexpr int kBandBlocks = 8;      // resident CTAs per SM: 128 registers a thread

// As synth_mixed_kernel, over rows (node, segment) of lpr lanes (lpr not a
// power of two in general: rpw = 32 / lpr rows a warp, the lanes left over
// idle) on the coarse sample grid.
__global__ void __launch_bounds__(kBandWarps * 32, kBandBlocks)
synth_band_kernel(SynthArgs A, MixConsts K, BandArgs b)
{
    constexpr int S = kBandS, S2 = S / 2;
    __shared__ RecM sRec[kBandWarps][32];
    __shared__ uint64_t sAcc[kBandWarps][4][S2][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int P = A.rd.P, Q = A.rd.Q;
    const int64_t F = A.F;
    const int total = b.item0[b.I * b.O];
    const uint64_t zero2 = pk2(0.f, 0.f);

    for (;;) {
    int item = 0;
    if (lane == 0) item = atomicAdd(b.item_counter, 1);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= total) break;
    const BandItem it = b.items[item];
    const int inst = it.v / b.O, o = it.v - inst * b.O;
    const BandPlan &pl = b.plan[inst];
    const BandM lay = b.sh.m[pl.im];
    const BandN chirps = b.sh.n[pl.in];
    const int lpr = lay.lpr, rpw = 32 / lpr;
    const int row = lane / lpr, col = lane - row * lpr;
    const int rs = it.grp * rpw + row;                 // (node, segment)
    const bool row_ok = row < rpw && rs < chirps.nj * lay.nseg;
    const int node = row_ok ? rs / lay.nseg : 0;
    const int seg = row_ok ? rs - node * lay.nseg : 0;
    const int tx = o / Q, rx = o % Q;
    const float d = lay.d;
    const float fm0 = fmaf(d, (float)((seg * lpr + col) * S), -lay.off);
    // chord of the quadratic phase over the lane, its error centred:
    // p2 d^2 s (s - 15) averages -35 p2 d^2
    const float fm0sq = fmaf(fm0, fm0, -35.f * d * d);
    const float eps_lane = 6.283185307179586f * d * fmaf((float)(S - 1), d, 2.f * fm0);
    MixRow w;
    {
        const float nf = b.nodes[chirps.node0 + node];
        const float slot = fmaf(nf, (float)A.rd.slots, A.rd.tdm ? (float)tx : 0.f);   // exact
        w.tn = slot * K.tc;
        w.ant_t = tx;
        w.ant_r = P + rx;
        const double t = (double)slot * A.rd.Tc;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const double vt = A.vel64[3 * inst + r] * t;
            const double xt = A.rd.ant[tx][r] - vt, xr = A.rd.ant[P + rx][r] - vt;
            w.ath[r] = (float)xt;
            w.atl[r] = (float)(xt - (double)w.ath[r]);
            w.arh[r] = (float)xr;
            w.arl[r] = (float)(xr - (double)w.arh[r]);
        }
        w.d = d;
        // with the reference off, the steps' angles lie about 0, where the
        // recurrence's rounding grows fastest (as the square of the steps);
        // an eighth of a turn per step puts its two-step angle about a quarter
        // turn; lanes start at whole turns, and band_reduce_kernel turns back
        w.turn = pl.rotate ? 0.125f : 0.f;
        w.ref = b.refn[(int64_t)it.v * b.sh.N + node];
    }
    uint64_t PR[S2], PI[S2];
#pragma unroll
    for (int k = 0; k < S2; ++k) {
        PR[k] = PI[k] = zero2;
        sAcc[warp][0][k][lane] = zero2;
        sAcc[warp][1][k][lane] = zero2;
        sAcc[warp][2][k][lane] = zero2;
        sAcc[warp][3][k][lane] = zero2;
    }
    const int32_t *list = A.vis_idx + (int64_t)o * F + b.vstart[it.v];
    int held = 0;                                      // facets in PR, PI
    for (int base = it.rbeg; base < it.rend; base += lpr) {
        const bool valid = row_ok && base + col < it.rend;
        int cls = -1;
        if (valid)
            cls = build_mixed_record<true>(A, K, w, list[base + col], sRec[warp][lane].f,
                                           pl.exact_u != 0);
        __syncwarp();
        const unsigned int mv = __ballot_sync(0xffffffffu, cls == kRecVertex);
        const unsigned int mp = __ballot_sync(0xffffffffu, cls == kRecPair);
        const unsigned int ms = __ballot_sync(0xffffffffu, cls == kRecSeries || cls == kRecEdge);
        const unsigned int mser = __ballot_sync(0xffffffffu, cls == kRecSeries);
        if (row_ok)
            for (int ii = 0; ii < lpr; ++ii) {
                const int i = row * lpr + ii;
                if ((mv >> i) & 1u)
                    vertex_form_lane<S>(sRec[warp][i].f, fm0, fm0sq, eps_lane, PR, PI);
                else if ((mp >> i) & 1u)
                    vertex_form_lane<S, true>(sRec[warp][i].f, fm0, fm0sq, eps_lane, PR, PI,
                                              K.kap_step, d);
                else if ((ms >> i) & 1u)
                    series_edge_lane<S>(sRec[warp][i].f, (mser >> i) & 1u, fm0, d, w.turn, K, PR, PI);
            }
        // Kahan-compensated accumulation, every 32 facets
        held += lpr;
        if (held + lpr > 32 || base + lpr >= it.rend) {
#pragma unroll
            for (int k = 0; k < S2; ++k) {
                kahan_pair(sAcc[warp][0][k][lane], sAcc[warp][2][k][lane], PR[k]);
                kahan_pair(sAcc[warp][1][k][lane], sAcc[warp][3][k][lane], PI[k]);
                PR[k] = PI[k] = zero2;
            }
            held = 0;
        }
        __syncwarp();
    }
    float4 *dst = b.partial + (int64_t)item * (S2 * 32) + lane;
#pragma unroll
    for (int k = 0; k < S2; ++k) {
        float r0, r1, i0, i1;
        upk2(sAcc[warp][0][k][lane], r0, r1);
        upk2(sAcc[warp][1][k][lane], i0, i1);
        dst[k * 32] = make_float4(r0, i0, r1, i1);
    }
    __syncwarp();
    }
}

// Coarse values of an (instance, channel): the items' partial sums, Kahan-
// compensated.  A thread takes a slice of the chunks of one value (in memory
// order, so that a warp's loads are one run), the slices are added in order.
// What bounds it is the chain of loads, so a slice is 4 chunks or more of up
// to eight: a sedan's 188 chunks one after the other, a value a thread, took
// 28 us, this takes 8.
constexpr int kRedThreads = 256;
constexpr int kRedSlices = 8;

__device__ __forceinline__ void kahan_add(float v, float &sum, float &c)
{
    const float y = v - c, t = sum + y;
    c = (t - sum) - y;
    sum = t;
}

__global__ void __launch_bounds__(kRedThreads) band_reduce_kernel(BandArgs b)
{
    __shared__ float4 s_part[kRedThreads];                // sums and their compensation
    const int v = blockIdx.x;
    const int cnt = b.vcnt[v];
    if (cnt == 0) return;
    const BandPlan &pl = b.plan[v / b.O];
    const BandM lay = b.sh.m[pl.im];
    const int rows = b.sh.n[pl.in].nj * lay.nseg;
    const int rpw = 32 / lay.lpr, groups = band_groups(b.sh, pl);
    const int chunks = (b.item0[v + 1] - b.item0[v]) / groups;
    const float2 *part = reinterpret_cast<const float2 *>(b.partial) +
                         (int64_t)b.item0[v] * (kBandS * 32);
    float2 *out = b.coarse + b.coff[v];
    const int lane_s = kBandS * lay.lpr;               // samples of a (node, segment) row
    int slices = 1;
    while (slices < kRedSlices && chunks >= 8 * slices) slices *= 2;
    const int per = kRedThreads / slices;              // values at once: a divisor of 512
    const int t = threadIdx.x & (per - 1), slice = threadIdx.x / per;
    const int j0 = chunks * slice / slices, j1 = chunks * (slice + 1) / slices;
    const int64_t step = (int64_t)groups * (kBandS * 32);
    const int tiles = kBandS * 32 / per;               // of a group
    for (int tile = blockIdx.y; tile < groups * tiles; tile += gridDim.y) {
        // position: [group][pair][lane][half]
        const int grp = tile / tiles, at = (tile - grp * tiles) * per + t;
        const int lane = (at & 63) >> 1, row = lane / lay.lpr;
        const int rs = grp * rpw + row;
        const int s = (lane - row * lay.lpr) * 16 + (at >> 6) * 2 + (at & 1);
        float sr = 0.f, si = 0.f, cr = 0.f, ci = 0.f;
        const float2 *src = part + (int64_t)grp * (kBandS * 32) + at;
#pragma unroll 4
        for (int j = j0; j < j1; ++j) {
            const float2 p = src[j * step];
            kahan_add(p.x, sr, cr);
            kahan_add(p.y, si, ci);
        }
        if (slices > 1) {
            s_part[threadIdx.x] = make_float4(sr, si, cr, ci);
            __syncthreads();
        }
        if (slice == 0 && row < rpw && rs < rows) {
            for (int k = 1; k < slices; ++k) {
                const float4 p = s_part[k * per + t];
                kahan_add(p.x, sr, cr);
                kahan_add(p.y, si, ci);
                cr += p.z;
                ci += p.w;
            }
            if (pl.rotate) {                               // the steps' eighth turns back
                const int k = s & 7;
                const float h = 0.70710678f;
                const float c = k == 0 ? 1.f : k == 4 ? -1.f : (k & 3) == 2 ? 0.f : (k == 1 || k == 7) ? h : -h;
                const float z = (k & 3) == 0 ? 0.f : k == 2 ? 1.f : k == 6 ? -1.f : k < 4 ? h : -h;
                const float x = fmaf(c, sr, z * si);
                si = fmaf(c, si, -z * sr);
                sr = x;
            }
            out[(int64_t)rs * lane_s + s] = make_float2(sr, si);
        }
        if (slices > 1) __syncthreads();
    }
}

// -------------------------------------------------------------------------
// expansion: each block writes kExpN chirps x kExpM samples of one channel
// of one scene: per instance, the chirps' interpolation of the coarse samples
// it needs into shared memory, then the samples' taps and the reference
// phase; the instances in order.  The taps' weights lie sample by sample
// (sample by tap, a warp's load was 20 cache lines), and a multiprocessor holds
// four blocks, some spills for 64 registers (two of 92: latency-bound, 24 % of
// the warps): a batch of eight scenes takes 132 us against 178.
// -------------------------------------------------------------------------
constexpr int kExpN = 8;
constexpr int kExpM = 256;

__global__ void __launch_bounds__(kExpM, 4)
band_expand_kernel(BandArgs b, MixConsts K, void *__restrict__ out, int out_c64)
{
    extern __shared__ float2 sT[];                     // [kExpN][width]
    __shared__ float sW[kExpN][128];
    const int N = b.sh.N, M = b.sh.M;
    const int mt = (M + kExpM - 1) / kExpM;
    const int n0 = (blockIdx.x / mt) * kExpN, m0 = (blockIdx.x % mt) * kExpM;
    const int nn = min(kExpN, N - n0);
    const int o = blockIdx.y, sc = blockIdx.z;
    const int tid = threadIdx.x;
    const int m = m0 + tid;
    const bool ok = m < M;
    const int m_last = min(M, m0 + kExpM) - 1;
    const float fm = (float)m;
    float ar[kExpN], ai[kExpN];
#pragma unroll
    for (int k = 0; k < kExpN; ++k) ar[k] = ai[k] = 0.f;
    for (int i = b.scene_inst[sc]; i < b.scene_inst[sc + 1]; ++i) {
        const int v = i * b.O + o;
        if (b.vcnt[v] == 0) continue;
        const BandPlan &pl = b.plan[i];
        const BandM lay = b.sh.m[pl.im];
        const BandN ch = b.sh.n[pl.in];
        const float2 *C = b.coarse + b.coff[v];
        const int *base = b.base + (int64_t)pl.im * M;
        const int s0 = pl.im ? base[m0] : m0;
        const int width = pl.im ? base[m_last] + kBandTaps - s0 : m_last + 1 - m0;
        __syncthreads();                               // sT and sW of the last instance
        if (pl.in > 1) {
            for (int e = tid; e < nn * ch.nj; e += kExpM)
                sW[e / ch.nj][e % ch.nj] = b.wn[ch.w0 + (int64_t)n0 * ch.nj + e];
            __syncthreads();
            for (int s = tid; s < width; s += kExpM) {
                float tr[kExpN], ti[kExpN];
#pragma unroll
                for (int k = 0; k < kExpN; ++k) tr[k] = ti[k] = 0.f;
#pragma unroll 4
                for (int j = 0; j < ch.nj; ++j) {
                    const float2 c = C[(int64_t)j * lay.Mi + s0 + s];
#pragma unroll
                    for (int k = 0; k < kExpN; ++k) {
                        tr[k] = fmaf(sW[k][j], c.x, tr[k]);
                        ti[k] = fmaf(sW[k][j], c.y, ti[k]);
                    }
                }
#pragma unroll
                for (int k = 0; k < kExpN; ++k) sT[k * width + s] = make_float2(tr[k], ti[k]);
            }
        } else {
            for (int s = tid; s < width; s += kExpM)
                for (int k = 0; k < nn; ++k)
                    sT[k * width + s] = C[(int64_t)(pl.in ? 0 : n0 + k) * lay.Mi + s0 + s];
        }
        __syncthreads();
        if (!ok) continue;
        float xr[kExpN], xi[kExpN];
        if (pl.im) {
            const float *wm = b.wm + (int64_t)pl.im * kBandTaps * M + m;
            const int off = base[m] - s0;
#pragma unroll
            for (int k = 0; k < kExpN; ++k) xr[k] = xi[k] = 0.f;
#pragma unroll 4
            for (int e = 0; e < kBandTaps; ++e) {
                const float w = wm[(int64_t)e * M];
#pragma unroll
                for (int k = 0; k < kExpN; ++k) {
                    const float2 c = sT[k * width + off + e];
                    xr[k] = fmaf(w, c.x, xr[k]);
                    xi[k] = fmaf(w, c.y, xi[k]);
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < kExpN; ++k) {
                const float2 c = k < nn ? sT[k * width + tid] : make_float2(0.f, 0.f);
                xr[k] = c.x;
                xi[k] = c.y;
            }
        }
        if (pl.rotate) {
            const float4 *ref = b.ref + (int64_t)v * N + n0;
#pragma unroll
            for (int k = 0; k < kExpN; ++k) {
                if (k >= nn) break;
                const float4 r = ref[k];
                const float th = red1(r.y * fm) + fmaf(r.z, fm, fmaf(r.w, fm * fm, r.x));
                float s_, c_;
                sincospif(2.f * red1(th), &s_, &c_);
                ar[k] += fmaf(c_, xr[k], -s_ * xi[k]);
                ai[k] += fmaf(c_, xi[k], s_ * xr[k]);
            }
        } else {
#pragma unroll
            for (int k = 0; k < kExpN; ++k) {
                ar[k] += xr[k];
                ai[k] += xi[k];
            }
        }
    }
    if (!ok) return;
    const float kp = fmaf(fm, K.kap_step, 1.f);
    const float scl = K.out_scale / (kp * kp);
    const int64_t row = (((int64_t)sc * b.O + o) * N + n0) * M + m;
#pragma unroll
    for (int k = 0; k < kExpN; ++k) {
        if (k >= nn) break;
        const float re = ar[k] * scl, im = ai[k] * scl;
        if (out_c64) reinterpret_cast<float2 *>(out)[row + (int64_t)k * M] = make_float2(re, im);
        else reinterpret_cast<double2 *>(out)[row + (int64_t)k * M] = make_double2(re, im);
    }
}

// the forms of every (facet, channel, chirp) record of the frame (stats)
__global__ void __launch_bounds__(128) count_records_kernel(SynthArgs A, MixConsts K)
{
    const int n = blockIdx.x, vrow = blockIdx.y;
    const int o = vrow % A.rd.O, P = A.rd.P, Q = A.rd.Q, tx = o / Q, rx = o % Q;
    const int64_t F = A.F;
    const int slot = n * A.rd.slots + (A.rd.tdm ? tx : 0);
    MixRow w;
    w.sl = slot;
    w.tau_s = (float)slot - K.s_mid;
    w.tn = (float)slot * K.tc;
    w.kin_t = A.kin + (int64_t)tx * F * kKinRow;
    w.kin_r = A.kin + (int64_t)(P + rx) * F * kKinRow;
    w.quad_t = A.kquad + (int64_t)tx * F * kKinQuadWords;
    w.quad_r = A.kquad + (int64_t)(P + rx) * F * kKinQuadWords;
    w.ant_t = tx;
    w.ant_r = P + rx;
    for (int r = 0; r < 3; ++r) {
        w.ptx[r] = K.ant[tx][r];
        w.prx[r] = K.ant[P + rx][r];
    }
    const int32_t *list = A.vis_idx + (int64_t)o * F + (A.vstart ? A.vstart[vrow] : 0);
    const int cnt = A.vcnt[vrow];
    int nf[3] = {0, 0, 0};
    for (int k = threadIdx.x; k < cnt; k += blockDim.x) {
        float R[24];
        const int cls = build_mixed_record(A, K, w, list[k], R);
        nf[0] += cls == kRecVertex;
        nf[1] += cls == kRecSeries;
        nf[2] += cls == kRecEdge;
    }
    for (int f = 0; f < 3; ++f) {
        const int sum = __reduce_add_sync(0xffffffffu, nf[f]);
        if ((threadIdx.x & 31) == 0 && sum) atomicAdd(A.counters + f, (unsigned long long)sum);
    }
}

}  // namespace

void launch_band_tables(const BandShape &sh, float *nodes, float *wn, int *base, float *wm,
                        cudaStream_t s)
{
    static const BandChol chol = [] {
        constexpr int T = kBandTaps;
        const double w2 = 1.0 / kBandOver;
        BandChol c{};
        double L[T][T] = {};
        for (int i = 0; i < T; ++i)
            for (int j = 0; j <= i; ++j) {
                double a = w2 * band_sinc(w2 * (i - j)) + (i == j ? 1e-12 : 0.0);
                for (int k = 0; k < j; ++k) a -= L[i][k] * L[j][k];
                L[i][j] = i == j ? sqrt(a) : a / L[j][j];
                c.L[i * (i + 1) / 2 + j] = i == j ? 1.0 / L[i][j] : L[i][j];
            }
        return c;
    }();
    band_table_kernel<<<dim3((unsigned int)(sh.n_n + sh.n_m), kTabRows), 32, 0, s>>>(sh, chol, nodes,
                                                                                    wn, base, wm);
}

void launch_band_plan(const BandArgs &b, const SynthArgs &a, cudaStream_t s)
{
    const MixConsts K = mix_consts(a.rd);
    band_plan_kernel<<<b.I, 32, 0, s>>>(b, a.rd, K, a.vel32, a.fac);
    dim3 g((unsigned int)((2 * b.sh.N + 127) / 128), (unsigned int)(b.I * b.O));
    band_ref_kernel<<<g, 128, 0, s>>>(b, a.rd, a.vel64);
}

void launch_synth_band(const BandArgs &b, const SynthArgs &a, cudaStream_t s)
{
    const MixConsts K = mix_consts(a.rd);
    const int V = b.I * b.O;
    if (V <= kBandSmall) {
        band_small_kernel<<<1, 1024, 0, s>>>(b, a.vis_idx, a.vis_cnt, a.F);
    } else {
        band_lists_kernel<<<(V + 3) / 4, 256, 0, s>>>(b, a.vis_idx, a.vis_cnt, a.F);
        band_items_kernel<<<1, 1024, 0, s>>>(b);
        band_fill_kernel<<<V, 64, 0, s>>>(b);
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t need = (b.max_items + kBandWarps - 1) / kBandWarps;
    const int grid = (int)std::min<int64_t>(need, (int64_t)kBandBlocks * sms);
    synth_band_kernel<<<grid, kBandWarps * 32, 0, s>>>(a, K, b);
    band_reduce_kernel<<<dim3((unsigned int)V, (unsigned int)std::max(8, std::min(32, 2048 / V))),
                         kRedThreads, 0, s>>>(b);
    const int mt = (b.sh.M + kExpM - 1) / kExpM, nt = (b.sh.N + kExpN - 1) / kExpN;
    const size_t sm = (size_t)kExpN * (kExpM + kBandTaps) * sizeof(float2);
    band_expand_kernel<<<dim3((unsigned int)(mt * nt), (unsigned int)b.O, (unsigned int)b.B), kExpM,
                         sm, s>>>(b, K, a.out, a.out_c64);
}

int launch_synth_band_count(const BandArgs &b) { return b.I * b.O <= kBandSmall ? 4 : 6; }

void launch_count_records(const SynthArgs &a, cudaStream_t s)
{
    const MixConsts K = mix_consts(a.rd);
    count_records_kernel<<<dim3((unsigned int)a.rd.N, (unsigned int)a.VO), 128, 0, s>>>(a, K);
}

}  // namespace bart
