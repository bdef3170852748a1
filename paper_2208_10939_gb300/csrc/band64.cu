// Band-limited FP64 echo synthesis (see band64.cuh): tables, plan, reference
// phases, work items, node sums, interpolation.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "band64.cuh"
#include "band_plan.cuh"
#include "record_fp64.cuh"

namespace bart {

// -------------------------------------------------------------------------
// layouts (host)
// -------------------------------------------------------------------------
void band64_shape(int N, int M, Band64Shape &sh)
{
    // nodes and the phase they carry: 4 sum_{k >= K-1} |J_k(a)| = 1e-13
    static const struct { int K; float a; } chirps[] = {
        {8, 0.077f}, {10, 0.255f}, {12, 0.569f}, {14, 1.01f}, {16, 1.59f}, {20, 3.05f},
        {24, 4.86f}, {28, 6.92f}, {32, 9.19f}, {40, 14.1f}, {48, 19.6f}, {64, 31.3f},
        {80, 43.8f}, {128, 83.7f}};
    static const struct { int K; float a; } samples[] = {
        {32, 9.19f}, {48, 19.6f}, {64, 31.3f}, {80, 43.8f}, {96, 56.8f}, {128, 83.7f}, {160, 111.f}, {192, 139.f},
        {224, 168.f}, {256, 197.f}, {320, 256.f}, {384, 316.f}, {448, 376.f}, {512, 437.f},
        {640, 558.f}, {768, 681.f}};
    sh = Band64Shape{};
    sh.N = N;
    sh.M = M;
    int x = 0;
    int64_t w = 0;
    auto chirp = [&](int K, float a, bool table) {
        const int l = sh.n_n++;
        sh.kn[l] = K;
        sh.an[l] = a;
        sh.xn[l] = x;
        sh.wn[l] = w;
        x += K;
        if (table) w += (int64_t)K * N;
    };
    chirp(N, 1e30f, false);
    chirp(1, 0.f, false);
    for (auto &c : chirps)
        if (5 * c.K <= 4 * N && sh.n_n < kB64N) chirp(c.K, c.a, true);
    x = 0;
    w = 0;
    auto sample = [&](int K, float a, bool table) {
        const int l = sh.n_m++;
        sh.km[l] = K;
        sh.am[l] = a;
        sh.xm[l] = x;
        sh.wm[l] = w;
        x += K;
        if (table) w += (int64_t)K * M;
    };
    sample(M, 1e30f, false);
    for (auto &c : samples)
        if (5 * c.K <= 4 * M && sh.n_m < kB64M) sample(c.K, c.a, true);
}

Band64Sizes band64_sizes(const Band64Shape &sh)
{
    Band64Sizes z{};
    for (int l = 0; l < sh.n_n; ++l) {
        z.xn += sh.kn[l];
        if (l > 1) z.wn += (int64_t)sh.kn[l] * sh.N;
    }
    for (int l = 0; l < sh.n_m; ++l) {
        z.xm += sh.km[l];
        if (l > 0) z.wm += (int64_t)sh.km[l] * sh.M;
    }
    return z;
}

void band64_tables(double *tab, Band64Args &b)
{
    const Band64Sizes z = band64_sizes(b.sh);
    b.turn = reinterpret_cast<double2 *>(tab);
    b.xn = tab + 512;
    b.xm = b.xn + z.xn;
    b.wn = b.xm + z.xm;
    b.wm = b.wn + z.wn;
}

namespace {

// -------------------------------------------------------------------------
// tables: the Chebyshev nodes of [0, len - 1] and their barycentric weights at
// the whole positions (a warp a position); block (0, 0) also the sines
// -------------------------------------------------------------------------
__device__ __forceinline__ double cheb_node(int j, int K, int len)
{
    return 0.5 * (len - 1) * (1.0 - cospi((j + 0.5) / K));
}

__global__ void __launch_bounds__(256) band64_table_kernel(Band64Shape sh, double *__restrict__ xn,
                                                           double *__restrict__ xm,
                                                           double *__restrict__ wn,
                                                           double *__restrict__ wm,
                                                           double2 *__restrict__ turn)
{
    const bool chirps = (int)blockIdx.x < sh.n_n;
    const int l = chirps ? blockIdx.x : blockIdx.x - sh.n_n;
    const int K = chirps ? sh.kn[l] : sh.km[l], len = chirps ? sh.N : sh.M;
    const bool whole = l == 0 || (chirps && l == 1);
    double *x = chirps ? xn + sh.xn[l] : xm + sh.xm[l];
    if (blockIdx.x == 0 && blockIdx.y == 0) {
        double s, c;
        sincospi(threadIdx.x / 128.0, &s, &c);
        turn[threadIdx.x] = make_double2(c, s);
    }
    if (blockIdx.y == 0)
        for (int j = threadIdx.x; j < K; j += blockDim.x) x[j] = whole ? j : cheb_node(j, K, len);
    if (whole) return;
    const int lane = threadIdx.x & 31;
    for (int n = blockIdx.y * 8 + (threadIdx.x >> 5); n < len; n += gridDim.y * 8) {
        double sum = 0.0;
        int hit = -1;
        for (int j = lane; j < K; j += 32) {
            const double d = n - cheb_node(j, K, len);
            if (d == 0.0) hit = j;
            else sum += (j & 1 ? -1.0 : 1.0) * sinpi((j + 0.5) / K) / d;
        }
        for (int off = 16; off > 0; off >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, off);
            hit = max(hit, __shfl_xor_sync(0xffffffffu, hit, off));
        }
        for (int j = lane; j < K; j += 32) {
            const double d = n - cheb_node(j, K, len);
            const double v = hit >= 0 ? (j == hit ? 1.0 : 0.0)
                                      : (j & 1 ? -1.0 : 1.0) * sinpi((j + 0.5) / K) / (d * sum);
            if (chirps) wn[sh.wn[l] + (int64_t)n * K + j] = v;
            else wm[sh.wm[l] + (int64_t)j * len + n] = v;
        }
    }
}

// Cells of an instance of nf facets: each at least 256, since a cell's
// interpolation costs about as much as the direct sum of one lit facet in it.
// A 5k-facet car on 12 channels of 32 x 256: a frame of 2.74 ms with one cell,
// 1.89 with four, and no less with eight (sums 1.52 and 1.46, interpolation 0.13
// and 0.21).
__device__ __forceinline__ int band64_cells(const Band64Args &b, int64_t nf)
{
    int n = 1;
    while (2 * n <= b.cells && nf >= 512 * (int64_t)n) n *= 2;
    return n;
}

// each facet's cell (by its centroid, the box halved along its longest sides)
// and the cells' boxes
__global__ void __launch_bounds__(128)
band64_cell_kernel(Band64Args b, const FacetRec *__restrict__ fac, int64_t F)
{
    const int64_t k = (int64_t)blockIdx.x * 128 + threadIdx.x;
    int body = -1;
    unsigned int bx[7] = {0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (k < F) {
        const FacetRec f = fac[k];
        const int n = band64_cells(b, b.ioff[f.inst + 1] - b.ioff[f.inst]);
        float lo[3], h[3];
        int cut[3] = {1, 1, 1}, at = 0;
        for (int r = 0; r < 3; ++r) {
            lo[r] = ord_f(~b.box[8 * f.inst + r]);
            h[r] = ord_f(b.box[8 * f.inst + 3 + r]) - lo[r];
        }
        for (int m = 1; m < n; m *= 2) {
            int r = 0;
            for (int q = 1; q < 3; ++q)
                if (h[q] * cut[r] > h[r] * cut[q]) r = q;
            cut[r] *= 2;
        }
        for (int r = 0; r < 3; ++r) {
            const float x = h[r] > 0.f ? (f.c[r] - lo[r]) / h[r] * (float)cut[r] : 0.f;
            at = at * cut[r] + min(cut[r] - 1, max(0, (int)x));
        }
        body = f.inst * b.cells + at;
        b.cell[k] = (uint8_t)at;
        float rad2 = 0.f;
        for (int r = 0; r < 3; ++r) {
            const float a0 = f.dv[r], a1 = f.dv[3 + r], a2 = f.dv[6 + r];
            const float pad = 1e-6f * fabsf(f.c[r]);            // the FP32 centroid's rounding
            bx[r] = ~ord_u(f.c[r] + fminf(fminf(a0, a1), a2) - pad);
            bx[3 + r] = ord_u(f.c[r] + fmaxf(fmaxf(a0, a1), a2) + pad);
        }
        for (int v = 0; v < 3; ++v)
            rad2 = fmaxf(rad2, f.dv[3 * v] * f.dv[3 * v] + f.dv[3 * v + 1] * f.dv[3 * v + 1] +
                                   f.dv[3 * v + 2] * f.dv[3 * v + 2]);
        bx[6] = ord_u(rad2);
    }
    const int b0 = __shfl_sync(0xffffffffu, body, 0);
    if (__all_sync(0xffffffffu, body == b0)) {
        for (int r = 0; r < 7; ++r) {
            const unsigned int m = __reduce_max_sync(0xffffffffu, bx[r]);
            if ((threadIdx.x & 31) == 0 && b0 >= 0) atomicMax(b.cbox + 8 * (int64_t)b0 + r, m);
        }
    } else if (body >= 0) {
        for (int r = 0; r < 7; ++r) atomicMax(b.cbox + 8 * (int64_t)body + r, bx[r]);
    }
}

// -------------------------------------------------------------------------
// plan and reference phases
// -------------------------------------------------------------------------
__global__ void band64_plan_kernel(Band64Args b, RadarDev rd, MixConsts K,
                                   const float *__restrict__ vel32, const FacetRec *__restrict__ fac)
{
    const int body = blockIdx.x, i = body / b.cells;
    const BandBounds q = band_bounds(b.cells > 1 ? b.cbox : b.box, body, i, rd, K, vel32);
    if (threadIdx.x != 0) return;
    Band64Plan pl;
    for (int r = 0; r < 3; ++r) pl.c[r] = q.c[r];
    pl.in = pl.im = 0;
    pl.rotate = q.ok;
    const float span = 3.1415927f * q.beta * (float)(b.sh.M - 1);
    if (q.ok)
        for (int l = 1; l < b.sh.n_m && pl.im == 0; ++l)
            if (span <= b.sh.am[l]) pl.im = l;
    // a facet lit from both sides has a kink where its obliquity changes sign:
    // every chirp is kept
    const bool smooth = b.ioff[i] < b.ioff[i + 1] && !fac[b.ioff[i]].two_sided;
    if (q.speed == 0.f) {
        pl.in = 1;
    } else if (q.ok && smooth) {
        for (int l = 2; l < b.sh.n_n && pl.in == 0; ++l)
            if (q.turn <= b.sh.an[l]) pl.in = l;
    }
    b.plan[body] = pl;
}

__device__ __forceinline__ double two_sum(double a, double b, double &e)
{
    const double s = a + b, t = s - a;
    e = (a - (s - t)) + (b - t);
    return s;
}

// The reference phase of (instance, channel) in a chirp that starts at tn, as
// a quadratic in the time from the middle of its samples, cycles: the box
// centre's path, its constant in double-double (its rounding is the whole
// instance's), reduced mod 1.
__device__ __forceinline__ double4 band64_ref(const RadarDev &rd, const float *c,
                                              const double *__restrict__ v, int p, int q, double tn)
{
    const double tc = 0.5 * (rd.M - 1) / rd.fs, t = rd.intra ? tn + tc : tn;
    const double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    double Lh = 0.0, Ll = 0.0, L1 = 0.0, L2 = 0.0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const double *pa = rd.ant[e == 0 ? p : rd.P + q];
        double qh = 0.0, ql = 0.0, sv = 0.0, er;
        for (int r = 0; r < 3; ++r) {
            double sl;
            const double s = two_sum(pa[r] - (double)c[r], -v[r] * t, sl);
            const double pr = s * s;
            ql += fma(s, s, -pr) + 2.0 * s * sl;
            qh = two_sum(qh, pr, er);
            ql += er;
            sv += s * v[r];
        }
        const double R = sqrt(qh);
        const double lo = 0.5 * (fma(-R, R, qh) + ql) / R;
        const double rr = -sv / R;
        Lh = two_sum(Lh, R, er);
        Ll += er + lo;
        L1 += rr;
        L2 += 0.5 * (v2 - rr * rr) / R;
    }
    if (!rd.intra) L1 = L2 = 0.0;
    const double F = (rd.f0 + rd.slope * tc) / kC0, mc = rd.slope / kC0;
    const double m2 = rd.slope / (2.0 * kC0 * kC0);
    const double ph = F * Lh, phe = fma(F, Lh, -ph);
    const double p0 = (ph - rint(ph)) + (phe + F * Ll) - m2 * Lh * Lh;
    return make_double4(p0 - rint(p0), F * L1 + mc * Lh - 2.0 * m2 * Lh * L1,
                        F * L2 + mc * L1 - m2 * (L1 * L1 + 2.0 * Lh * L2), 0.0);
}

__device__ __forceinline__ double chirp_start(const RadarDev &rd, double n, int tx)
{
    return (n * rd.slots + (rd.tdm ? tx : 0)) * rd.Tc;
}

__global__ void __launch_bounds__(128)
band64_ref_kernel(Band64Args b, RadarDev rd, const double *__restrict__ vel64)
{
    const int v = blockIdx.y, i = v / b.O, o = v % b.O;
    const Band64Plan pl = b.plan[i];
    const int N = b.sh.N, nj = b.sh.kn[pl.in];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const bool node = e >= N;                     // chirps first, then nodes
    const int k = node ? e - N : e;
    if (k >= (node ? nj : N)) return;
    double4 r = make_double4(0.0, 0.0, 0.0, 0.0);
    if (pl.rotate) {
        const int p = o / rd.Q, q = o % rd.Q;
        const double n = node ? b.xn[b.sh.xn[pl.in] + k] : (double)k;
        r = band64_ref(rd, pl.c, vel64 + 3 * (i / b.cells), p, q, chirp_start(rd, n, p));
    }
    (node ? b.refn : b.ref)[(int64_t)v * N + k] = r;
}

// -------------------------------------------------------------------------
// list parts and work items
// -------------------------------------------------------------------------
__global__ void band64_lists_kernel(Band64Args b, const int32_t *__restrict__ vis_idx,
                                    const int32_t *__restrict__ vis_cnt, int64_t F)
{
    const int lane = threadIdx.x & 31;
    const int v = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (v >= b.I * b.O) return;
    const int i = v / b.O, o = v % b.O;          // one cell an instance
    const int32_t *list = vis_idx + (int64_t)o * F;
    const int lo = warp_lower_bound(list, vis_cnt[o], b.ioff[i], lane);
    const int n = warp_lower_bound(list + lo, vis_cnt[o] - lo, b.ioff[i + 1], lane);
    if (lane == 0) {
        b.vstart[v] = lo;
        b.vcnt[v] = n;
    }
}

// the same with cells: a block per (instance, channel) puts its part of the
// list in cell order, each cell's facets in theirs
__global__ void __launch_bounds__(256)
band64_cell_lists_kernel(Band64Args b, const int32_t *__restrict__ vis_idx,
                         const int32_t *__restrict__ vis_cnt, int64_t F)
{
    __shared__ int s_lo, s_n, s_cnt[kB64Cells], s_w[8][kB64Cells], s_run[kB64Cells];
    const int i = blockIdx.x / b.O, o = blockIdx.x % b.O;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int32_t *list = vis_idx + (int64_t)o * F;
    if (warp == 0) {
        const int lo = warp_lower_bound(list, vis_cnt[o], b.ioff[i], lane);
        const int n = warp_lower_bound(list + lo, vis_cnt[o] - lo, b.ioff[i + 1], lane);
        if (lane == 0) {
            s_lo = lo;
            s_n = n;
        }
    }
    if (t < kB64Cells) s_cnt[t] = 0;
    __syncthreads();
    const int lo = s_lo, n = s_n;
    for (int e = t; e < n; e += 256) atomicAdd(&s_cnt[b.cell[list[lo + e]]], 1);
    __syncthreads();
    if (t == 0) {
        int at = lo;
        for (int c = 0; c < kB64Cells; ++c) {
            const int v = (i * b.cells + c) * b.O + o;
            b.vstart[v] = s_run[c] = at;
            b.vcnt[v] = s_cnt[c];
            at += s_cnt[c];
        }
    }
    __syncthreads();
    int32_t *out = b.list + (int64_t)o * F;
    for (int e0 = 0; e0 < n; e0 += 256) {
        const int e = e0 + t;
        const int32_t k = e < n ? list[lo + e] : 0;
        const int c = e < n ? (int)b.cell[k] : -1;
        int rank = 0;
        for (int q = 0; q < kB64Cells; ++q) {
            const unsigned int m = __ballot_sync(0xffffffffu, c == q);
            if (c == q) rank = __popc(m & ((1u << lane) - 1u));
            if (lane == 0) s_w[warp][q] = __popc(m);
        }
        __syncthreads();
        if (c >= 0) {
            int at = s_run[c] + rank;
            for (int w = 0; w < warp; ++w) at += s_w[w][c];
            out[at] = k;
        }
        __syncthreads();
        if (t < kB64Cells)
            for (int w = 0; w < 8; ++w) s_run[t] += s_w[w][t];
        __syncthreads();
    }
}

constexpr int kSeg = 64;             // nodes of a work item

// parts of an (instance, channel)'s facets, by its own list and layout alone:
// the sums do not depend on what else is in the call
__device__ __forceinline__ int band64_chunks(const Band64Args &b, const Band64Plan &pl, int cnt)
{
    const Band64Shape &sh = b.sh;
    const int64_t room = (int64_t)b.room * sh.N * sh.M / ((int64_t)sh.kn[pl.in] * sh.km[pl.im]);
    return (int)max((int64_t)1, min(room, (int64_t)min(kB64Chunks, (cnt + 127) / 128)));
}

__device__ __forceinline__ int band64_item_count(const Band64Args &b, const Band64Plan &pl, int cnt)
{
    return cnt == 0 ? 0 : b.sh.kn[pl.in] * ((b.sh.km[pl.im] + kSeg - 1) / kSeg) *
                              band64_chunks(b, pl, cnt);
}

// the adjoint's items: a chirp node and kAdjFacets facets each
constexpr int kAdjFacets = 128;

__device__ __forceinline__ int band64_adjoint_count(const Band64Shape &sh, const Band64Plan &pl,
                                                    int cnt)
{
    return sh.kn[pl.in] * ((cnt + kAdjFacets - 1) / kAdjFacets);
}

// item prefix (one block)
__global__ void __launch_bounds__(1024) band64_items_kernel(Band64Args b, int adjoint)
{
    __shared__ int s_w[32], s_run;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int V = b.I * b.O;
    if (t == 0) {
        s_run = 0;
        *b.ticket = 0;
    }
    __syncthreads();
    for (int v0 = 0; v0 < V; v0 += 1024) {
        const int v = v0 + t;
        const int items = v >= V ? 0
                          : adjoint ? band64_adjoint_count(b.sh, b.plan[v / b.O], b.vcnt[v])
                                    : band64_item_count(b, b.plan[v / b.O], b.vcnt[v]);
        int x = items;
        for (int off = 1; off < 32; off <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += u;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        int before = s_run, all = 0;
        for (int k = 0; k < 32; ++k) {
            if (k < warp) before += s_w[k];
            all += s_w[k];
        }
        if (v < V) b.item0[v] = before + x - items;
        __syncthreads();
        if (t == 0) s_run += all;
        __syncthreads();
    }
    if (t == 0) b.item0[V] = s_run;
}

// -------------------------------------------------------------------------
// phasors and records
// -------------------------------------------------------------------------

// exp(j 2 pi x): the nearest 256th of a turn from the table, the rest (at most
// 0.0123 rad) by the sine's and cosine's own series (next terms 8e-18, 1e-20).
// 14 FP64 operations.
__device__ __forceinline__ void turn_exp(double x, const double2 *turn, double &c, double &s)
{
    const double big = 6755399441055744.0;            // 1.5 2^52: rounds to whole numbers
    const double t = fma(x, 256.0, big);
    const double2 w = turn[__double2loint(t) & 255];
    const double r = fma(t - big, -1.0 / 256.0, x), r2 = r * r;
    const double p = 2.0 * kPi, p2 = p * p;
    const double es = r * fma(r2, fma(r2, p * p2 * p2 / 120.0, -p * p2 / 6.0), p);
    const double ec = fma(r2, fma(r2, fma(r2, -p2 * p2 * p2 / 720.0, p2 * p2 / 24.0), -p2 / 2.0), 1.0);
    c = fma(w.x, ec, -w.y * es);
    s = fma(w.x, es, w.y * ec);
}

__device__ __forceinline__ double frac1(double x)      // x - rint(x)
{
    const double big = 6755399441055744.0;
    return x - ((x + big) - big);
}

// path length over a chirp: sqrt(q(t)) of both legs as a quartic in the time
// from the middle of the samples where |q(t) / q(tc) - 1| stays below 1e-3
// (next term 7/256 1e-15), else evaluated as it stands
struct Rec64 {
    double L[5];                     // the quartic, or qt0 qt1 q2 qr0 qr1
    double d[16];
    int kind, flags;
    int quartic, pad;
};

struct Node64 {                      // a node's constants
    double t, tau, fmc, kp, rp;
};

__device__ __forceinline__ Node64 band64_node(const RadarDev &rd, double x, const double4 &ref)
{
    Node64 n;
    n.t = x / rd.fs;
    n.tau = (x - 0.5 * (rd.M - 1)) / rd.fs;
    const double fm = rd.f0 + rd.slope * n.t;
    n.fmc = fm / kC0;
    n.kp = fm / rd.f0;
    n.rp = frac1(fma(n.tau, fma(n.tau, ref.z, ref.y), ref.x));
    return n;
}

__device__ __forceinline__ void band64_record(const SynthArgs &A, int64_t k, double tn,
                                              const double *ptx, const double *prx, double k0,
                                              double kmax, Rec64 &R)
{
    const int inst = A.fac[k].inst;
    double tri[9], c0[3], rec[kRecEntries];
    for (int i = 0; i < 9; ++i) tri[i] = A.tri64[9 * k + i];
    for (int r = 0; r < 3; ++r) c0[r] = A.c64[3 * k + r];
    int flags = 0;
    R.kind = build_record<double>(tri, c0, A.vel64 + 3 * inst, tn, ptx, prx, (double)A.fac[k].rho,
                                  A.rd.intra, k0, kmax, kDelayFacet, nullptr, A.fac[k].two_sided,
                                  rec, &flags);
    R.flags = flags;
    for (int i = 0; i < 16; ++i) R.d[i] = rec[kRecD + i];
    const double h = 0.5 * (A.rd.M - 1) / A.rd.fs, q2 = rec[2];
    const double q1t = rec[1] + 2.0 * q2 * h, q1r = rec[4] + 2.0 * q2 * h;
    const double Qt = rec[0] + h * (rec[1] + h * q2), Qr = rec[3] + h * (rec[4] + h * q2);
    R.quartic = Qt > 0.0 && Qr > 0.0 && h * (fabs(q1t) + h * q2) < 1e-3 * Qt &&
                h * (fabs(q1r) + h * q2) < 1e-3 * Qr;
    if (!R.quartic) {
        for (int i = 0; i < 5; ++i) R.L[i] = rec[i];
        return;
    }
    // sqrt(Q + q1 tau + q2 tau^2) = sum l_k tau^k: 2 l0 l1 = q1, 2 l0 l2 + l1^2 = q2,
    // l0 l3 + l1 l2 = 0, 2 l0 l4 + 2 l1 l3 + l2^2 = 0
    const double st = sqrt(Qt), sr = sqrt(Qr), ht = 0.5 / st, hr = 0.5 / sr;
    const double t1 = q1t * ht, r1 = q1r * hr;
    const double t2 = (q2 - t1 * t1) * ht, r2 = (q2 - r1 * r1) * hr;
    const double t3 = -2.0 * t1 * t2 * ht, r3 = -2.0 * r1 * r2 * hr;
    R.L[0] = st + sr;
    R.L[1] = t1 + r1;
    R.L[2] = t2 + r2;
    R.L[3] = t3 + r3;
    R.L[4] = -(2.0 * t1 * t3 + t2 * t2) * ht - (2.0 * r1 * r3 + r2 * r2) * hr;
}

__device__ __forceinline__ double band64_path(const Rec64 &R, const Node64 &n)
{
    if (R.quartic)
        return fma(n.tau, fma(n.tau, fma(n.tau, fma(n.tau, R.L[4], R.L[3]), R.L[2]), R.L[1]), R.L[0]);
    return sqrt(R.L[0] + n.t * (R.L[1] + n.t * R.L[2])) + sqrt(R.L[3] + n.t * (R.L[4] + n.t * R.L[2]));
}

// the record's term at a node, its reference phase taken off, added to (re, im)
__device__ __forceinline__ void band64_eval(const Rec64 &R, const Node64 &n, double mu_2c2,
                                            const double2 *turn, double &re, double &im)
{
    const double L = band64_path(R, n);
    const double th = frac1(L * fma(-mu_2c2, L, n.fmc)) - n.rp;
    double c, s;
    if (R.kind == kRecVertex) {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            turn_exp(fma(-n.fmc, R.d[v], th), turn, c, s);
            re = fma(R.d[3 + v], c, re);
            im = fma(R.d[3 + v], s, im);
        }
    } else if (R.kind == kRecSeries) {
        turn_exp(fma(-n.fmc, R.d[0], th), turn, c, s);
        const double k2 = n.kp * n.kp;
        double a = R.d[8], bb = R.d[15];
#pragma unroll
        for (int q = 6; q >= 0; --q) a = fma(a, k2, R.d[1 + q]);
#pragma unroll
        for (int q = 5; q >= 0; --q) bb = fma(bb, k2, R.d[9 + q]);
        const double pr = a * k2, pi = bb * k2 * n.kp;
        re += c * pr - s * pi;
        im += c * pi + s * pr;
    } else {
        for (int e = 0; e < 3; ++e) {
            turn_exp(fma(-n.fmc, R.d[3 * e], th), turn, c, s);
            const double x = n.kp * R.d[3 * e + 1];
            double sn;
            if (R.flags & (1 << e)) {
                const double x2 = x * x;
                sn = 1.0 + x2 * (-1.0 / 6 + x2 * (1.0 / 120 + x2 * (-1.0 / 5040 +
                     x2 * (1.0 / 362880 + x2 * (-1.0 / 39916800)))));
            } else {
                sn = sin(x) / x;
            }
            const double coef = n.kp * R.d[3 * e + 2] * sn;
            re -= coef * s;
            im += coef * c;
        }
    }
}

// -------------------------------------------------------------------------
// node sums.  Work item = (instance, channel, chirp node, 64 sample nodes,
// part of the facets), handed out by a ticket: the FP64 pipe is shared by all
// blocks of a multiprocessor, so an equal count of items a multiprocessor is
// an equal load (48 nodes cost it what 64 do, but the interpolation less: 114 us
// against 127 on a 5k-facet car).  A warp takes a quarter of the part: a lane builds a
// facet's record, then the records go round with two nodes a lane; the four
// warps' sums are added in order.
// -------------------------------------------------------------------------
constexpr int kB64Warps = 4;

__device__ __forceinline__ int band64_find(const int32_t *__restrict__ item0, int V, int item)
{
    int lo = 0, hi = V - 1;                       // last v with item0[v] <= item
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (item0[mid] <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(kB64Warps * 32)
synth_band64_kernel(SynthArgs A, Band64Args b)
{
    __shared__ Rec64 s_rec[kB64Warps][32];
    __shared__ double2 s_turn[256];
    __shared__ double2 s_sum[kB64Warps - 1][kSeg];
    __shared__ int s_item;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s_turn[i] = b.turn[i];
    const RadarDev &rd = A.rd;
    const int V = b.I * b.O, total = b.item0[V];
    const double c = kC0;
    const double k0 = 2.0 * kPi * rd.f0 / c;
    const double kmax = 2.0 * kPi * (rd.f0 + rd.slope * (rd.M - 1) / rd.fs) / c;
    const double mu_2c2 = rd.slope / (2.0 * c * c);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(b.ticket, 1);
        __syncthreads();
        if (s_item >= total) return;
        const int v = band64_find(b.item0, V, s_item);
        const int i = v / b.O, o = v % b.O, cnt = b.vcnt[v];
        const Band64Plan pl = b.plan[i];
        const int nj = b.sh.kn[pl.in], Km = b.sh.km[pl.im], segs = (Km + kSeg - 1) / kSeg;
        const int C = band64_chunks(b, pl, cnt);
        int at = s_item - b.item0[v];
        const int chunk = at % C;
        at /= C;
        const int seg = at % segs, j = at / segs;
        const int tx = o / rd.Q, rx = o % rd.Q;
        const double tn = chirp_start(rd, b.xn[b.sh.xn[pl.in] + j], tx);
        const double *ptx = rd.ant[tx], *prx = rd.ant[rd.P + rx];
        const double4 ref = b.refn[(int64_t)v * b.sh.N + j];
        const int s0 = seg * kSeg + lane;
        const bool ok0 = s0 < Km, ok1 = s0 + 32 < Km;      // Km is a multiple of 16
        const double *xm = b.xm + b.sh.xm[pl.im];
        const Node64 n0 = band64_node(rd, xm[ok0 ? s0 : 0], ref);
        const Node64 n1 = band64_node(rd, xm[ok1 ? s0 + 32 : 0], ref);
        double re0 = 0.0, im0 = 0.0, re1 = 0.0, im1 = 0.0;
        const int32_t *list = (b.cells > 1 ? b.list : A.vis_idx) + (int64_t)o * A.F + b.vstart[v];
        const int part = chunk * kB64Warps + warp;
        const int beg = (int)((int64_t)cnt * part / (C * kB64Warps));
        const int end = (int)((int64_t)cnt * (part + 1) / (C * kB64Warps));
        for (int base = beg; base < end; base += 32) {
            const int m = min(32, end - base);
            __syncwarp();
            if (lane < m)
                band64_record(A, list[base + lane], tn, ptx, prx, k0, kmax, s_rec[warp][lane]);
            __syncwarp();
            for (int k = 0; k < m; ++k) {
                const Rec64 &R = s_rec[warp][k];
                if (ok0) band64_eval(R, n0, mu_2c2, s_turn, re0, im0);
                if (ok1) band64_eval(R, n1, mu_2c2, s_turn, re1, im1);
            }
        }
        if (warp > 0) {
            s_sum[warp - 1][lane] = make_double2(re0, im0);
            s_sum[warp - 1][lane + 32] = make_double2(re1, im1);
        }
        __syncthreads();
        if (warp == 0) {
            for (int k = 0; k < kB64Warps - 1; ++k) {
                re0 += s_sum[k][lane].x;
                im0 += s_sum[k][lane].y;
                re1 += s_sum[k][lane + 32].x;
                im1 += s_sum[k][lane + 32].y;
            }
            double2 *out = b.coarse + (int64_t)v * b.room * b.sh.N * b.sh.M +
                           ((int64_t)chunk * nj + j) * Km;
            if (ok0) out[s0] = make_double2(re0, im0);
            if (ok1) out[s0 + 32] = make_double2(re1, im1);
        }
    }
}

// the parts' sums into the first, in order
__global__ void __launch_bounds__(256) band64_reduce_kernel(Band64Args b)
{
    const int v = blockIdx.x, cnt = b.vcnt[v];
    if (cnt == 0) return;
    const Band64Plan pl = b.plan[v / b.O];
    const int C = band64_chunks(b, pl, cnt);
    if (C == 1) return;
    const int n = b.sh.kn[pl.in] * b.sh.km[pl.im];
    double2 *x = b.coarse + (int64_t)v * b.room * b.sh.N * b.sh.M;
    for (int e = blockIdx.y * 256 + threadIdx.x; e < n; e += gridDim.y * 256) {
        double2 a = x[e];
        for (int k = 1; k < C; ++k) {
            const double2 q = x[(int64_t)k * n + e];
            a.x += q.x;
            a.y += q.y;
        }
        x[e] = a;
    }
}

// -------------------------------------------------------------------------
// interpolation: a block makes 64 chirps x 16 samples of a channel, instance
// by instance: first along the samples (its 16 samples of every chirp node, in
// shared memory), then along the chirps, turned by the reference
// -------------------------------------------------------------------------
constexpr int kExpN = 64, kExpM = 16;

__global__ void __launch_bounds__(256)
band64_expand_kernel(Band64Args b, RadarDev rd, void *__restrict__ out, int out_c64)
{
    __shared__ double2 s_d[kB64MaxNodes][kExpM];
    __shared__ double2 s_turn[256];
    s_turn[threadIdx.x] = b.turn[threadIdx.x];
    const int N = b.sh.N, M = b.sh.M;
    const int mt = M / kExpM;                     // M is a multiple of 32
    const int m0 = (int)(blockIdx.x % mt) * kExpM, n0 = (int)(blockIdx.x / mt) * kExpN;
    const int o = blockIdx.y, scene = blockIdx.z;
    const int mm = threadIdx.x & (kExpM - 1), nn = threadIdx.x / kExpM, m = m0 + mm;
    const double tau = (m - 0.5 * (rd.M - 1)) / rd.fs;
    double2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_double2(0.0, 0.0);
    for (int i = b.scene_inst[scene] * b.cells; i < b.scene_inst[scene + 1] * b.cells; ++i) {
        const int v = i * b.O + o;
        if (b.vcnt[v] == 0) continue;
        const Band64Plan pl = b.plan[i];
        const int nj = b.sh.kn[pl.in], Km = b.sh.km[pl.im];
        const double2 *x = b.coarse + (int64_t)v * b.room * N * M;
        // rows: the chirp nodes, or (every chirp kept) the block's chirps
        const int j0 = pl.in == 0 ? n0 : 0, rows = pl.in == 0 ? min(kExpN, N - n0) : nj;
        __syncthreads();
        for (int j = nn; j < rows; j += 256 / kExpM) {
            const double2 *row = x + (int64_t)(j0 + j) * Km;
            double2 d = make_double2(0.0, 0.0);
            if (pl.im == 0) {
                d = row[m];
            } else {
                const double *w = b.wm + b.sh.wm[pl.im] + m;
#pragma unroll 8
                for (int s = 0; s < Km; ++s) {
                    const double ws = w[(int64_t)s * M];
                    const double2 cs = row[s];
                    d.x = fma(ws, cs.x, d.x);
                    d.y = fma(ws, cs.y, d.y);
                }
            }
            s_d[j][mm] = d;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int n = n0 + nn + k * (256 / kExpM);
            if (n >= N) break;
            double2 z = make_double2(0.0, 0.0);
            if (pl.in == 0) {
                z = s_d[n - n0][mm];
            } else if (pl.in == 1) {
                z = s_d[0][mm];
            } else {
                const double *w = b.wn + b.sh.wn[pl.in] + (int64_t)n * nj;
                for (int j = 0; j < nj; ++j) {
                    const double wj = w[j];
                    const double2 d = s_d[j][mm];
                    z.x = fma(wj, d.x, z.x);
                    z.y = fma(wj, d.y, z.y);
                }
            }
            if (pl.rotate) {
                const double4 r = b.ref[(int64_t)v * N + n];
                double c, s;
                turn_exp(frac1(fma(tau, fma(tau, r.z, r.y), r.x)), s_turn, c, s);
                z = make_double2(z.x * c - z.y * s, z.x * s + z.y * c);
            }
            acc[k].x += z.x;
            acc[k].y += z.y;
        }
    }
    const double fm = rd.f0 + rd.slope * (double)m / rd.fs;
    const double km = 2.0 * kPi * fm / kC0;
    const double sc = 2.0 * sqrt(kPi) / pow(4.0 * kPi, 1.5) / (km * km);
    const int64_t row = ((int64_t)scene * b.O + o) * N;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int n = n0 + nn + k * (256 / kExpM);
        if (n >= N) break;
        const int64_t e = (row + n) * M + m;
        if (out_c64)
            static_cast<float2 *>(out)[e] = make_float2((float)(acc[k].x * sc), (float)(acc[k].y * sc));
        else
            static_cast<double2 *>(out)[e] = make_double2(acc[k].x * sc, acc[k].y * sc);
    }
}

// per-form counts of every (facet, channel, chirp) record (stats)
__global__ void __launch_bounds__(128) count_records64_kernel(SynthArgs A)
{
    const int n = blockIdx.x, vrow = blockIdx.y, o = vrow % A.rd.O;
    const int tx = o / A.rd.Q, rx = o % A.rd.Q;
    const double c = kC0, k0 = 2.0 * kPi * A.rd.f0 / c;
    const double kmax = 2.0 * kPi * (A.rd.f0 + A.rd.slope * (A.rd.M - 1) / A.rd.fs) / c;
    const int32_t *list = A.vis_idx + (int64_t)o * A.F + (A.vstart ? A.vstart[vrow] : 0);
    unsigned int cnt[3] = {0, 0, 0};
    for (int e = threadIdx.x; e < A.vcnt[vrow]; e += 128) {
        Rec64 R;
        band64_record(A, list[e], chirp_start(A.rd, n, tx), A.rd.ant[tx], A.rd.ant[A.rd.P + rx], k0,
                      kmax, R);
        ++cnt[R.kind == kRecVertex ? 0 : R.kind == kRecSeries ? 1 : 2];
    }
    for (int k = 0; k < 3; ++k) {
        const unsigned int s = __reduce_add_sync(0xffffffffu, cnt[k]);
        if ((threadIdx.x & 31) == 0 && s) atomicAdd(A.counters + k, (unsigned long long)s);
    }
}

// -------------------------------------------------------------------------
// adjoint: the transposes of the interpolation, then each facet's reverse
// pass over its node terms.  With H[n][m] = conj(G) scale(m) exp(j 2 pi ref),
// the loss varies as Re sum_{j,s} Hc[j][s] dC[j][s],
//   Hc[j][s] = sum_n Wn[n][j] sum_m Wm[m][s] H[n][m].
// -------------------------------------------------------------------------

// Y[j][m] = sum_n Wn[n][j] H[n][m], 16 samples of an (instance, channel) a block
__global__ void __launch_bounds__(256)
band64_gather_kernel(Band64Args b, RadarDev rd, const void *__restrict__ grad, int grad_c64)
{
    constexpr int R = 256 / kExpM;                // rows at once
    __shared__ double2 s_h[R][kExpM];
    __shared__ double2 s_turn[256];
    s_turn[threadIdx.x] = b.turn[threadIdx.x];
    __syncthreads();
    const int v = blockIdx.y, i = v / b.O, o = v % b.O;
    if (b.vcnt[v] == 0) return;
    const Band64Plan pl = b.plan[i];
    const int N = b.sh.N, M = b.sh.M, nj = b.sh.kn[pl.in];
    const int mm = threadIdx.x & (kExpM - 1), nn = threadIdx.x / kExpM;
    const int m = blockIdx.x * kExpM + mm;
    int scene = 0;
    while (b.scene_inst[scene + 1] * b.cells <= i) ++scene;
    const double fm = rd.f0 + rd.slope * (double)m / rd.fs, km = 2.0 * kPi * fm / kC0;
    const double sc = 2.0 * sqrt(kPi) / pow(4.0 * kPi, 1.5) / (km * km);
    const double tau = (m - 0.5 * (rd.M - 1)) / rd.fs;
    const int64_t row = ((int64_t)scene * b.O + o) * N;
    double2 *Y = b.coarse + (int64_t)v * b.room * N * M;
    const auto h_at = [&](int n) -> double2 {
        double2 g;
        if (grad_c64) {
            const float2 f = static_cast<const float2 *>(grad)[(row + n) * M + m];
            g = make_double2(f.x, f.y);
        } else {
            g = static_cast<const double2 *>(grad)[(row + n) * M + m];
        }
        g = make_double2(g.x * sc, -g.y * sc);
        if (!pl.rotate) return g;
        const double4 r = b.ref[(int64_t)v * N + n];
        double c, s;
        turn_exp(frac1(fma(tau, fma(tau, r.z, r.y), r.x)), s_turn, c, s);
        return make_double2(g.x * c - g.y * s, g.x * s + g.y * c);
    };
    if (pl.in == 0) {
        for (int n = nn; n < N; n += R) Y[(int64_t)n * M + m] = h_at(n);
        return;
    }
    const double *w = b.wn + b.sh.wn[pl.in];
    for (int j0 = 0; j0 < nj; j0 += 2 * R) {
        const int ja = j0 + nn, jb = ja + R;
        double2 ya = make_double2(0.0, 0.0), yb = ya;
        for (int n0 = 0; n0 < N; n0 += R) {
            __syncthreads();
            if (n0 + nn < N) s_h[nn][mm] = h_at(n0 + nn);
            __syncthreads();
            const int lim = min(R, N - n0);
            for (int q = 0; q < lim; ++q) {
                const double2 h = s_h[q][mm];
                if (ja < nj) {
                    const double wa = pl.in == 1 ? 1.0 : w[(int64_t)(n0 + q) * nj + ja];
                    ya.x = fma(wa, h.x, ya.x);
                    ya.y = fma(wa, h.y, ya.y);
                }
                if (jb < nj) {
                    const double wb = w[(int64_t)(n0 + q) * nj + jb];
                    yb.x = fma(wb, h.x, yb.x);
                    yb.y = fma(wb, h.y, yb.y);
                }
            }
        }
        if (ja < nj) Y[(int64_t)ja * M + m] = ya;
        if (jb < nj) Y[(int64_t)jb * M + m] = yb;
    }
}

// Hc[j][s] = sum_m Wm[m][s] Y[j][m], a node a thread
__global__ void __launch_bounds__(128) band64_gather_samples_kernel(Band64Args b)
{
    const int v = blockIdx.y;
    if (b.vcnt[v] == 0) return;
    const Band64Plan pl = b.plan[v / b.O];
    const int M = b.sh.M, nj = b.sh.kn[pl.in], Km = b.sh.km[pl.im];
    const double2 *Y = b.coarse + (int64_t)v * b.room * b.sh.N * M;
    double2 *H = b.coarse + ((int64_t)v * b.room + 1) * b.sh.N * M;
    for (int e = blockIdx.x * 128 + threadIdx.x; e < nj * Km; e += gridDim.x * 128) {
        const int j = e / Km, s = e - j * Km;
        const double2 *y = Y + (int64_t)j * M;
        double2 h = make_double2(0.0, 0.0);
        if (pl.im == 0) {
            h = y[s];
        } else {
            const double *w = b.wm + b.sh.wm[pl.im] + (int64_t)s * M;
#pragma unroll 8
            for (int m = 0; m < M; ++m) {
                h.x = fma(w[m], y[m].x, h.x);
                h.y = fma(w[m], y[m].y, h.y);
            }
        }
        H[e] = h;
    }
}

struct V3 {
    double x, y, z;
};
__device__ __forceinline__ V3 v3(double x, double y, double z) { return V3{x, y, z}; }
__device__ __forceinline__ V3 v3(const double *p) { return V3{p[0], p[1], p[2]}; }
__device__ __forceinline__ V3 operator+(V3 a, V3 b) { return V3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 operator-(V3 a, V3 b) { return V3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 operator*(double s, V3 a) { return V3{s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(V3 a, V3 b) { return fma(a.x, b.x, fma(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ V3 cross(V3 a, V3 b)
{
    return V3{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// Reverse pass of build_record (facet delay form): gp[10] = sum over the record's
// entries of bar[entry] d entry / d (vertex coordinates, reflectivity); bq: bars of
// qt0, qt1, qr0, qr1; bd: of d[0..15].  The centroid is the vertices' mean.
__device__ __forceinline__ void record_reverse(const double *tri, const double *c0, const double *vel,
                                               double tn, const double *ptx, const double *prx,
                                               double rho, int intra, double k0, int two_sided,
                                               int kind, const double *bq, const double *bd,
                                               double *gp)
{
    const V3 c = v3(c0), vv = v3(vel);
    V3 dv[3], bdv[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dv[i] = v3(tri + 3 * i) - c;
        bdv[i] = v3(0.0, 0.0, 0.0);
    }
    const V3 cc = c + tn * vv;
    const V3 e1 = dv[1] - dv[0], e2 = dv[2] - dv[0], nr = cross(e1, e2);
    const double nl = sqrt(dot(nr, nr)), inl = 1.0 / nl, area = 0.5 * nl;
    const V3 n = inl * nr;
    const V3 dt = v3(ptx) - cc, dr = v3(prx) - cc;
    const double it = 1.0 / sqrt(dot(dt, dt)), ir = 1.0 / sqrt(dot(dr, dr));
    const V3 b = it * dt + ir * dr;
    const double bn = dot(b, n), sg = two_sided && bn < 0.0 ? -0.5 : 0.5;
    const double ok = sg * bn, g = rho * ok * it * ir;
    const V3 bt = b - bn * n;
    double u[3], bu[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 3; ++i) u[i] = dot(bt, dv[i]);
    const double A2 = 2.0 * area * g;
    double bA2 = 0.0, bg = 0.0;
    V3 bbt = v3(0.0, 0.0, 0.0), bnv = v3(0.0, 0.0, 0.0);
    if (kind == kRecVertex) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int i1 = (i + 1) % 3, i2 = (i + 2) % 3;
            const double p = 1.0 / (u[i] - u[i1]), q = 1.0 / (u[i] - u[i2]);
            const double f = -p * q, t = bd[3 + i] * A2 * f;
            bA2 += bd[3 + i] * f;
            bu[i] += bd[i] - t * (p + q);
            bu[i1] += t * p;
            bu[i2] += t * q;
        }
    } else if (kind == kRecSeries) {
        const double ub = (u[0] + u[1] + u[2]) / 3.0;
        const double y0 = k0 * (u[0] - ub), y1 = k0 * (u[1] - ub), y2 = k0 * (u[2] - ub);
        const double s2 = y0 * y1 + y0 * y2 + y1 * y2, s3 = y0 * y1 * y2;
        double h[15], bh[15];
        h[0] = 1.0;
        h[1] = 0.0;
        h[2] = -s2;
        for (int p = 3; p < 15; ++p) h[p] = -s2 * h[p - 2] + s3 * h[p - 3];
        const double sc = A2 * k0 * k0;
        double bsc = 0.0, b2 = 0.0, b3 = 0.0;
        for (int i = 0; i < 8; ++i) {
            const double w = ((i & 1) ? -1.0 : 1.0) * c_inv_fact[2 * i + 2] * bd[1 + i];
            bh[2 * i] = sc * w;
            bsc += h[2 * i] * w;
        }
        for (int i = 0; i < 7; ++i) {
            const double w = ((i & 1) ? 1.0 : -1.0) * c_inv_fact[2 * i + 3] * bd[9 + i];
            bh[2 * i + 1] = sc * w;
            bsc += h[2 * i + 1] * w;
        }
        for (int p = 14; p >= 3; --p) {
            b2 -= bh[p] * h[p - 2];
            bh[p - 2] -= s2 * bh[p];
            b3 += bh[p] * h[p - 3];
            bh[p - 3] += s3 * bh[p];
        }
        b2 -= bh[2];
        bA2 = bsc * k0 * k0;
        const double by0 = b2 * (y1 + y2) + b3 * y1 * y2, by1 = b2 * (y0 + y2) + b3 * y0 * y2,
                     by2 = b2 * (y0 + y1) + b3 * y0 * y1;
        const double m = (bd[0] - k0 * (by0 + by1 + by2)) / 3.0;
        bu[0] = k0 * by0 + m;
        bu[1] = k0 * by1 + m;
        bu[2] = k0 * by2 + m;
    } else {
        const double ib2 = 1.0 / dot(bt, bt), kg = k0 * g * ib2;
        const V3 nxb = cross(n, bt);
        V3 bx = v3(0.0, 0.0, 0.0);
        double bb2 = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int i1 = (i + 1) % 3;
            const V3 e = dv[i1] - dv[i];
            const double x = dot(e, nxb), w = bd[3 * i + 2], t = 0.5 * k0 * bd[3 * i + 1];
            bu[i] += 0.5 * bd[3 * i] - t;
            bu[i1] += 0.5 * bd[3 * i] + t;
            bg += w * k0 * x * ib2;
            bb2 -= w * kg * x * ib2;
            const V3 be = (w * kg) * nxb;
            bdv[i1] = bdv[i1] + be;
            bdv[i] = bdv[i] - be;
            bx = bx + (w * kg) * e;
        }
        bnv = cross(bt, bx);
        bbt = cross(bx, n) + (2.0 * bb2) * bt;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        bbt = bbt + bu[i] * dv[i];
        bdv[i] = bdv[i] + bu[i] * bt;
    }
    const double barea = 2.0 * g * bA2;
    bg += 2.0 * area * bA2;
    V3 bb = bbt;
    const double bbn = -dot(bbt, n) + sg * bg * rho * it * ir;   // through bt and the obliquity
    bnv = bnv - bn * bbt + bbn * b;
    bb = bb + bbn * n;
    const double bRt = -bg * g * it - dot(bb, dt) * it * it;
    const double bRr = -bg * g * ir - dot(bb, dr) * ir * ir;
    V3 bdt = it * bb + (2.0 * bq[0] + bRt * it) * dt;
    V3 bdr = ir * bb + (2.0 * bq[2] + bRr * ir) * dr;
    if (intra) {
        bdt = bdt - (2.0 * bq[1]) * vv;
        bdr = bdr - (2.0 * bq[3]) * vv;
    }
    const V3 bnr = inl * (bnv - dot(n, bnv) * n) + (0.5 * barea) * n;
    const V3 be1 = cross(e2, bnr), be2 = cross(bnr, e1);
    bdv[1] = bdv[1] + be1;
    bdv[2] = bdv[2] + be2;
    bdv[0] = bdv[0] - be1 - be2;
    const V3 bc = (1.0 / 3.0) * (v3(0.0, 0.0, 0.0) - bdt - bdr - bdv[0] - bdv[1] - bdv[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        gp[3 * i] = bdv[i].x + bc.x;
        gp[3 * i + 1] = bdv[i].y + bc.y;
        gp[3 * i + 2] = bdv[i].z + bc.z;
    }
    gp[9] = bg * ok * it * ir;
}

// Work item = (instance, channel, chirp node, 128 facets), a facet a lane: the
// nodes' constants go round through shared memory, so that a lane's sums need
// no exchange, and its reverse pass follows in registers.  The FP64 pipe
// bounds it (some 95 operations a node).
__global__ void __launch_bounds__(kAdjFacets)
adjoint_band64_kernel(SynthArgs A, Band64Args b, double *__restrict__ gfac)
{
    constexpr int kInv = 21;                      // entries of a lane's column
    __shared__ double s_r[kInv + 10][kAdjFacets]; // d[16], L[5], 1 / (2 leg) quartics
    __shared__ double2 s_turn[256];
    __shared__ Node64 s_node[kSeg];
    __shared__ double2 s_h[kSeg];
    __shared__ int s_item;
    const int t = threadIdx.x;
    for (int i = t; i < 256; i += blockDim.x) s_turn[i] = b.turn[i];
    const RadarDev &rd = A.rd;
    const int V = b.I * b.O, total = b.item0[V];
    const double c = kC0;
    const double k0 = 2.0 * kPi * rd.f0 / c;
    const double kmax = 2.0 * kPi * (rd.f0 + rd.slope * (rd.M - 1) / rd.fs) / c;
    const double mu_2c2 = rd.slope / (2.0 * c * c);
    for (;;) {
        __syncthreads();
        if (t == 0) s_item = atomicAdd(b.ticket, 1);
        __syncthreads();
        if (s_item >= total) return;
        const int v = band64_find(b.item0, V, s_item);
        const int i = v / b.O, o = v % b.O, cnt = b.vcnt[v];
        const Band64Plan pl = b.plan[i];
        const int Km = b.sh.km[pl.im], parts = (cnt + kAdjFacets - 1) / kAdjFacets;
        const int at = s_item - b.item0[v], j = at / parts;
        const int e = (at - j * parts) * kAdjFacets + t;
        const bool valid = e < cnt;
        const int tx = o / rd.Q, rx = o % rd.Q;
        const double tn = chirp_start(rd, b.xn[b.sh.xn[pl.in] + j], tx);
        const double *ptx = rd.ant[tx], *prx = rd.ant[rd.P + rx];
        const double4 ref = b.refn[(int64_t)v * b.sh.N + j];
        const double2 *H = b.coarse + ((int64_t)v * b.room + 1) * b.sh.N * b.sh.M + (int64_t)j * Km;
        const int64_t k = valid ? (b.cells > 1 ? b.list : A.vis_idx)[(int64_t)o * A.F + b.vstart[v] + e] : 0;
        int kind = -1, flags = 0, quartic = 0;
        if (valid) {
            Rec64 R;
            band64_record(A, k, tn, ptx, prx, k0, kmax, R);
            kind = R.kind;
            flags = R.flags;
            quartic = R.quartic;
            for (int q = 0; q < 16; ++q) s_r[q][t] = R.d[q];
            for (int q = 0; q < 5; ++q) s_r[16 + q][t] = R.L[q];
            if (quartic) {
                // 1 / (2 sqrt(Q + q1 tau + q2 tau^2)) = h (1 + u)^(-1/2) to tau^4,
                // u = a tau + a2 tau^2
                const int inst = A.fac[k].inst;
                const double *vel = A.vel64 + 3 * inst;
                const double hc = rd.intra ? 0.5 * (rd.M - 1) / rd.fs : 0.0;
                const double q2 = rd.intra ? vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2] : 0.0;
                for (int leg = 0; leg < 2; ++leg) {
                    const double *pa = leg ? prx : ptx;
                    double Q = 0.0, q1 = 0.0;
                    for (int r = 0; r < 3; ++r) {
                        const double x = pa[r] - (A.c64[3 * k + r] + vel[r] * (tn + hc));
                        Q += x * x;
                        q1 -= 2.0 * x * vel[r];
                    }
                    const double iQ = 1.0 / Q, a = rd.intra ? q1 * iQ : 0.0, a2 = q2 * iQ;
                    const double h = 0.5 * sqrt(iQ), aa = a * a;
                    double *w = &s_r[kInv + 5 * leg][t];
                    w[0] = h;
                    w[kAdjFacets] = -0.5 * a * h;
                    w[2 * kAdjFacets] = h * (0.375 * aa - 0.5 * a2);
                    w[3 * kAdjFacets] = h * a * (0.75 * a2 - 0.3125 * aa);
                    w[4 * kAdjFacets] = h * (0.375 * a2 * a2 - 0.9375 * aa * a2 + 0.2734375 * aa * aa);
                }
            }
        }
        double bd[16], bq[4];
#pragma unroll
        for (int q = 0; q < 16; ++q) bd[q] = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) bq[q] = 0.0;
        const auto D = [&](int q) { return s_r[q][t]; };
        for (int s0 = 0; s0 < Km; s0 += kSeg) {
            __syncthreads();
            const int ns = min(kSeg, Km - s0);
            for (int s = t; s < ns; s += blockDim.x) {
                s_node[s] = band64_node(rd, b.xm[b.sh.xm[pl.im] + s0 + s], ref);
                s_h[s] = H[s0 + s];
            }
            __syncthreads();
            if (!valid) continue;
            for (int s = 0; s < ns; ++s) {
                const Node64 &nd = s_node[s];
                const double gr = s_h[s].x, gi = s_h[s].y, tau = nd.tau;
                double L, it, ir;
                if (quartic) {
                    L = fma(tau, fma(tau, fma(tau, fma(tau, D(20), D(19)), D(18)), D(17)), D(16));
                    it = fma(tau, fma(tau, fma(tau, fma(tau, D(25), D(24)), D(23)), D(22)), D(21));
                    ir = fma(tau, fma(tau, fma(tau, fma(tau, D(30), D(29)), D(28)), D(27)), D(26));
                } else {
                    const double st = sqrt(D(16) + nd.t * (D(17) + nd.t * D(18)));
                    const double sr = sqrt(D(19) + nd.t * (D(20) + nd.t * D(18)));
                    L = st + sr;
                    it = 0.5 / st;
                    ir = 0.5 / sr;
                }
                const double fmc = nd.fmc, kp = nd.kp;
                const double th = frac1(L * fma(-mu_2c2, L, fmc)) - nd.rp;
                double ath = 0.0, cs, sn;             // d / d phase, over -2 pi
                if (kind == kRecVertex) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        turn_exp(fma(-fmc, D(q), th), s_turn, cs, sn);
                        const double zr = gr * cs - gi * sn, zi = D(3 + q) * (gr * sn + gi * cs);
                        bd[3 + q] += zr;
                        bd[q] = fma(fmc, zi, bd[q]);
                        ath += zi;
                    }
                } else if (kind == kRecSeries) {
                    turn_exp(fma(-fmc, D(0), th), s_turn, cs, sn);
                    const double zr = gr * cs - gi * sn, zi = gr * sn + gi * cs;
                    const double k2 = kp * kp;
                    double a = D(8), bb = D(15);
#pragma unroll
                    for (int q = 6; q >= 0; --q) a = fma(a, k2, D(1 + q));
#pragma unroll
                    for (int q = 5; q >= 0; --q) bb = fma(bb, k2, D(9 + q));
                    double pw = k2;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        bd[1 + q] = fma(zr, pw, bd[1 + q]);
                        if (q < 7) bd[9 + q] = fma(-zi * kp, pw, bd[9 + q]);
                        pw *= k2;
                    }
                    ath = zr * (bb * k2 * kp) + zi * (a * k2);
                    bd[0] = fma(fmc, ath, bd[0]);
                } else {
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        turn_exp(fma(-fmc, D(3 * q), th), s_turn, cs, sn);
                        const double zr = gr * cs - gi * sn, zi = gr * sn + gi * cs;
                        const double x = kp * D(3 * q + 1);
                        double f, fp;                 // sin x / x and its derivative
                        if (flags & (1 << q)) {
                            const double x2 = x * x;
                            f = 1.0 + x2 * (-1.0 / 6 + x2 * (1.0 / 120 + x2 * (-1.0 / 5040 +
                                x2 * (1.0 / 362880 + x2 * (-1.0 / 39916800)))));
                            fp = x * (-1.0 / 3 + x2 * (1.0 / 30 + x2 * (-1.0 / 840 +
                                 x2 * (1.0 / 45360 + x2 * (-1.0 / 3991680)))));
                        } else {
                            double sx, cx;
                            sincos(x, &sx, &cx);
                            const double ix = 1.0 / x;
                            f = sx * ix;
                            fp = (cx - f) * ix;
                        }
                        const double w = kp * D(3 * q + 2), coef = w * f;
                        bd[3 * q + 2] = fma(-zi * kp, f, bd[3 * q + 2]);
                        bd[3 * q + 1] = fma(-zi * w, fp * kp, bd[3 * q + 1]);
                        bd[3 * q] = fma(coef * fmc, zr, bd[3 * q]);
                        ath = fma(coef, zr, ath);
                    }
                }
                // phase -> path length -> the legs' squared-range coefficients
                const double aL = ath * fma(-2.0 * mu_2c2, L, fmc);
                const double wt = aL * it, wr = aL * ir;
                bq[0] += wt;
                bq[1] = fma(wt, nd.t, bq[1]);
                bq[2] += wr;
                bq[3] = fma(wr, nd.t, bq[3]);
            }
        }
        if (!valid) continue;
        const double p2 = 2.0 * kPi;
#pragma unroll
        for (int q = 0; q < 4; ++q) bq[q] *= -p2;
        if (kind == kRecVertex) {
#pragma unroll
            for (int q = 0; q < 3; ++q) bd[q] *= p2;
        } else if (kind == kRecSeries) {
            bd[0] *= p2;
        } else {
#pragma unroll
            for (int q = 0; q < 3; ++q) bd[3 * q] *= p2;
        }
        double tri[9], c0[3], gp[10];
        const int inst = A.fac[k].inst;
        for (int q = 0; q < 9; ++q) tri[q] = A.tri64[9 * k + q];
        for (int r = 0; r < 3; ++r) c0[r] = A.c64[3 * k + r];
        record_reverse(tri, c0, A.vel64 + 3 * inst, tn, ptx, prx, (double)A.fac[k].rho, rd.intra, k0,
                       A.fac[k].two_sided, kind, bq, bd, gp);
#pragma unroll
        for (int p = 0; p < 10; ++p) atomicAdd(gfac + 10 * k + p, gp[p]);
    }
}

}  // namespace

void launch_band64_tables(const Band64Args &b, cudaStream_t s)
{
    band64_table_kernel<<<dim3((unsigned int)(b.sh.n_n + b.sh.n_m), 16), 256, 0, s>>>(
        b.sh, const_cast<double *>(b.xn), const_cast<double *>(b.xm), const_cast<double *>(b.wn),
        const_cast<double *>(b.wm), const_cast<double2 *>(b.turn));
}

void launch_band64_plan(const Band64Args &b, const SynthArgs &a, cudaStream_t s)
{
    const MixConsts K = mix_consts(a.rd);
    if (b.cells > 1) {
        cudaMemsetAsync(b.cbox, 0, (size_t)b.I * 8 * sizeof(unsigned int), s);
        band64_cell_kernel<<<(unsigned int)((a.F + 127) / 128), 128, 0, s>>>(b, a.fac, a.F);
    }
    band64_plan_kernel<<<b.I, 32, 0, s>>>(b, a.rd, K, a.vel32, a.fac);
    const dim3 g((unsigned int)((2 * b.sh.N + 127) / 128), (unsigned int)(b.I * b.O));
    band64_ref_kernel<<<g, 128, 0, s>>>(b, a.rd, a.vel64);
}

static void launch_lists(const Band64Args &b, const SynthArgs &a, cudaStream_t s)
{
    const int V = b.I * b.O;
    if (b.cells > 1)
        band64_cell_lists_kernel<<<V / b.cells, 256, 0, s>>>(b, a.vis_idx, a.vis_cnt, a.F);
    else
        band64_lists_kernel<<<(V + 3) / 4, 128, 0, s>>>(b, a.vis_idx, a.vis_cnt, a.F);
}

void launch_synth_band64(const Band64Args &b, const SynthArgs &a, cudaStream_t s)
{
    const int V = b.I * b.O;
    launch_lists(b, a, s);
    band64_items_kernel<<<1, 1024, 0, s>>>(b, 0);
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, synth_band64_kernel, kB64Warps * 32, 0);
    synth_band64_kernel<<<std::max(1, sms) * std::max(1, per_sm), kB64Warps * 32, 0, s>>>(a, b);
    band64_reduce_kernel<<<dim3((unsigned int)V, 4), 256, 0, s>>>(b);
    const int tiles = (b.sh.M / kExpM) * ((b.sh.N + kExpN - 1) / kExpN);
    band64_expand_kernel<<<dim3((unsigned int)tiles, (unsigned int)b.O, (unsigned int)b.B), 256, 0,
                           s>>>(b, a.rd, a.out, a.out_c64);
}

void launch_adjoint_band64(const Band64Args &b, const SynthArgs &a, const void *grad, int grad_c64,
                           double *gfac, cudaStream_t s)
{
    const int V = b.I * b.O;
    cudaMemsetAsync(gfac, 0, (size_t)a.F * 10 * sizeof(double), s);
    launch_lists(b, a, s);
    band64_items_kernel<<<1, 1024, 0, s>>>(b, 1);
    band64_gather_kernel<<<dim3((unsigned int)(b.sh.M / kExpM), (unsigned int)V), 256, 0, s>>>(
        b, a.rd, grad, grad_c64);
    band64_gather_samples_kernel<<<dim3(8, (unsigned int)V), 128, 0, s>>>(b);
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, adjoint_band64_kernel, kAdjFacets, 0);
    adjoint_band64_kernel<<<std::max(1, sms) * std::max(1, per_sm), kAdjFacets, 0, s>>>(a, b, gfac);
}

void launch_count_records64(const SynthArgs &a, cudaStream_t s)
{
    count_records64_kernel<<<dim3((unsigned int)a.rd.N, (unsigned int)a.VO), 128, 0, s>>>(a);
}

}  // namespace bart
