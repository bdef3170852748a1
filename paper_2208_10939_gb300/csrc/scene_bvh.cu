// Scene flattening (world facets at the frame start) and the LBVH builder
// used by the BART visibility rays (Sec. 2.2 ray tracing).
//
// LBVH: 30-bit Morton codes of facet centroids, a stable LSD radix sort, the
// hierarchy of Karras (2012, "Maximizing parallelism in the construction of
// BVHs, octrees, and k-d trees"), each node's boxes from the boxes of aligned
// runs of the sorted leaves.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "bart_internal.cuh"

namespace bart {

// -------------------------------------------------------------------------
// world facets
// -------------------------------------------------------------------------
__device__ __forceinline__ unsigned int f2ord(float x)
{
    unsigned int b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned int u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Rigid transform with one IEEE rounding per operation, in a fixed order:
//   w = ((r0 x + r1 y) + r2 z) + p;  w = w + v t
__device__ __forceinline__ double world_coord(const double *r, double x, double y, double z,
                                              double p, double v, double t)
{
    double w = __dmul_rn(r[0], x);
    w = __dadd_rn(w, __dmul_rn(r[1], y));
    w = __dadd_rn(w, __dmul_rn(r[2], z));
    w = __dadd_rn(w, p);
    w = __dadd_rn(w, __dmul_rn(v, t));
    return w;
}

__global__ void build_facets_kernel(const MeshDesc *__restrict__ meshes,
                                    const InstDev *__restrict__ insts, int n_inst, int64_t F,
                                    double t0, double *__restrict__ tri64,
                                    float *__restrict__ tri32, float4 *__restrict__ trel,
                                    double *__restrict__ c64, FacetRec *__restrict__ fac,
                                    float *__restrict__ aabb, float *__restrict__ vel32,
                                    unsigned int *__restrict__ bounds,
                                    double *__restrict__ ref64, float *__restrict__ ref32,
                                    float *__restrict__ fac_lo, unsigned int *__restrict__ box)
{
    const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float cf[3] = {0.f, 0.f, 0.f};
    int inst = -1;
    unsigned int bx[7] = {0u, 0u, 0u, 0u, 0u, 0u, 0u};    // the facet's part of its box
    const bool valid = f < F;
    if (valid) {
        int lo = 0, hi = n_inst - 1;            // last instance with off <= f
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (insts[mid].off <= f) lo = mid;
            else hi = mid - 1;
        }
        const InstDev &in = insts[lo];
        const MeshDesc &m = meshes[in.mesh];
        const int64_t j = f - in.off;
        double v[9];
        for (int k = 0; k < 3; ++k) {
            const int64_t vi = m.tris[3 * j + k];
            const double x = m.verts[3 * vi], y = m.verts[3 * vi + 1], z = m.verts[3 * vi + 2];
            for (int r = 0; r < 3; ++r)
                v[3 * k + r] = world_coord(in.rot + 3 * r, x, y, z, in.pos[r], in.vel[r], t0);
        }
        inst = lo;
        float vmax = 0.f;
        for (int i = 0; i < 9; ++i) {
            tri64[9 * f + i] = v[i];
            const float vf = (float)v[i];
            if (tri32) tri32[12 * f + i] = vf;
            vmax = fmaxf(vmax, fabsf(vf));
        }
        if (tri32) {
            tri32[12 * f + 9] = vmax;
            tri32[12 * f + 10] = 0.f;
            tri32[12 * f + 11] = 0.f;
        }
        double c[3];
        for (int r = 0; r < 3; ++r) {
            c[r] = __ddiv_rn(__dadd_rn(__dadd_rn(v[r], v[3 + r]), v[6 + r]), 3.0);
            c64[3 * f + r] = c[r];
        }
        const double e1[3] = {v[3] - v[0], v[4] - v[1], v[5] - v[2]};
        const double e2[3] = {v[6] - v[0], v[7] - v[1], v[8] - v[2]};
        const float h0 = (float)v[0], h1 = (float)v[1], h2 = (float)v[2];
        trel[3 * f] = make_float4(h0, h1, h2, (float)e1[0]);
        trel[3 * f + 1] = make_float4((float)e1[1], (float)e1[2], (float)e2[0], (float)e2[1]);
        trel[3 * f + 2] = make_float4((float)e2[2], (float)(v[0] - (double)h0),
                                      (float)(v[1] - (double)h1), (float)(v[2] - (double)h2));
        const double nx = e1[1] * e2[2] - e1[2] * e2[1];
        const double ny = e1[2] * e2[0] - e1[0] * e2[2];
        const double nz = e1[0] * e2[1] - e1[1] * e2[0];
        const double nl = sqrt(nx * nx + ny * ny + nz * nz);
        FacetRec rec;
        for (int r = 0; r < 3; ++r) {
            rec.c[r] = (float)c[r];
            cf[r] = rec.c[r];
        }
        rec.area = (float)(0.5 * nl);
        for (int r = 0; r < 3; ++r) fac_lo[12 * f + r] = (float)(c[r] - (double)rec.c[r]);
        for (int k = 0; k < 3; ++k)
            for (int r = 0; r < 3; ++r) {
                const double d = v[3 * k + r] - c[r];
                rec.dv[3 * k + r] = (float)d;
                fac_lo[12 * f + 3 + 3 * k + r] = (float)(d - (double)rec.dv[3 * k + r]);
            }
        float rad2 = 0.f;
        for (int k = 0; k < 3; ++k)
            rad2 = fmaxf(rad2, rec.dv[3 * k] * rec.dv[3 * k] + rec.dv[3 * k + 1] * rec.dv[3 * k + 1] +
                                   rec.dv[3 * k + 2] * rec.dv[3 * k + 2]);
        bx[6] = f2ord(rad2);
        const double inl = nl > 0.0 ? 1.0 / nl : 0.0;
        rec.n[0] = (float)(nx * inl);
        rec.n[1] = (float)(ny * inl);
        rec.n[2] = (float)(nz * inl);
        rec.rho = m.rho ? m.rho[j] * in.rho_scale : in.rho_scale;
        rec.inst = lo;
        rec.two_sided = m.two_sided;
        rec.pad = 0.f;
        fac[f] = rec;
        // conservative FP32 box: outward rounding plus a pad covering the
        // FP32 slab test of a segment of <= ~200 m length
        float mx = 0.f;
        for (int r = 0; r < 3; ++r) {
            double lo_ = fmin(fmin(v[r], v[3 + r]), v[6 + r]);
            double hi_ = fmax(fmax(v[r], v[3 + r]), v[6 + r]);
            mx = fmaxf(mx, fmaxf(fabsf((float)lo_), fabsf((float)hi_)));
            aabb[6 * f + r] = __double2float_rd(lo_);
            aabb[6 * f + 3 + r] = __double2float_ru(hi_);
            bx[r] = ~f2ord(__double2float_rd(lo_));
            bx[3 + r] = f2ord(__double2float_ru(hi_));
        }
        const float pad = 1e-4f + 4e-6f * mx;
        for (int r = 0; r < 3; ++r) {
            aabb[6 * f + r] -= pad;
            aabb[6 * f + 3 + r] += pad;
        }
        if (j == 0) {
            for (int r = 0; r < 3; ++r) {
                vel32[4 * lo + r] = (float)in.vel[r];
                // the instance origin at t0 (reference point of the delay form)
                const double o = world_coord(in.rot + 3 * r, 0.0, 0.0, 0.0, in.pos[r], in.vel[r], t0);
                ref64[3 * lo + r] = o;
                ref32[4 * lo + r] = (float)o;
            }
            vel32[4 * lo + 3] = 0.f;
            ref32[4 * lo + 3] = 0.f;
        }
    }
    // the instances' boxes: a warp of one instance reduces before its atomics
    {
        const int i0 = __shfl_sync(0xffffffffu, inst, 0);
        if (__all_sync(0xffffffffu, inst == i0)) {
            for (int r = 0; r < 7; ++r) {
                const unsigned int m = __reduce_max_sync(0xffffffffu, bx[r]);
                if ((threadIdx.x & 31) == 0 && i0 >= 0) atomicMax(box + 8 * (int64_t)i0 + r, m);
            }
        } else if (inst >= 0) {
            for (int r = 0; r < 7; ++r) atomicMax(box + 8 * (int64_t)inst + r, bx[r]);
        }
    }
    // centroid bounds for the Morton grid
    __shared__ unsigned int s_b[6];
    if (threadIdx.x < 6) s_b[threadIdx.x] = threadIdx.x < 3 ? 0xffffffffu : 0u;
    __syncthreads();
    if (valid)
        for (int r = 0; r < 3; ++r) {
            atomicMin(&s_b[r], f2ord(cf[r]));
            atomicMax(&s_b[3 + r], f2ord(cf[r]));
        }
    __syncthreads();
    if (threadIdx.x < 3) atomicMin(&bounds[threadIdx.x], s_b[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&bounds[threadIdx.x], s_b[threadIdx.x]);
}

const void *build_facets_kernel_fn(int *t0_arg_index, int *n_args)
{
    *t0_arg_index = 4;      // meshes, insts, n_inst, F, t0, tri64, tri32, trel, c64, fac, aabb,
    *n_args = 17;           // vel32, bounds, ref64, ref32, fac_lo, box
    return reinterpret_cast<const void *>(build_facets_kernel);
}

void launch_build_facets(const MeshDesc *meshes, const InstDev *insts, int n_inst, int64_t F,
                         double t0, double *tri64, float *tri32, float4 *trel, double *c64,
                         FacetRec *fac,
                         float *aabb, float *vel32, unsigned int *bounds, double *ref64,
                         float *ref32, float *fac_lo, unsigned int *box, cudaStream_t s)
{
    cudaMemsetAsync(box, 0, (size_t)n_inst * 8 * sizeof(unsigned int), s);
    cudaMemsetAsync(bounds, 0xff, 3 * sizeof(unsigned int), s);
    cudaMemsetAsync(bounds + 3, 0, 3 * sizeof(unsigned int), s);
    // FP64 instructions issue at 1/64 of an SM's FP32 rate, so a block's warps
    // queue for them: small blocks spread the facets over all SMs (256 threads
    // a block: 19 us for 200 facets, 22 us for 20k)
    const int T = 64;
    const unsigned int G = (unsigned int)((F + T - 1) / T);
    build_facets_kernel<<<G, T, 0, s>>>(meshes, insts, n_inst, F, t0, tri64, tri32, trel, c64, fac,
                                        aabb, vel32, bounds, ref64, ref32, fac_lo, box);
}

// -------------------------------------------------------------------------
// Morton codes
// -------------------------------------------------------------------------
__device__ __forceinline__ uint32_t spread10(uint32_t x)
{
    x &= 0x3ffu;
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

__device__ __forceinline__ uint32_t morton_code(const FacetRec &f, const unsigned int *bounds)
{
    uint32_t code = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float lo = ord2f(bounds[r]), hi = ord2f(bounds[3 + r]);
        const float ext = hi - lo;
        float u = ext > 0.f ? (f.c[r] - lo) / ext : 0.f;
        u = fminf(fmaxf(u, 0.f), 1.f);
        const uint32_t q = (uint32_t)fminf(u * 1024.f, 1023.f);
        code |= spread10(q) << (2 - r);
    }
    return code;
}

__global__ void morton_kernel(const FacetRec *__restrict__ fac, int64_t F,
                              const unsigned int *__restrict__ bounds,
                              uint32_t *__restrict__ keys, int32_t *__restrict__ vals)
{
    const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= F) return;
    keys[f] = morton_code(fac[f], bounds);
    vals[f] = (int32_t)f;
}

void launch_morton(const FacetRec *fac, int64_t F, const unsigned int *bounds, uint32_t *keys,
                   int32_t *vals, cudaStream_t s)
{
    const int T = 256;
    morton_kernel<<<(unsigned int)((F + T - 1) / T), T, 0, s>>>(fac, F, bounds, keys, vals);
}

// -------------------------------------------------------------------------
// stable LSD radix sort, 8-bit digits
// -------------------------------------------------------------------------
constexpr int kSortThreads = 256;
constexpr int kSortTile = 2048;     // keys per block

static inline int64_t sort_blocks(int64_t n) { return (n + kSortTile - 1) / kSortTile; }

constexpr int kSortMaxPasses = 8;

int64_t radix_sort_temp_words(int64_t n) { return 256 * sort_blocks(n) + 256 * kSortMaxPasses; }

__global__ void rs_hist_kernel(const uint32_t *__restrict__ keys, int64_t n, int shift,
                               uint32_t *__restrict__ hist, int64_t nblk,
                               uint32_t *__restrict__ total)
{
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int i = threadIdx.x; i < kSortTile; i += kSortThreads) {
        const int64_t idx = base + i;
        if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & 0xffu], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblk + blockIdx.x] = h[threadIdx.x];
    if (h[threadIdx.x]) atomicAdd(total + threadIdx.x, h[threadIdx.x]);
}

// first position of every (digit, block): a block per digit adds the smaller
// digits' totals and scans its row (one block over all rows took 35 us at 169
// blocks, this takes 4)
__global__ void rs_scan_kernel(uint32_t *__restrict__ hist, int64_t nblk,
                               const uint32_t *__restrict__ total)
{
    __shared__ uint32_t s_w[8], s_run;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, d = blockIdx.x;
    uint32_t below = t < d ? total[t] : 0u;
    below = __reduce_add_sync(0xffffffffu, below);
    if (lane == 0) s_w[warp] = below;
    __syncthreads();
    if (t == 0) {
        s_run = 0;
        for (int w = 0; w < 8; ++w) s_run += s_w[w];
    }
    __syncthreads();
    uint32_t *row = hist + (int64_t)d * nblk;
    for (int64_t b0 = 0; b0 < nblk; b0 += 256) {
        const int64_t b = b0 + t;
        const uint32_t v = b < nblk ? row[b] : 0u;
        uint32_t x = v;
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        uint32_t run = s_run, all = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) run += s_w[w];
            all += s_w[w];
        }
        if (b < nblk) row[b] = run + x - v;
        __syncthreads();
        if (t == 0) s_run += all;
        __syncthreads();
    }
}

__global__ void rs_scatter_kernel(const uint32_t *__restrict__ keys_in,
                                  const int32_t *__restrict__ vals_in, int64_t n, int shift,
                                  const uint32_t *__restrict__ hist, int64_t nblk,
                                  uint32_t *__restrict__ keys_out, int32_t *__restrict__ vals_out)
{
    constexpr int W = kSortThreads / 32;
    __shared__ uint32_t s_base[256];
    __shared__ uint32_t s_wcnt[W][256];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    s_base[t] = hist[(int64_t)t * nblk + blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    const unsigned int lt = (1u << lane) - 1u;
    for (int r = 0; r < kSortTile / kSortThreads; ++r) {
        for (int w = 0; w < W; ++w) s_wcnt[w][t] = 0;
        __syncthreads();
        const int64_t idx = base + (int64_t)r * kSortThreads + t;
        const bool valid = idx < n;
        uint32_t key = 0;
        int32_t val = 0;
        int d = 256;                                   // invalid items form their own group
        if (valid) {
            key = keys_in[idx];
            val = vals_in[idx];
            d = (key >> shift) & 0xff;
        }
        const unsigned int peers = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(peers & lt);
        if (valid && rank == 0) s_wcnt[warp][d] = __popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t pos = s_base[d] + rank;
            for (int w = 0; w < warp; ++w) pos += s_wcnt[w][d];
            keys_out[pos] = key;
            vals_out[pos] = val;
        }
        __syncthreads();
        uint32_t tot = 0;
        for (int w = 0; w < W; ++w) tot += s_wcnt[w][t];
        s_base[t] += tot;
        __syncthreads();
    }
}

void radix_sort_pairs(uint32_t *keys, int32_t *vals, uint32_t *keys_tmp, int32_t *vals_tmp,
                      uint32_t *temp, int64_t n, int bits, cudaStream_t s)
{
    const int64_t nblk = sort_blocks(n);
    uint32_t *ka = keys, *kb = keys_tmp, *total = temp + 256 * nblk;
    int32_t *va = vals, *vb = vals_tmp;
    int passes = (bits + 7) / 8;
    if (passes & 1) passes += 1;                      // even: result lands in `keys`
    cudaMemsetAsync(total, 0, (size_t)256 * passes * sizeof(uint32_t), s);
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        rs_hist_kernel<<<(unsigned int)nblk, kSortThreads, 0, s>>>(ka, n, shift, temp, nblk,
                                                                   total + 256 * p);
        rs_scan_kernel<<<256, 256, 0, s>>>(temp, nblk, total + 256 * p);
        rs_scatter_kernel<<<(unsigned int)nblk, kSortThreads, 0, s>>>(ka, va, n, shift, temp,
                                                                      nblk, kb, vb);
        uint32_t *tk = ka; ka = kb; kb = tk;
        int32_t *tv = va; va = vb; vb = tv;
    }
}

// -------------------------------------------------------------------------
// One-launch sort of up to 96k facets: Morton codes, then stable 8-bit LSD
// passes over the code (and, batched, over the scene), with keys and values
// in the shared memory of one cluster of up to eight CTAs.  A pass ranks a
// CTA's keys by warp (match, then warp-private counts), adds the counts over
// the warps, reads the other CTAs' totals and scatters through distributed
// shared memory; the cluster's barrier is the only synchronisation.  What
// bounds the multi-launch sort at these sizes is its chain of twelve launches
// (and 10 to 40 blocks of serial rounds): 20k facets 93 us there; with batch
// scenes, 63k facets, 165 us.
// -------------------------------------------------------------------------
namespace cg = cooperative_groups;
constexpr int kCsThreads = 1024, kCsWarps = kCsThreads / 32, kCsMaxCtas = 8;
constexpr int kCsMaxPer = 12288;                      // keys per CTA: 16 B each of 227 KB

static size_t cs_smem(int per) { return (size_t)per * 16 + kCsWarps * 256 * 2 + 3 * 256 * 4; }

__device__ __forceinline__ uint32_t scene_of(const int64_t *foff, int B, int64_t f)
{
    int lo = 0, hi = B - 1;                 // last scene with foff <= f
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (foff[mid] <= f) lo = mid;
        else hi = mid - 1;
    }
    return (uint32_t)lo;
}

__global__ void __launch_bounds__(kCsThreads)
cluster_sort_kernel(const FacetRec *__restrict__ fac, int n, int per,
                    const unsigned int *__restrict__ bounds, const int64_t *__restrict__ foff,
                    int B, int scene_passes, uint32_t *__restrict__ keys_out,
                    int32_t *__restrict__ vals_out, uint32_t *__restrict__ skeys_out)
{
    extern __shared__ __align__(16) unsigned char cs_raw[];
    uint32_t *key = reinterpret_cast<uint32_t *>(cs_raw);            // [2][per]
    int32_t *val = reinterpret_cast<int32_t *>(key + 2 * per);       // [2][per]
    uint16_t *cnt = reinterpret_cast<uint16_t *>(val + 2 * per);     // [warp][digit]
    uint32_t *tot = reinterpret_cast<uint32_t *>(cnt + kCsWarps * 256);   // this CTA's totals
    uint32_t *base = tot + 256;                                      // first positions
    uint32_t *s_scan = base + 256;                                   // scan scratch
    cg::cluster_group cl = cg::this_cluster();
    const int ctas = (int)cl.num_blocks(), me = (int)cl.block_rank();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int first = me * per, mine = max(0, min(per, n - first));
    for (int i = t; i < mine; i += kCsThreads) {
        key[i] = morton_code(fac[first + i], bounds);
        val[i] = first + i;
    }
    const int wper = ((per + kCsThreads - 1) / kCsThreads) * 32;     // a warp's consecutive keys
    const int steps = wper / 32;
    const unsigned int lt = (1u << lane) - 1u;
    int cur = 0;
    for (int pass = 0; pass < 4 + scene_passes; ++pass) {
        for (int i = t; i < kCsWarps * 256 / 2; i += kCsThreads) reinterpret_cast<uint32_t *>(cnt)[i] = 0u;
        __syncthreads();
        const uint32_t *k0 = key + cur * per;
        const int32_t *v0 = val + cur * per;
        uint16_t *wc = cnt + warp * 256;
        uint32_t rank[kCsMaxPer / kCsThreads];                       // digit << 16 | rank in the warp
#pragma unroll
        for (int st = 0; st < kCsMaxPer / kCsThreads; ++st) {
            if (st >= steps) break;
            const int i = warp * wper + st * 32 + lane;
            const bool ok = i < mine;
            uint32_t d = 256u;
            if (ok)
                d = pass < 4 ? (k0[i] >> (8 * pass)) & 255u
                             : (scene_of(foff, B, v0[i]) >> (8 * (pass - 4))) & 255u;
            const unsigned int peers = __match_any_sync(0xffffffffu, d);
            const int r = __popc(peers & lt);
            uint32_t before = 0;
            if (ok) before = wc[d];
            rank[st] = ok ? (d << 16) | (before + (uint32_t)r) : 0xffffffffu;
            __syncwarp();
            if (ok && r == 0) wc[d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        if (t < 256) {                                               // over the warps
            uint32_t run = 0;
            for (int w = 0; w < kCsWarps; ++w) {
                const uint32_t c = cnt[w * 256 + t];
                cnt[w * 256 + t] = (uint16_t)run;
                run += c;
            }
            tot[t] = run;
        }
        cl.sync();
        if (t < 256) {                                               // over the CTAs, then the digits
            uint32_t all = 0, below = 0;
            for (int c = 0; c < ctas; ++c) {
                const uint32_t x = cl.map_shared_rank(tot, c)[t];
                if (c < me) below += x;
                all += x;
            }
            uint32_t x = all;
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
                if (lane >= off) x += y;
            }
            if (lane == 31) s_scan[warp] = x;
            base[t] = x - all + below;
        }
        __syncthreads();
        if (t < 256) {
            uint32_t add = 0;
            for (int w = 0; w < warp; ++w) add += s_scan[w];
            base[t] += add;
        }
        __syncthreads();
        uint32_t *k1 = key + (cur ^ 1) * per;
        int32_t *v1 = val + (cur ^ 1) * per;
#pragma unroll
        for (int st = 0; st < kCsMaxPer / kCsThreads; ++st) {
            if (st >= steps) break;
            const uint32_t e = rank[st];
            if (e != 0xffffffffu) {
                const int i = warp * wper + st * 32 + lane;
                const uint32_t d = e >> 16;
                const uint32_t pos = base[d] + wc[d] + (e & 0xffffu);
                const int c = (int)(pos / (uint32_t)per), off = (int)(pos - (uint32_t)c * per);
                cl.map_shared_rank(k1, c)[off] = k0[i];
                cl.map_shared_rank(v1, c)[off] = v0[i];
            }
        }
        cl.sync();
        cur ^= 1;
    }
    for (int i = t; i < mine; i += kCsThreads) {
        keys_out[first + i] = key[cur * per + i];
        vals_out[first + i] = val[cur * per + i];
        if (skeys_out) skeys_out[first + i] = scene_of(foff, B, val[cur * per + i]);
    }
}

static int scene_passes(int B)
{
    int p = 0;
    while (B > 1 && (1ll << (8 * p)) < B) ++p;
    return p;
}

// false: too large for one cluster
static bool launch_cluster_sort(const FacetRec *fac, int64_t F, const unsigned int *bounds,
                                const int64_t *foff, int B, uint32_t *keys, int32_t *vals,
                                uint32_t *skeys, cudaStream_t s)
{
    if (F > (int64_t)kCsMaxCtas * kCsMaxPer) return false;
    // one CTA up to 4096 facets (no cluster barrier), else eight
    const int ctas = F <= 4096 ? 1 : kCsMaxCtas;
    const int per = (int)(((F + ctas - 1) / ctas + 31) / 32 * 32);
    const size_t sm = cs_smem(per);
    if (cudaFuncSetAttribute(cluster_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)cs_smem(kCsMaxPer)) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)ctas);
    cfg.blockDim = dim3(kCsThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned int)ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, cluster_sort_kernel, fac, (int)F, per, bounds, foff, B,
                           scene_passes(B), keys, vals, B > 1 ? skeys : nullptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

// -------------------------------------------------------------------------
// Boxes of aligned runs of the sorted leaves: level l holds the boxes of
// leaves [j 2^l, (j + 1) 2^l), two float4 each (min, max), level after level.
// A node's box is then the union of at most two runs per level of its leaf
// range, read independently of one another; the bottom-up refit with atomics
// that this replaces is a chain of one atomic round trip per tree level (20k
// facets 40 us, 345k facets 100 us).
// -------------------------------------------------------------------------
constexpr int kLvLeaves = 1024;                      // leaves of a block: ten levels

int64_t leaf_levels_words(int64_t n)                 // float4
{
    int64_t c = n, sum = 0;
    for (;;) {
        sum += 2 * c;
        if (c <= 1) break;
        c = (c + 1) >> 1;
    }
    return sum;
}

struct Box {
    float4 lo, hi;
};
__device__ __forceinline__ void box_join(Box &a, const float4 lo, const float4 hi)
{
    a.lo.x = fminf(a.lo.x, lo.x);
    a.lo.y = fminf(a.lo.y, lo.y);
    a.lo.z = fminf(a.lo.z, lo.z);
    a.hi.x = fmaxf(a.hi.x, hi.x);
    a.hi.y = fmaxf(a.hi.y, hi.y);
    a.hi.z = fmaxf(a.hi.z, hi.z);
}
__device__ __forceinline__ Box box_empty()
{
    return Box{make_float4(INFINITY, INFINITY, INFINITY, 0.f),
               make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f)};
}
__device__ __forceinline__ Box box_xor(const Box &b, int mask)
{
    Box o = b;
    box_join(o,
             make_float4(__shfl_xor_sync(0xffffffffu, b.lo.x, mask),
                         __shfl_xor_sync(0xffffffffu, b.lo.y, mask),
                         __shfl_xor_sync(0xffffffffu, b.lo.z, mask), 0.f),
             make_float4(__shfl_xor_sync(0xffffffffu, b.hi.x, mask),
                         __shfl_xor_sync(0xffffffffu, b.hi.y, mask),
                         __shfl_xor_sync(0xffffffffu, b.hi.z, mask), 0.f));
    return o;
}

__global__ void __launch_bounds__(kLvLeaves)
leaf_levels_kernel(const int32_t *__restrict__ vals, const float *__restrict__ aabb, int64_t n,
                   float4 *lv, int *ticket)
{
    __shared__ Box s_box[32];
    __shared__ bool s_last;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t i = (int64_t)blockIdx.x * kLvLeaves + t;
    Box b = box_empty();
    if (i < n) {
        const float *a = aabb + 6 * (int64_t)vals[i];
        b.lo = make_float4(a[0], a[1], a[2], 0.f);
        b.hi = make_float4(a[3], a[4], a[5], 0.f);
        lv[2 * i] = b.lo;
        lv[2 * i + 1] = b.hi;
    }
    int64_t off = n, c = n;                          // level l at off; c boxes below it
    for (int l = 1; l <= 5; ++l) {
        b = box_xor(b, 1 << (l - 1));
        if (c > 1) {                                 // there is a level l
            c = (c + 1) >> 1;
            const int64_t j = i >> l;
            if ((t & ((1 << l) - 1)) == 0 && j < c) {
                lv[2 * (off + j)] = b.lo;
                lv[2 * (off + j) + 1] = b.hi;
            }
            off += c;
        }
    }
    if (lane == 0) s_box[warp] = b;
    __syncthreads();
    if (warp == 0) {
        b = s_box[lane];
        for (int l = 6; l <= 10; ++l) {
            b = box_xor(b, 1 << (l - 6));
            if (c > 1) {
                c = (c + 1) >> 1;
                const int64_t j = ((int64_t)blockIdx.x << (10 - l)) + (lane >> (l - 5));
                if ((lane & ((1 << (l - 5)) - 1)) == 0 && j < c) {
                    lv[2 * (off + j)] = b.lo;
                    lv[2 * (off + j) + 1] = b.hi;
                }
                off += c;
            }
        }
    }
    if (gridDim.x == 1) return;
    // the block that finishes last joins the blocks' boxes
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (t == 0) *ticket = 0;
    int64_t poff = 0, pc = n;                        // level 10, then up
    for (int l = 0; l < 10; ++l) {
        poff += pc;
        pc = (pc + 1) >> 1;
    }
    while (pc > 1) {
        const int64_t noff = poff + pc, nc = (pc + 1) >> 1;
        for (int64_t j = t; j < nc; j += kLvLeaves) {
            Box x{__ldcg(lv + 2 * (poff + 2 * j)), __ldcg(lv + 2 * (poff + 2 * j) + 1)};
            if (2 * j + 1 < pc)
                box_join(x, __ldcg(lv + 2 * (poff + 2 * j + 1)), __ldcg(lv + 2 * (poff + 2 * j + 1) + 1));
            __stcg(lv + 2 * (noff + j), x.lo);
            __stcg(lv + 2 * (noff + j) + 1, x.hi);
        }
        __syncthreads();
        poff = noff;
        pc = nc;
    }
}

// the box of sorted leaves a .. b
__device__ __forceinline__ Box range_box(const float4 *__restrict__ lv, int64_t n, int64_t a, int64_t b)
{
    Box x = box_empty();
    int64_t off = 0, c = n;
    while (a <= b) {
        if (a & 1) {
            box_join(x, lv[2 * (off + a)], lv[2 * (off + a) + 1]);
            ++a;
        }
        if (!(b & 1)) {
            box_join(x, lv[2 * (off + b)], lv[2 * (off + b) + 1]);
            --b;
        }
        a >>= 1;
        b >>= 1;
        off += c;
        c = (c + 1) >> 1;
    }
    return x;
}

// -------------------------------------------------------------------------
// Karras hierarchy
// -------------------------------------------------------------------------
// Common-prefix length of sorted leaves i and j (-1 outside [0, n)).  With
// batched scenes the key is (scene, Morton code, index): leaves of
// different scenes compare on the scene id alone (0..31), so every scene's
// leaves form one subtree; equal codes fall back to the index.
__device__ __forceinline__ int delta(const uint32_t *keys, const uint32_t *scene, int64_t n,
                                     int64_t i, int64_t j)
{
    if (j < 0 || j >= n) return -1;
    if (scene) {
        const uint32_t sa = scene[i], sb = scene[j];
        if (sa != sb) return __clz((int)(sa ^ sb));
    }
    const uint32_t a = keys[i], b = keys[j];
    if (a == b) return 64 + __clz((int)(i ^ j));      // index tie-break for equal codes
    return 32 + __clz((int)(a ^ b));
}

__global__ void lbvh_build_kernel(const uint32_t *__restrict__ keys,
                                  const uint32_t *__restrict__ scene,
                                  const int32_t *__restrict__ vals, int64_t n,
                                  const float4 *__restrict__ lv, BvhNode *__restrict__ nodes,
                                  int32_t *__restrict__ root)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    const int d = (delta(keys, scene, n, i, i + 1) - delta(keys, scene, n, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = delta(keys, scene, n, i, i - d);
    int64_t lmax = 2;
    while (delta(keys, scene, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int64_t l = 0;
    for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(keys, scene, n, i, i + (l + t) * d) > dmin) l += t;
    const int64_t j = i + l * d;
    const int dnode = delta(keys, scene, n, i, j);
    int64_t sp = 0;
    int64_t t = l;
    do {
        t = (t + 1) >> 1;
        if (delta(keys, scene, n, i, i + (sp + t) * d) > dnode) sp += t;
    } while (t > 1);
    const int64_t gamma = i + sp * d + (d < 0 ? -1 : 0);
    const int64_t lo = i < j ? i : j, hi = i < j ? j : i;
    const Box bl = range_box(lv, n, lo, gamma), br = range_box(lv, n, gamma + 1, hi);
    float4 *nd = reinterpret_cast<float4 *>(nodes + i);
    const int left = lo == gamma ? ~vals[gamma] : (int)gamma;
    const int right = hi == gamma + 1 ? ~vals[gamma + 1] : (int)(gamma + 1);
    nd[0] = make_float4(bl.lo.x, bl.lo.y, bl.lo.z, __int_as_float(left));
    nd[1] = make_float4(bl.hi.x, bl.hi.y, bl.hi.z, __int_as_float(right));
    nd[2] = make_float4(br.lo.x, br.lo.y, br.lo.z, 0.f);
    nd[3] = make_float4(br.hi.x, br.hi.y, br.hi.z, 0.f);
    if (scene) {
        // the node covering exactly one scene's leaves is that scene's root
        const uint32_t sc = scene[lo];
        if (scene[hi] == sc && (lo == 0 || scene[lo - 1] != sc) && (hi == n - 1 || scene[hi + 1] != sc))
            root[sc] = (int32_t)i;
    }
}

// Four-wide nodes for the visibility rays: wide node i holds the children of
// binary node i's children (a leaf child stands for itself), so that a ray
// makes half the dependent loads on its way down, each of four boxes.  Empty
// slots have a point box out of any ray's reach.
__global__ void lbvh_widen_kernel(const BvhNode *__restrict__ nodes, int64_t n,
                                  WideNode *__restrict__ wide)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    const BvhNode nd = nodes[i];
    WideNode w;
    int c = 0;
    auto put = [&](const float *a, const float *b, int code) {
        w.lo[c] = make_float4(a[0], a[1], a[2], __int_as_float(code));
        w.hi[c++] = make_float4(b[0], b[1], b[2], 0.f);
    };
    auto side = [&](const float *a, const float *b, int code) {
        if (code < 0) {
            put(a, b, code);
        } else {
            const BvhNode m = nodes[code];
            put(m.lmin, m.lmax, m.left);
            put(m.rmin, m.rmax, m.right);
        }
    };
    side(nd.lmin, nd.lmax, nd.left);
    side(nd.rmin, nd.rmax, nd.right);
    while (c < 4) {
        const float far[3] = {1e30f, 1e30f, 1e30f};
        put(far, far, 0);
    }
    wide[i] = w;
}

// scene of each sorted leaf: facets [foff[b], foff[b+1]) belong to scene b
__global__ void scene_keys_kernel(const int32_t *__restrict__ vals, int64_t n,
                                  const int64_t *__restrict__ foff, int B,
                                  uint32_t *__restrict__ skeys)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    skeys[i] = scene_of(foff, B, vals[i]);
}

__global__ void gather_keys_kernel(const int32_t *__restrict__ vals, int64_t n,
                                   const uint32_t *__restrict__ by_facet, uint32_t *__restrict__ keys)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) keys[i] = by_facet[vals[i]];
}

// one-facet scenes have their leaf as root; the others get theirs from the build
__global__ void scene_root_init_kernel(const int64_t *__restrict__ foff, int B,
                                       int32_t *__restrict__ root)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) root[b] = foff[b + 1] - foff[b] == 1 ? ~(int32_t)foff[b] : 0;
}

int launch_lbvh(const FacetRec *fac, const float *aabb, int64_t F, const unsigned int *bounds,
                const int64_t *foff, int B, uint32_t *keys, int32_t *vals, uint32_t *keys_tmp,
                int32_t *vals_tmp, uint32_t *temp, uint32_t *mkeys, uint32_t *skeys, float4 *levels,
                int *ticket, BvhNode *nodes, WideNode *wide, int32_t *root, cudaStream_t s)
{
    const int T = 256;
    const unsigned int G = (unsigned int)((F + T - 1) / T);
    int launches = 1;
    if (!launch_cluster_sort(fac, F, bounds, foff, B, keys, vals, skeys, s)) {
        launch_morton(fac, F, bounds, keys, vals, s);
        if (B > 1)
            cudaMemcpyAsync(mkeys, keys, (size_t)F * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
        radix_sort_pairs(keys, vals, keys_tmp, vals_tmp, temp, F, 30, s);
        launches += 3 * 4;
        if (B > 1) {
            scene_keys_kernel<<<G, T, 0, s>>>(vals, F, foff, B, skeys);
            const int p = scene_passes(B), q = p + (p & 1);
            radix_sort_pairs(skeys, vals, keys_tmp, vals_tmp, temp, F, 8 * p, s);   // stable
            gather_keys_kernel<<<G, T, 0, s>>>(vals, F, mkeys, keys);
            launches += 2 + 3 * q;
        }
    }
    if (B > 1) {
        scene_root_init_kernel<<<(B + T - 1) / T, T, 0, s>>>(foff, B, root);
        ++launches;
    }
    if (F < 2) return launches;
    leaf_levels_kernel<<<(unsigned int)((F + kLvLeaves - 1) / kLvLeaves), kLvLeaves, 0, s>>>(
        vals, aabb, F, levels, ticket);
    lbvh_build_kernel<<<(unsigned int)((F - 1 + T - 1) / T), T, 0, s>>>(
        keys, B > 1 ? skeys : nullptr, vals, F, levels, nodes, root);
    lbvh_widen_kernel<<<(unsigned int)((F - 1 + 127) / 128), 128, 0, s>>>(nodes, F, wide);
    return launches + 3;
}

}  // namespace bart
