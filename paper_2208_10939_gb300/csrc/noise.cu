// Additive white complex Gaussian noise at a given signal-to-noise ratio
// (Sec. 3.2: Gaussian white noise "with a certain signal-to-noise ratio").
//
//   x[e] += sigma * n[e],   sigma^2 = P / 10^(SNR/10),   P = mean |x|^2 of the cube
//   n[e] = (g1 + j g2) / sqrt(2),  (g1, g2) = Box-Muller(u1, u2)
//   u_i = (w_i + 1) 2^-32,  (w0, w1, w2, w3) = Philox4x32-10(ctr, key)
//   ctr = (e mod 2^32, e div 2^32, frame, 0),  key = (seed mod 2^32, seed div 2^32)
//
// Philox4x32-10 is the counter-based generator of Salmon, Moraes, Dror and
// Shaw (SC 2011), written here from its published round function.
#include <cuda_runtime.h>
#include <stdint.h>

#include "bart_internal.cuh"

namespace bart {

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned int hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const unsigned int hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

// Partial powers of the cube, one a block: two blocks on each of 152
// multiprocessors, few enough for every block of noise_add_* to sum them
// itself (one value or two a thread) instead of a launch between the two that
// does nothing else (one thread over 1024 partials took 60 us; the whole noise
// of a 12 x 128 x 256 cube takes 19 us against 76).
constexpr int kPowBlocks = 304;
constexpr int kPowThreads = 256;

// sum over the block's kPowThreads threads (the same tree whatever the
// values), in thread 0
__device__ __forceinline__ double block_sum(double v)
{
    __shared__ double s[kPowThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) s[warp] = v;
    __syncthreads();
    if (warp > 0) return 0.0;
    double t = lane < kPowThreads / 32 ? s[lane] : 0.0;
    for (int o = kPowThreads / 64; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    return t;
}

// four loads in flight a thread
template <typename C>
__global__ void __launch_bounds__(kPowThreads)
noise_power_kernel(const C *__restrict__ x, int64_t n, double *__restrict__ part)
{
    constexpr int64_t kStride = (int64_t)kPowBlocks * kPowThreads;
    double acc = 0.0;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * kPowThreads + threadIdx.x; i < n; i += kStride) {
        const C v = x[i];
        acc += (double)v.x * (double)v.x + (double)v.y * (double)v.y;
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// sigma from the partials: the same value in every block
__device__ __forceinline__ double noise_sigma(const double *__restrict__ part, int64_t n,
                                              double inv_snr)
{
    __shared__ double sigma;
    double p = 0.0;
    for (int b = threadIdx.x; b < kPowBlocks; b += kPowThreads) p += part[b];
    p = block_sum(p);
    if (threadIdx.x == 0) sigma = sqrt(p / (double)n * inv_snr);
    __syncthreads();
    return sigma;
}

__device__ __forceinline__ float2 noisy(float2 v, uint4 w, double sigma)
{
    const float u1 = ((float)w.x + 1.f) * 2.3283064e-10f;     // (w + 1) 2^-32
    const float u2 = ((float)w.y + 1.f) * 2.3283064e-10f;
    const float r = sqrtf(-2.f * logf(u1));
    float sn, cs;
    sincospif(2.f * u2, &sn, &cs);
    const float sg = (float)sigma * 0.70710678f;
    return make_float2(fmaf(sg * r, cs, v.x), fmaf(sg * r, sn, v.y));
}

__device__ __forceinline__ double2 noisy(double2 v, uint4 w, double sigma)
{
    const double u1 = ((double)w.x + 1.0) * 2.3283064365386963e-10;
    const double u2 = ((double)w.y + 1.0) * 2.3283064365386963e-10;
    const double r = sqrt(-2.0 * log(u1));
    double sn, cs;
    sincospi(2.0 * u2, &sn, &cs);
    const double sg = sigma * 0.70710678118654752;
    return make_double2(v.x + sg * r * cs, v.y + sg * r * sn);
}

template <typename C>
__global__ void __launch_bounds__(kPowThreads)
noise_add_kernel(C *__restrict__ x, int64_t n, uint2 key, unsigned int frame, double inv_snr,
                 const double *__restrict__ part)
{
    const double sigma = noise_sigma(part, n, inv_snr);
    for (int64_t e = (int64_t)blockIdx.x * kPowThreads + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * kPowThreads) {
        const uint4 w = philox4x32_10(
            make_uint4((unsigned int)e, (unsigned int)((uint64_t)e >> 32), frame, 0u), key);
        x[e] = noisy(x[e], w, sigma);
    }
}

int64_t noise_scratch_words() { return kPowBlocks; }

template <typename C>
static void add_noise(C *x, int64_t n, double inv_snr, uint2 key, unsigned int frame,
                      double *scratch, cudaStream_t s)
{
    // blocks of the sum: resident at once, so that each forms sigma once
    const int64_t blocks = (n + kPowThreads - 1) / kPowThreads, cap = 8 * 152;
    noise_power_kernel<C><<<kPowBlocks, kPowThreads, 0, s>>>(x, n, scratch);
    noise_add_kernel<C><<<(unsigned int)(blocks < cap ? blocks : cap), kPowThreads, 0, s>>>(
        x, n, key, frame, inv_snr, scratch);
}

void launch_add_noise(void *adc, int dtype, int64_t n, double snr_db, uint64_t seed,
                      unsigned int frame, double *scratch, cudaStream_t s)
{
    const uint2 key = make_uint2((unsigned int)seed, (unsigned int)(seed >> 32));
    const double inv = pow(10.0, -snr_db / 10.0);
    if (dtype == BART_C64) add_noise(static_cast<float2 *>(adc), n, inv, key, frame, scratch, s);
    else add_noise(static_cast<double2 *>(adc), n, inv, key, frame, scratch, s);
}

}  // namespace bart
