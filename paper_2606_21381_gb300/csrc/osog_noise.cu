// Sensor noise epilogue (Sec. III.C: the digitised output carries Poisson
// photon shot noise plus Gaussian read noise).
//
// out_i = (Poisson(g max(I_i, 0)) + sigma Z_i) / g, g photo-electrons per
// unit intensity, sigma the read noise in electrons, Z_i standard normal.
// Random numbers come from the counter-based Philox4x32-10 generator
// (Salmon, Moraes, Dror and Shaw, SC 2011) keyed by the 64-bit seed, one
// counter (i, round, tag) per element and round, so every element's draw is
// independent of the launch shape and reproducible.  Round 0 gives the two
// uniforms of the Box-Muller normal and the first Poisson attempt; rounds
// 1.. two more attempts each.  Poisson: inversion by sequential search for
// rates below 10, Hormann's transformed rejection with squeeze (PTRS, 1993)
// above.  Decisions and the result are those of double precision: an element
// is drawn on the FP32 pipes with bounds on its errors (osog_noise_fast.h),
// and in double precision when a bound leaves a decision open.
#include <math.h>
#include <stdint.h>

#include "osog.h"
#include "osog_noise_fast.h"

namespace osog {
namespace noise {
namespace {

constexpr uint32_t kTag = 0x6E6F6973u;  // fourth counter word
constexpr int kRounds = 64;            // attempts cap (2 per round)

__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
        const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

__device__ __forceinline__ double unit_open(uint32_t x) {
    return ((double)x + 0.5) * (1.0 / 4294967296.0);
}

__device__ __forceinline__ void uniforms(uint64_t seed, int64_t i, uint32_t round, double u[4]) {
    uint32_t c[4] = {(uint32_t)(uint64_t)i, (uint32_t)((uint64_t)i >> 32), round, kTag};
    philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
#pragma unroll
    for (int k = 0; k < 4; ++k) u[k] = unit_open(c[k]);
}

__device__ int64_t poisson(double lam, uint64_t seed, int64_t i, const double u0[4]) {
    if (!(lam > 0.0)) return 0;
    if (lam < 10.0) {
        double p = exp(-lam), F = p;
        int64_t k = 0;
        while (u0[2] > F && k < 1000) {
            ++k;
            p *= lam / (double)k;
            F += p;
        }
        return k;
    }
    const double slam = sqrt(lam), loglam = log(lam);
    const double b = 0.931 + 2.53 * slam;
    const double a = -0.059 + 0.02483 * b;
    const double invalpha = 1.1239 + 1.1328 / (b - 3.4);
    const double vr = 0.9277 - 3.6224 / (b - 2.0);
    double u[4] = {u0[0], u0[1], u0[2], u0[3]};
    for (int r = 0; r < kRounds; ++r) {
        if (r > 0) uniforms(seed, i, (uint32_t)r, u);
        for (int h = (r == 0 ? 1 : 0); h < 2; ++h) {
            const double U = u[2 * h] - 0.5, V = u[2 * h + 1];
            const double us = 0.5 - fabs(U);
            const double k = floor((2.0 * a / us + b) * U + lam + 0.43);
            if (us >= 0.07 && V <= vr) return (int64_t)k;
            if (k < 0.0 || (us < 0.013 && V > us)) continue;
            if (log(V * invalpha / (a / (us * us) + b)) <= -lam + k * loglam - lgamma(k + 1.0))
                return (int64_t)k;
        }
    }
    return (int64_t)floor(lam);
}

// One element in double precision.
__device__ __noinline__ float draw_exact(float v, int64_t i, double g, double sigma,
                                         uint64_t seed) {
    const double pi2 = 6.283185307179586476925286766559;
    double u[4];
    uniforms(seed, i, 0, u);
    const double lam = g * (v > 0.f ? (double)v : 0.0);
    const double z = sqrt(-2.0 * log(u[0])) * cos(pi2 * u[1]);
    return (float)(((double)poisson(lam, seed, i, u) + sigma * z) / g);
}

// Gain and read noise of a launch: in double precision, and as float-float
// for the FP32 draw (fast = 0: outside its range, every element is drawn in
// double precision).
struct NoiseArgs {
    const float *img;
    float *out;
    int64_t count;
    uint64_t seed;
    double g, sigma;
    ff g_ff, inv_g, sigma_ff;
    int32_t fast;
};

// One element on the FP32 pipes; false when a decision is left open.
__device__ __forceinline__ bool draw_fast(const NoiseArgs &a, float v, int64_t i, float *out) {
    uint32_t c[4] = {(uint32_t)(uint64_t)i, (uint32_t)((uint64_t)i >> 32), 0u, kTag};
    philox4x32_10(c, (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
    ff z = {0.f, 0.f};
    if (a.sigma_ff.h > 0.f) {
        if (c[0] == 0u) return false;
        z = normal_ff(c[0], c[1]);
    }
    float k = 0.f;
    if (v > 0.f) {
        ff lam = two_prod(a.g_ff.h, v);
        lam = fast_two_sum(lam.h, f_fma(a.g_ff.l, v, lam.l));
        // below 10 inverts; the rate is exact when the gain has 24 bits
        const float side = f_add(f_sub(lam.h, 10.f), lam.l);
        if (a.g_ff.l != 0.f && fabsf(side) < 1e-10f) return false;
        if (side < 0.f) {
            if (poisson_small(lam.h, c[2], &k) != kYes) return false;
        } else {
            if (!(lam.h < 4194304.f)) return false;
            const Ptrs p = ptrs_of(lam);
            int s = ptrs_attempt(p, c[2], c[3], &k);
            for (uint32_t r = 1; s == kNo; ++r) {
                if (r == kRounds) return false;
                c[0] = (uint32_t)(uint64_t)i;
                c[1] = (uint32_t)((uint64_t)i >> 32);
                c[2] = r;
                c[3] = kTag;
                philox4x32_10(c, (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
                s = ptrs_attempt(p, c[0], c[1], &k);
                if (s == kNo) s = ptrs_attempt(p, c[2], c[3], &k);
            }
            if (s != kYes) return false;
        }
    }
    return noisy_value(k, a.sigma_ff, z, a.inv_g, out);
}

// Bound by instruction issue: about 900 warp instructions per 32 elements
// (Philox 100 a round, the normal 155, about 80 per rejection attempt, and a
// warp runs as many attempts as its unluckiest lane needs).  All of it in
// double precision was bound by the FP64 pipe, 11.54 ms for 16 images of
// 1024 x 1024 at 1,000 photons; this kernel takes 0.574 ms, with the same bits.
__global__ void __launch_bounds__(256) k_sensor_noise(const __grid_constant__ NoiseArgs a) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float v = a.img[i];
        float y;
        if (!(a.fast && draw_fast(a, v, i, &y))) y = draw_exact(v, i, a.g, a.sigma, a.seed);
        a.out[i] = y;
    }
}

}  // namespace
}  // namespace noise
}  // namespace osog

extern "C" int osog_sensor_noise(const float *image, int64_t count, double photons_per_unit,
                                 double read_sigma, uint64_t seed, float *out,
                                 osog_stream_t stream) {
    if (count < 0 || (count > 0 && (!image || !out))) return OSOG_ERR_INVALID_ARG;
    if (!(photons_per_unit > 0.0) || !(photons_per_unit <= 1e12) || !(read_sigma >= 0.0) ||
        !isfinite(read_sigma))
        return OSOG_ERR_INVALID_ARG;
    if (count == 0) return OSOG_OK;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return OSOG_ERR_CUDA;
    const int64_t want = (count + 255) / 256;
    const int blocks = (int)(want < (int64_t)sms * 8 ? want : (int64_t)sms * 8);
    osog::noise::NoiseArgs a;
    a.img = image;
    a.out = out;
    a.count = count;
    a.seed = seed;
    a.g = photons_per_unit;
    a.sigma = read_sigma;
    // the range where no float-float part under- or overflows
    a.fast = photons_per_unit >= 1e-6 && (read_sigma == 0.0 || (read_sigma >= 1e-6 && read_sigma <= 1e6));
    a.g_ff = osog::noise::split(photons_per_unit);
    a.inv_g = osog::noise::split(1.0 / photons_per_unit);
    a.sigma_ff = osog::noise::split(read_sigma);
    osog::noise::k_sensor_noise<<<blocks, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(a);
    return cudaGetLastError() == cudaSuccess ? OSOG_OK : OSOG_ERR_CUDA;
}
