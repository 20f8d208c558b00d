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
        const uint64_t p0 = (uint64_t)0xD2511F53u * c[0], p1 = (uint64_t)0xCD9E8D57u * c[2];
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c[1] ^ k0, n2 = (uint32_t)(p0 >> 32) ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = (uint32_t)p1;
        c[2] = n2;
        c[3] = (uint32_t)p0;
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
// for the FP32 draw.
struct NoiseArgs {
    const float *img;
    float *out;
    int64_t count;
    uint64_t seed;
    double g, sigma;
    ff g_ff, inv_g, sigma_ff;
};

// Gains and read noises outside the FP32 draw's range: every element in double
// precision.
__global__ void __launch_bounds__(256) k_sensor_noise_exact(const __grid_constant__ NoiseArgs a) {
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < a.count; i += (int64_t)gridDim.x * 256)
        a.out[i] = draw_exact(a.img[i], i, a.g, a.sigma, a.seed);
}

// An element whose first rejection attempt was not accepted at once: its
// candidate (n = 0: rejected already), its rate, sigma z and place in the tile.
struct Pending {
    float k;
    uint32_t n, xv;
    ff lam, noise;
    uint32_t at;
};

// The attempts of the rounds after the first one: kYes with the count or
// kUndecided.
__device__ __forceinline__ int more_attempts(const NoiseArgs &a, ff lam, int64_t i, float *k) {
    const Ptrs p = ptrs_of(lam);
    int s = kNo;
    for (uint32_t r = 1; s == kNo && r < kRounds; ++r) {
        uint32_t c[4] = {(uint32_t)(uint64_t)i, (uint32_t)((uint64_t)i >> 32), r, kTag};
        philox4x32_10(c, (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
        s = ptrs_attempt(p, c[0], c[1], k);
        if (s == kNo) s = ptrs_attempt(p, c[2], c[3], k);
    }
    return s == kNo ? kUndecided : s;
}

constexpr int kNoiseThreads = 256, kPerThread = 4;
constexpr int kNoiseCtas = 4;  // resident on an SM

// A CTA draws tiles of PER elements a thread in three sweeps.  Every element gets its
// normal and the quick part of its first attempt (about 68% of rates above ten
// end there); the others queue up in shared memory and take their acceptance
// test as full warps; those it rejects queue up again for further attempts.  A
// warp would otherwise run every step for its unluckiest lane.  Undecided
// elements collect over the tiles and are drawn in double precision by the CTA
// together, as are rates from 2^22 (of 1,048,576 such pixels 830 us; a thread per element,
// as in k_sensor_noise_exact, 739).
//
// PER = kPerThread, or 1 where every such tile has a place on the chip: an element
// drawn in double precision costs as much as a hundred others, and 4,096 of 10^8
// photons took 114 us in four tiles, 33 in sixteen; 65,536 at 1,000 photons 23.0 and
// 20.1.
//
// Bound by instruction issue.  16 images of 1024 x 1024 at 1,000 photons (the
// same bits): all in double precision 11.54 ms, bound by the FP64 pipe; on the
// FP32 pipes without queues 0.560 ms, about 1,000 warp instructions per 32
// elements; this kernel 0.45 ms, about 740.
template <int PER>
__global__ void __launch_bounds__(kNoiseThreads, kNoiseCtas)
k_sensor_noise(const __grid_constant__ NoiseArgs a) {
    constexpr int kTile = kNoiseThreads * PER;
    __shared__ Pending queue[kTile];
    __shared__ uint16_t again[kTile];
    __shared__ int64_t open[kTile + kNoiseThreads];
    __shared__ int npend, nagain, nopen;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    if (threadIdx.x == 0) npend = nagain = nopen = 0;
    __syncthreads();
    // a warp's lanes with `take` reserve consecutive places of a list
    auto reserve = [&](int *count, bool take) {
        const unsigned m = __ballot_sync(0xffffffffu, take);
        int base = 0;
        if (lane == 0 && m) base = atomicAdd(count, __popc(m));
        return __shfl_sync(0xffffffffu, base, 0) + __popc(m & below);
    };
    const int64_t tiles = (a.count + kTile - 1) / kTile;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t i0 = tile * kTile;
        for (int u = 0; u < PER; ++u) {
            const int at = u * kNoiseThreads + threadIdx.x;
            const int64_t i = i0 + at;
            Pending e;
            bool pend = false, undecided = false;
            if (i < a.count) {
                const float v = a.img[i];
                uint32_t c[4] = {(uint32_t)(uint64_t)i, (uint32_t)((uint64_t)i >> 32), 0u, kTag};
                philox4x32_10(c, (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
                e.noise = {0.f, 0.f};
                if (a.sigma_ff.h > 0.f) {
                    undecided = undecided || c[0] == 0u;
                    e.noise = mul_lazy(a.sigma_ff, normal_ff(c[0], c[1]));
                }
                e.k = 0.f;
                if (v > 0.f) {
                    e.lam = two_prod(a.g_ff.h, v);
                    e.lam = fast_two_sum(e.lam.h, f_fma(a.g_ff.l, v, e.lam.l));
                    // below 10 inverts; the rate is exact when the gain has 24 bits
                    const float side = f_add(f_sub(e.lam.h, 10.f), e.lam.l);
                    if (a.g_ff.l != 0.f && fabsf(side) < 1e-10f) undecided = true;
                    if (side < 0.f) {
                        if (!undecided) undecided = poisson_small(e.lam.h, c[2], &e.k) != kYes;
                    } else if (!(e.lam.h < 4194304.f)) {
                        undecided = true;
                    } else {
                        const Ptrs p = ptrs_of(e.lam);
                        e.n = 0u;
                        e.xv = c[3];
                        int s = ptrs_candidate(p, c[2], c[3], &e.k, &e.n);
                        if (s == kYes) s = ptrs_quick(p, e.n, c[3]);
                        pend = s == kNo;
                        undecided = undecided || s == kUndecided;
                    }
                }
                if (undecided) {
                    pend = false;
                } else if (!pend) {
                    float y;
                    undecided = !noisy_value(e.k, e.noise, a.inv_g, &y);
                    if (!undecided) a.out[i] = y;
                }
                e.at = (uint32_t)at;
            }
            const int q = reserve(&npend, pend);
            if (pend) queue[q] = e;
            if (__any_sync(0xffffffffu, undecided)) {
                const int o = reserve(&nopen, undecided);
                if (undecided) open[o] = i;
            }
        }
        __syncthreads();
        const int np = npend;
        for (int q = threadIdx.x; q - lane < np; q += kNoiseThreads) {
            int s = kYes;
            int64_t i = 0;
            if (q < np) {
                const Pending e = queue[q];
                i = i0 + e.at;
                s = e.n ? ptrs_accept_float(e.lam, e.k, e.n, e.xv) : kNo;
                if (s == kYes) {
                    float y;
                    if (noisy_value(e.k, e.noise, a.inv_g, &y))
                        a.out[i] = y;
                    else
                        s = kUndecided;
                }
            }
            const int r = reserve(&nagain, s == kNo);
            if (s == kNo) again[r] = (uint16_t)q;
            const int o = reserve(&nopen, s == kUndecided);
            if (s == kUndecided) open[o] = i;
        }
        __syncthreads();
        const int na = nagain;
        for (int q = threadIdx.x; q - lane < na; q += kNoiseThreads) {
            bool undecided = false;
            int64_t i = 0;
            if (q < na) {
                const Pending e = queue[again[q]];
                i = i0 + e.at;
                float k, y;
                undecided = more_attempts(a, e.lam, i, &k) != kYes || !noisy_value(k, e.noise, a.inv_g, &y);
                if (!undecided) a.out[i] = y;
            }
            const int o = reserve(&nopen, undecided);
            if (undecided) open[o] = i;
        }
        __syncthreads();
        // room for a whole tile stays in the list of undecided elements
        if (nopen >= kNoiseThreads) {
            for (int o = threadIdx.x; o < nopen; o += kNoiseThreads)
                a.out[open[o]] = draw_exact(a.img[open[o]], open[o], a.g, a.sigma, a.seed);
            __syncthreads();
            if (threadIdx.x == 0) nopen = 0;
        }
        if (threadIdx.x == 0) npend = nagain = 0;
        __syncthreads();
    }
    for (int o = threadIdx.x; o < nopen; o += kNoiseThreads)
        a.out[open[o]] = draw_exact(a.img[open[o]], open[o], a.g, a.sigma, a.seed);
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
    osog::noise::NoiseArgs a;
    a.img = image;
    a.out = out;
    a.count = count;
    a.seed = seed;
    a.g = photons_per_unit;
    a.sigma = read_sigma;
    const cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int64_t rows = (count + osog::noise::kNoiseThreads - 1) / osog::noise::kNoiseThreads;
    // the range where no float-float part under- or overflows
    const bool fast = photons_per_unit >= 1e-6 && (read_sigma == 0.0 || (read_sigma >= 1e-6 && read_sigma <= 1e6));
    a.g_ff = osog::noise::split(photons_per_unit);
    a.inv_g = osog::noise::split(1.0 / photons_per_unit);
    a.sigma_ff = osog::noise::split(read_sigma);
    if (!fast) {
        const int64_t most = (int64_t)sms * 8;
        osog::noise::k_sensor_noise_exact<<<(unsigned)(rows < most ? rows : most), 256, 0, st>>>(a);
        return cudaGetLastError() == cudaSuccess ? OSOG_OK : OSOG_ERR_CUDA;
    }
    const int64_t ctas = (int64_t)sms * osog::noise::kNoiseCtas;
    if (rows <= ctas) {
        osog::noise::k_sensor_noise<1><<<(unsigned)rows, osog::noise::kNoiseThreads, 0, st>>>(a);
    } else {
        const int64_t tiles = (rows + osog::noise::kPerThread - 1) / osog::noise::kPerThread;
        osog::noise::k_sensor_noise<osog::noise::kPerThread>
            <<<(unsigned)(tiles < ctas ? tiles : ctas), osog::noise::kNoiseThreads, 0, st>>>(a);
    }
    return cudaGetLastError() == cudaSuccess ? OSOG_OK : OSOG_ERR_CUDA;
}
