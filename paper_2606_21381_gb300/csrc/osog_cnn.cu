// Convolutions of the learned warm start as implicit GEMMs on the tensor
// cores (BF16 operands, FP32 accumulation): the C ABI, the warp-level MMA
// kernels (mma.sync).  The convolutions and their gradients run on tcgen05 in
// osog_conv_tma.cu unless the warp-level engine is selected or a forward
// reduction is too short to feed it.
//
//   forward  Y[m = (n,p,q)][k]   = sum_{j = (r,s,c)} X(im2col)[m][j] W[k][j]
//   data     dX[m = (n,h,w)][c]  = sum_{j = (r,s,k)} dY(gathered)[m][j] Wt[c][j]
//   filter   dW[k][j = (r,s,c)]  = sum_{m = (n,p,q)} dY[m][k] X(im2col)[m][j]
//
// A CTA computes a 64 x 64 tile of the product from 32-wide slices of the
// reduction: both operands are gathered from NHWC tensors (8 channels per
// 16-byte vector, zero outside the image or for strides that skip a tap),
// staged in shared memory as [row][reduction] and fed to mma.m16n8k16
// through ldmatrix; four warps each own a 32 x 32 sub-tile.  The filter
// gradient splits its pixel reduction across CTAs and sums the partial tiles
// in a fixed order, so every result is bitwise reproducible.
#include <cuda_bf16.h>

#include "osog_cnn.h"
#include "osog_conv_tma.h"

namespace osog {
namespace cnn {
namespace {

constexpr int BM = 64, BN = 64, BK = 32, LDS = BK + 8;  // smem row: 40 bf16 = 80 bytes
constexpr int NT = 128;
constexpr int kSplitPixels = 2048;  // pixels per CTA in the filter-gradient reduction

// kDgrad2: the data gradient of a stride-2 convolution for the input
// pixels of one parity class (h mod 2, w mod 2), reduced over the taps that
// reach them only (the other taps of that class are zero).
enum Pass { kFwd = 0, kDgrad = 1, kWgrad = 2, kDgrad2 = 3 };

struct Args {
    Geo g;
    const __nv_bfloat16 *x;     // fwd: X, dgrad: dY, wgrad: dY
    const __nv_bfloat16 *w;     // fwd: W [K][RSC], dgrad: Wt [C][RSK], wgrad: X
    const float *bias;
    const __nv_bfloat16 *mask;  // dgrad: activation whose ReLU derivative applies
    __nv_bfloat16 *y;
    float *y32;
    float *part;                // wgrad partial tiles [splits][M][N]
    int relu;
    int M, Ncols, Kred;         // GEMM sizes
    // kDgrad2: parity class, its pixel grid and its taps
    int ph, pw, Hc, Wc, nr, ns;
    int rtap[4], stap[4];
};

__device__ __forceinline__ uint4 zero4() { return make_uint4(0u, 0u, 0u, 0u); }

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void ldsm_x4(unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3,
                                        const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(smem_u32(p)));
}

__device__ __forceinline__ void ldsm_x4_t(unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3,
                                          const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(smem_u32(p)));
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------- gathers
// Forward A: 8 reduction entries j..j+7 (same tap, 8 channels) of output
// pixel m.
__device__ __forceinline__ const __nv_bfloat16 *fwd_a_src(const Args &a, int m, int j) {
    const Geo &g = a.g;
    if (m >= a.M || j >= a.Kred) return nullptr;
    const int q = m % g.Q, t = m / g.Q, p = t % g.P, n = t / g.P;
    const int rs = j / g.C, c = j - rs * g.C, r = rs / g.S, s = rs - r * g.S;
    const int h = p * g.stride + r - g.pad, w = q * g.stride + s - g.pad;
    if (h < 0 || h >= g.H || w < 0 || w >= g.W) return nullptr;
    return a.x + (((size_t)n * g.H + h) * g.W + w) * g.C + c;
}
__device__ __forceinline__ uint4 fwd_a(const Args &a, int m, int j) {
    const __nv_bfloat16 *p = fwd_a_src(a, m, j);
    return p ? *reinterpret_cast<const uint4 *>(p) : zero4();
}

// Data-gradient A: dY at the output pixel that tap (r, s) of input pixel m
// reads, 8 output channels; zero where the stride skips it.
__device__ __forceinline__ const __nv_bfloat16 *dgrad_a_src(const Args &a, int m, int j) {
    const Geo &g = a.g;
    if (m >= a.M || j >= a.Kred) return nullptr;
    const int w = m % g.W, t = m / g.W, h = t % g.H, n = t / g.H;
    const int rs = j / g.K, k = j - rs * g.K, r = rs / g.S, s = rs - r * g.S;
    const int hp = h + g.pad - r, wq = w + g.pad - s;
    if (hp < 0 || wq < 0 || hp % g.stride || wq % g.stride) return nullptr;
    const int p = hp / g.stride, q = wq / g.stride;
    if (p >= g.P || q >= g.Q) return nullptr;
    return a.x + (((size_t)n * g.P + p) * g.Q + q) * g.K + k;
}
__device__ __forceinline__ uint4 dgrad_a(const Args &a, int m, int j) {
    const __nv_bfloat16 *p = dgrad_a_src(a, m, j);
    return p ? *reinterpret_cast<const uint4 *>(p) : zero4();
}

// Stride-2 data gradient, parity class (ph, pw): class pixel m = (n, i, j)
// is input pixel (n, 2 i + ph, 2 j + pw); reduction entry (tap, k) with tap
// = (ri, si) reads dY at ((h + pad - r) / 2, (w + pad - s) / 2), which the
// class's taps make exact.
__device__ __forceinline__ const __nv_bfloat16 *dgrad2_a_src(const Args &a, int m, int j) {
    const Geo &g = a.g;
    if (m >= a.M || j >= a.Kred) return nullptr;
    const int wi = m % a.Wc, t = m / a.Wc, hi = t % a.Hc, n = t / a.Hc;
    const int tap = j / g.K, k = j - tap * g.K, ri = tap / a.ns, si = tap - ri * a.ns;
    const int p = (2 * hi + a.ph + g.pad - a.rtap[ri]) >> 1;
    const int q = (2 * wi + a.pw + g.pad - a.stap[si]) >> 1;
    if (p < 0 || q < 0 || p >= g.P || q >= g.Q) return nullptr;
    return a.x + (((size_t)n * g.P + p) * g.Q + q) * g.K + k;
}
__device__ __forceinline__ uint4 dgrad2_a(const Args &a, int m, int j) {
    const __nv_bfloat16 *p = dgrad2_a_src(a, m, j);
    return p ? *reinterpret_cast<const uint4 *>(p) : zero4();
}

// Filters reordered [C][R][S][K], row c, reduction entry (tap, k) of the
// class's taps.
__device__ __forceinline__ const __nv_bfloat16 *dgrad2_b_src(const Args &a, int c, int j) {
    const Geo &g = a.g;
    if (c >= a.Ncols || j >= a.Kred) return nullptr;
    const int tap = j / g.K, k = j - tap * g.K, ri = tap / a.ns, si = tap - ri * a.ns;
    const int rs = a.rtap[ri] * g.S + a.stap[si];
    return a.w + ((size_t)c * g.R * g.S + rs) * g.K + k;
}
__device__ __forceinline__ uint4 dgrad2_b(const Args &a, int c, int j) {
    const __nv_bfloat16 *p = dgrad2_b_src(a, c, j);
    return p ? *reinterpret_cast<const uint4 *>(p) : zero4();
}

// Row-major operand rows (8 consecutive reduction entries of row r).
__device__ __forceinline__ const __nv_bfloat16 *rows_src(const __nv_bfloat16 *base, int rows, int ld,
                                                         int r, int j) {
    if (r >= rows || j >= ld) return nullptr;
    return base + (size_t)r * ld + j;
}
__device__ __forceinline__ uint4 rows_b(const __nv_bfloat16 *base, int rows, int ld, int r, int j) {
    const __nv_bfloat16 *p = rows_src(base, rows, ld, r, j);
    return p ? *reinterpret_cast<const uint4 *>(p) : zero4();
}

// Filter gradient: A(k, pixel) = dY[pixel][k..k+7] (a vector across 8 rows
// of the A tile); B(j, pixel) = X(im2col)[pixel][j..j+7] (across 8 rows of
// the B tile).
__device__ __forceinline__ uint4 wgrad_a(const Args &a, int k, int pix) {
    if (k >= a.M || pix >= a.Kred) return zero4();
    return *reinterpret_cast<const uint4 *>(a.x + (size_t)pix * a.g.K + k);
}
__device__ __forceinline__ uint4 wgrad_b(const Args &a, int j, int pix) {
    const Geo &g = a.g;
    if (j >= a.Ncols || pix >= a.Kred) return zero4();
    const int q = pix % g.Q, t = pix / g.Q, p = t % g.P, n = t / g.P;
    const int rs = j / g.C, c = j - rs * g.C, r = rs / g.S, s = rs - r * g.S;
    const int h = p * g.stride + r - g.pad, w = q * g.stride + s - g.pad;
    if (h < 0 || h >= g.H || w < 0 || w >= g.W) return zero4();
    return *reinterpret_cast<const uint4 *>(a.w + (((size_t)n * g.H + h) * g.W + w) * g.C + c);
}

// Output of two adjacent columns (col, col + 1) of GEMM row `row`.
template <int PASS>
__device__ __forceinline__ void epilogue_pair(const Args &a, int row, int col, float v0, float v1) {
    size_t o = (size_t)row * a.Ncols + col;
    if constexpr (PASS == kDgrad2) {  // class pixel -> input pixel
        const int wi = row % a.Wc, t = row / a.Wc, hi = t % a.Hc, n = t / a.Hc;
        o = (((size_t)n * a.g.H + 2 * hi + a.ph) * a.g.W + 2 * wi + a.pw) * a.Ncols + col;
    }
    if constexpr (PASS == kFwd) {
        v0 += a.bias[col];
        v1 += a.bias[col + 1];
        if (a.relu) {
            v0 = fmaxf(v0, 0.f);
            v1 = fmaxf(v1, 0.f);
        }
        *reinterpret_cast<__nv_bfloat162 *>(a.y + o) = __floats2bfloat162_rn(v0, v1);
        if (a.y32) *reinterpret_cast<float2 *>(a.y32 + o) = make_float2(v0, v1);
    } else if constexpr (PASS == kDgrad || PASS == kDgrad2) {
        if (a.mask) {
            const __nv_bfloat162 mk = *reinterpret_cast<const __nv_bfloat162 *>(a.mask + o);
            if (!(__bfloat162float(mk.x) > 0.f)) v0 = 0.f;
            if (!(__bfloat162float(mk.y) > 0.f)) v1 = 0.f;
        }
        *reinterpret_cast<__nv_bfloat162 *>(a.y + o) = __floats2bfloat162_rn(v0, v1);
    } else {
        *reinterpret_cast<float2 *>(a.part + (size_t)blockIdx.z * a.M * a.Ncols + o) =
            make_float2(v0, v1);
    }
}

// ---------------------------------------------------------------- GEMM
// The filter gradient reduces over pixels, the outer index of both NHWC
// operands: its tiles are kept as [pixel][row] (16-byte vector stores) and
// its fragments are read transposed (ldmatrix .trans).
constexpr int LDT = BM + 8;  // 72 bf16 = 144 bytes per pixel row

template <int PASS>
__global__ void __launch_bounds__(NT) k_conv_gemm(const __grid_constant__ Args a) {
    constexpr bool T = PASS == kWgrad;
    __shared__ __align__(16) __nv_bfloat16 smA[2 * (T ? BK * LDT : BM * LDS)];
    __shared__ __align__(16) __nv_bfloat16 smB[2 * (T ? BK * LDT : BN * LDS)];
    // element (row, k) of stage buf: [row][k] tiles, or [k][row] for T
    auto As = [&](int buf, int row, int k) -> __nv_bfloat16 * {
        return T ? smA + buf * BK * LDT + k * LDT + row : smA + buf * BM * LDS + row * LDS + k;
    };
    auto Bs = [&](int buf, int row, int k) -> __nv_bfloat16 * {
        return T ? smB + buf * BK * LDT + k * LDT + row : smB + buf * BN * LDS + row * LDS + k;
    };
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    int kbeg = 0, kend = a.Kred;
    if constexpr (PASS == kWgrad) {
        kbeg = blockIdx.z * kSplitPixels;
        kend = min(a.Kred, kbeg + kSplitPixels);
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wm = warp & 1, wn = warp >> 1;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[i][j][k] = 0.f;
    uint4 ra[2], rb[2];

    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int v = tid + i * NT;
            if constexpr (PASS == kWgrad) {
                const int kc = v & 31, rg = v >> 5;
                ra[i] = wgrad_a(a, m0 + rg * 8, k0 + kc);
                rb[i] = wgrad_b(a, n0 + rg * 8, k0 + kc);
            } else {
                const int row = v >> 2, kv = v & 3;
                if constexpr (PASS == kDgrad2) {
                    ra[i] = dgrad2_a(a, m0 + row, k0 + kv * 8);
                    rb[i] = dgrad2_b(a, n0 + row, k0 + kv * 8);
                } else {
                    ra[i] = PASS == kFwd ? fwd_a(a, m0 + row, k0 + kv * 8)
                                         : dgrad_a(a, m0 + row, k0 + kv * 8);
                    rb[i] = rows_b(a.w, a.Ncols, a.Kred, n0 + row, k0 + kv * 8);
                }
            }
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int v = tid + i * NT;
            if constexpr (PASS == kWgrad) {
                const int kc = v & 31, rg = v >> 5;
                *reinterpret_cast<uint4 *>(As(buf, rg * 8, kc)) = ra[i];
                *reinterpret_cast<uint4 *>(Bs(buf, rg * 8, kc)) = rb[i];
            } else {
                const int row = v >> 2, kv = v & 3;
                *reinterpret_cast<uint4 *>(As(buf, row, kv * 8)) = ra[i];
                *reinterpret_cast<uint4 *>(Bs(buf, row, kv * 8)) = rb[i];
            }
        }
    };

    load(kbeg);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = kbeg; k0 < kend; k0 += BK) {
        const bool more = k0 + BK < kend;
        if (more) load(k0 + BK);  // global loads in flight during the MMAs
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            unsigned af[2][4], bf[4][2];
            const int q = lane >> 3, r8 = lane & 7;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                if constexpr (T)  // 8x8 blocks (m 0-7 | 8-15) x (k 0-7 | 8-15), stored [k][m]
                    ldsm_x4_t(af[mt][0], af[mt][1], af[mt][2], af[mt][3],
                              As(buf, wm * 32 + mt * 16 + (q & 1) * 8, kk + r8 + (q >> 1) * 8));
                else
                    ldsm_x4(af[mt][0], af[mt][1], af[mt][2], af[mt][3],
                            As(buf, wm * 32 + mt * 16 + (lane & 15), kk + (lane >> 4) * 8));
            }
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                if constexpr (T)  // (n 0-7, k 0-7), (n 0-7, k 8-15), (n 8-15, k 0-7), (n 8-15, k 8-15)
                    ldsm_x4_t(bf[2 * np][0], bf[2 * np][1], bf[2 * np + 1][0], bf[2 * np + 1][1],
                              Bs(buf, wn * 32 + np * 16 + (q >> 1) * 8, kk + r8 + (q & 1) * 8));
                else
                    ldsm_x4(bf[2 * np][0], bf[2 * np][1], bf[2 * np + 1][0], bf[2 * np + 1][1],
                            Bs(buf, wn * 32 + np * 16 + (lane & 7) + (lane >> 4) * 8,
                               kk + ((lane >> 3) & 1) * 8));
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) mma_bf16(acc[mt][nt], af[mt], bf[nt][0], bf[nt][1]);
        }
        if (more) store(buf ^ 1);
        __syncthreads();
        buf ^= 1;
    }

    // epilogue: thread holds rows (lane / 4) and (lane / 4 + 8) of each
    // 16 x 8 tile, columns 2 (lane % 4) and +1
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int row = m0 + wm * 32 + mt * 16 + (lane >> 2) + half * 8;
                const int col = n0 + wn * 32 + nt * 8 + (lane & 3) * 2;
                if (row >= a.M || col >= a.Ncols) continue;
                epilogue_pair<PASS>(a, row, col, acc[mt][nt][half * 2], acc[mt][nt][half * 2 + 1]);
            }
}

// Sum of the filter-gradient partial tiles over the pixel splits, in split
// order.
// out[i] = sum over z of part[z][i] for i < count, in a fixed order: a CTA
// takes 32 consecutive outputs (one per lane); warp w adds the splits z = w,
// w + kSumWarps, ... in ascending order (four loads in flight per lane), and
// warp 0 adds the warps' sums in warp order.  Coalesced 128-byte loads and
// count / 32 CTAs, where one thread per output walked every split alone.
constexpr int kSumWarps = 16;

__global__ void __launch_bounds__(32 * kSumWarps)
k_sum_splits(const float *part, int splits, int64_t count, float *out) {
    __shared__ float red[kSumWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    float s = 0.f;
    if (i < count) {
        int z = warp;
        for (; z + 3 * kSumWarps < splits; z += 4 * kSumWarps) {
            const float a0 = part[(int64_t)z * count + i];
            const float a1 = part[(int64_t)(z + kSumWarps) * count + i];
            const float a2 = part[(int64_t)(z + 2 * kSumWarps) * count + i];
            const float a3 = part[(int64_t)(z + 3 * kSumWarps) * count + i];
            s += a0;
            s += a1;
            s += a2;
            s += a3;
        }
        for (; z < splits; z += kSumWarps) s += part[(int64_t)z * count + i];
    }
    red[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && i < count) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kSumWarps; ++w) t += red[w][lane];
        out[i] = t;
    }
}

// Launch of k_sum_splits over count outputs.
static void sum_splits(const float *part, int splits, int64_t count, float *out, cudaStream_t st) {
    if (count > 0)
        k_sum_splits<<<(unsigned)((count + 31) / 32), 32 * kSumWarps, 0, st>>>(part, splits, count, out);
}

// Partial bias gradients for K dividing 256: CTA c sums the pixels
// [c chunk, (c + 1) chunk), chunk = kBiasIter 256 / K, with 256 / K pixel
// lanes per channel (coalesced rows), then a fixed tree over the lanes:
// part[c][k].
constexpr int kBiasIter = 64;
__host__ __device__ constexpr int bias_chunk(int K) { return kBiasIter * (256 / K); }
__global__ void k_bias_partial(const __nv_bfloat16 *dy, int64_t pixels, int K, float *part) {
    __shared__ float red[256];
    const int lanes = 256 / K, t = threadIdx.x, k = t % K, pl = t / K;
    const int64_t p0 = (int64_t)blockIdx.x * bias_chunk(K);
    const int64_t p1 = p0 + bias_chunk(K) < pixels ? p0 + bias_chunk(K) : pixels;
    float acc = 0.f;
    for (int64_t p = p0 + pl; p < p1; p += lanes) acc += __bfloat162float(dy[p * K + k]);
    red[t] = acc;
    __syncthreads();
    for (int d = lanes / 2; d > 0; d >>= 1) {
        if (pl < d) red[t] += red[t + d * K];
        __syncthreads();
    }
    if (pl == 0) part[(int64_t)blockIdx.x * K + k] = red[t];
}

// dbias[k] = sum over pixels of dy[pixel][k] for other K: one CTA per
// channel, a fixed strided partition and a fixed tree.
__global__ void k_bias_grad(const __nv_bfloat16 *dy, int64_t pixels, int K, float *db) {
    __shared__ float red[256];
    const int k = blockIdx.x;
    float s = 0.f;
    for (int64_t p = threadIdx.x; p < pixels; p += blockDim.x) s += __bfloat162float(dy[p * K + k]);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int d = blockDim.x / 2; d > 0; d >>= 1) {
        if (threadIdx.x < d) red[threadIdx.x] += red[threadIdx.x + d];
        __syncthreads();
    }
    if (threadIdx.x == 0) db[k] = red[0];
}

// W [K][R][S][C] -> Wt [C][R][S][K].
__global__ void k_filter_transpose(const __nv_bfloat16 *w, int K, int RS, int C, __nv_bfloat16 *wt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t total = (int64_t)K * RS * C;
    if (i >= total) return;
    const int c = i % C;
    const int64_t t = i / C;
    const int rs = t % RS, k = t / RS;
    wt[((int64_t)c * RS + rs) * K + k] = w[i];
}

__global__ void k_relu_backward(const __nv_bfloat16 *dy, const __nv_bfloat16 *act, int64_t n,
                                __nv_bfloat16 *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = __bfloat162float(act[i]) > 0.f ? dy[i] : __float2bfloat16(0.f);
}

}  // namespace
}  // namespace cnn
}  // namespace osog

using namespace osog::cnn;

namespace {

bool shape_ok(const osog_conv_shape_t *s) {
    return s && s->N > 0 && s->H > 0 && s->W > 0 && s->C > 0 && s->C % 8 == 0 && s->K > 0 &&
           s->K % 8 == 0 && s->R > 0 && s->S > 0 && s->R <= 8 && s->S <= 8 &&
           (s->stride == 1 || s->stride == 2) &&
           s->pad >= 0 && s->H + 2 * s->pad >= s->R && s->W + 2 * s->pad >= s->S;
}

Geo geo_of(const osog_conv_shape_t *s) {
    Geo g;
    g.N = s->N;
    g.H = s->H;
    g.W = s->W;
    g.C = s->C;
    g.K = s->K;
    g.R = s->R;
    g.S = s->S;
    g.stride = s->stride;
    g.pad = s->pad;
    g.P = (s->H + 2 * s->pad - s->R) / s->stride + 1;
    g.Q = (s->W + 2 * s->pad - s->S) / s->stride + 1;
    return g;
}

int splits_of(const Geo &g) {
    const int64_t pix = (int64_t)g.N * g.P * g.Q;
    return (int)((pix + kSplitPixels - 1) / kSplitPixels);
}

int status_of(cudaError_t e) { return e == cudaSuccess ? OSOG_OK : OSOG_ERR_CUDA; }

// Engine of the forward and data-gradient convolutions: the tcgen05 kernel
// (1, default) or the warp-level MMA kernel (0).
int g_use_tcgen05 = 1;

const __nv_bfloat16 *bf(const uint16_t *p) { return reinterpret_cast<const __nv_bfloat16 *>(p); }
__nv_bfloat16 *bf(uint16_t *p) { return reinterpret_cast<__nv_bfloat16 *>(p); }

}  // namespace

extern "C" {

int32_t osog_conv_out_h(const osog_conv_shape_t *s) { return shape_ok(s) ? geo_of(s).P : 0; }
int32_t osog_conv_out_w(const osog_conv_shape_t *s) { return shape_ok(s) ? geo_of(s).Q : 0; }

int osog_conv2d_forward(const osog_conv_shape_t *shape, const uint16_t *x, const uint16_t *w,
                        const float *bias, int32_t relu, uint16_t *y, float *y_f32,
                        osog_stream_t stream) {
    if (!shape_ok(shape) || !x || !w || !bias || !y) return OSOG_ERR_INVALID_ARG;
    Args a{};
    a.g = geo_of(shape);
    a.x = bf(x);
    a.w = bf(w);
    a.bias = bias;
    a.y = bf(y);
    a.y32 = y_f32;
    a.relu = relu;
    a.M = a.g.N * a.g.P * a.g.Q;
    a.Ncols = a.g.K;
    a.Kred = a.g.R * a.g.S * a.g.C;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // reductions shorter than 128 stay on the warp-level MMA (the 8-channel
    // first layer and the 1 x 1 head)
    if (g_use_tcgen05 && a.Kred >= 128) {
        const cudaError_t e = conv_forward_tma(a.g, x, w, bias, relu != 0, y, y_f32, st);
        if (e != cudaErrorNotSupported) return status_of(e);
    }
    dim3 grid((a.M + BM - 1) / BM, (a.Ncols + BN - 1) / BN);
    k_conv_gemm<kFwd><<<grid, NT, 0, st>>>(a);
    return status_of(cudaGetLastError());
}

int osog_conv2d_backward_data(const osog_conv_shape_t *shape, const uint16_t *dy,
                              const uint16_t *w, const uint16_t *x_act, uint16_t *dx,
                              uint16_t *w_t, osog_stream_t stream) {
    if (!shape_ok(shape) || !dy || !w || !dx || !w_t) return OSOG_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const Geo g = geo_of(shape);
    if (g_use_tcgen05) {  // reads the filters in place: w_t stays untouched
        const cudaError_t e = conv_dgrad_tma(g, dy, w, x_act, dx, st);
        if (e != cudaErrorNotSupported) return status_of(e);
    }
    const int64_t nw = (int64_t)g.K * g.R * g.S * g.C;
    k_filter_transpose<<<(unsigned)((nw + 255) / 256), 256, 0, st>>>(bf(w), g.K, g.R * g.S, g.C, bf(w_t));
    Args a{};
    a.g = g;
    a.x = bf(dy);
    a.w = bf(w_t);
    a.mask = x_act ? bf(x_act) : nullptr;
    a.y = bf(dx);
    a.Ncols = g.C;
    if (g.stride == 2) {  // four parity classes, each over its own taps
        for (int ph = 0; ph < 2; ++ph)
            for (int pw = 0; pw < 2; ++pw) {
                a.ph = ph;
                a.pw = pw;
                a.Hc = (g.H - ph + 1) / 2;
                a.Wc = (g.W - pw + 1) / 2;
                a.nr = a.ns = 0;
                for (int r = 0; r < g.R; ++r)
                    if (((ph + g.pad - r) & 1) == 0) a.rtap[a.nr++] = r;
                for (int sx = 0; sx < g.S; ++sx)
                    if (((pw + g.pad - sx) & 1) == 0) a.stap[a.ns++] = sx;
                a.M = g.N * a.Hc * a.Wc;
                a.Kred = a.nr * a.ns * g.K;
                if (a.M == 0) continue;
                dim3 grid((a.M + BM - 1) / BM, (a.Ncols + BN - 1) / BN);
                k_conv_gemm<kDgrad2><<<grid, NT, 0, st>>>(a);
            }
        return status_of(cudaGetLastError());
    }
    a.M = g.N * g.H * g.W;
    a.Kred = g.R * g.S * g.K;
    dim3 grid((a.M + BM - 1) / BM, (a.Ncols + BN - 1) / BN);
    k_conv_gemm<kDgrad><<<grid, NT, 0, st>>>(a);
    return status_of(cudaGetLastError());
}

static int bias_chunks(const Geo &g) {
    if (256 % g.K) return 0;
    return (int)(((int64_t)g.N * g.P * g.Q + bias_chunk(g.K) - 1) / bias_chunk(g.K));
}

size_t osog_conv2d_backward_filter_workspace(const osog_conv_shape_t *shape) {
    if (!shape_ok(shape)) return 0;
    const Geo g = geo_of(shape);
    const size_t warp = ((size_t)splits_of(g) * g.K * g.R * g.S * g.C +
                         (size_t)bias_chunks(g) * g.K) * sizeof(float);
    const size_t tma = conv_wgrad_tma_workspace(g);
    return warp > tma ? warp : tma;  // whichever engine the call runs on
}

int osog_conv2d_backward_filter(const osog_conv_shape_t *shape, const uint16_t *dy,
                                const uint16_t *x, float *dw, float *dbias, void *ws,
                                size_t ws_bytes, osog_stream_t stream) {
    if (!shape_ok(shape) || !dy || !x || !dw || !dbias) return OSOG_ERR_INVALID_ARG;
    if (!ws || ws_bytes < osog_conv2d_backward_filter_workspace(shape)) return OSOG_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const Geo g = geo_of(shape);
    if (g_use_tcgen05) {
        const cudaError_t e = conv_wgrad_tma(g, dy, x, dw, dbias, static_cast<float *>(ws), st);
        if (e != cudaErrorNotSupported) return status_of(e);
    }
    Args a{};
    a.g = g;
    a.x = bf(dy);
    a.w = bf(x);
    a.part = static_cast<float *>(ws);
    a.M = g.K;
    a.Ncols = g.R * g.S * g.C;
    a.Kred = g.N * g.P * g.Q;
    const int splits = splits_of(g);
    dim3 grid((a.M + BM - 1) / BM, (a.Ncols + BN - 1) / BN, splits);
    k_conv_gemm<kWgrad><<<grid, NT, 0, st>>>(a);
    const int64_t count = (int64_t)a.M * a.Ncols;
    sum_splits(a.part, splits, count, dw, st);
    const int64_t pixels = (int64_t)g.N * g.P * g.Q;
    if (256 % g.K == 0) {
        float *bpart = a.part + (size_t)splits * count;
        const int chunks = bias_chunks(g);
        k_bias_partial<<<chunks, 256, 0, st>>>(bf(dy), pixels, g.K, bpart);
        sum_splits(bpart, chunks, g.K, dbias, st);
    } else {
        k_bias_grad<<<g.K, 256, 0, st>>>(bf(dy), pixels, g.K, dbias);
    }
    return status_of(cudaGetLastError());
}

int osog_relu_backward(const uint16_t *dy, const uint16_t *act, uint16_t *dy_out, int64_t count,
                       osog_stream_t stream) {
    if (!dy || !act || !dy_out || count < 0) return OSOG_ERR_INVALID_ARG;
    if (count == 0) return OSOG_OK;
    k_relu_backward<<<(unsigned)((count + 255) / 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        bf(dy), bf(act), count, bf(dy_out));
    return status_of(cudaGetLastError());
}

void osog_conv_use_tcgen05(int32_t enable) { g_use_tcgen05 = enable ? 1 : 0; }

int osog_conv_test_wait_limit(int32_t polls) {
    const int v = polls > 0 ? polls : 0;
    return status_of(conv_tma_set_probe(v));
}

int osog_conv_sync_status(osog_stream_t stream) {
    if (cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess) return OSOG_ERR_CUDA;
    int t = 0;
    if (conv_tma_take_status(&t) != cudaSuccess) return OSOG_ERR_CUDA;
    return t ? OSOG_ERR_TIMEOUT : OSOG_OK;
}

}  // extern "C"
