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

#include <initializer_list>

#include "osog_cnn.h"
#include "osog_conv_tma.h"

namespace osog {
namespace cnn {
namespace {

constexpr int BM = 64, BN = 64, BK = 32, LDS = BK + 8;  // smem row: 40 bf16 = 80 bytes
constexpr int NT = 128;

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
    pdl_enter();
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

// ---------------------------------------------------------------- 8 channels
// The first layer (8 input channels, nine or ten taps): its reduction is too
// short for tcgen05, and the tiles of k_conv_gemm spend their time on gathers
// (every pixel is fetched once per tap through L1, 120 us of a 20 us HBM floor
// on 64 images of 256 x 256).  A pixel is one 16-byte vector, which is also one
// row of an ldmatrix 8 x 8 block: so the input patch of a tile is copied to
// shared memory once and every tap's fragment is read from it in place.  For
// stride 2 the patch's even and odd columns are kept apart, so that eight
// output pixels of one tap are 128 contiguous bytes.  The products are added in
// the order of k_conv_gemm (two taps per k16 step): the same bits.  On those
// images forward 120 -> 48 us, filter gradient 167 (110 by k_wgrad_patch, whose
// products of 16 columns are bound by their reads of dY) -> 54 us, at a quarter
// to a third of HBM: two or three CTAs of an SM do not cover the copies' latency
// and the issue of fragments.
constexpr int kC8Taps = 10, kC8W = 32, kC8Threads = 256;

struct PatchC8 {
    int stride, pad, S, RS;
    int pw, ph, half, pitch;  // pixels; half: columns of one parity; pitch: pixels per row
};

__host__ __device__ inline PatchC8 patch_c8(const Geo &g, int rows) {
    PatchC8 p;
    p.stride = g.stride;
    p.pad = g.pad;
    p.S = g.S;
    p.RS = g.R * g.S;
    p.pw = (kC8W - 1) * g.stride + g.S;
    p.ph = (rows - 1) * g.stride + g.R;
    p.half = (p.pw + 1) / 2;
    p.pitch = g.stride == 2 ? 2 * p.half : p.pw;
    return p;
}

// 16-byte asynchronous copy to shared memory; a NULL source writes zeros.
__device__ __forceinline__ void cp16(void *dst, const __nv_bfloat16 *src, const void *any) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n"
                 :: "r"(smem_u32(dst)), "l"(src ? (const void *)src : any), "r"(src ? 16 : 0)
                 : "memory");
}

// Copy of the input patch of the output tile (oy0, ox0) of image n.
__device__ __forceinline__ void load_patch_c8(const Geo &g, const PatchC8 &p, const __nv_bfloat16 *x,
                                              int n, int oy0, int ox0, uint4 *dst) {
    const int h0 = oy0 * p.stride - p.pad, w0 = ox0 * p.stride - p.pad;
    const __nv_bfloat16 *img = x + (size_t)n * g.H * g.W * 8;
    const float inv = 1.f / (float)p.pw;
    for (int e = threadIdx.x; e < p.ph * p.pw; e += kC8Threads) {
        int r = (int)((float)e * inv);  // e / pw, corrected below (e < 2^24)
        int c = e - r * p.pw;
        if (c >= p.pw) {
            ++r;
            c -= p.pw;
        } else if (c < 0) {
            --r;
            c += p.pw;
        }
        const int h = h0 + r, w = w0 + c;
        const bool in = h >= 0 && h < g.H && w >= 0 && w < g.W;
        const int at = p.stride == 2 ? (c & 1) * p.half + (c >> 1) : c;
        cp16(dst + r * p.pitch + at, in ? img + ((size_t)h * g.W + w) * 8 : nullptr, x);
    }
}

// Shared address of tap t's pixel for output pixel (row, x) of the tile.
__device__ __forceinline__ uint32_t tap_c8(const PatchC8 &p, uint32_t patch, int t, int row, int x) {
    const int r = t / p.S, s = t - r * p.S;
    const int col = p.stride == 2 ? (s & 1) * p.half + x + (s >> 1) : x + s;
    return patch + (uint32_t)((row * p.stride + r) * p.pitch + col) * 16u;
}

__device__ __forceinline__ void ldsm_x4_at(unsigned (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm_x4_t_at(unsigned (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}

// Forward: a CTA computes 32 x 16 output pixels of 32 output channels, warp w
// the rows w and w + 8, 16 pixels at a time; the filters' fragments stay in
// registers.
constexpr int kC8Rows = 16;
__global__ void __launch_bounds__(kC8Threads, 3) k_conv_c8(const __grid_constant__ Args a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(16) unsigned char out[kC8Threads / 32][16 * 80];
    __shared__ __align__(16) uint4 zero;
    pdl_enter();
    const Geo &g = a.g;
    const PatchC8 p = patch_c8(g, kC8Rows);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tx = (g.Q + kC8W - 1) / kC8W, ty = (g.P + kC8Rows - 1) / kC8Rows;
    const int n = blockIdx.x / (tx * ty), tile = blockIdx.x - n * tx * ty;
    const int oy0 = tile / tx * kC8Rows, ox0 = tile % tx * kC8W, n0 = blockIdx.y * 32;
    if (threadIdx.x == 0) zero = zero4();
    load_patch_c8(g, p, a.x, n, oy0, ox0, reinterpret_cast<uint4 *>(smem));
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    // fragments of the filters: column n = lane / 4 of each block of 8, entries
    // 2 (lane % 4), + 1 and those + 8 of every k16 step
    unsigned bf[kC8Taps / 2][4][2];
#pragma unroll
    for (int ks = 0; ks < kC8Taps / 2; ++ks)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int col = n0 + nt * 8 + (lane >> 2), j = ks * 16 + h * 8 + (lane & 3) * 2;
                bf[ks][nt][h] = col < a.Ncols && j < a.Kred
                                    ? *reinterpret_cast<const unsigned *>(a.w + (size_t)col * a.Kred + j)
                                    : 0u;
            }
    float2 bias[4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int col = n0 + nt * 8 + (lane & 3) * 2;
        bias[nt] = col < a.Ncols ? make_float2(a.bias[col], a.bias[col + 1]) : make_float2(0.f, 0.f);
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const uint32_t patch = smem_u32(smem), none = smem_u32(&zero);
    const int q = lane >> 3, r8 = lane & 7;
    // this lane's row of each k16 step's blocks (pixels 0-7 | 8-15) x (tap 2 ks
    // | 2 ks + 1); a tap past the last reads zeros
    uint32_t src[kC8Taps / 2];
    bool tap[kC8Taps / 2];
#pragma unroll
    for (int ks = 0; ks < kC8Taps / 2; ++ks) {
        const int t = 2 * ks + (q >> 1);
        tap[ks] = t < p.RS;
        src[ks] = tap[ks] ? tap_c8(p, patch, t, 0, (q & 1) * 8 + r8) : none;
    }
    const uint32_t row_step = (uint32_t)(p.stride * p.pitch) * 16u;
    unsigned char *st = out[warp];
    for (int row = warp; row < kC8Rows; row += kC8Threads / 32) {
        const int oy = oy0 + row;
        if (oy >= g.P) break;
#pragma unroll
        for (int xb = 0; xb < kC8W; xb += 16) {
            if (ox0 + xb >= g.Q) break;
            float acc[4][4];
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[nt][j] = 0.f;
#pragma unroll
            for (int ks = 0; ks < kC8Taps / 2; ++ks) {
                unsigned af[4];
                ldsm_x4_at(af, src[ks] + (tap[ks] ? row * row_step + xb * 16u : 0u));
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) mma_bf16(acc[nt], af, bf[ks][nt][0], bf[ks][nt][1]);
            }
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float v0 = acc[nt][2 * h] + bias[nt].x, v1 = acc[nt][2 * h + 1] + bias[nt].y;
                    if (a.relu) {
                        v0 = fmaxf(v0, 0.f);
                        v1 = fmaxf(v1, 0.f);
                    }
                    *reinterpret_cast<__nv_bfloat162 *>(st + ((lane >> 2) + 8 * h) * 80 + nt * 16 +
                                                        (lane & 3) * 4) = __floats2bfloat162_rn(v0, v1);
                }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int px = i * 8 + (lane >> 2), vec = lane & 3;
                const int ox = ox0 + xb + px, col = n0 + vec * 8;
                if (ox < g.Q && col < a.Ncols)
                    *reinterpret_cast<uint4 *>(a.y + (((size_t)n * g.P + oy) * g.Q + ox) * a.Ncols + col) =
                        *reinterpret_cast<const uint4 *>(st + px * 80 + vec * 16);
            }
            __syncwarp();
        }
    }
}

// Filter and bias gradient: a CTA adds the tiles z, z + splits, ... of 32 x 8
// output pixels; warp w takes row w, 16 pixels to a k16 step, with the output
// channels (16 MT) as the rows and every tap's 8 channels as one block of
// columns.  The next tile's copies run during a tile's products.  Partial sums
// in the layout of k_sum_parts.
constexpr int kC8GradRows = kC8Threads / 32;
template <int MT>
__global__ void __launch_bounds__(kC8Threads, MT == 2 ? 2 : 1)
k_wgrad_c8(const __grid_constant__ Args a, int splits) {
    constexpr int KP = MT * 16, VECS = KP / 8, kPix = kC8W * kC8GradRows;
    static_assert(kPix == kC8Threads, "a thread sums VECS vectors of a tile");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(16) uint4 zero;
    pdl_enter();
    const Geo &g = a.g;
    const PatchC8 p = patch_c8(g, kC8GradRows);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tx = (g.Q + kC8W - 1) / kC8W, ty = (g.P + kC8GradRows - 1) / kC8GradRows;
    const int tiles = g.N * tx * ty, z = blockIdx.x;
    const int patch_bytes = p.pitch * p.ph * 16, stage = kPix * KP * 2 + patch_bytes;
    if (threadIdx.x == 0) zero = zero4();
    // vector v of pixel px: rows of KP / 8 vectors, rotated so that eight
    // consecutive pixels of one vector fall on different banks
    auto at = [](int px, int v) { return px * VECS + (VECS == 4 ? v ^ ((px >> 1) & 3) : v ^ (px & 7)); };
    auto load = [&](int tile, unsigned char *dst) {
        const int n = tile / (tx * ty), t = tile - n * tx * ty;
        const int oy0 = t / tx * kC8GradRows, ox0 = t % tx * kC8W;
        uint4 *d = reinterpret_cast<uint4 *>(dst);
        for (int e = threadIdx.x; e < kPix * VECS; e += kC8Threads) {
            const int v = e % VECS, px = e / VECS, oy = oy0 + px / kC8W, ox = ox0 + px % kC8W;
            const bool in = oy < g.P && ox < g.Q && v * 8 < g.K;
            cp16(d + at(px, v), in ? a.x + (((size_t)n * g.P + oy) * g.Q + ox) * g.K + v * 8 : nullptr, a.x);
        }
        load_patch_c8(g, p, a.w, n, oy0, ox0, reinterpret_cast<uint4 *>(dst + kPix * KP * 2));
    };
    float acc[MT][kC8Taps][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int t = 0; t < kC8Taps; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[mt][t][j] = 0.f;
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int q = lane >> 3, r8 = lane & 7;
    // this lane's row of the blocks (tap 2 tp | 2 tp + 1) x (pixels 0-7 | 8-15)
    // of the warp's image row, relative to a stage; a tap past the last reads
    // zeros
    const uint32_t none = smem_u32(&zero);
    uint32_t src[kC8Taps / 2];
    bool tap[kC8Taps / 2];
#pragma unroll
    for (int tp = 0; tp < kC8Taps / 2; ++tp) {
        const int t = 2 * tp + (q >> 1);
        tap[tp] = t < p.RS;
        src[tp] = tap[tp] ? tap_c8(p, kPix * KP * 2, t, warp, (q & 1) * 8 + r8) : none;
    }
    load(z, smem);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    int buf = 0;
    for (int tile = z; tile < tiles; tile += splits) {
        if (tile + splits < tiles) load(tile + splits, smem + (buf ^ 1) * stage);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncthreads();
        const uint32_t dy = smem_u32(smem + buf * stage);
#pragma unroll
        for (int xb = 0; xb < kC8W; xb += 16) {
            unsigned af[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)  // (channels 0-7 | 8-15) x (pixels 0-7 | 8-15)
                ldsm_x4_t_at(af[mt], dy + 16u * at(warp * kC8W + xb + r8 + (q >> 1) * 8, mt * 2 + (q & 1)));
#pragma unroll
            for (int tp = 0; tp < kC8Taps / 2; ++tp) {
                unsigned bf[4];
                ldsm_x4_t_at(bf, src[tp] + (tap[tp] ? dy + xb * 16u : 0u));
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    mma_bf16(acc[mt][2 * tp], af[mt], bf[0], bf[1]);
                    mma_bf16(acc[mt][2 * tp + 1], af[mt], bf[2], bf[3]);
                }
            }
        }
        // bias: thread u sums vector u % VECS over the pixels u / VECS, ... of the tile,
        // then adds that to the tiles before
        const uint4 *d = reinterpret_cast<const uint4 *>(smem + buf * stage);
        uint4 v[VECS];
#pragma unroll
        for (int i = 0; i < VECS; ++i)
            v[i] = d[at(threadIdx.x / VECS + i * (kC8Threads / VECS), threadIdx.x % VECS)];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 t = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < VECS; ++i)
                t = cadd(t, __bfloat1622float2(reinterpret_cast<const __nv_bfloat162 *>(&v[i])[j]));
            sum[2 * j] += t.x;
            sum[2 * j + 1] += t.y;
        }
        __syncthreads();
        buf ^= 1;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    // the warps' sums in warp order, then the pixel lanes of the bias
    float *red = reinterpret_cast<float *>(smem);          // [KP][80]
    float *bred = red + KP * kC8Taps * 8;                  // [lanes][KP]
#pragma unroll
    for (int j = 0; j < 8; ++j)
        bred[(threadIdx.x / VECS) * KP + (threadIdx.x % VECS) * 8 + j] = sum[j];
    for (int w = 0; w < kC8Threads / 32; ++w) {
        if (warp == w) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int t = 0; t < kC8Taps; ++t)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float *r = red + (mt * 16 + (lane >> 2) + (j >> 1) * 8) * (kC8Taps * 8) + t * 8 +
                                   (lane & 3) * 2 + (j & 1);
                        *r = w ? *r + acc[mt][t][j] : acc[mt][t][j];
                    }
        }
        __syncthreads();
    }
    float *part = a.part + (size_t)z * ((size_t)g.K * a.Ncols + g.K);
    for (int i = threadIdx.x; i < g.K * a.Ncols; i += kC8Threads)
        part[i] = red[(i / a.Ncols) * (kC8Taps * 8) + i % a.Ncols];
    if ((int)threadIdx.x < g.K) {
        float v = 0.f;
        for (int l = 0; l < kC8Threads / VECS; ++l) v += bred[l * KP + threadIdx.x];
        part[(size_t)g.K * a.Ncols + threadIdx.x] = v;
    }
}

// Both take nine or ten taps (five k16 steps); the filter gradient up to 64
// output channels.
bool fits_c8(const Geo &g) {
    const PatchC8 p = patch_c8(g, kC8Rows);
    return g.C == 8 && g.R * g.S >= 9 && g.R * g.S <= kC8Taps && p.pitch * p.ph * 16 <= 96 * 1024;
}
int splits_c8(const Geo &g) {
    const int64_t tiles = (int64_t)g.N * ((g.Q + kC8W - 1) / kC8W) * ((g.P + kC8GradRows - 1) / kC8GradRows);
    // two CTAs on each SM, and more where one of a CTA's eight warps would add more
    // than kSplitPixels pixels
    const int64_t fill = 2 * kSms, warps = kC8Threads / 32 * kSplitPixels;
    const int64_t least = ((int64_t)g.N * g.P * g.Q + warps - 1) / warps;
    const int64_t splits = fill > least ? fill : least;
    return (int)(tiles < splits ? tiles : splits);
}

cudaError_t launch_conv_c8(const Args &a, cudaStream_t st) {
    const Geo &g = a.g;
    const PatchC8 p = patch_c8(g, kC8Rows);
    static osog::DeviceOnce once;
    const cudaError_t e = opt_in_smem(once, k_conv_c8, 96 * 1024);
    if (e != cudaSuccess) return e;
    const dim3 grid(g.N * ((g.Q + kC8W - 1) / kC8W) * ((g.P + kC8Rows - 1) / kC8Rows), (g.K + 31) / 32);
    return launch_conv(k_conv_c8, grid, kC8Threads, p.pitch * p.ph * 16, st, a);
}

template <int MT>
cudaError_t launch_wgrad_c8(const Args &a, cudaStream_t st) {
    const PatchC8 p = patch_c8(a.g, kC8GradRows);
    const int red = (MT * 16 * kC8Taps * 8 + kC8Threads * 8) * 4;
    int smem = 2 * (kC8W * kC8GradRows * MT * 32 + p.pitch * p.ph * 16);
    if (smem < red) smem = red;
    static osog::DeviceOnce once;
    const cudaError_t e = opt_in_smem(once, k_wgrad_c8<MT>, 200 * 1024);
    if (e != cudaSuccess) return e;
    const int splits = splits_c8(a.g);
    return launch_conv(k_wgrad_c8<MT>, dim3(splits), kC8Threads, smem, st, a, splits);
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

// True if every pointer is a multiple of `bytes` (a NULL is).
bool aligned(uintptr_t bytes, std::initializer_list<const void *> ptrs) {
    uintptr_t any = 0;
    for (const void *p : ptrs) any |= reinterpret_cast<uintptr_t>(p);
    return any % bytes == 0;
}

const __nv_bfloat16 *bf(const uint16_t *p) { return reinterpret_cast<const __nv_bfloat16 *>(p); }
__nv_bfloat16 *bf(uint16_t *p) { return reinterpret_cast<__nv_bfloat16 *>(p); }

}  // namespace

extern "C" {

int32_t osog_conv_out_h(const osog_conv_shape_t *s) { return shape_ok(s) ? geo_of(s).P : 0; }
int32_t osog_conv_out_w(const osog_conv_shape_t *s) { return shape_ok(s) ? geo_of(s).Q : 0; }

int osog_conv2d_forward(const osog_conv_shape_t *shape, const uint16_t *x, const uint16_t *w,
                        const float *bias, int32_t relu, uint16_t *y, float *y_f32,
                        osog_stream_t stream) {
    if (!shape_ok(shape) || !x || !w || !bias || !y || !aligned(16, {x})) return OSOG_ERR_INVALID_ARG;
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
    // first layer and the 1 x 1 head), and so do 8 channels up to 25 taps: the patch
    // kernel spends a product of 16 on each tap's 8 and a TMA row on each of its
    // filters' 16 bytes (81 x 154, 8 -> 216, 4 x 4: 21.6 us, k_conv_gemm 11.6; 16 images
    // of 23 x 42, 8 -> 24, 5 x 5: 14.9 and 14.1; at 49 taps 19.5 and 21.1).  The patch
    // kernels store 16-byte vectors; k_conv_gemm takes the outputs that are not so
    // aligned (pairs of columns).
    const bool deep = a.g.C == 8 ? a.Kred > 200 : a.Kred >= 128;
    if (g_use_tcgen05 && deep && aligned(16, {w, y, y_f32})) {
        const cudaError_t e = conv_forward_tma(a.g, x, w, bias, relu != 0, y, y_f32, st);
        if (e != cudaErrorNotSupported) return status_of(e);
    }
    if (!y_f32 && fits_c8(a.g) && aligned(16, {y}) && aligned(4, {w}))
        return status_of(launch_conv_c8(a, st));
    if (!aligned(16, {w}) || !aligned(4, {y}) || !aligned(8, {y_f32})) return OSOG_ERR_INVALID_ARG;
    dim3 grid((a.M + BM - 1) / BM, (a.Ncols + BN - 1) / BN);
    // early dispatch for grids of one CTA per SM at most (1 x 11 x 11, 16 -> 8 channels,
    // 1 x 1: 2.5 us, 3.0 without): the CTAs of more share the SMs with the next kernel's
    // waiting ones (16 x 40 x 40, 112 -> 16: 8.9 us, 7.0 without)
    const bool early = (int64_t)grid.x * grid.y <= osog::kSms;
    return status_of(osog::launch_pdl(k_conv_gemm<kFwd>, early, grid, NT, 0, st, a));
}

int osog_conv2d_backward_data(const osog_conv_shape_t *shape, const uint16_t *dy,
                              const uint16_t *w, const uint16_t *x_act, uint16_t *dx,
                              uint16_t *w_t, osog_stream_t stream) {
    if (!shape_ok(shape) || !dy || !w || !dx || !w_t || !aligned(16, {dy})) return OSOG_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const Geo g = geo_of(shape);
    // reads the filters in place, by TMA: w_t stays untouched.  Filters at any
    // address are transposed element by element into w_t below.
    if (g_use_tcgen05 && aligned(16, {w, x_act, dx})) {
        const cudaError_t e = conv_dgrad_tma(g, dy, w, x_act, dx, st);
        if (e != cudaErrorNotSupported) return status_of(e);
    }
    if (!aligned(16, {w_t}) || !aligned(4, {x_act, dx})) return OSOG_ERR_INVALID_ARG;
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
    const size_t c8 = fits_c8(g) && g.K <= 64
                          ? (size_t)splits_c8(g) * ((size_t)g.K * g.R * g.S * g.C + g.K) * sizeof(float)
                          : 0;
    const size_t most = warp > tma ? warp : tma;
    return most > c8 ? most : c8;  // whichever kernel the call runs on
}

int osog_conv2d_backward_filter(const osog_conv_shape_t *shape, const uint16_t *dy,
                                const uint16_t *x, float *dw, float *dbias, void *ws,
                                size_t ws_bytes, osog_stream_t stream) {
    if (!shape_ok(shape) || !dy || !x || !dw || !dbias || !aligned(16, {dy, x})) return OSOG_ERR_INVALID_ARG;
    if (!ws || ws_bytes < osog_conv2d_backward_filter_workspace(shape)) return OSOG_ERR_WORKSPACE;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const Geo g = geo_of(shape);
    Args a{};
    a.g = g;
    a.x = bf(dy);
    a.w = bf(x);
    a.part = static_cast<float *>(ws);
    a.M = g.K;
    a.Ncols = g.R * g.S * g.C;
    a.Kred = g.N * g.P * g.Q;
    const bool vectors = aligned(16, {ws, dw, dbias});  // of k_sum_parts
    if (vectors && fits_c8(g) && g.K <= 64) {
        cudaError_t e = g.K <= 32 ? launch_wgrad_c8<2>(a, st) : launch_wgrad_c8<4>(a, st);
        const bool ragged = g.P % kC8GradRows || g.Q % kC8W;
        if (e == cudaSuccess)
            e = conv_sum_parts(g, splits_c8(g), a.part, dw, dbias, ragged ? dy : nullptr, x, kC8GradRows,
                               kC8W, st);
        return status_of(e);
    }
    if (g_use_tcgen05 && vectors) {
        const cudaError_t e = conv_wgrad_tma(g, dy, x, dw, dbias, static_cast<float *>(ws), st);
        if (e != cudaErrorNotSupported) return status_of(e);
    }
    if (!aligned(8, {ws}) || !aligned(4, {dw, dbias})) return OSOG_ERR_INVALID_ARG;
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
