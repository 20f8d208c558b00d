// Convolutions as implicit GEMMs on the fifth-generation tensor cores, with
// the operands staged by the TMA unit (BF16 operands, FP32 accumulation).
//
// What bounds such a convolution is not the tensor pipe but the traffic into
// shared memory: an im2col tile holds every input pixel once per filter tap
// (nine times for 3 x 3).  Here a tile of output pixels is 8 wide and 16 high
// and its input is loaded once, as the patch of pixels that all taps touch
// ((8 + S - 1) x (16 + R - 1) for stride 1).  A patch row is one pixel's 64
// channels, 128 bytes, in the TMA unit's 128-byte swizzle, which is a function
// of the shared address alone; so the operand of a tap is the same patch read
// from a start address shifted by the tap's rows, with the patch's pitch as
// the stride between the groups of eight rows (one image row of the tile) that
// the matrix descriptor describes.  Padding and ragged edges are the TMA
// unit's zero fill.
//
//   forward   Y[(y, x)][k]  = sum_{r, s, c} X[(y st + r - pad, ...)][c] W[k][r, s][c]
//   data      dX[(y, x)][c] = sum_{r, s, k} dY[(y + pad - r, ...)][k] W[k][r, s][c]
//
// Stride 2, forward: the taps of one row and column parity read every second
// pixel, which the TMA unit gathers (traversal stride 2) into a patch of its
// own, one per parity.  Stride 2, data gradient: the input pixels of one parity
// class are reached by the taps of that parity only and form a stride-1
// problem on dY; one CTA computes the four classes of its tile from one patch.
// The data gradient reads the filters as they are stored ([K][R][S][C], the
// reduction index outermost: an MN-major operand), so no transposed copy of
// them is made.
//
// Measured on 64 images (us, before / now, the copies through 16-byte cp.async
// that this replaces): 128 -> 128 channels, 32 x 32: forward 104 / 21 (925
// TFLOP/s), data gradient 113 / 22; 32 -> 64, stride 2, 128 x 128 (100 to 167 MB
// of activations): forward 90 / 32, data gradient 209 / 55; 64 -> 128, stride 2:
// 59 / 20 and 132 / 23.  What bounds the wide layers now is the part of a CTA
// that its neighbour on the SM does not cover (launch, first patch, epilogue);
// the strided ones also write and read several HBM floors' worth of
// activations at partial overlap.
#include <cuda.h>
#include <cuda_bf16.h>

#include "osog_common.cuh"
#include "osog_conv_tma.h"

namespace osog {
namespace cnn {
namespace {

constexpr int kTileW = 8, kTileH = 16;   // pixels of a sub-tile: the 128 rows of one MMA
// A patch row is CH channels of one pixel: 64 (128 bytes, 128-byte swizzle), or
// 32 (64 bytes, 64-byte swizzle) when the source has no more, which halves the
// patch.
constexpr int kMaxTaps = 64;
constexpr int kCtaThreads = 256;
constexpr int kSmemMax = 232448;         // shared memory a CTA may opt in to (227 KB)
constexpr int kSpinLimit = 1 << 22;
constexpr int kMaxRing = 4;

__device__ int g_status;        // a bounded wait ran out
__device__ int g_probe_polls;   // failure-detection hook (osog_conv_test_wait_limit)

// One filter tap of a launch: the patch plane it reads, its shift inside the
// plane, its index in the filters and the output class it adds to.
struct Tap {
    uint8_t plane, sy, sx, cls;
    int16_t wt;
    int16_t first;   // 1: the first tap of its class (overwrites the accumulator)
};

struct PatchArgs {
    int tiles_x, tiles_y;      // CTA tiles per image
    int tx, ty;                // sub-tiles of a CTA, across and down
    int classes;               // 1, or 4 output parity classes (stride-2 data gradient)
    int taps;
    int planes, pw, ph;        // patch planes and their pixels
    int plane_bytes;           // of one plane and chunk (1024-byte multiple)
    int mul, off_y, off_x;     // patch origin: tile origin times mul, plus off, plus parity
    int ch;                    // channels of a patch row: 64 or 32
    int chunks, group;         // chunks of ch channels of the source; those held at a time
    int src_ch;                // source channels
    int bn, ncols;             // columns of a CTA and of the result
    int b_bytes;               // filters of one (tap, chunk) step
    int per, ring;             // steps of a stage, stages
    int mn_major;              // 1: filters as [reduction][column] (data gradient)
    uint32_t tmem_cols;
    // result
    int out_h, out_w;          // result image
    int cls_mul;               // 2: class (a, b) pixel (i, j) is result pixel (2 i + a, 2 j + b)
    const float *bias;
    const __nv_bfloat16 *mask;
    __nv_bfloat16 *y;
    float *y32;
    int relu;
    uint32_t live;             // bit c: class c has a tap
    Tap tap[kMaxTaps];
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, int limit = kSpinLimit) {
    for (int it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     "selp.u32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
        if (it > 64) __nanosleep(32);
    }
    return false;
}
// True in one lane of the (converged) warp.  The warps that issue TMA loads and
// matrix instructions run their loops with all lanes and issue from the elected
// one, so that loop state and descriptors stay warp-uniform (uniform
// registers); a loop inside a single-lane branch moves every operand there
// first, 80 to 100 cycles a matrix instruction.
__device__ __forceinline__ bool elect_lane() {
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void expect_bytes(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void init_bar(uint32_t bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void commit_to(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                 ::"r"(bar) : "memory");
}
__device__ __forceinline__ void load_4d(uint32_t dst, const CUtensorMap *m, int c, int x, int y,
                                        int n, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3, %4, %5}], [%6];\n"
                 ::"r"(dst), "l"(m), "r"(c), "r"(x), "r"(y), "r"(n), "r"(bar) : "memory");
}
__device__ __forceinline__ void load_3d(uint32_t dst, const CUtensorMap *m, int c, int t, int k,
                                        uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3, %4}], [%5];\n"
                 ::"r"(dst), "l"(m), "r"(c), "r"(t), "r"(k), "r"(bar) : "memory");
}

// Matrix descriptor of a swizzled tile, in two words: the low one holds the
// start address (16-byte units, so operands are moved by adding to it) and the
// byte stride between 64-element groups of the row index (MN-major tiles only),
// the high one the byte stride between groups of eight rows, the version and
// the swizzle (128-byte rows, or 64-byte ones).
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lead) {
    return ((addr >> 4) & 0x3FFF) | (lead >> 4) << 16;
}
template <int ROW = 128>
__device__ __forceinline__ uint32_t desc_hi(uint32_t stride) {
    return (stride >> 4) | 1u << 14 | (ROW == 128 ? 2u : 4u) << 29;
}
// kind::f16 instruction descriptor: FP32 accumulator, BF16 operands, M 128.
__device__ __forceinline__ uint32_t instr_desc(int n, bool a_mn, bool b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn ? 1u << 15 : 0u) | (b_mn ? 1u << 16 : 0u) |
           ((uint32_t)(n >> 3) << 17) | (8u << 24);
}
__device__ __forceinline__ void mma(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                    uint32_t b_hi, uint32_t idesc, uint32_t add) {
    asm volatile("{\n.reg .pred p;\n.reg .b64 ad, bd;\nsetp.ne.b32 p, %6, 0;\n"
                 "mov.b64 ad, {%1, %2};\nmov.b64 bd, {%3, %4};\n"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], ad, bd, %5, p;\n}\n"
                 ::"r"(d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(add)
                 : "memory");
}
__device__ __forceinline__ void tmem_load32(uint32_t addr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
        "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
          "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
          "=r"(v[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// Result columns of one pixel (this lane's), eight of them from v, as bf16.
template <bool FWD>
__device__ __forceinline__ uint4 finish8(const PatchArgs &a, const uint32_t *v, const float *bias,
                                         float *y32) {
    float x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = __uint_as_float(v[j]);
    if constexpr (FWD) {
        const float4 b0 = *reinterpret_cast<const float4 *>(bias);
        const float4 b1 = *reinterpret_cast<const float4 *>(bias + 4);
        const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            x[j] += bb[j];
            if (a.relu) x[j] = fmaxf(x[j], 0.f);
        }
        if (y32) {
            *reinterpret_cast<float4 *>(y32) = make_float4(x[0], x[1], x[2], x[3]);
            *reinterpret_cast<float4 *>(y32 + 4) = make_float4(x[4], x[5], x[6], x[7]);
        }
    }
    uint4 out;
    __nv_bfloat162 *o2 = reinterpret_cast<__nv_bfloat162 *>(&out);
#pragma unroll
    for (int j = 0; j < 4; ++j) o2[j] = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
    return out;
}

// v with the entries whose activation is not above zero cleared.
__device__ __forceinline__ uint4 relu_mask(uint4 v, uint4 act) {
    __nv_bfloat16 *x = reinterpret_cast<__nv_bfloat16 *>(&v);
    const __nv_bfloat16 *m = reinterpret_cast<const __nv_bfloat16 *>(&act);
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (!(__bfloat162float(m[j]) > 0.f)) x[j] = __float2bfloat16(0.f);
    return v;
}

// Staging of one warp in the epilogue: 32 pixels x 64 columns, rows of 144
// bytes (conflict-free for 16-byte accesses by consecutive rows).
constexpr int kStageCols = 64;
constexpr int kStageRow = 2 * kStageCols + 16;
constexpr int kStageBytes = 32 * kStageRow;
constexpr int kEpilogueSmem = kCtaThreads / 32 * kStageBytes;

// A CTA owns tx x ty sub-tiles of 8 x 16 output pixels of one image and bn
// result columns; accumulator (class, sub-tile) has bn columns of tensor
// memory.  Warp 0 issues the TMA loads (the patch, then the filters of the
// (tap, chunk) steps, `per` of them to a stage of the ring), warp 1 the matrix
// instructions; the steps run over the taps, each over the channel chunks, so
// that products are added in the order (tap, channel).  Then all eight warps
// read the accumulators back and write the result.
template <bool FWD, int CH>
__global__ void __launch_bounds__(kCtaThreads, 2)
k_conv_patch(const __grid_constant__ CUtensorMap src, const __grid_constant__ CUtensorMap flt,
             const __grid_constant__ PatchArgs a) {
    constexpr int kRow = 2 * CH;  // bytes of a patch row
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t bars[2 * kMaxRing + 4];
    __shared__ __align__(16) float bias[128];  // of this CTA's columns
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t patch = smem_addr(smem);
    const uint32_t ring = patch + (uint32_t)(a.group * a.planes * a.plane_bytes);
    const uint32_t full = smem_addr(bars), empty = full + 8u * kMaxRing;
    const uint32_t patch_full = empty + 8u * kMaxRing, group_done = patch_full + 8u,
                   all_done = patch_full + 16u, probe = patch_full + 24u;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     ::"r"(smem_addr(&tmem_slot)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < 2 * kMaxRing + 4; ++i) init_bar(full + 8u * i);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    pdl_enter();  // after the allocation: see launch_conv
    const int tile = blockIdx.x % (a.tiles_x * a.tiles_y), img = blockIdx.x / (a.tiles_x * a.tiles_y);
    const int oy0 = (tile / a.tiles_x) * a.ty * kTileH, ox0 = (tile % a.tiles_x) * a.tx * kTileW;
    const int n0 = blockIdx.y * a.bn;
    const int subs = a.tx * a.ty;
    const int groups = (a.chunks + a.group - 1) / a.group;
    const int per = a.per, stages = a.ring, taps = a.taps;
    const uint32_t stage_bytes = (uint32_t)(per * a.b_bytes);
    bool ok = true;
    if (warp == 0) {
        int st = 0;
        uint32_t ph = 0;
        bool filled = false;  // every stage used once: waits on its consumer from then on
        for (int g = 0; g < groups && ok; ++g) {
            const int c0 = g * a.group, nc = min(a.group, a.chunks - c0);
            if (g > 0) ok = wait_bar(group_done, (uint32_t)(g - 1) & 1u);
            if (!ok) break;
            if (elect_lane()) {
                expect_bytes(patch_full, (uint32_t)(nc * a.planes * a.pw * a.ph * kRow));
                for (int p = 0; p < a.planes; ++p)
                    for (int c = 0; c < nc; ++c)
                        load_4d(patch + (uint32_t)((c * a.planes + p) * a.plane_bytes), &src,
                                (c0 + c) * CH, ox0 * a.mul + a.off_x + (p & 1),
                                oy0 * a.mul + a.off_y + (p >> 1), img, patch_full);
            }
            __syncwarp();
            int t = 0, c = 0;
            for (int left = taps * nc; left > 0 && ok; left -= per) {
                if (filled) ok = wait_bar(empty + 8u * st, ph ^ 1u);
                if (!ok) break;
                const int n = min(per, left);
                const uint32_t bar = full + 8u * st;
                uint32_t dst = ring + (uint32_t)st * stage_bytes;
                const bool lead = elect_lane();
                if (lead) expect_bytes(bar, (uint32_t)(n * a.b_bytes));
                for (int i = 0; i < n; ++i) {
                    const int wt = a.tap[t].wt;
                    if (lead) {
                        if (a.mn_major) {
                            for (int b = 0; b * 64 < a.bn; ++b)
                                load_3d(dst + (uint32_t)(b * CH * 128), &flt, n0 + b * 64, wt,
                                        (c0 + c) * CH, bar);
                        } else {
                            load_3d(dst, &flt, (c0 + c) * CH, wt, n0, bar);
                        }
                    }
                    dst += (uint32_t)a.b_bytes;
                    if (++c == nc) {
                        c = 0;
                        ++t;
                    }
                }
                __syncwarp();
                if (++st == stages) {
                    st = 0;
                    ph ^= 1u;
                    filled = true;
                }
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc = instr_desc(a.bn, false, a.mn_major != 0);
        const uint32_t pitch = (uint32_t)(a.pw * kRow);
        // K-major filters have the patch's row width, MN-major ones rows of 64
        // result columns
        const uint32_t a_hi = desc_hi<kRow>(pitch),
                       b_hi = a.mn_major ? desc_hi<128>(1024u) : desc_hi<kRow>(8u * kRow);
        const uint32_t pitch16 = pitch >> 4, chunk16 = (uint32_t)(a.planes * a.plane_bytes) >> 4,
                       plane16 = (uint32_t)a.plane_bytes >> 4, bn = (uint32_t)a.bn;
        const uint32_t b_step = a.mn_major ? 2048u >> 4 : 32u >> 4;  // 16 reduction entries
        const uint32_t b_first = desc_lo(ring, a.mn_major ? CH * 128 : 16u);
        const uint32_t b16 = (uint32_t)a.b_bytes >> 4;
        uint32_t sub16[4];
#pragma unroll
        for (int s = 0; s < 4; ++s)
            sub16[s] = (uint32_t)(s / a.tx) * kTileH * pitch16 +
                       (uint32_t)(s % a.tx) * (kTileW * kRow >> 4);
        const int last_ch = a.src_ch;
        int st = 0;
        uint32_t ph = 0;
        for (int g = 0; g < groups && ok; ++g) {
            const int c0 = g * a.group, nc = min(a.group, a.chunks - c0);
            ok = wait_bar(patch_full, (uint32_t)g & 1u);
            int t = 0, c = 0;
            Tap now = a.tap[0], next = a.tap[min(1, taps - 1)];
            uint32_t a_lo = desc_lo(patch, 16u) + now.plane * plane16 + now.sy * pitch16 +
                            now.sx * (kRow >> 4);
            for (int left = taps * nc; left > 0 && ok; left -= per) {
                ok = wait_bar(full + 8u * st, ph);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                uint32_t b_lo = b_first + (uint32_t)(st * per) * b16;
                const int n = min(per, left);
                const bool lead = elect_lane();
                for (int i = 0; i < n; ++i) {
                    const uint32_t add = now.first && g == 0 && c == 0 ? 0u : 1u;
                    const int rest = last_ch - (c0 + c) * CH;
                    const uint32_t acc = tmem + now.cls * (uint32_t)subs * bn;
                    if (lead) {
#pragma unroll
                        for (int s = 0; s < 4; ++s) {
                            if (s >= subs) break;
                            const uint32_t as = a_lo + sub16[s], d = acc + (uint32_t)s * bn;
                            mma(d, as, a_hi, b_lo, b_hi, idesc, add);
                            if (rest > 16) mma(d, as + 2u, a_hi, b_lo + b_step, b_hi, idesc, 1u);
                            if constexpr (CH == 64) {
                                if (rest > 32) mma(d, as + 4u, a_hi, b_lo + 2u * b_step, b_hi, idesc, 1u);
                                if (rest > 48) mma(d, as + 6u, a_hi, b_lo + 3u * b_step, b_hi, idesc, 1u);
                            }
                        }
                    }
                    b_lo += b16;
                    a_lo += chunk16;
                    if (++c == nc) {
                        c = 0;
                        ++t;
                        now = next;
                        next = a.tap[min(t + 1, taps - 1)];  // read ahead of its use
                        a_lo = desc_lo(patch, 16u) + now.plane * plane16 + now.sy * pitch16 +
                               now.sx * (kRow >> 4);
                    }
                }
                if (lead) commit_to(empty + 8u * st);
                __syncwarp();
                if (++st == stages) {
                    st = 0;
                    ph ^= 1u;
                }
            }
            if (ok && g + 1 < groups && elect_lane()) commit_to(group_done);
            __syncwarp();
        }
        if (ok && elect_lane()) commit_to(all_done);
    } else if (FWD && tid >= kCtaThreads - 128) {  // meanwhile
        const int col = tid - (kCtaThreads - 128);
        if (col < a.bn && n0 + col < a.ncols) bias[col] = __ldg(a.bias + n0 + col);
    }
    __syncwarp();
    ok = wait_bar(all_done, 0u) && ok;
    __syncthreads();
    if (tid == 0 && g_probe_polls > 0)  // a wait made to run out (test hook)
        ok = wait_bar(probe, 0u, g_probe_polls) && ok;
    if (!ok) atomicExch(&g_status, 1);
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    // Warp w reads the tensor-memory lanes 32 (w % 4) .. + 31 (pixels) of the
    // (accumulator, 64 columns) units of its half (w / 4).  A lane holds one
    // pixel; written from there, the 16-byte stores of a warp would fall on 32
    // different lines, so a unit goes through the warp's own shared-memory
    // rows (the operands are consumed by now) and leaves as whole pixels.
    const int quarter = warp & 3, half = warp >> 2;
    unsigned char *stage = smem + warp * kStageBytes;
    const int units = (a.bn + kStageCols - 1) / kStageCols;
    for (int u = half; u < a.classes * subs * units; u += 2) {
        const int acc = u / units, cc = (u % units) * kStageCols;
        const int cls = acc / subs, s = acc % subs;
        const int ncol = min(kStageCols, min(a.bn - cc, a.ncols - n0 - cc));  // a multiple of 8
        if (ncol <= 0) continue;
        int oy = oy0 + (s / a.tx) * kTileH + quarter * 4, ox = ox0 + (s % a.tx) * kTileW;
        if (a.cls_mul == 2) {
            oy = 2 * oy + (cls >> 1);
            ox = 2 * ox + (cls & 1);
        }
        // pixel i of the warp: (oy + (i / 8) cls_mul, ox + (i % 8) cls_mul)
        const size_t img_row = (size_t)img * a.out_h;
        const int my = oy + (lane >> 3) * a.cls_mul, mx = ox + (lane & 7) * a.cls_mul;
        float *y32 = FWD && a.y32 && my < a.out_h && mx < a.out_w
                         ? a.y32 + ((img_row + my) * a.out_w + mx) * a.ncols + n0 + cc
                         : nullptr;
        // this lane's 16-byte vectors of the result: pixels first + i step; the
        // activations of the mask are read ahead of everything else
        const int vecs = ncol >> 3;                            // of a pixel
        const int lanes = vecs > 4 ? 8 : vecs > 2 ? 4 : vecs;  // of a pixel (1, 2, 4 or 8)
        const int sh = lanes == 8 ? 3 : lanes == 4 ? 2 : lanes - 1;
        const int vec = lane & (lanes - 1), first = lane >> sh, step = 32 >> sh;
        int64_t at[8];
        uint4 act[FWD ? 1 : 8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int p = first + i * step;
            const int py = oy + (p >> 3) * a.cls_mul, px = ox + (p & 7) * a.cls_mul;
            const bool in = p < 32 && vec < vecs && py < a.out_h && px < a.out_w;
            at[i] = in ? (int64_t)(((img_row + py) * a.out_w + px) * a.ncols + n0 + cc + vec * 8) : -1;
            if constexpr (!FWD)
                if (a.mask && in) act[i] = __ldg(reinterpret_cast<const uint4 *>(a.mask + at[i]));
        }
#pragma unroll
        for (int h = 0; h < kStageCols; h += 32) {
            if (h >= ncol) break;
            uint32_t v[32];
            tmem_load32(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * a.bn + cc + h), v);
            if (!((a.live >> cls) & 1u)) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = 0u;
            }
#pragma unroll
            for (int j = 0; j < 32; j += 8)
                if (h + j < ncol)
                    *reinterpret_cast<uint4 *>(stage + lane * kStageRow + (h + j) * 2) =
                        finish8<FWD>(a, v + j, bias + cc + h + j, y32 ? y32 + h + j : nullptr);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (at[i] >= 0) {
                uint4 v = *reinterpret_cast<const uint4 *>(stage + (first + i * step) * kStageRow + vec * 16);
                if (!FWD && a.mask) v = relu_mask(v, act[i]);
                *reinterpret_cast<uint4 *>(a.y + at[i]) = v;
            }
        __syncwarp();
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(a.tmem_cols)
                     : "memory");
}

// Filter gradient: dW[k][r, s][c] = sum over output pixels of dY[pixel][k]
// X[pixel st + (r, s) - pad][c], and dbias[k] = sum of dY[pixel][k].
//
// The pixels are the reduction.  A tile of 8 x 16 output pixels of dY (rows of
// 64 output channels) and the patches of X it touches are loaded once and feed
// every tap of the CTA's group: tap (r, s) multiplies the same dY rows with the
// patch rows shifted by the tap, both operands with the reduction outermost
// (MN-major).  A CTA adds the tiles z, z + splits, ... of its split into one
// tensor-memory accumulator per tap (128 output channels by up to 128 input
// channels, 512 columns in all) and writes its partial sums; k_sum_parts adds
// the splits in order.  The warps that neither load nor issue sum dY over the
// pixels of the tile for the bias gradient while it is in shared memory.
//
// Measured with the sums over the splits and the bias gradient (us, 64 images,
// before / now): 128 -> 128, 32 x 32: 123 / 23; 64 -> 128, stride 2: 116 / 20;
// 32 -> 64, stride 2: 138 / 37 (bound by the reads of dY from shared memory, 4 KB
// per product however few its columns); 128 -> 64: 96 / 21.
//
// The accumulators round (to FP32, towards zero) at every 16 pixels, so the error of a
// sum grows with their number; a split has at most about kSplitPixels pixels of one
// accumulator, whatever the layer and however many images.  Without that limit the
// 3 x 3 layer of 256 -> 256 channels on 64 images of 64 x 64 added 21,800 pixels: its
// error was 3.2e-5 of the gradient's norm, now 1.8e-6 (the general kernel's 2.0e-6), for
// 314 us instead of 200 (1,461 with the copies through cp.async); the network's layers
// have shorter chains anyway.  The bias gradient is summed tile by tile for the same
// reason.
struct WgradArgs {
    int tiles_x, tiles, splits;        // tiles of all images
    int tiles_y;
    int pw, ph, plane_bytes;           // X patch planes
    int stride, pad;
    int chunks;                        // ch-channel chunks of a column block
    int k64;                           // 64-channel blocks of dY in a row block (1 or 2)
    int ring, stage_bytes;
    int bn, cblk;                      // columns of an accumulator, channels of a column block
    int cblocks, groups;               // column blocks, tap groups
    int K, C, RS;
    uint32_t tmem_cols;
    float *part;                       // [splits][K RS C + K]
    int group0[kMaxTaps + 1];          // first tap of each group
    uint8_t planes[kMaxTaps];          // per group: the planes its taps read, bit set
    Tap tap[kMaxTaps];                 // sorted by group
};

constexpr int kSumThreads = kCtaThreads - 64;  // warps 2..7: the bias gradient

template <int CH>
__global__ void __launch_bounds__(kCtaThreads, 1)
k_wgrad_patch(const __grid_constant__ CUtensorMap mdy, const __grid_constant__ CUtensorMap mx,
              const __grid_constant__ WgradArgs a) {
    constexpr int kRow = 2 * CH;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ uint64_t bars[2 * kMaxRing + 2];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t full = smem_addr(bars), empty = full + 8u * kMaxRing,
                   all_done = empty + 8u * kMaxRing, probe = all_done + 8u;
    const int blocks = gridDim.x / a.splits, z = blockIdx.x / blocks;
    const int group = blockIdx.x % blocks % a.groups, blk = blockIdx.x % blocks / a.groups;
    const int c0 = (blk % a.cblocks) * a.cblk, k0 = (blk / a.cblocks) * 128;
    const bool sums_bias = group == 0 && c0 == 0;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     ::"r"(smem_addr(&tmem_slot)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kMaxRing; ++i) {
            init_bar(full + 8u * i);
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n"
                         ::"r"(empty + 8u * i), "r"(sums_bias ? 1 + kSumThreads / 32 : 1) : "memory");
        }
        init_bar(all_done);
        init_bar(probe);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    pdl_enter();
    const uint32_t base = smem_addr(smem);
    const int dy_bytes = a.k64 * kTileW * kTileH * 128;
    const uint32_t planes = a.planes[group];
    const int nplanes = __popc(planes);
    const int t0 = a.group0[group], nt = a.group0[group + 1] - t0;
    const int ntiles = (a.tiles - z + a.splits - 1) / a.splits;
    bool ok = true;
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (warp == 0) {
        int st = 0;
        uint32_t ph = 0;
        for (int i = 0; i < ntiles && ok; ++i) {
            if (i >= a.ring) ok = wait_bar(empty + 8u * st, ph ^ 1u);
            if (!ok) break;
            const int tile = z + i * a.splits;
            const int img = tile / (a.tiles_x * a.tiles_y), t = tile - img * a.tiles_x * a.tiles_y;
            const int oy = (t / a.tiles_x) * kTileH, ox = (t % a.tiles_x) * kTileW;
            const uint32_t dst = base + (uint32_t)st * a.stage_bytes, bar = full + 8u * st;
            if (elect_lane()) {
                expect_bytes(bar, (uint32_t)(dy_bytes + nplanes * a.chunks * a.pw * a.ph * kRow));
                for (int b = 0; b < a.k64; ++b)
                    load_4d(dst + (uint32_t)(b * kTileW * kTileH * 128), &mdy, k0 + b * 64, ox, oy, img, bar);
                int slot = 0;
                for (int p = 0; p < 4; ++p) {
                    if (!((planes >> p) & 1u)) continue;
                    for (int c = 0; c < a.chunks; ++c)
                        load_4d(dst + dy_bytes + (uint32_t)((c * nplanes + slot) * a.plane_bytes), &mx,
                                c0 + c * CH, ox * a.stride - a.pad + (p & 1),
                                oy * a.stride - a.pad + (p >> 1), img, bar);
                    ++slot;
                }
            }
            __syncwarp();
            if (++st == a.ring) {
                st = 0;
                ph ^= 1u;
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc = instr_desc(a.bn, true, true);
        const uint32_t pitch = (uint32_t)(a.pw * kRow), pitch16 = pitch >> 4;
        const uint32_t a_hi = desc_hi<128>(1024u), b_hi = desc_hi<kRow>(pitch);
        const uint32_t b_lead = (uint32_t)(nplanes * a.plane_bytes);
        const uint32_t plane16 = (uint32_t)a.plane_bytes >> 4, bn = (uint32_t)a.bn;
        int st = 0;
        uint32_t ph = 0;
        for (int i = 0; i < ntiles && ok; ++i) {
            ok = wait_bar(full + 8u * st, ph);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t src = base + (uint32_t)st * a.stage_bytes;
            const uint32_t a_lo = desc_lo(src, kTileW * kTileH * 128);
            const uint32_t x_lo = desc_lo(src + dy_bytes, b_lead);
            const bool lead = elect_lane();
            Tap next = a.tap[t0];
            for (int t = 0; t < nt; ++t) {
                const Tap now = next;
                next = a.tap[min(t0 + t + 1, t0 + nt - 1)];
                const uint32_t slot = __popc(planes & ((1u << now.plane) - 1u));
                const uint32_t b_lo = x_lo + slot * plane16 + now.sy * pitch16 + now.sx * (kRow >> 4);
                const uint32_t acc = tmem + (uint32_t)t * bn;
                if (lead) {
#pragma unroll
                    for (int k = 0; k < kTileH / 2; ++k)  // 16 pixels: two rows of the tile
                        mma(acc, a_lo + k * (2048u >> 4), a_hi, b_lo + k * 2u * pitch16, b_hi, idesc,
                            i > 0 || k > 0 ? 1u : 0u);
                }
            }
            if (lead) commit_to(empty + 8u * st);
            __syncwarp();
            if (++st == a.ring) {
                st = 0;
                ph ^= 1u;
            }
        }
        if (ok && elect_lane()) commit_to(all_done);
    } else if (sums_bias) {
        // thread u sums the 8 channels of vector u % vecs over the pixels u /
        // vecs, + lanes, ...
        const int u = tid - 64, vecs = a.k64 * 8, lanes = kSumThreads / vecs;
        const int vec = u % vecs, p0 = u / vecs;
        int st = 0;
        uint32_t ph = 0;
        for (int i = 0; i < ntiles && ok; ++i) {
            ok = wait_bar(full + 8u * st, ph);
            if (!ok) break;
            const unsigned char *src = smem + (size_t)st * a.stage_bytes +
                                       (vec >> 3) * (kTileW * kTileH * 128);
            float part[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            for (int p = p0; p < kTileW * kTileH; p += lanes) {
                const uint4 v = *reinterpret_cast<const uint4 *>(src + p * 128 + (((vec ^ p) & 7) << 4));
                const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 f = __bfloat1622float2(h[j]);
                    part[2 * j] += f.x;
                    part[2 * j + 1] += f.y;
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) sum[j] += part[j];
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(empty + 8u * st) : "memory");
            if (++st == a.ring) {
                st = 0;
                ph ^= 1u;
            }
        }
    }
    __syncwarp();
    ok = wait_bar(all_done, 0u) && ok;
    if (tid == 0 && g_probe_polls > 0)  // a wait made to run out (test hook)
        ok = wait_bar(probe, 0u, g_probe_polls) && ok;
    if (!ok) atomicExch(&g_status, 1);
    __syncthreads();  // every stage is consumed: shared memory is free
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    float *part = a.part + (size_t)z * ((size_t)a.K * a.RS * a.C + a.K);
    if (sums_bias) {  // the pixel lanes of a channel in order
        float *red = reinterpret_cast<float *>(smem);  // [lanes][8 vecs]
        const int u = tid - 64, vecs = a.k64 * 8, lanes = kSumThreads / vecs;
        if (u >= 0)
#pragma unroll
            for (int j = 0; j < 8; ++j) red[(u / vecs) * vecs * 8 + (u % vecs) * 8 + j] = sum[j];
        __syncthreads();
        if (tid < vecs * 8 && k0 + tid < a.K) {
            float v = 0.f;
            for (int l = 0; l < lanes; ++l) v += red[l * vecs * 8 + tid];
            part[(size_t)a.K * a.RS * a.C + k0 + tid] = v;
        }
        __syncthreads();
    }
    // accumulators to the partial sums: warp w holds output channels 32 (w % 4)
    // .. + 31 (one per lane); pieces of 32 input channels leave through the
    // warp's shared rows so that the stores are whole lines
    const int quarter = warp & 3, half = warp >> 2;
    unsigned char *stage = smem + warp * kStageBytes;
    const int pieces = (a.bn + 31) / 32;
    const int kfirst = k0 + quarter * 32;
    if (kfirst < a.K && quarter * 32 < a.k64 * 64)
        for (int u = half; u < nt * pieces; u += 2) {
            const int t = u / pieces, cc = (u % pieces) * 32;
            uint32_t v[32];
            tmem_load32(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(t * a.bn + cc), v);
#pragma unroll
            for (int j = 0; j < 32; j += 4)
                *reinterpret_cast<uint4 *>(stage + lane * kStageRow + j * 4) =
                    make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            __syncwarp();
            const int wt = a.tap[t0 + t].wt;
            const int c = c0 + cc + (lane & 7) * 4;
            if (c < a.C && cc + (lane & 7) * 4 < a.cblk) {
#pragma unroll
                for (int r = lane >> 3; r < 32; r += 4) {
                    if (kfirst + r >= a.K) continue;
                    *reinterpret_cast<uint4 *>(part + ((size_t)(kfirst + r) * a.RS + wt) * a.C + c) =
                        *reinterpret_cast<const uint4 *>(stage + r * kStageRow + (lane & 7) * 16);
                }
            }
            __syncwarp();
        }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(a.tmem_cols)
                     : "memory");
}

// Sums over the splits, out[i] = sum over z of part[z][i], i < count (out = dw) or
// count <= i < count + extra (out2 = dbias), four outputs per thread (count and
// extra are multiples of 8), the splits in order within each of kSumLanes
// interleaved partial sums, which are then added in order.
//
// Tiles that reach past the image pair its missing output pixels, zeros of dY, with
// whatever X holds there for other taps: 0 inf is NaN, in entries that those pixels
// are no part of.  Only a product of a zero can do that, and only to make a partial
// sum NaN; so where tiles are ragged (RAGGED) a warp whose sum is NaN adds its splits
// again, and takes the NaN entries of a split from the existing pixels of the split's
// tiles (an entry whose own products give NaN stays so, and is left at that).
// Sums without a NaN, all but those of a diverged network, keep their bits and pay one
// vote; the other path goes entry by entry, so that the kernel keeps its 32 registers
// (8 images of 255 x 249, 64 -> 64: 99 us; all of X NaN 261, one pixel infinite in every
// channel 1,170).
constexpr int kSumLanes = 8;
struct EdgeFix {
    const __nv_bfloat16 *dy, *x;
    Geo g;
    int tile_h, tile_w;
};
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// Entry e of split z's partial sum from the existing pixels (of the lanes that want it;
// all lanes of the warp call it).
__device__ __forceinline__ float split_of_pixels(const EdgeFix &f, int z, int splits, int64_t e, bool want) {
    const Geo &g = f.g;
    const int c = (int)(e % g.C), t = (int)(e / g.C), rs = t % (g.R * g.S), k = t / (g.R * g.S);
    const int dh = rs / g.S - g.pad, dw = rs % g.S - g.pad;
    const int tx = (g.Q + f.tile_w - 1) / f.tile_w, ty = (g.P + f.tile_h - 1) / f.tile_h;
    float s = 0.f;
    for (int tile = z; tile < g.N * tx * ty && __any_sync(0xffffffffu, want); tile += splits) {
        const int n = tile / (tx * ty), p0 = tile % (tx * ty) / tx * f.tile_h, q0 = tile % tx * f.tile_w;
        for (int p = p0; p < min(p0 + f.tile_h, g.P); ++p) {
            if (!want) continue;
            const int h = p * g.stride + dh;
            const __nv_bfloat16 *dy = f.dy + ((size_t)n * g.P + p) * g.Q * g.K + k;
            const __nv_bfloat16 *x = f.x + ((size_t)n * g.H + h) * g.W * g.C + c;
#pragma unroll 4
            for (int q = q0; q < min(q0 + f.tile_w, g.Q); ++q) {
                const int u = q * g.stride + dw;
                const bool in = h >= 0 && h < g.H && u >= 0 && u < g.W;  // else padding
                s = fmaf(__bfloat162float(dy[(size_t)q * g.K]), in ? __bfloat162float(x[(size_t)u * g.C]) : 0.f, s);
            }
            want = !isnan(s);
        }
    }
    return s;
}

template <bool RAGGED>
__global__ void __launch_bounds__(32 * kSumLanes, 8)
k_sum_parts(const float4 *part, int splits, int64_t count4, int64_t extra4, float4 *out,
            float4 *out2, const __grid_constant__ EdgeFix fix) {
    __shared__ float4 red[kSumLanes][32];
    pdl_enter();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane, row = count4 + extra4;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < row) {
#pragma unroll 4
        for (int z = w; z < splits; z += kSumLanes) s = add4(s, __ldg(part + (size_t)z * row + i));
    }
    red[w][lane] = s;
    if constexpr (RAGGED) {
        if (__any_sync(0xffffffffu, i < count4 && isnan(s.x + s.y + s.z + s.w))) {
            for (int j = 0; j < 4; ++j) {
                float *mine = &red[w][lane].x + j;
                const bool bad = i < count4 && isnan(*mine);
                float t = 0.f;
                for (int z = w; z < splits; z += kSumLanes) {
                    float v = bad ? reinterpret_cast<const float *>(part + (size_t)z * row + i)[j] : 0.f;
                    const bool want = isnan(v) && !isnan(t);
                    if (__any_sync(0xffffffffu, want)) {
                        const float u = split_of_pixels(fix, z, splits, want ? 4 * i + j : 0, want);
                        if (want) v = u;
                    }
                    t += v;
                }
                if (bad) *mine = t;
            }
        }
    }
    __syncthreads();
    if (w == 0 && i < row) {
        s = red[0][lane];
        for (int l = 1; l < kSumLanes; ++l) s = add4(s, red[l][lane]);
        if (i < count4)
            out[i] = s;
        else
            out2[i - count4] = s;
    }
}

// ------------------------------------------------------------------ host
using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                              const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                              const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
    static const EncodeFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeFn>(p);
    }();
    return fn;
}

// Tensor map of a bf16 tensor with `rank` dimensions (innermost first), boxes
// of the given extents (the innermost 64 or 32: 128- or 64-byte swizzle),
// traversal strides es, zero fill.
cudaError_t encode(CUtensorMap *m, const void *base, int rank, const uint64_t *dims,
                   const uint32_t *box, const uint32_t *es) {
    const EncodeFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    cuuint64_t d[5], strides[5];
    cuuint32_t b[5], e[5];
    uint64_t bytes = 2;
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        bytes *= dims[i];
        strides[i] = bytes;  // of dimension i + 1
        b[i] = box[i];
        e[i] = es[i];
    }
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank,
                          const_cast<void *>(base), d, strides, b, e, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          box[0] == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }
int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Result columns of a forward CTA: as few blocks of at most 128 as there can be, of
// equal width (136 columns as 80 + 56, not 128 + 8: 64 images of 40 x 46, 16 -> 136, 5 x
// 5, stride 2, 46.7 -> 31.3 us; 43.2 with the copies through cp.async).  The data
// gradient's filters come in groups of 64 columns and keep 128.
int column_block(int n) { return round_up(ceil_div(n, ceil_div(n, 128)), 16); }

uint32_t tmem_columns(int need) {
    uint32_t c = 32;  // need is at most 512, what an SM has
    while ((int)c < need) c *= 2;
    return c;
}

int patch_smem(const PatchArgs &a) {
    const int operands = a.group * a.planes * a.plane_bytes + a.ring * a.per * a.b_bytes;
    return operands > kEpilogueSmem ? operands : kEpilogueSmem;
}

// Sub-tiles per CTA and the shared-memory plan of a launch over an oh x ow
// pixel grid of `images` images.  More sub-tiles share one stage of filters and
// one patch, but leave fewer CTAs to fill the SMs and to hide one another's
// fixed parts.  The choice minimises a count of cycles: the larger of what the
// SM's rates allow (bytes into shared memory at 64 a cycle, tensor cycles at N /
// 2 for a 128 x N x 16 product) and of the waves of CTAs times the length of one
// (launch and allocation 1400, the patch's latency, 150 for a stage, 900 for an
// epilogue unit of a warp; measured with clock reads on the 128 -> 128 and 32 ->
// 64 channel layers).  False if no plan fits.
bool conv_patch_plan(PatchArgs &a, int images, int oh, int ow, int reach_y, int reach_x) {
    static const int shapes[3][2] = {{1, 1}, {2, 1}, {2, 2}};
    const int col_blocks = ceil_div(a.ncols, a.bn);
    double best = 0;
    bool found = false;
    PatchArgs pick = a;
    for (const auto &sh : shapes) {
        PatchArgs t = a;
        t.tx = sh[0];
        t.ty = sh[1];
        const int subs = t.tx * t.ty;
        if (subs > 1 && ((t.tx - 1) * kTileW >= ow || (t.ty - 1) * kTileH >= oh)) continue;
        const int cols = (t.classes * subs - 1) * t.bn + round_up(t.bn, 32);
        if (cols > 512) continue;
        t.tmem_cols = tmem_columns(cols);
        t.pw = t.tx * kTileW + reach_x;
        t.ph = t.ty * kTileH + reach_y;
        if ((t.pw - 1) * t.mul + 1 > 256 || (t.ph - 1) * t.mul + 1 > 256) continue;
        t.plane_bytes = round_up(t.pw * t.ph * 2 * t.ch, 1024);
        t.tiles_x = ceil_div(ow, t.tx * kTileW);
        t.tiles_y = ceil_div(oh, t.ty * kTileH);
        const double per_sm_ctas = (double)images * t.tiles_x * t.tiles_y * col_blocks / kSms;
        const int steps = t.taps * t.chunks;
        const double mma = (double)steps * (t.ch / 16) * t.bn / 2.0 * subs;
        const double units = (t.classes * subs * ceil_div(t.bn, 64) + 1) / 2;
        for (t.ring = 2; t.ring <= 4; ++t.ring)
            for (t.per = 1; t.per <= 9; ++t.per) {
                if (t.per > 1 && (t.ring - 1) * t.per >= steps) continue;
                int group = t.chunks;
                const int stages = t.ring * t.per * t.b_bytes;
                while (group > 1 && group * t.planes * t.plane_bytes + stages > kSmemMax - 2048)
                    group = (group + 1) / 2;
                if (group * t.planes * t.plane_bytes + stages > kSmemMax - 2048) continue;
                t.group = group;
                int co = (kSmemMax + 1024) / (patch_smem(t) + 2048);
                co = co > 512 / (int)t.tmem_cols ? 512 / (int)t.tmem_cols : co;
                co = co > 2 ? 2 : co;  // registers
                const double bytes = (double)t.chunks * t.planes * t.plane_bytes +
                                     (double)steps * t.b_bytes;
                const double rate = per_sm_ctas * (bytes / 64.0 > mma ? bytes / 64.0 : mma);
                // a stage's filters arrive about 1200 cycles after they are asked for
                const double turn = 1200.0 / (t.ring - 1);
                const double stage_mma = mma / steps * t.per + 150.0;
                const double len = 1400.0 + 1000.0 + (double)t.chunks * t.planes * t.plane_bytes / 64.0 +
                                   (stage_mma > turn ? stage_mma : turn) * ceil_div(steps, t.per) +
                                   1500.0 + 900.0 * units;
                const double waves = per_sm_ctas / co;
                const double whole = waves < 3 ? (double)(long)(waves + 0.999) : waves + 0.5;
                double cost = whole * len;
                if (cost < rate) cost = rate;
                cost += 0.2 * rate;
                if (group < t.chunks) cost *= 1.5;
                if (!found || cost < best) {
                    found = true;
                    best = cost;
                    pick = t;
                }
            }
    }
    if (found) a = pick;
    return found;
}

template <bool FWD, int CH>
cudaError_t launch_patch_ch(const CUtensorMap &src, const CUtensorMap &flt, const PatchArgs &a,
                            int images, cudaStream_t st) {
    static DeviceOnce once;
    const cudaError_t e = opt_in_smem(once, k_conv_patch<FWD, CH>, kSmemMax - 2048);
    if (e != cudaSuccess) return e;
    const dim3 grid(images * a.tiles_x * a.tiles_y, ceil_div(a.ncols, a.bn));
    return launch_conv(k_conv_patch<FWD, CH>, grid, kCtaThreads, patch_smem(a), st, src, flt, a);
}

template <bool FWD>
cudaError_t launch_patch(const CUtensorMap &src, const CUtensorMap &flt, const PatchArgs &a,
                         int images, cudaStream_t st) {
    return a.ch == 64 ? launch_patch_ch<FWD, 64>(src, flt, a, images, st)
                      : launch_patch_ch<FWD, 32>(src, flt, a, images, st);
}

}  // namespace

cudaError_t conv_forward_tma(const Geo &g, const uint16_t *x, const uint16_t *w, const float *bias,
                             bool relu, uint16_t *y, float *y32, cudaStream_t st) {
    PatchArgs a{};
    a.classes = 1;
    a.live = 1u;
    a.cls_mul = 1;
    a.mul = g.stride;
    a.off_y = a.off_x = -g.pad;
    a.src_ch = g.C;
    a.ch = g.C <= 32 ? 32 : 64;
    a.chunks = ceil_div(g.C, a.ch);
    a.ncols = g.K;
    a.bn = column_block(g.K);
    a.b_bytes = a.bn * 2 * a.ch;
    a.planes = g.stride == 1 || (g.R == 1 && g.S == 1) ? 1 : 4;
    for (int r = 0; r < g.R; ++r)
        for (int s = 0; s < g.S; ++s) {
            Tap &t = a.tap[a.taps];
            t.plane = g.stride == 1 ? 0 : (uint8_t)((r & 1) * 2 + (s & 1));
            t.sy = (uint8_t)(g.stride == 1 ? r : r >> 1);
            t.sx = (uint8_t)(g.stride == 1 ? s : s >> 1);
            t.cls = 0;
            t.wt = (int16_t)(r * g.S + s);
            t.first = a.taps == 0;
            ++a.taps;
        }
    const int ry = g.stride == 1 ? g.R - 1 : (g.R - 1) / 2, rx = g.stride == 1 ? g.S - 1 : (g.S - 1) / 2;
    if (!conv_patch_plan(a, g.N, g.P, g.Q, ry, rx)) return cudaErrorNotSupported;
    a.out_h = g.P;
    a.out_w = g.Q;
    a.bias = bias;
    a.relu = relu;
    a.y = reinterpret_cast<__nv_bfloat16 *>(y);
    a.y32 = y32;
    CUtensorMap src, flt;
    const uint64_t sd[4] = {(uint64_t)g.C, (uint64_t)g.W, (uint64_t)g.H, (uint64_t)g.N};
    const uint32_t sb[4] = {(uint32_t)a.ch, (uint32_t)((a.pw - 1) * g.stride + 1),
                            (uint32_t)((a.ph - 1) * g.stride + 1), 1};
    const uint32_t se[4] = {1, (uint32_t)g.stride, (uint32_t)g.stride, 1};
    cudaError_t e = encode(&src, x, 4, sd, sb, se);
    const uint64_t fd[3] = {(uint64_t)g.C, (uint64_t)(g.R * g.S), (uint64_t)g.K};
    const uint32_t fb[3] = {(uint32_t)a.ch, 1, (uint32_t)a.bn}, fe[3] = {1, 1, 1};
    if (e == cudaSuccess) e = encode(&flt, w, 3, fd, fb, fe);
    return e == cudaSuccess ? launch_patch<true>(src, flt, a, g.N, st) : e;
}

cudaError_t conv_dgrad_tma(const Geo &g, const uint16_t *dy, const uint16_t *w,
                           const uint16_t *mask, uint16_t *dx, cudaStream_t st) {
    PatchArgs a{};
    const bool two = g.stride == 2;
    a.classes = two ? 4 : 1;
    a.cls_mul = two ? 2 : 1;
    a.mul = 1;
    a.src_ch = g.K;
    a.ch = g.K <= 32 ? 32 : 64;
    a.chunks = ceil_div(g.K, a.ch);
    a.ncols = g.C;
    a.bn = g.C > 128 ? 128 : round_up(g.C, 16);
    a.b_bytes = ceil_div(a.bn, 64) * a.ch * 128;
    a.mn_major = 1;
    a.planes = 1;
    // tap (r, s) of class (ph, pw): dY row i + (ph + pad - r) / 2 (stride 2,
    // matching parity) or i + pad - r; shifts are counted from the smallest
    int lo_y = 1 << 20, hi_y = -(1 << 20), lo_x = lo_y, hi_x = hi_y;
    auto offset = [&](int cls, int tap, int &o) {
        if (!two) {
            o = g.pad - tap;
            return true;
        }
        if ((cls + g.pad - tap) & 1) return false;
        o = (cls + g.pad - tap) / 2;  // exact: an even number
        return true;
    };
    for (int pass = 0; pass < 2; ++pass) {
        a.taps = 0;
        a.live = 0;
        for (int c = 0; c < a.classes; ++c)
            for (int r = 0; r < g.R; ++r)
                for (int s = 0; s < g.S; ++s) {
                    int oy, ox;
                    if (!offset(c >> 1, r, oy) || !offset(c & 1, s, ox)) continue;
                    if (pass == 0) {
                        lo_y = oy < lo_y ? oy : lo_y;
                        hi_y = oy > hi_y ? oy : hi_y;
                        lo_x = ox < lo_x ? ox : lo_x;
                        hi_x = ox > hi_x ? ox : hi_x;
                        continue;
                    }
                    Tap &t = a.tap[a.taps];
                    t.plane = 0;
                    t.sy = (uint8_t)(oy - lo_y);
                    t.sx = (uint8_t)(ox - lo_x);
                    t.cls = (uint8_t)c;
                    t.wt = (int16_t)(r * g.S + s);
                    t.first = !((a.live >> c) & 1u);
                    a.live |= 1u << c;
                    ++a.taps;
                }
    }
    a.off_y = lo_y;
    a.off_x = lo_x;
    const int oh = two ? (g.H + 1) / 2 : g.H, ow = two ? (g.W + 1) / 2 : g.W;
    if (!conv_patch_plan(a, g.N, oh, ow, hi_y - lo_y, hi_x - lo_x)) return cudaErrorNotSupported;
    a.out_h = g.H;
    a.out_w = g.W;
    a.mask = reinterpret_cast<const __nv_bfloat16 *>(mask);
    a.y = reinterpret_cast<__nv_bfloat16 *>(dx);
    CUtensorMap src, flt;
    const uint64_t sd[4] = {(uint64_t)g.K, (uint64_t)g.Q, (uint64_t)g.P, (uint64_t)g.N};
    const uint32_t sb[4] = {(uint32_t)a.ch, (uint32_t)a.pw, (uint32_t)a.ph, 1}, ones[4] = {1, 1, 1, 1};
    cudaError_t e = encode(&src, dy, 4, sd, sb, ones);
    const uint64_t fd[3] = {(uint64_t)g.C, (uint64_t)(g.R * g.S), (uint64_t)g.K};
    const uint32_t fb[3] = {64, 1, (uint32_t)a.ch};
    if (e == cudaSuccess) e = encode(&flt, w, 3, fd, fb, ones);
    return e == cudaSuccess ? launch_patch<false>(src, flt, a, g.N, st) : e;
}

namespace {

// Plan of the filter gradient; false if no stage fits in shared memory.
bool wgrad_plan(const Geo &g, WgradArgs &a, int &ch) {
    ch = g.C <= 32 ? 32 : 64;
    a.K = g.K;
    a.C = g.C;
    a.RS = g.R * g.S;
    a.stride = g.stride;
    a.pad = g.pad;
    a.k64 = g.K <= 64 ? 1 : 2;
    a.tiles_x = ceil_div(g.Q, kTileW);
    a.tiles_y = ceil_div(g.P, kTileH);
    a.tiles = g.N * a.tiles_x * a.tiles_y;
    const bool two = g.stride == 2;
    a.pw = kTileW + (two ? (g.S - 1) / 2 : g.S - 1);
    a.ph = kTileH + (two ? (g.R - 1) / 2 : g.R - 1);
    if ((a.pw - 1) * g.stride + 1 > 256 || (a.ph - 1) * g.stride + 1 > 256) return false;
    a.plane_bytes = round_up(a.pw * a.ph * 2 * ch, 1024);
    const int dy = a.k64 * kTileW * kTileH * 128;
    for (a.chunks = g.C > 64 ? 2 : 1; a.chunks >= 1; --a.chunks) {
        a.cblk = a.chunks * ch;
        a.bn = round_up(g.C < a.cblk ? g.C : a.cblk, 16);
        a.cblocks = ceil_div(g.C, a.cblk);
        // taps by the plane they read, in the order that pairs the plane of four
        // taps with that of one; groups of as many accumulators as tensor
        // memory holds, spread evenly
        static const int order[4] = {0, 3, 1, 2};
        // (an accumulator is read back in pieces of 32 columns)
        const int fit = (512 - round_up(a.bn, 32)) / a.bn + 1;
        const int most = fit < a.RS ? fit : a.RS;
        a.groups = ceil_div(a.RS, most);
        // and more groups while the tiles leave SMs idle: a CTA then reads fewer
        // accumulators back (2 images of 12 x 7, 16 -> 48, 5 x 5: 14.4 -> 5.2 us)
        const int idle = kSms / (ceil_div(g.K, 128) * a.cblocks) / a.tiles;
        if (idle > a.groups) a.groups = idle;
        const int each = ceil_div(a.RS, a.groups);
        a.groups = ceil_div(a.RS, each);
        int n = 0;
        for (int o = 0; o < 4; ++o)
            for (int r = 0; r < g.R; ++r)
                for (int s = 0; s < g.S; ++s) {
                    const int plane = two ? (r & 1) * 2 + (s & 1) : 0;
                    if (plane != order[o]) continue;
                    Tap &t = a.tap[n++];
                    t.plane = (uint8_t)plane;
                    t.sy = (uint8_t)(two ? r >> 1 : r);
                    t.sx = (uint8_t)(two ? s >> 1 : s);
                    t.wt = (int16_t)(r * g.S + s);
                }
        int planes = 0;
        for (int gr = 0; gr <= a.groups; ++gr) a.group0[gr] = gr * each < a.RS ? gr * each : a.RS;
        for (int gr = 0; gr < a.groups; ++gr) {
            a.planes[gr] = 0;
            for (int t = a.group0[gr]; t < a.group0[gr + 1]; ++t) a.planes[gr] |= 1u << a.tap[t].plane;
            const int np = __builtin_popcount(a.planes[gr]);
            planes = np > planes ? np : planes;
        }
        a.stage_bytes = dy + planes * a.chunks * a.plane_bytes;
        a.ring = (kSmemMax - 2048) / a.stage_bytes;
        if (a.ring > kMaxRing) a.ring = kMaxRing;
        if (a.ring < 1) continue;
        a.tmem_cols = tmem_columns((each - 1) * a.bn + round_up(a.bn, 32));
        // a CTA per SM, and more where a split would add more pixels in one accumulator
        // than kSplitPixels less a tile
        constexpr int kMost = kSplitPixels - kTileW * kTileH;
        const int64_t pixels = (int64_t)g.N * g.P * g.Q;
        const int blocks = ceil_div(g.K, 128) * a.cblocks * a.groups;
        const int fill = kSms / blocks, least = (int)((pixels + kMost - 1) / kMost);
        // (the last of several waves is filled, too: 64 images of 44 x 67, 8 -> 8, 7 x 7
        // 175 -> 126 us)
        const int waves = (least * blocks + kSms - 1) / kSms;
        a.splits = fill > least ? fill : waves * kSms / blocks > least ? waves * kSms / blocks : least;
        if (a.splits > a.tiles) a.splits = a.tiles;
        return true;
    }
    return false;
}

// The matrix instructions read 128 rows of dY, two 64-channel blocks, also when
// a stage holds one (the rows of the second are not used): the last stage's
// reads end inside the allocation too.
int wgrad_smem(const WgradArgs &a) {
    const int n = a.ring * a.stage_bytes;
    const int reach = (a.ring - 1) * a.stage_bytes + 2 * kTileW * kTileH * 128;
    const int m = n > reach ? n : reach;
    return m > kEpilogueSmem ? m : kEpilogueSmem;
}

template <int CH>
cudaError_t launch_wgrad(const CUtensorMap &mdy, const CUtensorMap &mx, const WgradArgs &a,
                         cudaStream_t st) {
    static DeviceOnce once;
    const cudaError_t e = opt_in_smem(once, k_wgrad_patch<CH>, kSmemMax - 2048);
    if (e != cudaSuccess) return e;
    // (one dimension: the others end at 65,535, which the splits may pass)
    const dim3 grid(ceil_div(a.K, 128) * a.cblocks * a.groups * a.splits);
    return launch_conv(k_wgrad_patch<CH>, grid, kCtaThreads, wgrad_smem(a), st, mdy, mx, a);
}

}  // namespace

size_t conv_wgrad_tma_workspace(const Geo &g) {
    WgradArgs a{};
    int ch;
    if (!wgrad_plan(g, a, ch)) return 0;
    return (size_t)a.splits * ((size_t)a.K * a.RS * a.C + a.K) * sizeof(float);
}

cudaError_t conv_wgrad_tma(const Geo &g, const uint16_t *dy, const uint16_t *x, float *dw,
                           float *dbias, float *ws, cudaStream_t st) {
    WgradArgs a{};
    int ch;
    if (!wgrad_plan(g, a, ch)) return cudaErrorNotSupported;
    a.part = ws;
    CUtensorMap mdy, mx;
    const uint64_t yd[4] = {(uint64_t)g.K, (uint64_t)g.Q, (uint64_t)g.P, (uint64_t)g.N};
    const uint32_t yb[4] = {64, kTileW, kTileH, 1}, ones[4] = {1, 1, 1, 1};
    cudaError_t e = encode(&mdy, dy, 4, yd, yb, ones);
    const uint64_t xd[4] = {(uint64_t)g.C, (uint64_t)g.W, (uint64_t)g.H, (uint64_t)g.N};
    const uint32_t xb[4] = {(uint32_t)ch, (uint32_t)((a.pw - 1) * g.stride + 1),
                            (uint32_t)((a.ph - 1) * g.stride + 1), 1};
    const uint32_t xe[4] = {1, (uint32_t)g.stride, (uint32_t)g.stride, 1};
    if (e == cudaSuccess) e = encode(&mx, x, 4, xd, xb, xe);
    if (e != cudaSuccess) return e;
    e = ch == 64 ? launch_wgrad<64>(mdy, mx, a, st) : launch_wgrad<32>(mdy, mx, a, st);
    if (e != cudaSuccess) return e;
    const bool ragged = g.P % kTileH || g.Q % kTileW;
    return conv_sum_parts(g, a.splits, ws, dw, dbias, ragged ? dy : nullptr, x, kTileH, kTileW, st);
}

cudaError_t conv_sum_parts(const Geo &g, int splits, const float *part, float *dw, float *dbias,
                           const uint16_t *ragged_dy, const uint16_t *x, int tile_h, int tile_w,
                           cudaStream_t st) {
    const int64_t count4 = (int64_t)g.K * g.R * g.S * g.C / 4, extra4 = g.K / 4;
    return launch_conv(ragged_dy ? k_sum_parts<true> : k_sum_parts<false>,
                       dim3((unsigned)((count4 + extra4 + 31) / 32)), 32 * kSumLanes, 0, st,
                       reinterpret_cast<const float4 *>(part), splits, count4, extra4,
                       reinterpret_cast<float4 *>(dw), reinterpret_cast<float4 *>(dbias),
                       EdgeFix{reinterpret_cast<const __nv_bfloat16 *>(ragged_dy),
                               reinterpret_cast<const __nv_bfloat16 *>(x), g, tile_h, tile_w});
}

cudaError_t conv_tma_take_status(int *timed_out) {
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_status, sizeof v);
    if (e == cudaSuccess && v) {
        const int zero = 0;
        e = cudaMemcpyToSymbol(g_status, &zero, sizeof zero);
    }
    *timed_out = v;
    return e;
}

cudaError_t conv_tma_set_probe(int polls) {
    return cudaMemcpyToSymbol(g_probe_polls, &polls, sizeof polls);
}

}  // namespace cnn
}  // namespace osog
