// Shared-memory Stockham FFT for sets of lines held by one CTA.
//
// A CTA owns L lines of N complex samples (N a power of two, 32..2048) in
// shared memory, line l at buf + l * line_stride(N), sample i at pad16(i).
// The transform runs as a few radix-P passes (P in {4, 8, 16}).  In each
// pass every thread loads whole butterflies into registers, the CTA
// synchronises, and the results are written back in Stockham (self-sorting)
// order, so no bit reversal is needed and a single buffer suffices.
//
// Stockham radix-P pass with sub-transform length Ns (product of the radices
// of the earlier passes), for butterfly j in [0, N/P), k = j mod Ns:
//     v_r = x[j + r N/P] * w^{r k},   w = exp(-+ 2 pi i / (Ns P))
//     V   = DFT_P(v)
//     x'[(j - k) P + k + r Ns] = V_r
// (the self-sorting formulation of Stockham's autosort FFT, e.g.
// Govindaraju et al., "High performance discrete Fourier transforms on
// graphics processors", SC 2008).  The twiddles w^{rk} come from per-pass
// tables laid out [r - 1][k] (so the lanes of a warp, which hold
// consecutive k, read consecutive entries) that the host builds in double
// precision and rounds to float once; the tables of all passes of an
// N-point transform fit in N entries.  Inverse transforms use the conjugate
// twiddles and are unnormalised.
#pragma once

#include <math.h>

#include <type_traits>

#include "osog_common.cuh"

namespace osog {

// cos and sin of 2 pi m / 16, m = 0..15 (cos(pi/8) = sqrt(2 + sqrt 2) / 2,
// sin(pi/8) = sqrt(2 - sqrt 2) / 2, cos(pi/4) = sqrt(1/2)).
__host__ __device__ constexpr float quarter_cos16(int m) {  // m in 0..4
    return m == 0 ? 1.0f
         : m == 1 ? 0.92387953251128674f
         : m == 2 ? 0.70710678118654752f
         : m == 3 ? 0.38268343236508977f
         : 0.0f;
}
__host__ __device__ constexpr float cos16(int m) {
    m &= 15;
    return m <= 4 ? quarter_cos16(m)
         : m <= 8 ? -quarter_cos16(8 - m)
         : m <= 12 ? -quarter_cos16(m - 8)
         : quarter_cos16(16 - m);
}
__host__ __device__ constexpr float sin16(int m) { return cos16(m - 4); }

// x * exp(-+ 2 pi i K / P) with K, P compile-time (P divides 16).
template <int P, int K, bool INV>
__device__ __forceinline__ float2 twc(float2 x) {
    constexpr int m = (K * 16 / P) & 15;
    if constexpr (m == 0) {
        return x;
    } else if constexpr (m == 4) {
        return INV ? make_float2(-x.y, x.x) : make_float2(x.y, -x.x);
    } else if constexpr (m == 8) {
        return make_float2(-x.x, -x.y);
    } else if constexpr (m == 12) {
        return INV ? make_float2(x.y, -x.x) : make_float2(-x.y, x.x);
    } else {
        constexpr float c = cos16(m);
        constexpr float s = INV ? sin16(m) : -sin16(m);
        return make_float2(fmaf(x.x, c, -__fmul_rn(x.y, s)), fmaf(x.x, s, __fmul_rn(x.y, c)));
    }
}

template <int P, bool INV, int K = 0>
__device__ __forceinline__ void twiddle_odds(float2 *o) {
    if constexpr (K < P / 2) {
        o[K] = twc<P, K, INV>(o[K]);
        twiddle_odds<P, INV, K + 1>(o);
    }
}

// In-register DFT of P points (radix-2 decimation in time, unrolled).
template <int P, bool INV>
__device__ __forceinline__ void dft(float2 *v) {
    if constexpr (P == 2) {
        float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else {
        float2 e[P / 2], o[P / 2];
#pragma unroll
        for (int k = 0; k < P / 2; ++k) {
            e[k] = v[2 * k];
            o[k] = v[2 * k + 1];
        }
        dft<P / 2, INV>(e);
        dft<P / 2, INV>(o);
        twiddle_odds<P, INV>(o);
#pragma unroll
        for (int k = 0; k < P / 2; ++k) {
            v[k] = cadd(e[k], o[k]);
            v[k + P / 2] = csub(e[k], o[k]);
        }
    }
}

// Radix plans: 32 = 8.4, 64 = 8.8, 128 = 8.4.4, 256 = 8.8.4, 512 = 8.8.8,
// 1024 = 16.8.8, 2048 = 16.16.8.  Below 512 points a set has two samples or
// fewer per thread, and a radix-16 pass would leave all but one or two warps
// idle while those work through 16 samples each (128 = 16.8 and 256 = 16.16,
// 256 x 256 scene: the whole
// render 22.2 -> 18.8 us).
__host__ __device__ constexpr int fft_passes(int n) { return n >= 128 ? 3 : 2; }
__host__ __device__ constexpr int fft_radix(int n, int p) {
    return n == 32 ? (p == 0 ? 8 : 4)
         : n == 64 ? 8
         : n == 128 ? (p == 0 ? 8 : 4)
         : n == 256 ? (p < 2 ? 8 : 4)
         : n == 512 ? 8
         : n == 1024 ? (p == 0 ? 16 : 8)
         : (p < 2 ? 16 : 8);
}
__host__ __device__ constexpr int fft_ns(int n, int p) {  // sub-transform length before pass p
    return p == 0 ? 1 : fft_ns(n, p - 1) * fft_radix(n, p - 1);
}
__host__ __device__ constexpr int fft_twoff(int n, int p) {  // start of pass p's table
    return p == 0 ? 0
                  : fft_twoff(n, p - 1) +
                        (fft_ns(n, p - 1) > 1 ? (fft_radix(n, p - 1) - 1) * fft_ns(n, p - 1) : 0);
}

// pad16(base + r * stride) - pad16(base) for the bases the Stockham passes
// write from: with stride >= 16 (a power of two) the carry into the padding
// term is r * stride / 16; with stride 8 the base's low part k < 8 never
// carries, leaving r / 2; with stride 1 the base is a multiple of the radix
// P <= 16 and base % 16 + r < 16.  Every offset folds to a constant once the
// r loop is unrolled.
__device__ __forceinline__ constexpr int stride_off(int stride, int r) {
    return stride >= 16 ? r * (stride + stride / 16) : stride == 8 ? 8 * r + (r >> 1) : r;
}

// Synchronisation of the threads that own line l when each line of the set
// belongs to its own group of kThreads / L threads (a named barrier per
// line, or the warp when a line has one warp).
template <int L>
__device__ __forceinline__ void line_sync(int l) {
    constexpr int TPL = kThreads / L;
    if constexpr (TPL == 32) {
        __syncwarp();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(1 + l), "r"(TPL) : "memory");
    }
}

// How the threads of a pass synchronise: the whole CTA, the group of a line
// (line_sync), or the first kThreads threads of a larger CTA.
enum FftSync { kSyncCta = 0, kSyncLine = 1, kSyncThreads = 2 };
template <int G, int L>
__device__ __forceinline__ void pass_sync(int l) {
    if constexpr (G == kSyncLine)
        line_sync<L>(l);
    else if constexpr (G == kSyncThreads)
        asm volatile("bar.sync 15, %0;" ::"n"(kThreads) : "memory");
    else
        __syncthreads();
}

// True when the passes of an N-point transform can run with one thread
// group per line: every pass has at least one butterfly per thread of the
// group (sets of 8192 samples, N >= 1024).
__host__ __device__ constexpr bool fft_grouped(int n) {
    return set_elems(n) == kMaxSetElems && n >= 1024;
}

// Butterfly q of this thread in a pass of NB butterflies per line over L
// lines: grouped, the threads [l TPL, (l + 1) TPL) take line l; otherwise
// consecutive threads take consecutive butterflies of the whole set.
template <int L, int NB, bool LINE>
__device__ __forceinline__ void butterfly_of(int q, int &l, int &j) {
    if constexpr (LINE) {
        constexpr int TPL = kThreads / L;
        l = threadIdx.x / TPL;
        j = threadIdx.x % TPL + q * TPL;
    } else {
        const int b = threadIdx.x + q * kThreads;
        l = b / NB;
        j = b % NB;
    }
}

// The same for the passes that read or write global memory; FAST > 0: consecutive
// threads take FAST consecutive lines, then the butterflies of those lines.
template <int L, int NB, int G, int FAST>
__device__ __forceinline__ void line_butterfly(int q, int &l, int &j) {
    if constexpr (FAST > 0) {
        static_assert(L % FAST == 0, "whole groups of lines");
        const int b = threadIdx.x + q * kThreads;
        l = b % FAST + b / (FAST * NB) * FAST;
        j = b / FAST % NB;
    } else {
        butterfly_of<L, NB, G == kSyncLine>(q, l, j);
    }
}

// Row strips read and write column-blocked arrays, whose block of one strip is R x B
// samples end to end.  Consecutive threads over four lines cover 128 bytes of 4 x 4
// samples and more; along one line they would take 32 or 64 bytes of every block
// (inverse rows of a 2048 x 2048 image 11.6 -> 10.6 us; 32 whole images 1607 -> 1550,
// sixteen DIC images of 1024 x 1024 305 -> 303).  Four lines are also as many as lie
// on different banks (line_stride).
constexpr int kRowFast = 4;

// Largest radix whose twiddles are formed as products (0: all read from the
// table).  A radix-P pass needs w^{r k}, r = 1..P-1: the table entries at
// r = 1, 2, 4 (and 8) are read and the others formed as products of two of
// them, which takes those reads off the load path at the cost of a few
// fused multiply-adds and a rounding error of a few units in the last place.
constexpr int kTwiddleProducts = 16;

// v[r] *= w^{r k} (conjugated for the inverse transform), r = 1..P-1, with
// t the pass's table at entry [0][k] (entries [r - 1][k] at stride NS).
template <int P, bool INV, int NS>
__device__ __forceinline__ void apply_twiddles(float2 *v, const float2 *__restrict__ t) {
    auto mul = [](float2 a, float2 w) { return INV ? cmulc(a, w) : cmul(a, w); };
    if constexpr (P == 8 && kTwiddleProducts >= 8) {
        const float2 w1 = __ldg(t), w2 = __ldg(t + NS), w4 = __ldg(t + 3 * NS);
        const float2 w3 = cmul(w2, w1);
        v[1] = mul(v[1], w1);
        v[2] = mul(v[2], w2);
        v[3] = mul(v[3], w3);
        v[4] = mul(v[4], w4);
        v[5] = mul(v[5], cmul(w4, w1));
        v[6] = mul(v[6], cmul(w4, w2));
        v[7] = mul(v[7], cmul(w4, w3));
    } else if constexpr (P == 16 && kTwiddleProducts >= 16) {
        const float2 w1 = __ldg(t), w2 = __ldg(t + NS), w4 = __ldg(t + 3 * NS),
                     w8 = __ldg(t + 7 * NS);
        const float2 w3 = cmul(w2, w1), w5 = cmul(w4, w1), w6 = cmul(w4, w2), w7 = cmul(w4, w3);
        v[1] = mul(v[1], w1);
        v[2] = mul(v[2], w2);
        v[3] = mul(v[3], w3);
        v[4] = mul(v[4], w4);
        v[5] = mul(v[5], w5);
        v[6] = mul(v[6], w6);
        v[7] = mul(v[7], w7);
        v[8] = mul(v[8], w8);
        v[9] = mul(v[9], cmul(w8, w1));
        v[10] = mul(v[10], cmul(w8, w2));
        v[11] = mul(v[11], cmul(w8, w3));
        v[12] = mul(v[12], cmul(w8, w4));
        v[13] = mul(v[13], cmul(w8, w5));
        v[14] = mul(v[14], cmul(w8, w6));
        v[15] = mul(v[15], cmul(w8, w7));
    } else {
#pragma unroll
        for (int r = 1; r < P; ++r) v[r] = mul(v[r], __ldg(t + (r - 1) * NS));
    }
}

// One Stockham pass over L lines of N points.  G: one thread group per line
// (fft_grouped(N)); the pass then synchronises only the line's group.
template <int N, int L, int P, int NS, bool INV, int G = kSyncCta>
__device__ __forceinline__ void stockham_pass(float2 *buf, const float2 *__restrict__ tw) {
    static_assert(NS == 1 || NS == 8 || NS % 16 == 0, "unsupported Stockham stride");
    constexpr int NB = N / P;
    constexpr int TOT = L * NB;
    constexpr int PER = (TOT + kThreads - 1) / kThreads;
    constexpr int LS = line_stride(N);
    static_assert(G != kSyncLine || (NB % (kThreads / L) == 0 && kThreads % L == 0), "grouped pass");
    float2 v[PER][P];
    int l = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int j;
        butterfly_of<L, NB, G == kSyncLine>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            if constexpr (NB % 16 == 0) {
                const float2 *src = buf + l * LS + pad16(j);
#pragma unroll
                for (int r = 0; r < P; ++r) v[q][r] = src[r * (NB + NB / 16)];
            } else {
                const float2 *src = buf + l * LS;
#pragma unroll
                for (int r = 0; r < P; ++r) v[q][r] = src[pad16(j + r * NB)];
            }
        }
    }
    pass_sync<G, L>(l);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int j;
        butterfly_of<L, NB, G == kSyncLine>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            const int k = j & (NS - 1);
            if constexpr (NS > 1) apply_twiddles<P, INV, NS>(v[q], tw + k);  // entries [r - 1][k]
            dft<P, INV>(v[q]);
            float2 *dst = buf + l * LS + pad16((j - k) * P + k);
#pragma unroll
            for (int r = 0; r < P; ++r) dst[stride_off(NS, r)] = v[q][r];
        }
    }
    pass_sync<G, L>(l);
}

// Full FFT of the L lines (forward: exp(-2 pi i jk/N); inverse: conjugate,
// unnormalised), following the radix plan above.  tw is the N-point
// transform's table block.
template <int N, int L, bool INV, int G = kSyncCta, int PASS = 0>
__device__ __forceinline__ void fft_lines(float2 *buf, const float2 *__restrict__ tw) {
    if constexpr (PASS < fft_passes(N)) {
        stockham_pass<N, L, fft_radix(N, PASS), fft_ns(N, PASS), INV, G>(buf,
                                                                         tw + fft_twoff(N, PASS));
        fft_lines<N, L, INV, G, PASS + 1>(buf, tw);
    }
}

// Passes [PASS, END) of the radix plan, each an in-place Stockham pass
// (G: grouped, see stockham_pass).
template <int N, int L, bool INV, int PASS, int END, int G = kSyncCta>
__device__ __forceinline__ void fft_pass_range(float2 *buf, const float2 *__restrict__ tw) {
    if constexpr (PASS < END) {
        stockham_pass<N, L, fft_radix(N, PASS), fft_ns(N, PASS), INV, G>(buf,
                                                                         tw + fft_twoff(N, PASS));
        fft_pass_range<N, L, INV, PASS + 1, END, G>(buf, tw);
    }
}

// The first pass of the plan (stride 1, no twiddles) with its inputs taken
// from ld(l, i), sample i of line l, instead of from buf: the kernels fold
// the step that produces a line (a global load, the exit wave, a transfer
// function) into the pass.  The butterflies and the order of every
// operation are those of stockham_pass, so the results are bitwise the same.
// IN_PLACE: ld reads buf itself, and the threads synchronise between the
// loads and the writes.  G: grouped (see stockham_pass); ld(l, i) may then
// read only line l of buf.  FAST: as in fft_last_pass.  Ends with a barrier
// (the line's, grouped).
template <int N, int L, bool INV, bool IN_PLACE, int G, int FAST = 0, class Ld>
__device__ __forceinline__ void fft_first_pass(float2 *buf, Ld ld) {
    constexpr int P = fft_radix(N, 0);
    constexpr int NB = N / P;
    constexpr int TOT = L * NB;
    constexpr int PER = (TOT + kThreads - 1) / kThreads;
    constexpr int LS = line_stride(N);
    static_assert(G != kSyncLine || (NB % (kThreads / L) == 0 && kThreads % L == 0), "grouped pass");
    static_assert(!(FAST > 0 && G == kSyncLine), "one thread mapping");
    float2 v[PER][P];
    int l = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int j;
        line_butterfly<L, NB, G, FAST>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
#pragma unroll
            for (int r = 0; r < P; ++r) v[q][r] = ld(l, j + r * NB);
        }
    }
    if constexpr (IN_PLACE) {
        pass_sync<G, L>(l);
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int j;
        line_butterfly<L, NB, G, FAST>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            dft<P, INV>(v[q]);
            float2 *dst = buf + l * LS + pad16(j * P);
#pragma unroll
            for (int r = 0; r < P; ++r) dst[r] = v[q][r];
        }
    }
    pass_sync<G, L>(l);
}

// The last pass of the plan with its outputs handed to st(l, i, value),
// sample i of line l, instead of written back to buf (the kernels store
// straight to global memory).  Arithmetic as in stockham_pass.  FAST > 0:
// consecutive threads take FAST consecutive lines (columns of a block, rows of a
// strip, interleaved in global memory; the pass before must end with a CTA
// barrier); G: grouped (see stockham_pass); else consecutive butterflies of
// the whole set.  buf is only read, so there is no barrier.  st may take a
// fourth argument, the number of the output among the thread's own (a constant
// once the loops are unrolled; fft_last_outputs of them).
template <int N, int L>
__host__ __device__ constexpr int fft_last_outputs() {
    constexpr int P = fft_radix(N, fft_passes(N) - 1);
    return (L * (N / P) + kThreads - 1) / kThreads * P;
}
template <int N, int L, bool INV, int FAST, int G, class St>
__device__ __forceinline__ void fft_last_pass(const float2 *buf, const float2 *__restrict__ tw,
                                              St st) {
    constexpr int PASS = fft_passes(N) - 1;
    constexpr int P = fft_radix(N, PASS), NS = fft_ns(N, PASS);
    static_assert(NS * P == N && NS > 1, "the last pass of the plan");
    static_assert(!(FAST > 0 && G == kSyncLine), "one thread mapping");
    constexpr int NB = N / P;
    constexpr int TOT = L * NB;
    constexpr int PER = (TOT + kThreads - 1) / kThreads;
    constexpr int LS = line_stride(N);
    const float2 *__restrict__ t = tw + fft_twoff(N, PASS);
    float2 v[PER][P];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int l, j;
        line_butterfly<L, NB, G, FAST>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            if constexpr (NB % 16 == 0) {
                const float2 *src = buf + l * LS + pad16(j);
#pragma unroll
                for (int r = 0; r < P; ++r) v[q][r] = src[r * (NB + NB / 16)];
            } else {
                const float2 *src = buf + l * LS;
#pragma unroll
                for (int r = 0; r < P; ++r) v[q][r] = src[pad16(j + r * NB)];
            }
        }
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int l, j;
        line_butterfly<L, NB, G, FAST>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            apply_twiddles<P, INV, NS>(v[q], t + j);
            dft<P, INV>(v[q]);
#pragma unroll
            for (int r = 0; r < P; ++r) {
                if constexpr (std::is_invocable_v<St, int, int, float2, int>)
                    st(l, j + r * NS, v[q][r], q * P + r);
                else
                    st(l, j + r * NS, v[q][r]);
            }
        }
    }
}

// ------------------------------------------------------- transposed passes
// The DFT matrix is symmetric, so the plan's passes transposed and in reverse order
// are the same transform: pass p loads from where the pass above stores, transforms,
// multiplies by the same twiddles and stores to where that pass loads from.  Its first
// pass takes samples j + r NS of the plan's last, which are the outputs a thread of
// fft_last_pass holds: what follows a transform (a product with a transfer function)
// and the transform back need no pass over shared memory in between, and the slots
// are the thread's own, so no barrier either.
template <int N, int L, int PASS, bool LOAD>
__device__ __forceinline__ void line_slots(float2 *buf, int l, int j, float2 *v) {
    constexpr int P = fft_radix(N, PASS), NB = N / P;  // samples j + r NB of line l
    float2 *b = buf + l * line_stride(N) + (NB % 16 == 0 ? pad16(j) : 0);
#pragma unroll
    for (int r = 0; r < P; ++r) {
        float2 &x = b[NB % 16 == 0 ? r * (NB + NB / 16) : pad16(j + r * NB)];
        if constexpr (LOAD)
            v[r] = x;
        else
            x = v[r];
    }
}

// First transposed pass, inputs from ld(l, i), or ld(l, i, the number of the input
// among the thread's own: as in fft_last_pass); ld may read any memory but other
// threads' slots of buf.  Ends with a barrier (the line's, grouped).
template <int N, int L, bool INV, int G, class Ld>
__device__ __forceinline__ void fft_t_first_pass(float2 *buf, const float2 *__restrict__ tw, Ld ld) {
    constexpr int PASS = fft_passes(N) - 1;
    constexpr int P = fft_radix(N, PASS), NS = fft_ns(N, PASS);
    constexpr int TOT = L * NS, PER = (TOT + kThreads - 1) / kThreads;
    const float2 *__restrict__ t = tw + fft_twoff(N, PASS);
    int l = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int j;
        butterfly_of<L, NS, G == kSyncLine>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            float2 v[P];
#pragma unroll
            for (int r = 0; r < P; ++r) {
                if constexpr (std::is_invocable_v<Ld, int, int, int>)
                    v[r] = ld(l, j + r * NS, q * P + r);
                else
                    v[r] = ld(l, j + r * NS);
            }
            dft<P, INV>(v);
            apply_twiddles<P, INV, NS>(v, t + j);
            line_slots<N, L, PASS, false>(buf, l, j, v);
        }
    }
    pass_sync<G, L>(l);
}

// The plan's last pass, f(l, i, value) on its outputs, and the first transposed
// pass of the transform back, in registers (INV: the first one is the inverse).
template <int N, int L, bool INV, int G, class F>
__device__ __forceinline__ void fft_turn_pass(float2 *buf, const float2 *__restrict__ tw, F f) {
    constexpr int PASS = fft_passes(N) - 1;
    constexpr int P = fft_radix(N, PASS), NS = fft_ns(N, PASS);
    constexpr int TOT = L * NS, PER = (TOT + kThreads - 1) / kThreads;
    const float2 *__restrict__ t = tw + fft_twoff(N, PASS);
    int l = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int j;
        butterfly_of<L, NS, G == kSyncLine>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            float2 v[P];
            line_slots<N, L, PASS, true>(buf, l, j, v);
            apply_twiddles<P, INV, NS>(v, t + j);
            dft<P, INV>(v);
#pragma unroll
            for (int r = 0; r < P; ++r) v[r] = f(l, j + r * NS, v[r]);
            dft<P, !INV>(v);
            apply_twiddles<P, !INV, NS>(v, t + j);
            line_slots<N, L, PASS, false>(buf, l, j, v);
        }
    }
    pass_sync<G, L>(l);
}

// The transposed passes between the first and the last.
template <int N, int L, bool INV, int G, int PASS = fft_passes(N) - 2>
__device__ __forceinline__ void fft_t_mid_passes(float2 *buf, const float2 *__restrict__ tw) {
    if constexpr (PASS >= 1) {
        constexpr int P = fft_radix(N, PASS), NS = fft_ns(N, PASS), NB = N / P;
        constexpr int TOT = L * NB, PER = (TOT + kThreads - 1) / kThreads;
        float2 v[PER][P];
        int l = 0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            int j;
            butterfly_of<L, NB, G == kSyncLine>(q, l, j);
            if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
                const int k = j & (NS - 1);
                const float2 *src = buf + l * line_stride(N) + pad16((j - k) * P + k);
#pragma unroll
                for (int r = 0; r < P; ++r) v[q][r] = src[stride_off(NS, r)];
            }
        }
        pass_sync<G, L>(l);
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            int j;
            butterfly_of<L, NB, G == kSyncLine>(q, l, j);
            if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
                dft<P, INV>(v[q]);
                apply_twiddles<P, INV, NS>(v[q], tw + fft_twoff(N, PASS) + (j & (NS - 1)));
                line_slots<N, L, PASS, false>(buf, l, j, v[q]);
            }
        }
        pass_sync<G, L>(l);
        fft_t_mid_passes<N, L, INV, G, PASS - 1>(buf, tw);
    }
}

// The last transposed pass, outputs to st(l, i, value); FAST, G as in fft_last_pass.
template <int N, int L, bool INV, int FAST, int G, class St>
__device__ __forceinline__ void fft_t_last_pass(const float2 *buf, St st) {
    constexpr int P = fft_radix(N, 0), NB = N / P;
    constexpr int TOT = L * NB, PER = (TOT + kThreads - 1) / kThreads;
    static_assert(!(FAST > 0 && G == kSyncLine), "one thread mapping");
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        int l, j;
        line_butterfly<L, NB, G, FAST>(q, l, j);
        if (G == kSyncLine || TOT % kThreads == 0 || threadIdx.x + q * kThreads < TOT) {
            float2 v[P];
            const float2 *src = buf + l * line_stride(N) + pad16(j * P);
#pragma unroll
            for (int r = 0; r < P; ++r) v[r] = src[r];
            dft<P, INV>(v);
#pragma unroll
            for (int r = 0; r < P; ++r) st(l, j + r * NB, v[r]);
        }
    }
}

// Host: the twiddle tables of an n-point transform, n entries, in double
// precision rounded once to float: pass p's block holds
// exp(-2 pi i r k / (Ns P)) at [(r - 1) Ns + k], r = 1..P-1, k = 0..Ns-1.
__host__ inline void fill_twiddles(int n, float2 *out) {
    const double two_pi = 6.283185307179586476925286766559;
    for (int i = 0; i < n; ++i) out[i] = make_float2(0.f, 0.f);
    for (int p = 0; p < fft_passes(n); ++p) {
        const int P = fft_radix(n, p), NS = fft_ns(n, p);
        if (NS == 1) continue;
        float2 *t = out + fft_twoff(n, p);
        for (int r = 1; r < P; ++r)
            for (int k = 0; k < NS; ++k) {
                const long m = (long)r * k % (long)(NS * P);
                const double ang = two_pi * (double)m / (double)(NS * P);
                t[(r - 1) * NS + k] = make_float2((float)cos(ang), (float)-sin(ang));
            }
    }
}

}  // namespace osog
