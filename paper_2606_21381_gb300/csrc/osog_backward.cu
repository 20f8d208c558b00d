// Adjoint of the render (osog_render_backward): gradients of a loss of the
// images with respect to every particle field and to the optics scalars
// (defocus, shear length, shear angle, DIC bias).
//
// With E the exit wave, G its row DFT, E^ = DFT_cols(G), Q_m =
// IDFT_cols(E^ H_m) and E_m = IDFT_rows(Q_m), I_m = |E_m|^2, and complex
// gradients g = dL/dRe + i dL/dIm, the chain runs backwards as
//   rows    dL/dQ_m = DFT_rows(2 gI_m E_m)               (E_m recomputed)
//   column  dL/dZ_m = DFT_cols(dL/dQ_m),  dL/dE^ = sum_m conj(H_m) dL/dZ_m,
//           dL/dG = IDFT_cols(dL/dE^);  dL/d(optics) = sum Re(conj(dL/dZ_m)
//           E^ dH_m/d(optics))                             (E^ recomputed)
//   strip   dL/dE = IDFT_rows(dL/dG); OPD and ATT re-rasterised, E recomputed;
//           dL/dOPD = (2 pi / lambda) Re(conj(dL/dE) i E),
//           dL/dATT = -Re(conj(dL/dE) E); each particle's pixels are then
//           gathered by one warp into a partial per (band slot, strip)
//   reduce  fixed-order sums of the partials per particle and of the
//           per-block optics partials.
// The intermediates G and Q_m of the recomputed forward pass are overwritten
// in place by dL/dG and dL/dQ_m.  Every sum runs in a fixed order, so the
// gradients are bitwise reproducible.
#include "osog_strip.cuh"

namespace osog {

namespace {

// Deterministic warp sum (fixed butterfly pattern).
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
    return v;
}

// The sums of eight values over the lanes of a warp: lanes exchange halves of
// the values while they add (nine shuffles instead of forty), in a fixed order.
// Lane l ends with the sum of value (l >> 2) & 7 as 4 b4 + 2 b3 + b2 of its bits.
__device__ __forceinline__ float warp_sum8(float (&v)[8], int lane) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = lane & 16;
        const float give = up ? v[i] : v[i + 4], keep = up ? v[i + 4] : v[i];
        v[i] = keep + __shfl_xor_sync(kFull, give, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool up = lane & 8;
        const float give = up ? v[i] : v[i + 2], keep = up ? v[i + 2] : v[i];
        v[i] = keep + __shfl_xor_sync(kFull, give, 8);
    }
    const bool up = lane & 4;
    const float give = up ? v[0] : v[1], keep = up ? v[1] : v[0];
    float s = keep + __shfl_xor_sync(kFull, give, 4);
    s += __shfl_xor_sync(kFull, s, 2);
    return s + __shfl_xor_sync(kFull, s, 1);
}

// The thread groups of the passes (see fft_grouped).
template <int N>
constexpr int kGroup = fft_grouped(N) ? kSyncLine : kSyncCta;

// Rows: the inverse transform's first pass takes Q from global memory, its last
// multiplies by 2 gI and goes on as the first (transposed) pass of the forward
// transform, whose last stores the result over Q.
template <int N>
__global__ void __launch_bounds__(kThreads, 2) k_bwd_rows(const __grid_constant__ BwdRowsArgs a) {
    pdl_enter_spread(a.geo, a.S);
    constexpr int L = set_elems(N) / N, G = kGroup<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *bufE = reinterpret_cast<float2 *>(smem_raw);
    const Geometry &geo = a.geo;
    const int sm = blockIdx.y, K = a.K, R = geo.R, B = geo.B, lb = ilog2(B), H = geo.H;
    const int y0 = blockIdx.x * R;
    float2 *Qm = a.w.Q + (size_t)sm * geo.nblocks * H * B;
    const int2 cr = a.w.hull[sm / K];
    fft_first_pass<N, L, true, false, kSyncCta, kRowFast>(bufE, [&](int l, int kx) -> float2 {
        const int fx = kx < N / 2 ? kx : kx - N;
        return l < R && fx >= cr.x && fx <= cr.y
                   ? Qm[((size_t)(kx >> lb) * H + y0 + l) * B + (kx & (B - 1))]
                   : make_float2(0.f, 0.f);
    });
    fft_pass_range<N, L, true, 1, fft_passes(N) - 1, G>(bufE, a.tw);  // E_m rows
    const float *gI = a.grad_image + ((size_t)sm * H + y0) * N;
    fft_turn_pass<N, L, true, G>(bufE, a.tw, [&](int l, int x, float2 v) {
        const float g2 = l < R ? 2.f * gI[(size_t)l * N + x] : 0.f;
        return make_float2(g2 * v.x, g2 * v.y);
    });
    fft_t_mid_passes<N, L, false, G>(bufE, a.tw);  // adjoint of the inverse row DFT
    if constexpr (G == kSyncLine) __syncthreads();
    fft_t_last_pass<N, L, false, kRowFast, kSyncCta>(bufE, [&](int l, int kx, float2 v) {
        const int fx = kx < N / 2 ? kx : kx - N;
        if (l < R && fx >= cr.x && fx <= cr.y)
            Qm[((size_t)(kx >> lb) * H + y0 + l) * B + (kx & (B - 1))] = v;
    });
}

// Columns: the last pass of each modality's transform hands dL/dZ_m to the
// accumulation in registers, and the last of the inverse one stores over G.
template <int N>
__global__ void __launch_bounds__(kThreads, 1) k_bwd_column(const __grid_constant__ BwdColumnArgs a) {
    pdl_enter_spread(a.geo, a.S);
    constexpr int L = set_elems(N) / N;
    constexpr int LS = line_stride(N);
    constexpr int NW = kThreads / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *bufE = reinterpret_cast<float2 *>(smem_raw);
    float2 *bufZ = bufE + L * LS;
    int2 *chords = reinterpret_cast<int2 *>(bufZ + L * LS);
    float *red = reinterpret_cast<float *>(chords + kMaxModes * L);
    const Geometry &geo = a.geo;
    const int s = blockIdx.y, bk = blockIdx.x, K = a.K;
    const int B = geo.B, lb = ilog2(B), half = geo.W / 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *opart = a.opart + ((size_t)s * geo.nblocks + bk) * 4;
    const int2 cr = a.w.hull[s];
    if (!block_active(geo, bk, cr)) {  // no pupil passes these columns: no gradient
        if (threadIdx.x < 4) opart[threadIdx.x] = 0.f;
        return;
    }
    float2 *Gb = a.w.G + ((size_t)s * geo.nblocks + bk) * N * B;
    // The first pass of a block's columns, read from its global layout: as a copy to
    // shared memory and a pass the kernel took 19.3 us on a 1024 x 1024 image and the
    // whole adjoint 106.2 us; so 104.8 (107.4 with the strips' copy of G, too).
    auto first_pass = [&](float2 *buf, const float2 *src) {
        fft_first_pass<N, L, false, false, kSyncCta, L>(buf, [&](int c, int y) -> float2 {
            const int kx = bk * B + c, fx = kx < half ? kx : kx - geo.W;
            return c < B && fx >= cr.x && fx <= cr.y ? src[(size_t)y * B + c] : make_float2(0.f, 0.f);
        });
    };
    for (int j = threadIdx.x; j < K * B; j += kThreads) {  // this block's chords
        const int m = j >> lb, c = j & (B - 1), kx = bk * B + c;
        chords[m * L + c] = mode_chord(a.md[s][m], kx < half ? kx : kx - geo.W, N);
    }
    first_pass(bufE, Gb);
    first_pass(bufZ, a.w.Q + (((size_t)s * K) * geo.nblocks + bk) * N * B);
    fft_pass_range<N, L, false, 1, fft_passes(N)>(bufE, a.tw);  // E^ of the block's columns
    constexpr int OUT = fft_last_outputs<N, L>();
    float2 acc[OUT];
#pragma unroll
    for (int i = 0; i < OUT; ++i) acc[i] = make_float2(0.f, 0.f);
    float po[4] = {0.f, 0.f, 0.f, 0.f};
    for (int m = 0; m < K; ++m) {
        const ModeDev md = live_mode(a.md[s][m]);
        if (m > 0) {
            __syncthreads();  // the modality before has read bufZ
            first_pass(bufZ, a.w.Q + (((size_t)s * K + m) * geo.nblocks + bk) * N * B);
        }
        // dL/dZ_m (adjoint of the inverse column DFT)
        fft_pass_range<N, L, false, 1, fft_passes(N) - 1>(bufZ, a.tw);
        fft_last_pass<N, L, false, 0, kSyncCta>(bufZ, a.tw, [&](int c, int y, float2 gz, int i) {
            if (c >= B) return;
            const int kx = bk * B + c;
            const int fx = kx < half ? kx : kx - geo.W;
            const int fy = y < N / 2 ? y : y - N;
            const int2 ch = chords[m * L + c];
            if (fy >= ch.x && fy <= ch.y) {
                float2 h, dh[4];
                transfer_grad(md, fx, fy, h, dh);
                const float2 eh = bufE[c * LS + pad16(y)];
                acc[i] = cadd(acc[i], cmulc(gz, h));  // conj(H) dL/dZ
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 w = cmul(eh, dh[k]);
                    po[k] = fmaf(gz.x, w.x, fmaf(gz.y, w.y, po[k]));
                }
            }
        });
    }
    // dL/dG (adjoint of the forward column DFT), from acc's own places
    fft_t_first_pass<N, L, true, kSyncCta>(bufE, a.tw, [&](int, int, int i) { return acc[i]; });
    fft_t_mid_passes<N, L, true, kSyncCta>(bufE, a.tw);
    fft_t_last_pass<N, L, true, L, kSyncCta>(bufE, [&](int c, int y, float2 v) {
        if (c < B) Gb[(size_t)y * B + c] = v;
    });
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float v = warp_sum(po[k]);
        if (lane == 0) red[warp * 4 + k] = v;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        float v = 0.f;
        for (int w = 0; w < NW; ++w) v += red[w * 4 + threadIdx.x];
        opart[threadIdx.x] = v;
    }
}

// WIDE as in k_strip_forward: 1024 threads rasterise and gather, the first
// kThreads of them transform.
template <int N, bool WIDE>
__global__ void __launch_bounds__(WIDE ? kWideThreads : kThreads, 1)
k_bwd_strip(const __grid_constant__ BwdStripArgs a) {
    constexpr int NT = WIDE ? kWideThreads : kThreads;
    pdl_enter_spread(a.geo, a.S);
    constexpr int L = set_elems(N) / N;
    constexpr int LS = line_stride(N);
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *bufG = reinterpret_cast<float2 *>(smem_raw);
    float2 *bufO = bufG + L * LS;
    PRec *srec = reinterpret_cast<PRec *>(bufO + L * LS);
    RRec *srrec = reinterpret_cast<RRec *>(srec + kThreads);
    Rect *srect = reinterpret_cast<Rect *>(srrec + kThreads);
    int *sslot = reinterpret_cast<int *>(srect + kThreads);
    int *wsum = sslot + kThreads;
    const Geometry &geo = a.geo;
    const int s = blockIdx.y;
    const int y0 = blockIdx.x * geo.R, ylast = y0 + geo.R - 1;
    const int RN = geo.R * N;
    const SceneDev &sc = a.sc[s];
    const int2 cr = a.w.hull[s];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4 *o4 = reinterpret_cast<float4 *>(bufO);
    for (int i = threadIdx.x; i < geo.R * LS / 2; i += NT) o4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!WIDE || threadIdx.x < kThreads) {  // dL/dE (the raster's barriers order it and the zeros)
        constexpr int G = WIDE ? kSyncThreads : kSyncCta;
        const int B = geo.B, lb = ilog2(B), H = geo.H, R = geo.R;
        const float2 *Gs = a.w.G + (size_t)s * H * N;
        fft_first_pass<N, L, true, false, G, kRowFast>(bufG, [&](int l, int kx) -> float2 {
            const int fx = kx < N / 2 ? kx : kx - N;
            return l < R && fx >= cr.x && fx <= cr.y
                       ? Gs[((size_t)(kx >> lb) * H + y0 + l) * B + (kx & (B - 1))]
                       : make_float2(0.f, 0.f);
        });
        fft_pass_range<N, L, true, 1, fft_passes(N), G>(bufG, a.tw);
    }
    // OPD and ATT as fixed-point accumulators in bufO (its staging shares
    // the gather's staging area below, used only after the raster)
    raster_strip<N, kAccPhase, NT>(geo, a.w, sc, s, y0, geo.R, bufO,
                               reinterpret_cast<unsigned char *>(srec));
    __syncthreads();
    const float k2pi = 3.14159265358979323846f * sc.two_over_lambda;   // 2 pi / lambda
    for (int e = threadIdx.x; e < RN; e += NT) {
        {
            const int idx = (e / N) * LS + pad16(e % N);
            const float2 g = bufG[idx];
            const float2 E = exit_wave_fixed(PhaseSlot<N>::load(bufO, e / N, e % N));
            const float ex = E.x, ey = E.y;
            bufG[idx] = make_float2(k2pi * fmaf(g.y, ex, -g.x * ey), -fmaf(g.x, ex, g.y * ey));
        }
    }
    __syncthreads();
    // Gather: one warp per staged particle, partial per (band slot, strip).
    const int band = y0 / geo.BH;
    const int spb = geo.BH / geo.R, kstrip = (y0 - band * geo.BH) / geo.R;
    const int32_t *off = a.w.band_off + (size_t)s * (geo.nbands + 1);
    const int hi = min(off[band + 1], sc.pair_cap);
    const int lo = min(off[band], hi);
    const int32_t *ids = a.w.pairs + sc.pair0;
    const unsigned lt = lanemask_lt();
    for (int base = lo; base < hi; base += kThreads) {
        // the first kThreads threads stage kThreads entries
        const int i = WIDE && threadIdx.x >= kThreads ? hi : base + threadIdx.x;
        int id = 0;
        Rect q = {1, 0, 1, 0};
        if (i < hi) {
            id = ids[i];
            q = a.w.rect[id];
        }
        const bool keep = i < hi && q.y0 <= ylast && q.y1 >= y0;
        const unsigned m = __ballot_sync(kFull, keep);
        if (lane == 0 && warp < kThreads / 32) wsum[warp] = __popc(m);
        __syncthreads();
        int before = 0, nl = 0;
#pragma unroll
        for (int k = 0; k < kThreads / 32; ++k) {
            const int c = wsum[k];
            before += k < warp ? c : 0;
            nl += c;
        }
        if (keep) {
            const int slot = before + __popc(m & lt);
            srect[slot] = q;
            srec[slot] = a.w.rec[id];
            srrec[slot] = a.w.rrec[id];
            sslot[slot] = i;
        }
        __syncthreads();
        for (int k = warp; k < nl; k += NW) {
            const PRec r = srec[k];
            const RRec rr = srrec[k];
            const Rect rq = srect[k];
            const int ya = max((int)rq.y0, y0), yb = min((int)rq.y1, ylast);
            const int bh = yb - ya + 1;  // at most R <= 32 rows
            const int lyn = bh <= 1 ? 1 : 1 << (32 - __clz(bh - 1));
            const int lxn = 32 / lyn, shx = ilog2(lxn);
            const int lx = lane & (lxn - 1), ly = lane >> shx;
            // lane l finds the span of row ya + l (as in the raster); a pixel's
            // lanes take it from there
            RowItem it;
            it.hdr = 0u;
            it.f[0] = it.f[1] = it.f[2] = it.f[3] = 0.f;
            if (lane >= bh || !make_row_item<kAccPhase>(rr, rq.x0, rq.x1, ya + lane, 0, 1.f, it))
                it.hdr = 0u;
            const uint32_t hdr = __shfl_sync(kFull, it.hdr, ly);
            const int yy = ya + ly;
            const float ey = (float)yy + 0.5f - r.cy;
            const int xe = (int)(hdr & 0xFFFu) + (int)((hdr >> 12) & 0xFFFu);
            const float2 *row = bufG + (min(yy, ylast) - y0) * LS;
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (rr.kind == 0) {
                const float xlh = __shfl_sync(kFull, it.f[0], ly), xll = __shfl_sync(kFull, it.f[1], ly);
                const float xrh = __shfl_sync(kFull, it.f[2], ly), xrl = __shfl_sync(kFull, it.f[3], ly);
                const EllipseGrad e = ellipse_grad(r, rr.p[2]);
                for (int xx = (int)(hdr & 0xFFFu) + lx; xx < xe; xx += lxn) {
                    const float X = (float)xx + 0.5f;
                    const float ep = __fadd_rn(__fsub_rn(xrh, X), xrl);
                    const float en = __fsub_rn(__fsub_rn(X, xlh), xll);
                    const float qq = __fmul_rn(ep, en);
                    if (qq > 1e-30f) {
                        const float2 g = row[pad16(xx)];
                        ellipse_pixel_grad(r, e, qq, X - r.cx, ey, g.x, g.y, acc);
                    }
                }
            } else {
                for (int xx = (int)(hdr & 0xFFFu) + lx; xx < xe; xx += lxn) {
                    const float2 g = row[pad16(xx)];
                    prism_grad(r, (float)xx + 0.5f - r.cx, ey, g.x, g.y, acc);
                }
            }
            const float v = warp_sum8(acc, lane);
            float *dst = a.part + ((size_t)(sc.pair0 + sslot[k]) * spb + kstrip) * 8;
            if ((lane & 3) == 0) dst[((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = v;
        }
        __syncthreads();
    }
}

// Eight lanes per particle, one per field, kReduceParticles particles per CTA:
// lane f adds entry f of the particle's partials (a 32-byte line) in band and
// strip order, loading eight partials at a time before it adds them.
constexpr int kReduceParticles = kChunk / 8;

__global__ void __launch_bounds__(kChunk) k_bwd_reduce(const __grid_constant__ BwdReduceArgs a) {
    pdl_enter();
    const Geometry &geo = a.geo;
    const int pblocks = a.nchunks * (kChunk / kReduceParticles);
    if ((int)blockIdx.x >= pblocks) {  // optics: sum the per-block partials
        // Warp f sums component f: lane l adds blocks l, l + 32, ... in
        // double, then a fixed butterfly combines the lanes (same order on
        // every run).
        const int s = blockIdx.x - pblocks;
        const int f = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (f < 4) {
            double v = 0.0;
            for (int bk = lane; bk < geo.nblocks; bk += 32)
                v += (double)a.opart[((size_t)s * geo.nblocks + bk) * 4 + f];
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
            if (lane == 0) a.grad_optics[s * 4 + f] = (float)v;
        }
        return;
    }
    const int chunk = blockIdx.x / (kChunk / kReduceParticles);
    int s = 0;
    for (int t = 1; t < a.S; ++t)
        if (a.sc[t].chunk0 <= chunk) s = t;
    const SceneDev &sc = a.sc[s];
    const int f = threadIdx.x & 7;
    const int local = (chunk - sc.chunk0) * kChunk +
                      (blockIdx.x % (kChunk / kReduceParticles)) * kReduceParticles + (threadIdx.x >> 3);
    if (local >= sc.n) return;
    const int p = sc.p0 + local;
    const Rect q = a.w.rect[p];
    float acc = 0.f;
    if (q.x0 <= q.x1 && q.y0 <= q.y1) {
        const int spb = geo.BH / geo.R;
        const int b0 = q.y0 / geo.BH;
        const int nb = min(q.y1 / geo.BH - b0 + 1, a.w.slotmap_ppp);
        const int32_t *sm = a.w.slotmap + (size_t)p * a.w.slotmap_ppp;
        for (int e0 = 0; e0 < nb * spb; e0 += 8) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int e = e0 + i, j = e / spb, k = e - j * spb;
                const int r0 = (b0 + j) * geo.BH + k * geo.R;
                v[i] = 0.f;
                if (e < nb * spb && r0 <= q.y1 && r0 + geo.R - 1 >= q.y0) {
                    const int slot = sm[j];
                    if (slot >= 0) v[i] = a.part[((size_t)(sc.pair0 + slot) * spb + k) * 8 + f];
                }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) acc += v[i];
        }
    }
    a.grad_soa[(int64_t)f * a.ld + p] = acc;
    if (f == 0) a.grad_soa[(int64_t)8 * a.ld + p] = 0.f;
}

// Shared memory of a strip of the adjoint: two sets, then the raster's items or
// the gather's staged particles (kThreads of them).
constexpr size_t bwd_strip_smem(int W, int threads) {
    const int L = set_elems(W) / W;
    const size_t gather = kThreads * (sizeof(PRec) + sizeof(RRec) + sizeof(Rect) + sizeof(int)) + 64;
    const size_t raster = threads == kThreads ? raster_smem<kThreads>() : raster_smem<kWideThreads>();
    return (size_t)2 * L * line_stride(W) * sizeof(float2) + (gather > raster ? gather : raster);
}

// Where 1024 threads pay: strips of 8 rows and more pixels (a strip of the dense
// 1024 x 1024 image 41.5 -> 36.7 us; 512 x 512 with 200 particles 11.5 -> 11.8).
constexpr bool bwd_strip_wide(int W) { return W >= 1024; }

template <int N>
struct BwdLaunch {
    static cudaError_t rows(const BwdRowsArgs &a, cudaStream_t st) {
        const dim3 grid(a.geo.nstrips, a.S * a.K);
        return launch_chain(k_bwd_rows<N>, grid, kThreads, strip_inverse_smem(N), st, a);
    }
    static cudaError_t column(const BwdColumnArgs &a, cudaStream_t st) {
        return launch_chain(k_bwd_column<N>, dim3(a.geo.nblocks, a.S), kThreads, bwd_column_smem(N),
                            st, a);
    }
    static cudaError_t strip(const BwdStripArgs &a, cudaStream_t st) {
        const dim3 grid(a.geo.nstrips, a.S);
        if constexpr (bwd_strip_wide(N))
            if ((int)(grid.x * grid.y) <= kSms)
                return launch_chain(k_bwd_strip<N, true>, grid, kWideThreads,
                                    bwd_strip_smem(N, kWideThreads), st, a);
        return launch_chain(k_bwd_strip<N, false>, grid, kThreads, bwd_strip_smem(N, kThreads), st, a);
    }
    static cudaError_t prepare(int which) {
        if (which == 0)
            return cudaFuncSetAttribute(k_bwd_rows<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)strip_inverse_smem(N));
        if (which == 1)
            return cudaFuncSetAttribute(k_bwd_column<N>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)bwd_column_smem(N));
        cudaError_t e = cudaFuncSetAttribute(k_bwd_strip<N, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)bwd_strip_smem(N, kThreads));
        if constexpr (bwd_strip_wide(N))
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_bwd_strip<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bwd_strip_smem(N, kWideThreads));
        return e;
    }
};

template <int N>
struct BwdRows {
    static cudaError_t run(const BwdRowsArgs &a, cudaStream_t st) { return BwdLaunch<N>::rows(a, st); }
};
template <int N>
struct BwdColumn {
    static cudaError_t run(const BwdColumnArgs &a, cudaStream_t st) { return BwdLaunch<N>::column(a, st); }
};
template <int N>
struct BwdStrip {
    static cudaError_t run(const BwdStripArgs &a, cudaStream_t st) { return BwdLaunch<N>::strip(a, st); }
};
template <int N>
struct BwdPrepare {
    static cudaError_t run(int which) { return BwdLaunch<N>::prepare(which); }
};

}  // namespace

size_t bwd_column_smem(int H) {
    const int L = set_elems(H) / H;
    return (size_t)2 * L * line_stride(H) * sizeof(float2) + (size_t)kMaxModes * L * sizeof(int2) +
           (kThreads / 32) * 4 * sizeof(float);
}

cudaError_t prepare_backward(int H, int W) {
    cudaError_t e = dispatch_n<BwdPrepare>(W, 0);
    if (e == cudaSuccess) e = dispatch_n<BwdPrepare>(H, 1);
    if (e == cudaSuccess) e = dispatch_n<BwdPrepare>(W, 2);
    return e;
}

cudaError_t launch_bwd_rows(const BwdRowsArgs &a, cudaStream_t st) {
    return dispatch_n<BwdRows>(a.geo.W, a, st);
}
cudaError_t launch_bwd_column(const BwdColumnArgs &a, cudaStream_t st) {
    return dispatch_n<BwdColumn>(a.geo.H, a, st);
}
cudaError_t launch_bwd_strip(const BwdStripArgs &a, cudaStream_t st) {
    return dispatch_n<BwdStrip>(a.geo.W, a, st);
}
cudaError_t launch_bwd_reduce(const BwdReduceArgs &a, cudaStream_t st) {
    return launch_chain(k_bwd_reduce, dim3(a.nchunks * (kChunk / kReduceParticles) + a.S), kChunk, 0, st, a);
}

}  // namespace osog
