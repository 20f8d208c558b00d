// Rows of a column that a (shifted) pupil circle passes: the signed row
// frequencies fy with (fx / (W dx) + ox)^2 + (fy / (H dx) + oy)^2 <= r2.
//
// The interval's ends are those of the double-precision formula
// (pupil_chord_exact).  A chain of FP64 operations costs a column block over a
// thousand cycles (66 a multiply-add, 600 a square root), so the ends are taken
// in float-float first, with an error below 1e-7 rows, and in double precision
// only when one lies within 1e-6 of an integer or the column grazes the circle.
//
// Header of plain operations, so that the host can check the same code.
#pragma once

#include "osog_ff.h"

namespace osog {

struct RowRange {
    int lo, hi;  // empty: lo > hi
};

// The circle's constants as float-float pairs (split on the host): column
// pitch and centre in cycles / um, squared radius, rows per cycle / um.
struct PupilFF {
    ff fx_scale, ox, oy, r2, fy_span;
};

OSOG_HD RowRange pupil_chord_exact(double r2, double ox, double oy, double fx_scale,
                                   double fy_span, int fx) {
    const double ax = (double)fx * fx_scale + ox;
    const double rem = r2 - ax * ax;
    if (rem < 0.0) return {1, 0};
    const double root = sqrt(rem);
    const double lo = (-root - oy) * fy_span;
    const double hi = (root - oy) * fy_span;
    return {(int)ceil(lo), (int)floor(hi)};
}

// True with the interval when the float-float ends decide it.
OSOG_HD bool pupil_chord_ff(const PupilFF &p, int fx, RowRange *out) {
    const ff ax = ff_add(ff_mul(p.fx_scale, ff{(float)fx, 0.f}), p.ox);
    const ff rem = ff_add(p.r2, ff_neg(ff_mul(ax, ax)));
    const float edge = f_mul(p.r2.h, 1e-7f);
    if (rem.h < -edge) {
        *out = {1, 0};
        return true;
    }
    if (!(rem.h > edge)) return false;
#if defined(__CUDA_ARCH__)
    const float r = rsqrtf(rem.h);
#else
    const float r = 1.0f / sqrtf(rem.h);
#endif
    const float s = f_mul(rem.h, r);
    const float e = f_add(f_fma(-s, s, rem.h), rem.l);
    const ff root = fast_two_sum(s, f_mul(e, f_mul(0.5f, r)));
    const ff lo = ff_mul(ff_neg(ff_add(root, p.oy)), p.fy_span);
    const ff hi = ff_mul(ff_add(root, ff_neg(p.oy)), p.fy_span);
    const float rl = rintf(lo.h), rh = rintf(hi.h);
    const float dl = f_add(f_sub(lo.h, rl), lo.l), dh = f_add(f_sub(hi.h, rh), hi.l);
    if (!(fabsf(dl) > 1e-6f) || !(fabsf(dh) > 1e-6f) || !(fabsf(rl) < 1e6f) || !(fabsf(rh) < 1e6f))
        return false;
    *out = {(int)rl + (dl > 0.f ? 1 : 0), (int)rh - (dh < 0.f ? 1 : 0)};
    return true;
}

}  // namespace osog
