// The viewing frame of one image and the plane-synchronous walk chosen for
// it: one function for the device, which walks by it, and for the host, which
// leaves out the layout passes and the per-ray forward that no image needs.
#pragma once

#include <math.h>

#include "tomo_internal.cuh"

namespace tomo {

__host__ __device__ inline Frame image_frame(const tomo_pointing &p)
{
    Frame f;
    const double cl = cos(p.lat), sl = sin(p.lat);
    const double co = cos(p.lon), so = sin(p.lon);
    f.o[0] = p.d_obs * cl * co;
    f.o[1] = p.d_obs * cl * so;
    f.o[2] = p.d_obs * sl;
    f.w[0] = -cl * co;
    f.w[1] = -cl * so;
    f.w[2] = -sl;
    // w x z = (w_y, -w_x, 0), of length cos(lat)
    const double n1 = sqrt(f.w[0] * f.w[0] + f.w[1] * f.w[1]);
    const double a1[3] = { f.w[1] / n1, -f.w[0] / n1, 0.0 };
    const double a2[3] = { a1[1] * f.w[2] - a1[2] * f.w[1],
                           a1[2] * f.w[0] - a1[0] * f.w[2],
                           a1[0] * f.w[1] - a1[1] * f.w[0] };
    const double cr = cos(p.roll), sr = sin(p.roll);
    for (int a = 0; a < 3; ++a) {
        f.e1[a] = cr * a1[a] + sr * a2[a];
        f.e2[a] = -sr * a1[a] + cr * a2[a];
    }
    return f;
}

// code: the hint bits of ImgParam.pad.  With a tolerance: layouts, the
// layouts (bit L) that the hint may name if it may be valid (0: certainly not
// valid); fwd_may, fwd_sure: whether it may and whether it certainly selects
// the plane forward.  With tolerance 0 they repeat what code says.
struct PlaneHint {
    int32_t code;
    unsigned layouts;
    bool fwd_may, fwd_sure;
};

// Hint for the plane-synchronous walk of one image: M = the axis along
// which the line of sight of the image centre advances fastest, its
// direction, and L = the axis (other than M) along which neighbouring pixels
// of a row move at a fixed M plane.  Moving along the row turns the
// direction by ~e1; at a fixed M plane the ray through u + e1 d is displaced
// along e1 - u e1_M / u_M.  The hint is marked valid only when neighbouring
// pixels are at least rules.min_pitch voxels of L apart at the distance of
// Sun centre; the forward and walk-variant bits follow the other rules
// (defaults: the measured thresholds in tomo_internal.cuh; tomo_autotune
// can tune them per size bucket).  The device calls it with tolerance 0; the
// host, whose sines and contractions round differently, with a tolerance
// (relative to unit vectors and thresholds) within which a comparison counts
// as open.  Of tied axes the first is taken.
__host__ __device__ inline PlaneHint plane_hint(const tomo_pointing &p,
                                                const Frame &f, int nu, int nv,
                                                double3 vox,
                                                const tomo_plane_rules &rules,
                                                double tol)
{
    const double tu = tan((0.5 * (nu - 1) - p.crpix_u) * p.cdelt_u + p.crval_u);
    const double tv = tan((0.5 * (nv - 1) - p.crpix_v) * p.cdelt_v + p.crval_v);
    const double d[3] = { vox.x, vox.y, vox.z };
    const double step = p.d_obs * fabs(tan(p.cdelt_u));
    const double under = 1.0 - tol, over = 1.0 + tol;
    double u[3];
    for (int a = 0; a < 3; ++a) u[a] = f.w[a] + tu * f.e1[a] + tv * f.e2[a];
    const double most = fmax(fabs(u[0]), fmax(fabs(u[1]), fabs(u[2])));
    PlaneHint h = { -1, 0u, false, true };
    for (int M = 0; M < 3; ++M) {
        if (fabs(u[M]) < most * under) continue;
        double lat[3] = { 0.0, 0.0, 0.0 }, best = 0.0;
        double lo = INFINITY;  // the less steep minor component
        for (int a = 0; a < 3; ++a) {
            if (a == M) continue;
            lat[a] = fabs(f.e1[a] - u[a] * f.e1[M] / u[M]);
            best = fmax(best, lat[a]);
            lo = fmin(lo, fabs(u[a]));
        }
        lo /= fabs(u[M]);
        for (int L = 0; L < 3; ++L) {
            if (L == M || lat[L] < best - tol) continue;
            const double pitch = step / d[L];
            const bool may = pitch >= rules.min_pitch * under;
            const bool sure = pitch >= rules.min_pitch * over;
            const bool fwd = may && (pitch >= rules.fwd_min_pitch * under ||
                                     lo < rules.fwd_max_ratio + tol);
            if (h.code < 0)
                h.code = (may ? kPlaneHintValid : 0) | (fwd ? kPlaneFwdBit : 0) |
                         (lo >= rules.general_ratio ? kPlaneGeneralBit : 0) | M |
                         (L << 2) | ((u[M] < 0.0) ? 16 : 0);
            if (may) h.layouts |= 1u << L;
            h.fwd_may |= fwd;
            h.fwd_sure &= sure && (pitch >= rules.fwd_min_pitch * over ||
                                   lo < rules.fwd_max_ratio - tol);
        }
    }
    return h;
}

}  // namespace tomo
