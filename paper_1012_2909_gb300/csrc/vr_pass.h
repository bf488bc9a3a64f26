// Shape of a staged-cell pass (host code): lanes per ray segment and row bands per cell, by
// how closely the rays of its views lie.
#pragma once

#include <algorithm>
#include <cmath>

#include "vr_internal.cuh"

namespace vr {

// Area of a pixel, in square voxels, at the point c.
inline double pixel_area(const double c[3], const CamDev& cd) {
    auto len2 = [](const double* v) { return v[0] * v[0] + v[1] * v[1] + v[2] * v[2]; };
    double scale = 1.0;  // of the window at c
    if (cd.type == 1) {
        scale = 0.0;
        for (int a = 0; a < 3; ++a) scale += (c[a] - cd.eye[a]) * cd.fwd[a];
        scale = std::fabs(scale) / len2(cd.fwd);
    }
    return std::fabs(cd.du * cd.dv) * std::sqrt(len2(cd.right) * len2(cd.up)) * scale * scale;
}

struct PassShape {
    int group;  // lanes per ray segment
    int bands;  // most row bands of a staged cell's pixels (BrickParams::max_bands)
};

// The rule, for a pass over n cameras of one size around a cube's centre c.  It goes by the
// mean number of pixels a square voxel over the cameras, in any order: segments number as
// pixels do, so among near and far views of one batch the near ones decide.
//
// Lanes: fewer waste less on a segment's last step, and pay where neighbouring groups march
// segments of one length: in the short segments of FP32 cells (16 voxels thick: 1721 x 1721 x
// 1025 at 1.0 voxels a pixel 18.9 ms with 4 lanes and 19.7 with 8; equal within 1 % up to 3
// voxels a pixel; 1269 x 339 x 736 at 7.8 voxels a pixel 0.313 and 0.301; not measured
// between), and with 16-bit cells where the rays are at most a voxel apart (2048 x 2048 x 1024
// on 25 panels: 0.66 voxels 49.4 and 53.3 ms, 0.99 25.6 and 26.0; 1.31 16.6 and 16.3; 1024 x
// 1024 x 2048 at 2.7 voxels 2.57 and 2.27).
//
// Bands: a 32^3 cell covers some 1500 square voxels, and a band should keep 512 pixels.
inline PassShape pass_rule(const double c[3], const CamDev* cams, int n, bool f32) {
    double density = 0.0;
    for (int i = 0; i < n; ++i) density += 1.0 / std::max(pixel_area(c, cams[i]), 1e-3);
    density /= n;
    return PassShape{density >= (f32 ? 1.0 / 9.0 : 1.0) ? 4 : 8,
                     (int)std::min(64.0, std::max(1.0, 1500.0 * density / 512.0))};
}

}  // namespace vr
