// When a brick's projected footprint may stand for its voxels.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace tsdf {

// The brick culling projects the corners of a brick, padded by half a voxel;
// the geometry update projects each voxel centre, in another order of binary32
// operations.  True when rounding cannot take a voxel out of the hull of the
// corners, in depth or in the image: only then may a brick that projects
// inside the image skip its voxels' image tests, and one in front of every
// measurement its voxels' depths.
//
// Each computed projection is the exact one, K (R p + t), of a point displaced
// in the camera frame.  With u = 2^-24, A the sum of the largest |p_a| and |t_r|
// that enter the sums, D the largest camera coordinate of the volume, G the
// largest row sum of |K^-1| |K| (which turns the roundings of K X into a
// displacement of X) and s the voxel edge, the displacement per axis is at most
//   voxel   u (3 A + D) from p and three fused steps, 3 u G D from K
//   corner  u (7 A + 15 D) from p, six operations and the edge sums,
//           u G (8 D + 240 s) from K and its edge sums
// A voxel centre lies a whole voxel inside the padded brick, so it stays in the
// hull while sqrt(3) times their sum is below s.  (The quotients' roundings
// are below a hundredth of a pixel, of the one and a half that are kept.)  For 4 mm
// voxels, a 525-pixel focal length and a 640x480 image it holds up to about
// 1.8 km from the world's origin.
inline bool footprint_holds(const float R[9], const float t[3], const float K[9], const float Kinv[9],
                            const float origin[3], const int32_t nb[3], int32_t z0, float s) {
    double lo[3], hi[3], A = 0.0, at = 0.0, D = 0.0, G = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double first = a == 2 ? z0 : 0;
        lo[a] = (double)origin[a] + (first - 0.5) * (double)s;
        hi[a] = (double)origin[a] + (first + 8.0 * nb[a] + 0.5) * (double)s;
        A += std::max(std::fabs((double)origin[a]), std::max(std::fabs(lo[a]), std::fabs(hi[a])));
        at = std::max(at, std::fabs((double)t[a]));
    }
    A += at;
    for (int k = 0; k < 8; ++k)
        for (int r = 0; r < 3; ++r) {
            double x = t[r];
            for (int a = 0; a < 3; ++a) x += (double)R[3 * r + a] * (((k >> a) & 1) ? hi[a] : lo[a]);
            D = std::max(D, std::fabs(x));
        }
    for (int r = 0; r < 3; ++r) {
        double g = 0.0;
        for (int q = 0; q < 3; ++q)
            for (int a = 0; a < 3; ++a) g += std::fabs((double)Kinv[3 * r + a] * (double)K[3 * a + q]);
        if (!(g < 1e9)) return false;  // (an inverse that overflows binary32 makes it infinite or not a number)
        G = std::max(G, g);
    }
    // the reciprocal of K's third row times a camera point is exact between 2^-126 and 2^126
    const double k3 = std::max(std::fabs((double)K[6]), std::max(std::fabs((double)K[7]), std::fabs((double)K[8])));
    if (!(k3 > 1e-20 && k3 * D < 1e30)) return false;
    // sqrt(3) 2^-24 = 1.033e-7; 1e-30: far above what underflow adds
    const double moved = 1.1e-7 * (10.0 * A + 16.0 * D + 11.0 * G * D + 240.0 * G * (double)s) + 1e-30;
    return moved <= (double)s;  // (false when something is not finite)
}

}  // namespace tsdf
