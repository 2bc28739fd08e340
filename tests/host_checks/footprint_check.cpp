// Random cameras and bricks, near the world's origin and far from it: the two
// binary32 projections of the geometry update (the culling's padded corners and
// the voxels' centres), written out as the kernels compute them, compared
// voxel by voxel.  Where footprint_holds, a brick whose corners project inside
// the image may have no voxel outside it and none deeper than its corners;
// where it does not hold, such bricks have to be among the samples.
#include <cfloat>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "footprint_bound.h"

struct Camera {
    float R[9], t[3], K[9], Ki[9];
    int w, h;
    bool pinhole;
};

static float row(const float* a, float x, float y, float z) { return a[0] * x + a[1] * y + a[2] * z; }

int main(int argc, char** argv) {
    const int samples = argc > 1 ? std::atoi(argv[1]) : 100000;
    std::mt19937_64 rng(7);
    auto uni = [&](double lo, double hi) { return std::uniform_real_distribution<double>(lo, hi)(rng); };
    auto logu = [&](double lo, double hi) { return std::pow(10.0, uni(std::log10(lo), std::log10(hi))); };
    {  // intrinsics whose inverse overflows, a camera at infinity, voxels of no size
        const float I[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, o[3] = {0, 0, 0}, t[3] = {0, 0, 2}, far[3] = {0, 0, INFINITY};
        const float K[9] = {500, 0, 320, 0, 500, 240, 0, 0, 1}, Ki[9] = {0.002f, 0, -0.64f, 0, 0.002f, -0.48f, 0, 0, 1};
        const float Kz[9] = {1e-39f, 0, 320, 0, 500, 240, 0, 0, 1}, Kzi[9] = {INFINITY, 0, -INFINITY, 0, 0.002f, -0.48f, 0, 0, 1};
        const int32_t nb[3] = {8, 8, 8};
        if (!tsdf::footprint_holds(I, t, K, Ki, o, nb, 0, 0.01f) || tsdf::footprint_holds(I, t, Kz, Kzi, o, nb, 0, 0.01f) ||
            tsdf::footprint_holds(I, far, K, Ki, o, nb, 0, 0.01f) || tsdf::footprint_holds(I, t, K, Ki, o, nb, 0, 1e-9f))
            return 2;
    }
    long inner_holds = 0, inner_not = 0, wrong_holds = 0, wrong_not = 0, near_not = 0, near = 0;
    for (int n = 0; n < samples; ++n) {
        Camera c{};
        c.pinhole = n % 3 != 0;
        c.w = (int)logu(16, 4096);
        c.h = (int)logu(16, 4096);
        const double f = logu(0.3, 3.0) * c.w, fx = f, fy = f * uni(0.8, 1.25);
        double K[9] = {fx, 0, uni(0.2, 0.8) * c.w, 0, fy, uni(0.2, 0.8) * c.h, 0, 0, 1};
        if (!c.pinhole) {
            K[1] = uni(-0.1, 0.1) * fx, K[3] = uni(-0.1, 0.1) * fy, K[6] = uni(-0.2, 0.2), K[7] = uni(-0.2, 0.2);
            const double k = logu(0.1, 10.0);
            for (double& x : K) x *= k;
        }
        for (int i = 0; i < 9; ++i) c.K[i] = (float)K[i];
        {
            const float* k = c.K;
            const double a = k[0], b = k[1], d = k[2], e = k[3], g = k[4], h = k[5], i = k[6], j = k[7], l = k[8];
            const double A = g * l - h * j, B = h * i - e * l, C = e * j - g * i, det = a * A + b * B + d * C;
            const double adj[9] = {A, d * j - b * l, b * h - d * g, B, a * l - d * i, d * e - a * h, C, b * i - a * j, a * g - b * e};
            for (int q = 0; q < 9; ++q) c.Ki[q] = (float)(adj[q] / det);
        }
        // a rotation from a random quaternion
        double q[4], qn = 0;
        for (double& x : q) x = std::normal_distribution<double>()(rng), qn += x * x;
        for (double& x : q) x /= std::sqrt(qn);
        const double w = q[0], x = q[1], y = q[2], z = q[3];
        const double Rd[9] = {1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z), 1 - 2 * (x * x + z * z),
                              2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)};
        for (int i = 0; i < 9; ++i) c.R[i] = (float)Rd[i];
        // the volume, one of its bricks, and a camera that sees it near the image's middle or edge
        const float s = (float)logu(3e-4, 0.3);
        const int32_t nb[3] = {(int)logu(1, 64), (int)logu(1, 64), (int)logu(1, 64)};
        const int32_t z0 = n % 5 == 0 ? (int)uni(0, 3000) : 0;
        const double off = n % 2 ? logu(0.1, 1e6) : 0.0;
        float origin[3];
        for (int a = 0; a < 3; ++a) origin[a] = (float)(uni(-1, 1) * off - 4.0 * nb[a] * s);
        const int b[3] = {(int)uni(0, nb[0]), (int)uni(0, nb[1]), (int)uni(0, nb[2])};
        const double dist = logu(10.0 * s, 3000.0 * s);
        const double px = uni(0.0, 1.0) * c.w, py = uni(0.0, 1.0) * c.h;
        double cam[3];
        for (int r = 0; r < 3; ++r) cam[r] = c.Ki[3 * r] * px + c.Ki[3 * r + 1] * py + c.Ki[3 * r + 2];
        const double cz = cam[2];
        for (double& v : cam) v *= dist / cz;
        double T[3];  // camera centre: brick centre - R^T cam
        for (int a = 0; a < 3; ++a) {
            const double bc = origin[a] + ((a == 2 ? z0 : 0) + 8.0 * b[a] + 4.0) * s;
            T[a] = bc - (Rd[a] * cam[0] + Rd[3 + a] * cam[1] + Rd[6 + a] * cam[2]);
        }
        for (int r = 0; r < 3; ++r) {
            double v = 0;
            for (int a = 0; a < 3; ++a) v += (double)c.R[3 * r + a] * (double)(float)T[a];
            c.t[r] = (float)-v;
        }
        const bool holds = tsdf::footprint_holds(c.R, c.t, c.K, c.Ki, origin, nb, z0, s);
        // a camera within 4 m of what it sees, voxels of 1 mm and more within some metres of the origin
        if (c.pinhole && off <= 10.0 && s >= 1e-3f && dist <= 4.0 && c.w < 3 * c.h && c.h < 3 * c.w)
            ++near, near_not += holds ? 0 : 1;
        // the culling's footprint
        float lo[3], hi[3];
        for (int a = 0; a < 3; ++a) {
            const int v0 = 8 * b[a] + (a == 2 ? z0 : 0);
            lo[a] = origin[a] + ((float)v0 - 0.5f) * s;
            hi[a] = origin[a] + ((float)(v0 + 8) + 0.5f) * s;
        }
        float X0[3], dX[3][3], h0[3], dh[3][3];
        for (int r = 0; r < 3; ++r) {
            X0[r] = row(c.R + 3 * r, lo[0], lo[1], lo[2]) + c.t[r];
            for (int a = 0; a < 3; ++a) dX[r][a] = c.R[3 * r + a] * (hi[a] - lo[a]);
        }
        for (int r = 0; r < 3; ++r) {
            h0[r] = row(c.K + 3 * r, X0[0], X0[1], X0[2]);
            for (int a = 0; a < 3; ++a) dh[r][a] = row(c.K + 3 * r, dX[0][a], dX[1][a], dX[2][a]);
        }
        float umin = FLT_MAX, umax = -FLT_MAX, vmin = FLT_MAX, vmax = -FLT_MAX, zmax = -FLT_MAX;
        bool straddle = false;
        for (int k = 0; k < 8; ++k) {
            float Z = X0[2], xh = h0[0], yh = h0[1], zh = h0[2];
            for (int a = 0; a < 3; ++a)
                if ((k >> a) & 1) Z += dX[2][a], xh += dh[0][a], yh += dh[1][a], zh += dh[2][a];
            zmax = std::fmax(zmax, Z);
            if (zh <= 1e-4f) straddle = true;
            else {
                const float rz = 1.0f / zh, u = xh * rz, v = yh * rz;
                umin = std::fmin(umin, u), umax = std::fmax(umax, u), vmin = std::fmin(vmin, v), vmax = std::fmax(vmax, v);
            }
        }
        if (straddle || !(umin > 1.0f && vmin > 1.0f && umax < (float)c.w - 2.0f && vmax < (float)c.h - 2.0f)) continue;
        // the update's voxels
        bool out = false;
        for (int k = 0; k < 512; ++k) {
            const float p[3] = {std::fmaf((float)(8 * b[0] + (k & 7)) + 0.5f, s, origin[0]),
                                std::fmaf((float)(8 * b[1] + ((k >> 3) & 7)) + 0.5f, s, origin[1]),
                                std::fmaf((float)(8 * b[2] + (k >> 6) + z0) + 0.5f, s, origin[2])};
            float X[3];
            for (int r = 0; r < 3; ++r)
                X[r] = std::fmaf(c.R[3 * r], p[0], std::fmaf(c.R[3 * r + 1], p[1], std::fmaf(c.R[3 * r + 2], p[2], c.t[r])));
            float hm[3];
            for (int r = 0; r < 3; ++r) {
                const float* a = c.K + 3 * r;
                if (c.pinhole) hm[r] = r == 2 ? X[2] : std::fmaf(a[r], X[r], a[2] * X[2]);
                else hm[r] = std::fmaf(a[0], X[0], std::fmaf(a[1], X[1], a[2] * X[2]));
            }
            const float rz = 1.0f / hm[2], u = hm[0] * rz + 0.5f, v = hm[1] * rz + 0.5f;
            out = out || !(hm[2] > 0.0f && u >= 0.0f && u < (float)c.w && v >= 0.0f && v < (float)c.h) || X[2] > zmax;
        }
        (holds ? inner_holds : inner_not) += 1;
        if (out) (holds ? wrong_holds : wrong_not) += 1;
    }
    std::printf("bricks inside the image: %ld where the footprint holds, %ld of them with a voxel out; "
                "%ld where it does not, %ld with one; it does not hold for %ld of %ld ordinary views\n",
                inner_holds, wrong_holds, inner_not, wrong_not, near_not, near);
    return wrong_holds == 0 && inner_holds > samples / 10 && wrong_not > 0 && near_not == 0 && near > samples / 50 ? 0 : 1;
}
