// Ray casting of the fused volumes (tsdf_raycast): the paper's real-time
// feedback (ray casting both volumes, abstract) and the predicted surface
// vertex map for tracking (ray tracing the geometry volume, Section III).
//
// One thread per pixel, a warp per 8x4 pixels (neighbouring rays walk nearby
// bricks, which keeps their gathers in L1/L2).  Operation order as stated in
// tsdf.h; compiled with --fmad=false so only the written fmaf() fuse.
//
// Sampled step by step, what bounded it was the chain of a ray's dependent
// samples: a sample's position needs the step its predecessor decided on, and
// each costs a memory round trip (several hundred per ray).  Most samples lie
// in free space (value exactly 1) or
// unobserved space (no value), where the step is step_far whatever the exact
// position, so the march first builds a map from the brick summaries
// (k_ray_map) and crosses a whole uniform cube of 1, 2, 4 or 8 bricks on a
// side with one map read: within it only t is advanced, by the same additions
// t + step_far that the samples would have made.  The samples before a ray
// enters the volume, which have no value either, are passed the same way, and
// the march ends where the ray leaves the volume for good.  What is left is
// bound by instruction issue: 30-40 samples per ray whose eight corners are
// read (about 130 instructions each), then the hit's six gradient samples,
// which the lanes of a warp finish together after the march (inside it, lanes
// that hit at different samples had run them one after another).
// Measured, the kernel alone, on one scene (24 frames around 20 primitives in
// a 2 m cube): 640x480 rays through 512^3, 1064 -> 256 us and 5.6 us for the map;
// 1920x1080 through 192^3, 1936 -> 703 us and 3 us; on another scene 341 and
// 960 us.  The three prediction levels of a tracked frame at 512^3, 2454 -> 613
// us one after another, about 430 us beside one another (launch_raycast,
// RayLink).  Eight blocks per SM; 7, 10 and 12 were slower.
#include <cfloat>
#include <cstdint>

#include "common.cuh"

namespace tsdf {
namespace {

constexpr int RC_THREADS = 128;  // 4 warps of 8x4 pixels: 16x8 pixels
constexpr int RC_BX = 16, RC_BY = 8;

// ------------------------------------------------------------- brick map --
// What a sample whose cell has its lower corner in brick b is worth, by the
// axes on which the cell reaches into the next brick (bit a of m: axis a):
// over the bricks the cell touches,
//   RAY_NONE  one holds no observed voxel: the trilinear value does not exist
//   RAY_ONE   all are wholly observed with every F equal to 1: it is exactly 1
//             (each lerp computes fmaf(f, 0, 1))
//   RAY_SEEN  all are wholly observed: F decides
//   RAY_CELL  F and w decide
// The entry of b holds the code of m at bits 2 m.  At bits 14-15 (m = 7),
// RAY_ONE and RAY_NONE say more: every cell of b has that code (RAY_NONE: b
// itself holds no observed voxel; where only a neighbour does, m = 7 is left
// RAY_CELL), and bits 0-1 then hold the largest l <= 3 such that the same is
// true of all bricks of the aligned 2^l-brick cube around b.  Without plain_f
// (some F is NaN, infinite or huge, which the summaries do not tell) only
// cells inside one brick are coded.
enum : uint32_t { RAY_CELL = 0u, RAY_ONE = 1u, RAY_NONE = 2u, RAY_SEEN = 3u };
constexpr int MAP_EDGE = 8;  // bricks per axis of a map block
constexpr int HALO_EDGE = MAP_EDGE + 1;

__global__ void __launch_bounds__(MAP_EDGE * MAP_EDGE * MAP_EDGE) k_ray_map(const BrickSummary* __restrict__ summ,
                                                                          int nbx, int nby, int nbz, int plain_f,
                                                                          uint16_t* __restrict__ map) {
    __shared__ uint8_t kind[HALO_EDGE * HALO_EDGE * HALO_EDGE];  // bit 0 none observed, 1 not all 1, 2 not all observed
    __shared__ uint8_t cube[3][MAP_EDGE * MAP_EDGE * MAP_EDGE];  // per aligned cube of 1, 2, 4 bricks: its code (3: outside)
    const int tid = threadIdx.x;
    const int ox = blockIdx.x * MAP_EDGE, oy = blockIdx.y * MAP_EDGE, oz = blockIdx.z * MAP_EDGE;
    for (int i = tid; i < HALO_EDGE * HALO_EDGE * HALO_EDGE; i += MAP_EDGE * MAP_EDGE * MAP_EDGE) {
        const int x = ox + i % HALO_EDGE, y = oy + (i / HALO_EDGE) % HALO_EDGE, z = oz + i / (HALO_EDGE * HALO_EDGE);
        uint8_t k = 0;  // outside the volume: no cell reaches it
        if (x < nbx && y < nby && z < nbz) {
            const BrickSummary s = summ[((int64_t)z * nby + y) * nbx + x];
            k = (s.fmin <= FLT_MAX ? 0 : 1) | (s.fmin == 1.0f && s.fmax == 1.0f ? 0 : 2) | (s.wmin > 0u ? 0 : 4);
        }
        kind[i] = k;
    }
    __syncthreads();
    const int lx = tid & 7, ly = (tid >> 3) & 7, lz = tid >> 6;
    const bool in = ox + lx < nbx && oy + ly < nby && oz + lz < nbz;
    uint32_t entry = 0, code = 0;
    {
        const int at = (lz * HALO_EDGE + ly) * HALO_EDGE + lx;
        uint32_t k[8];
#pragma unroll
        for (int m = 0; m < 8; ++m)
            k[m] = kind[at + (m & 1) + ((m >> 1) & 1) * HALO_EDGE + (m >> 2) * HALO_EDGE * HALO_EDGE];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            uint32_t any = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if ((q & m) == q) any |= k[q];
            code = (any & 1u) ? RAY_NONE : ((any & 6u) == 0u ? RAY_ONE : ((any & 4u) ? RAY_CELL : RAY_SEEN));
            if (!plain_f && (m != 0 || code == RAY_SEEN)) code = RAY_CELL;
            if (m == 7 && code == RAY_NONE && !(k[0] & 1u)) code = RAY_CELL;
            entry |= code << (2 * m);
        }
    }
    // a cube is uniform when its eight halves are: the bitwise AND of the codes 1 and 2, with 3 for cubes outside
    cube[0][tid] = in ? (code == RAY_SEEN ? 0 : (uint8_t)code) : 3;
    __syncthreads();
#pragma unroll
    for (int l = 1; l < 3; ++l) {
        const int e = MAP_EDGE >> l;  // cubes of 2^l bricks per axis
        if (tid < e * e * e) {
            const int x = tid % e, y = (tid / e) % e, z = tid / (e * e), e2 = 2 * e;
            uint8_t a = 3;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                a &= cube[l - 1][((2 * z + (q >> 2)) * e2 + 2 * y + ((q >> 1) & 1)) * e2 + 2 * x + (q & 1)];
            cube[l][tid] = a;
        }
        __syncthreads();
    }
    if (!in) return;
    if (code == RAY_ONE || code == RAY_NONE) {
        uint32_t level = 0;
        if (cube[1][((lz >> 1) * 4 + (ly >> 1)) * 4 + (lx >> 1)] == code) {
            level = 1;
            if (cube[2][((lz >> 2) * 2 + (ly >> 2)) * 2 + (lx >> 2)] == code) {
                uint32_t a = 3;
#pragma unroll
                for (int q = 0; q < 8; ++q) a &= cube[2][q];
                level = a == code ? 3 : 2;
            }
        }
        entry = (entry & ~3u) | level;
    }
    map[((int64_t)(oz + lz) * nby + oy + ly) * nbx + ox + lx] = (uint16_t)entry;
}

// --------------------------------------------------------------- samples --
__device__ __forceinline__ float rc_lerp(float a, float b, float t) { return fmaf(t, b - a, a); }

// The trilinear cell of a world point.
struct RayCell {
    int i0[3];    // lower corner voxel
    float fr[3];  // fractions
    bool in;      // the eight corners lie in the volume
};

__device__ __forceinline__ RayCell rc_cell(const RayConst& c, const float p[3]) {
    RayCell s;
    s.in = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float g = fmaf(p[a] - c.origin[a], c.inv_sg, -0.5f);
        const float fl = floorf(g);
        s.in = s.in && fl >= 0.0f && fl + 1.0f <= (float)(c.ng[a] - 1);
        s.i0[a] = (int)fl;
        s.fr[a] = g - fl;
    }
    return s;
}

__device__ __forceinline__ int rc_brick(const RayConst& c, const RayCell& s) {
    return ((s.i0[2] >> 3) * c.nb[1] + (s.i0[1] >> 3)) * c.nb[0] + (s.i0[0] >> 3);
}

// Axes on which the cell reaches into the next brick.
__device__ __forceinline__ int rc_mask(const RayCell& s) {
    return ((s.i0[0] & 7) == 7 ? 1 : 0) | ((s.i0[1] & 7) == 7 ? 2 : 0) | ((s.i0[2] & 7) == 7 ? 4 : 0);
}

// The code of the cell from its brick's map entry.
__device__ __forceinline__ uint32_t rc_code(uint32_t entry, int m) {
    const uint32_t all = entry >> 14;
    return all == RAY_ONE || all == RAY_NONE ? all : (entry >> (2 * m)) & 3u;
}

// The eight corners' F and (RAY_CELL) w of a cell in the volume; every read is
// issued before the first is used.
struct RayCorners {
    float q[8];
    uint32_t wmin;
};
__device__ __forceinline__ void rc_corners(const RayConst& c, const float* __restrict__ F,
                                           const uint8_t* __restrict__ W, const RayCell& s, int b, uint32_t code,
                                           RayCorners& r) {
    const int lx = s.i0[0] & 7, ly = s.i0[1] & 7, lz = s.i0[2] & 7;
    const int64_t base = (int64_t)b * BRICK_VOX + (lz * BRICK + ly) * BRICK + lx;
    const int dx = lx == 7 ? BRICK_VOX - 7 : 1;
    const int dy = ly == 7 ? c.nb[0] * BRICK_VOX - 7 * BRICK : BRICK;
    const int dz = lz == 7 ? c.nb[0] * c.nb[1] * BRICK_VOX - 7 * BRICK * BRICK : BRICK * BRICK;
    uint32_t w[8];
    if (code == RAY_CELL) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            w[k] = __ldg(W + base + ((k & 1) ? dx : 0) + ((k & 2) ? dy : 0) + ((k & 4) ? dz : 0));
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
        r.q[k] = __ldg(F + base + ((k & 1) ? dx : 0) + ((k & 2) ? dy : 0) + ((k & 4) ? dz : 0));
    r.wmin = 255u;
    if (code == RAY_CELL) {
#pragma unroll
        for (int k = 0; k < 8; ++k) r.wmin = min(r.wmin, w[k]);
    }
}

__device__ __forceinline__ float rc_trilinear(const RayCorners& r, const float fr[3]) {
    const float c00 = rc_lerp(r.q[0], r.q[1], fr[0]), c10 = rc_lerp(r.q[2], r.q[3], fr[0]);
    const float c01 = rc_lerp(r.q[4], r.q[5], fr[0]), c11 = rc_lerp(r.q[6], r.q[7], fr[0]);
    const float c0 = rc_lerp(c00, c10, fr[1]), c1 = rc_lerp(c01, c11, fr[1]);
    return rc_lerp(c0, c1, fr[2]);
}

// Trilinear TSDF at two world points (the two ends of a central difference),
// the reads of both in flight together; false when either does not exist.
__device__ __forceinline__ bool rc_pair(const RayConst& c, const float* __restrict__ F, const uint8_t* __restrict__ W,
                                        const uint16_t* __restrict__ map, const float p[3], const float m[3],
                                        float& fp, float& fm) {
    const RayCell s[2] = {rc_cell(c, p), rc_cell(c, m)};
    if (!s[0].in || !s[1].in) return false;
    const int b[2] = {rc_brick(c, s[0]), rc_brick(c, s[1])};
    const uint32_t e[2] = {__ldg(map + b[0]), __ldg(map + b[1])};
    const uint32_t code[2] = {rc_code(e[0], rc_mask(s[0])), rc_code(e[1], rc_mask(s[1]))};
    if (code[0] == RAY_NONE || code[1] == RAY_NONE) return false;
    RayCorners r[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        r[i].wmin = 1u;
        if (code[i] != RAY_ONE) rc_corners(c, F, W, s[i], b[i], code[i], r[i]);
    }
    if (r[0].wmin == 0u || r[1].wmin == 0u) return false;
    fp = code[0] == RAY_ONE ? 1.0f : rc_trilinear(r[0], s[0].fr);
    fm = code[1] == RAY_ONE ? 1.0f : rc_trilinear(r[1], s[1].fr);
    return true;
}

// CHAIN: the casts launched beside one another (launch_raycast, RayLink).
// They read nothing of one another: the next one's blocks may start at once,
// filling the SMs this one's last rays leave, and one block ends only after
// the cast before it has, so the last cast's end is the end of all.  A cast
// by itself runs without these, which held eight bytes more per thread
// (spilled): whole calls, over several scenes, 640x480 through 512^3 328 -> 310
// us, 1920x1080 through 192^3 883 -> 789 us; three chained casts 25 us less
// with one waiting thread instead of all.
template <bool CHAIN>
__global__ void __launch_bounds__(RC_THREADS, 8) k_raycast(RayConst c, const float* __restrict__ F,
                                                        const uint8_t* __restrict__ W, const uint32_t* __restrict__ C,
                                                        const uint16_t* __restrict__ map, float* __restrict__ range,
                                                        float* __restrict__ vertex, float* __restrict__ normal,
                                                        uint32_t* __restrict__ rgbw) {
    if constexpr (CHAIN) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = blockIdx.x * RC_BX + (warp & 1) * 8 + (lane & 7);
    const int y = blockIdx.y * RC_BY + (warp >> 1) * 4 + (lane >> 3);
    if (x >= c.width || y >= c.height) return;
    const float fx = (float)x, fy = (float)y;
    const float dc0 = fmaf(c.Kinv[0], fx, fmaf(c.Kinv[1], fy, c.Kinv[2]));
    const float dc1 = fmaf(c.Kinv[3], fx, fmaf(c.Kinv[4], fy, c.Kinv[5]));
    const float dc2 = fmaf(c.Kinv[6], fx, fmaf(c.Kinv[7], fy, c.Kinv[8]));
    const float nd = __fdiv_rn(1.0f, __fsqrt_rn(fmaf(dc0, dc0, fmaf(dc1, dc1, dc2 * dc2))));
    float d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = fmaf(c.R[3 * a], dc0, fmaf(c.R[3 * a + 1], dc1, c.R[3 * a + 2] * dc2)) * nd;

    // The grid coordinate of a sample is the rounded A + B t; `slack` (voxels)
    // bounds that rounding (the sums of |o|, |t d| and |origin| carry at most
    // a few ulp each, scaled to voxels) and that of the bounds on t below.  A
    // sample's rounded coordinate is non-decreasing in t where d >= 0 (and
    // non-increasing where d <= 0), since each of its operations is, so a cube
    // entered by a sample is left only through its far sides.  A bound that is
    // not a number compares false and skips nothing.
    float A[3], rB[3], slack = 0.0f;
    float t_in = -FLT_MAX, t_end = c.far_;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        A[a] = fmaf(c.t[a] - c.origin[a], c.inv_sg, -0.5f);
        rB[a] = __frcp_rn(d[a] * c.inv_sg);
        slack = fmaxf(slack, fmaf((fabsf(c.t[a]) + fabsf(c.origin[a]) + c.far_) * c.inv_sg, 2e-6f, 1e-3f));
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // where the ray enters and leaves [0, ng - 1) on this axis, widened by the slack
        const float lo = (-slack - A[a]) * rB[a], hi = ((float)(c.ng[a] - 1) + slack - A[a]) * rB[a];
        if (d[a] > 0.0f || d[a] < 0.0f) {
            const float enter = d[a] > 0.0f ? lo : hi, leave = d[a] > 0.0f ? hi : lo;
            if (enter > t_in) t_in = enter;
            if (leave < t_end) t_end = leave;
        }
    }

    float t = c.near_, tp = 0.0f, Fp = 0.0f, hit_t = 0.0f;
    bool has_prev = false, hit = false;
    uint32_t it = 0;
    // the samples at t, t + step_far, ... up to t_last; tp is the last of them
    auto pass = [&](float t_last) {
        for (;;) {  // four at a time
            const float t1 = t + c.step_far, t2 = t1 + c.step_far, t3 = t2 + c.step_far;
            if (!(t3 <= t_last && it + 4u <= c.max_iter)) break;
            tp = t3;
            t = t3 + c.step_far;
            it += 4u;
        }
        while (it < c.max_iter && t <= t_last) {
            tp = t;
            t = t + c.step_far;
            ++it;
        }
    };
    // those before the volume have no value
    if (t <= t_in) pass(fminf(t_in, t_end));
    int b_at = -1;  // the brick whose map entry is held
    uint32_t entry = 0;
    for (;;) {
        // cross uniform space, up to a sample that the voxels decide; the
        // lanes of a warp then read theirs together
        bool decide = false;
        RayCell s;
        int b = 0;
        uint32_t code = RAY_NONE;
        while (it < c.max_iter && t <= t_end) {
            const float p[3] = {fmaf(t, d[0], c.t[0]), fmaf(t, d[1], c.t[1]), fmaf(t, d[2], c.t[2])};
            s = rc_cell(c, p);
            float t_last = t_end;
            if (s.in) {
                b = rc_brick(c, s);
                if (b != b_at) {
                    entry = __ldg(map + b);
                    b_at = b;
                }
                const int m = rc_mask(s);
                const uint32_t all = entry >> 14;
                const bool cube = all == RAY_ONE || all == RAY_NONE;
                code = cube ? all : (entry >> (2 * m)) & 3u;
                if (code == RAY_CELL || code == RAY_SEEN) {
                    decide = true;
                    break;
                }
                // the cells of this code: the cube around b, or b's cells of
                // the same m; the side on each axis by which the ray leaves
                // them bounds the samples known to lie inside
                const int l = (int)(entry & 3u) + 3;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const bool last = !cube && ((m >> a) & 1);
                    const int lo = cube ? (s.i0[a] >> l) << l : (last ? s.i0[a] : s.i0[a] & ~7);
                    const int hi = min(lo + (cube ? 1 << l : (last ? 1 : 7)), c.ng[a] - 1);
                    const float side = d[a] > 0.0f ? (float)hi - slack : (float)lo + slack;
                    const float tx = (side - A[a]) * rB[a];
                    if ((d[a] > 0.0f || d[a] < 0.0f) && !(tx >= t_last)) t_last = tx;
                }
            } else {
                code = RAY_NONE;
                t_last = t;
            }
            tp = t;  // this sample, and those known to be like it
            t = t + c.step_far;
            ++it;
            pass(t_last);
            has_prev = code == RAY_ONE;
            Fp = 1.0f;
        }
        if (!decide) break;
        RayCorners r;
        rc_corners(c, F, W, s, b, code, r);
        const bool ok = r.wmin != 0u;
        const float Fs = rc_trilinear(r, s.fr);
        if (ok && has_prev && Fp > 0.0f && Fs <= 0.0f) {
            hit_t = fmaf(t - tp, __fdiv_rn(Fp, Fp - Fs), tp);
            hit = true;
            break;
        }
        has_prev = ok;
        if (ok) {
            Fp = Fs;
            tp = t;
        }
        t = t + ((ok && Fs < 1.0f) ? c.step_near : c.step_far);
        ++it;
    }

    // the hits of a warp are finished together
    float out_t = 0.0f, v[3] = {0.0f, 0.0f, 0.0f}, n[3] = {0.0f, 0.0f, 0.0f};
    uint32_t col = 0u;
    if (hit) {
        out_t = hit_t;
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fmaf(hit_t, d[a], c.t[a]);
        if (normal) {
            float g[3];
            bool good = true;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                float pp[3] = {v[0], v[1], v[2]}, pm[3] = {v[0], v[1], v[2]};
                pp[a] = v[a] + c.s_g;
                pm[a] = v[a] - c.s_g;
                float fp = 0.0f, fm = 0.0f;
                good = rc_pair(c, F, W, map, pp, pm, fp, fm) && good;
                g[a] = fp - fm;
            }
            if (good) {
                const float l2 = fmaf(g[0], g[0], fmaf(g[1], g[1], g[2] * g[2]));
                if (l2 > 0.0f) {
                    const float l = __fsqrt_rn(l2);
#pragma unroll
                    for (int a = 0; a < 3; ++a) n[a] = __fdiv_rn(g[a], l);
                }
            }
        }
        if (rgbw) {
            int k[3];
            bool in = true;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float q = floorf((v[a] - c.origin[a]) * c.inv_sc);
                in = in && q >= 0.0f && q < (float)c.nc[a];
                k[a] = in ? (int)q : 0;
            }
            if (in) col = C[brick_offset(k[0], k[1], k[2], c.ncb)];
        }
    }
    const size_t i = (size_t)y * c.width + x;
    if (range) range[i] = out_t;
    if (vertex) {
        vertex[3 * i] = v[0];
        vertex[3 * i + 1] = v[1];
        vertex[3 * i + 2] = v[2];
    }
    if (normal) {
        normal[3 * i] = n[0];
        normal[3 * i + 1] = n[1];
        normal[3 * i + 2] = n[2];
    }
    if (rgbw) rgbw[i] = col;
    if constexpr (CHAIN) {
        if (x == 0 && y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    }
}

}  // namespace

cudaError_t launch_ray_map(const BrickSummary* summ, const int32_t nb[3], bool plain_f, uint16_t* map,
                           cudaStream_t stream) {
    const dim3 grid((nb[0] + MAP_EDGE - 1) / MAP_EDGE, (nb[1] + MAP_EDGE - 1) / MAP_EDGE,
                    (nb[2] + MAP_EDGE - 1) / MAP_EDGE);
    k_ray_map<<<grid, MAP_EDGE * MAP_EDGE * MAP_EDGE, 0, stream>>>(summ, nb[0], nb[1], nb[2], plain_f ? 1 : 0, map);
    return cudaGetLastError();
}

cudaError_t launch_raycast(const RayConst& c, const float* F, const uint8_t* W, const uint32_t* C, const uint16_t* map,
                           float* range, float* vertex, float* normal, uint32_t* rgbw, RayLink link,
                           cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((c.width + RC_BX - 1) / RC_BX, (c.height + RC_BY - 1) / RC_BY);
    cfg.blockDim = dim3(RC_THREADS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = link == RayLink::BEHIND ? 1 : 0;
    auto k = link == RayLink::ALONE ? k_raycast<false> : k_raycast<true>;
    return cudaLaunchKernelEx(&cfg, k, c, F, W, C, map, range, vertex, normal, rgbw);
}

}  // namespace tsdf
