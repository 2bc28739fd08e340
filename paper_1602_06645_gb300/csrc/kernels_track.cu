// Camera tracking (Section III: the KinectFusion loop the paper builds on):
// a depth pyramid with its vertex and normal maps, projective data
// association against the surface predicted by ray casting the geometry
// volume, and point-to-plane Gauss-Newton steps T <- exp(xi^) T.  Operation
// order as stated in tsdf.h (tsdf_track); compiled with --fmad=false so only
// the written fmaf() fuse.  The normal equations are reduced in binary64 in a
// fixed order, and solved and applied on the device, so every step of a
// frame is queued without a host round trip.
#include <cstdint>

#include "common.cuh"
#include "ffloat.cuh"

namespace tsdf {
namespace {

constexpr int TRACK_THREADS = 256;

// ------------------------------------------------------------ pyramid ----
__global__ void k_depth_metres(const uint16_t* __restrict__ depth, int n, float* __restrict__ d) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const uint32_t D = depth[i];
        d[i] = D ? (float)D * 0.001f : 0.0f;
    }
}

// Level l + 1 pixel from the 2 x 2 block of level l, in the order (0,0),
// (1,0), (0,1), (1,1): the mean of the valid depths within 0.03 m of the
// block's first valid depth, summed in that order.
__global__ void k_pyr_down(const float* __restrict__ src, int w, float* __restrict__ dst, int w2, int h2) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= w2 || y >= h2) return;
    float first = 0.0f, sum = 0.0f;
    int n = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float d = src[(size_t)(2 * y + (k >> 1)) * w + 2 * x + (k & 1)];
        if (d == 0.0f) continue;
        if (n == 0) first = d;
        if (fabsf(d - first) <= 0.03f) {
            sum = sum + d;
            ++n;
        }
    }
    dst[(size_t)y * w2 + x] = n ? __fdiv_rn(sum, (float)n) : 0.0f;
}

// Vertex d (fmaf(1/fx, x, -cx/fx), fmaf(1/fy, y, -cy/fy), 1) of pixel (x, y).
__device__ __forceinline__ float3 vertex_at(const float* __restrict__ d, int w, int x, int y, const float4 ki) {
    const float z = d[(size_t)y * w + x];
    return make_float3(z * fmaf(ki.x, (float)x, ki.z), z * fmaf(ki.y, (float)y, ki.w), z);
}

// Vertex and normal maps (camera frame): n = b x a with a = V(x+1, y) - V,
// b = V(x, y+1) - V, divided by sqrt(n . n); no normal on the last row or
// column, next to a pixel without depth, or when |n| = 0.
__global__ void k_maps(const float* __restrict__ d, int w, int h, float4 ki, float* __restrict__ V,
                       float* __restrict__ N) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= w || y >= h) return;
    const size_t i = (size_t)y * w + x;
    const float3 v0 = vertex_at(d, w, x, y, ki);
    V[3 * i] = v0.x;
    V[3 * i + 1] = v0.y;
    V[3 * i + 2] = v0.z;
    float n0 = 0.0f, n1 = 0.0f, n2 = 0.0f;
    if (x + 1 < w && y + 1 < h && v0.z != 0.0f) {
        const float3 v1 = vertex_at(d, w, x + 1, y, ki), v2 = vertex_at(d, w, x, y + 1, ki);
        if (v1.z != 0.0f && v2.z != 0.0f) {
            const float a0 = v1.x - v0.x, a1 = v1.y - v0.y, a2 = v1.z - v0.z;
            const float b0 = v2.x - v0.x, b1 = v2.y - v0.y, b2 = v2.z - v0.z;
            const float c0 = b1 * a2 - b2 * a1, c1 = b2 * a0 - b0 * a2, c2 = b0 * a1 - b1 * a0;
            const float len = __fsqrt_rn(fmaf(c0, c0, fmaf(c1, c1, c2 * c2)));
            if (len > 0.0f) {
                n0 = __fdiv_rn(c0, len);
                n1 = __fdiv_rn(c1, len);
                n2 = __fdiv_rn(c2, len);
            }
        }
    }
    N[3 * i] = n0;
    N[3 * i + 1] = n1;
    N[3 * i + 2] = n2;
}

// ------------------------------------------------------ normal equations --
// Sums of one step: the 21 entries of the upper triangle of A = sum J J^T
// (row by row), g = sum J r (6), sum r^2 and the count.
constexpr int NSUM = 29;

__device__ __forceinline__ void rigid3(const float* R, const float* t, float x, float y, float z, float& X, float& Y,
                                       float& Z) {
    X = fmaf(R[0], x, fmaf(R[1], y, fmaf(R[2], z, t[0])));
    Y = fmaf(R[3], x, fmaf(R[4], y, fmaf(R[5], z, t[1])));
    Z = fmaf(R[6], x, fmaf(R[7], y, fmaf(R[8], z, t[2])));
}

// What bounds a step is the binary64 pipe, which takes about 64 cycles per
// warp instruction on each quarter of an SM whatever the number of active
// lanes, so both parts keep off it where they can:
//  * terms: the 28 sums of products are kept per thread as error-free triples
//    of binary32 numbers (fsum3: 22 instructions per product, more bits than
//    a binary64 sum), the count as an integer; the sums of a warp's lanes are
//    reduced by halves (each exchange halves the sums a lane holds: 31
//    additions instead of 5 per sum, 145) and turned into binary64 one per
//    lane, the warps' and blocks' sums added with one lane per sum;
//  * solve: by the last block to finish, one warp, a lane per row or matrix
//    entry (one thread alone took 28 us per step).
// One launch per step; its blocks start while the previous step finishes and
// read their first pixels before waiting for that step's pose.
// Measured per step: 24.0 us at 640x480, 17.8 at 320x240, 14.2 at 160x120
// (some 14 us of each is the fixed chain of wait, reduction and solve); with
// the sums in binary64, one fused multiply-add per product, 27.6, 19.2 and
// 16.8 us; with separate kernels for the terms and a one-thread solve 57 us on
// average over a frame's 19 steps.
constexpr int NSLOT = 32;  // the 29 sums, padded

// Sums of a warp's lanes: lane l gets the sum of v[l].
__device__ __forceinline__ double warp_sums(fsum3 (&v)[NSLOT], int lane) {
#pragma unroll
    for (int h = NSLOT / 2; h >= 1; h >>= 1) {
        const bool up = (lane & h) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const fsum3 give = up ? v[k] : v[k + h], keep = up ? v[k + h] : v[k];
            v[k] = fsum3_merge(keep, fsum3_shfl_xor(give, h));
        }
    }
    return fsum3_value(v[0]);
}

// exp coefficients of a rotation by angle a: row 0 sin(a)/a, row 1
// (1 - cos(a))/a^2, row 2 (a - sin(a))/a^3, as power series in a^2
// ((-1)^k / (2k + 1 + row)!, exact to binary64 for a <= 1/2: the first term
// left out is below 0.25^8 / 17!).
__constant__ double c_exp_series[3][8] = {
    {1.0, -1.0 / 6, 1.0 / 120, -1.0 / 5040, 1.0 / 362880, -1.0 / 39916800, 1.0 / 6227020800.0,
     -1.0 / 1307674368000.0},
    {1.0 / 2, -1.0 / 24, 1.0 / 720, -1.0 / 40320, 1.0 / 3628800, -1.0 / 479001600, 1.0 / 87178291200.0,
     -1.0 / 20922789888000.0},
    {1.0 / 6, -1.0 / 120, 1.0 / 5040, -1.0 / 362880, 1.0 / 39916800, -1.0 / 6227020800.0, 1.0 / 1307674368000.0,
     -1.0 / 355687428096000.0}};

struct SolveShared {
    double s[NSLOT], L[6][6], xi[6], coef[3], R[9], V[9], pose[16];
};

// One warp: solves A xi = -g by Cholesky (binary64; lane i holds row i) from
// the sums in S.s and applies T <- exp(xi^) T; a matrix that is not positive
// definite leaves T as it is.  The step's sums (29), its starting pose (16),
// its xi (6) and whether it was solved go to record.
__device__ void icp_solve(SolveShared& S, double* __restrict__ pose, double* __restrict__ record, int lane) {
    const unsigned full = 0xffffffffu;
    if (lane < 16) S.pose[lane] = pose[lane];
    __syncwarp();
    if (lane < NSUM) record[lane] = S.s[lane];
    if (lane < 16) record[NSUM + lane] = S.pose[lane];
    const int row = min(lane, 5);
    double a[6];  // the row's lower part, then its factor's
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const int lo = min(row, j), hi = max(row, j);
        a[j] = S.s[lo * 6 - lo * (lo - 1) / 2 + hi - lo];  // the upper triangle, row by row
    }
    double z = -S.s[21 + row], inv = 1.0;
    bool ok = true;
    // a pivot that is not positive marks the step unsolved and is replaced by
    // 1 so the remaining arithmetic stays finite (its result is not used)
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double v = __shfl_sync(full, a[j], j);
        if (!(v > 0.0)) {
            ok = false;
            v = 1.0;
        }
        const double y = rsqrt(v);  // 1 / L_jj
        if (lane == j) inv = y;
        a[j] = a[j] * y;
#pragma unroll
        for (int q = j + 1; q < 6; ++q) a[q] = __fma_rn(-a[j], __shfl_sync(full, a[j], q), a[q]);
    }
    if (lane < 6) {
#pragma unroll
        for (int j = 0; j < 6; ++j) S.L[lane][j] = a[j];
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {  // L y = -g: lane j's z becomes y_j
        const double y = z * inv, yj = __shfl_sync(full, y, j);
        z = lane == j ? y : (lane > j ? __fma_rn(-a[j], yj, z) : z);
    }
    __syncwarp();
#pragma unroll
    for (int j = 5; j >= 0; --j) {  // L^T xi = y
        const double x = z * inv, xj = __shfl_sync(full, x, j);
        z = lane == j ? x : (lane < j ? __fma_rn(-S.L[j][row], xj, z) : z);
    }
    if (lane < 6) S.xi[lane] = ok ? z : 0.0;
    __syncwarp();
    if (ok) {
        // exp(xi^): Rodrigues rotation, V(phi) rho translation
        const double p0 = S.xi[3], p1 = S.xi[4], p2 = S.xi[5];
        const double a2 = __fma_rn(p0, p0, __fma_rn(p1, p1, p2 * p2));
        if (a2 <= 0.25) {
            const double* cs = c_exp_series[min(lane, 2)];
            double v = cs[7];
#pragma unroll
            for (int k = 6; k >= 0; --k) v = __fma_rn(v, a2, cs[k]);
            if (lane < 3) S.coef[lane] = v;
        } else if (lane == 0) {
            const double an = sqrt(a2);
            S.coef[0] = sin(an) / an;
            S.coef[1] = (1.0 - cos(an)) / a2;
            S.coef[2] = (an - sin(an)) / (a2 * an);
        }
        __syncwarp();
        if (lane < 9) {  // entry (i, j) of R = I + cA W + cB W^2 and V = I + cB W + cC W^2, W = phi^
            const int i = lane / 3, j = lane % 3;
            const double pi = S.xi[3 + i], pj = S.xi[3 + j], pk = S.xi[3 + (i == j ? (i + 1) % 3 : 3 - i - j)],
                         pl = S.xi[3 + (i + 2) % 3];
            const double w = i == j ? 0.0 : ((j - i + 3) % 3 == 1 ? -pk : pk);
            const double w2 = i == j ? -__fma_rn(pk, pk, pl * pl) : pi * pj;
            const double e = i == j ? 1.0 : 0.0;
            S.R[lane] = e + __fma_rn(S.coef[0], w, S.coef[1] * w2);
            S.V[lane] = e + __fma_rn(S.coef[1], w, S.coef[2] * w2);
        }
        __syncwarp();
        if (lane < 12) {
            const int i = lane >> 2, j = lane & 3;
            double v = 0.0;
            if (j == 3) {
#pragma unroll
                for (int q = 0; q < 3; ++q) v = __fma_rn(S.V[i * 3 + q], S.xi[q], v);
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) v = __fma_rn(S.R[i * 3 + q], S.pose[q * 4 + j], v);
            pose[lane] = v;
        }
    }
    if (lane < 6) record[NSUM + 16 + lane] = S.xi[lane];
    if (lane == 0) record[NSUM + 22] = ok ? 1.0 : 0.0;
}

// Per pixel: p = R V + t, m = R N; the prediction pixel of Rp p + tp through
// Kl (nearest, inside, Z > 0, with a predicted normal); the distance and
// normal gates; r = (p - q) . nq and J = (nq, p x nq).  The pose of the step
// is read from the device (binary64, rounded once to binary32 here).  Each
// block writes its binary64 partial sums, threads combined in a fixed order;
// the last block to finish sums the blocks' in a fixed order, solves and
// updates the pose, and resets the count of finished blocks.
__global__ void __launch_bounds__(TRACK_THREADS) k_icp_step(TrackLevel L, double* __restrict__ pose,
                                                            double* __restrict__ partials,
                                                            unsigned* __restrict__ finished,
                                                            double* __restrict__ record) {
    constexpr int NW = TRACK_THREADS / 32;
    __shared__ double red[NW][NSLOT];
    __shared__ SolveShared S;
    __shared__ bool last;
    const int npx = L.w * L.h;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    // the vertex and normal maps are older than the previous step: read
    // before waiting for it
    float vx = 0.0f, vy = 0.0f, vz = 0.0f, nx = 0.0f, ny = 0.0f, nz = 0.0f;
    auto fetch = [&](int k) {
        vx = L.V[3 * k], vy = L.V[3 * k + 1], vz = L.V[3 * k + 2];
        nx = L.N[3 * k], ny = L.N[3 * k + 1], nz = L.N[3 * k + 2];
    };
    if (i < npx) fetch(i);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float R[9], t[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
#pragma unroll
        for (int k = 0; k < 3; ++k) R[r * 3 + k] = (float)pose[r * 4 + k];
        t[r] = (float)pose[r * 4 + 3];
    }
    fsum3 acc[NSLOT];
#pragma unroll
    for (int k = 0; k < NSLOT; ++k) acc[k] = {0.0f, 0.0f, 0.0f};
    unsigned pairs = 0;
    for (; i < npx; i += gridDim.x * blockDim.x) {
        const float v0 = vx, v1 = vy, v2 = vz, m0 = nx, m1 = ny, m2 = nz;
        const int next = i + gridDim.x * blockDim.x;
        if (next < npx) fetch(next);
        if (v2 == 0.0f || (m0 == 0.0f && m1 == 0.0f && m2 == 0.0f)) continue;
        float p[3], m[3], qc[3];
        rigid3(R, t, v0, v1, v2, p[0], p[1], p[2]);
        const float zero[3] = {0.0f, 0.0f, 0.0f};
        rigid3(R, zero, m0, m1, m2, m[0], m[1], m[2]);
        rigid3(L.Rp, L.tp, p[0], p[1], p[2], qc[0], qc[1], qc[2]);
        if (!(qc[2] > 0.0f)) continue;
        const float rz = __frcp_rn(qc[2]);
        const float ux = fmaf(L.K[0], qc[0], L.K[2] * qc[2]) * rz;
        const float uy = fmaf(L.K[4], qc[1], L.K[5] * qc[2]) * rz;
        const float fu = floorf(ux + 0.5f), fv = floorf(uy + 0.5f);
        if (!(fu >= 0.0f && fu <= (float)(L.w - 1) && fv >= 0.0f && fv <= (float)(L.h - 1))) continue;
        const size_t j = (size_t)fv * L.w + (size_t)fu;
        const float q0 = L.PV[3 * j], q1 = L.PV[3 * j + 1], q2 = L.PV[3 * j + 2];
        const float n0 = L.PN[3 * j], n1 = L.PN[3 * j + 1], n2 = L.PN[3 * j + 2];
        if (n0 == 0.0f && n1 == 0.0f && n2 == 0.0f) continue;
        const float e0 = p[0] - q0, e1 = p[1] - q1, e2 = p[2] - q2;
        if (fmaf(e0, e0, fmaf(e1, e1, e2 * e2)) > L.max_dist2) continue;
        if (!(fmaf(m[0], n0, fmaf(m[1], n1, m[2] * n2)) >= L.min_cos)) continue;
        const float r = fmaf(e0, n0, fmaf(e1, n1, e2 * n2));
        const float J[7] = {n0, n1, n2, p[1] * n2 - p[2] * n1, p[2] * n0 - p[0] * n2, p[0] * n1 - p[1] * n0, r};
        int k = 0;
#pragma unroll
        for (int a = 0; a < 6; ++a)
#pragma unroll
            for (int b = a; b < 6; ++b, ++k) fsum3_add_product(acc[k], J[a], J[b]);
#pragma unroll
        for (int a = 0; a < 7; ++a) fsum3_add_product(acc[21 + a], J[a], J[6]);
        ++pairs;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pairs = __reduce_add_sync(0xffffffffu, pairs);
    const double sum = warp_sums(acc, lane);
    red[warp][lane] = lane == 28 ? (double)pairs : sum;
    __syncthreads();
    if (warp == 0) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) v += red[w][lane];
        partials[(size_t)blockIdx.x * NSLOT + lane] = v;
        __threadfence();
        __syncwarp();
        if (lane == 0) last = atomicAdd(finished, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // lane l of warp w: sum l of blocks w, w + 8, ... in order, then the warps'
    double v = 0.0;
#pragma unroll 4
    for (int b = warp; b < (int)gridDim.x; b += NW) v += __ldcg(partials + (size_t)b * NSLOT + lane);
    red[warp][lane] = v;
    __syncthreads();
    if (warp != 0) return;
    v = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) v += red[w][lane];
    S.s[lane] = v;
    if (lane == 0) *finished = 0u;
    __syncwarp();
    icp_solve(S, pose, record, lane);
}

}  // namespace

cudaError_t launch_track_pyramid(const uint16_t* depth, int W, int H, int levels, float* const* d,
                                 cudaStream_t stream) {
    k_depth_metres<<<(W * H + 255) / 256, 256, 0, stream>>>(depth, W * H, d[0]);
    int w = W, h = H;
    for (int l = 1; l < levels; ++l) {
        const int w2 = w / 2, h2 = h / 2;
        const dim3 blk(32, 8), grd((w2 + 31) / 32, (h2 + 7) / 8);
        k_pyr_down<<<grd, blk, 0, stream>>>(d[l - 1], w, d[l], w2, h2);
        w = w2;
        h = h2;
    }
    return cudaGetLastError();
}

cudaError_t launch_track_maps(const float* d, int w, int h, const float Kinv4[4], float* V, float* N,
                              cudaStream_t stream) {
    const dim3 blk(32, 8), grd((w + 31) / 32, (h + 7) / 8);
    k_maps<<<grd, blk, 0, stream>>>(d, w, h, make_float4(Kinv4[0], Kinv4[1], Kinv4[2], Kinv4[3]), V, N);
    return cudaGetLastError();
}

// Blocks of a step's launch: one thread per pixel up to one block per SM of a
// GB300, then each thread takes several pixels.  Every block reduces its
// threads' sums, so more blocks cost more than their pixels gain.
constexpr int TRACK_MAX_BLOCKS = 152;
int track_blocks(int npx) {
    const int want = (npx + TRACK_THREADS - 1) / TRACK_THREADS;
    return want < TRACK_MAX_BLOCKS ? (want > 0 ? want : 1) : TRACK_MAX_BLOCKS;
}

size_t track_partial_doubles(int npx) { return (size_t)track_blocks(npx) * NSLOT; }
size_t track_record_doubles() { return NSUM + 16 + 6 + 1; }

cudaError_t launch_track_step(const TrackLevel& L, double* pose, double* partials, unsigned* finished, double* record,
                              cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)track_blocks(L.w * L.h));
    cfg.blockDim = dim3(TRACK_THREADS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_icp_step, L, pose, partials, finished, record);
}

}  // namespace tsdf
