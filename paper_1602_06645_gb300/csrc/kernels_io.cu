// Layout conversion between the brick-major device volumes and linear
// x-fastest arrays (read-out / restore), and brick summaries of a restored
// volume.
#include <cfloat>
#include <cstdint>

#include "common.cuh"

namespace tsdf {
namespace {

// Bound by HBM: each voxel is read once and written once.  A warp moves the
// 8 rows of 32 voxels (4 bricks) of one z slice in accesses of VE voxels, the
// widest that both addresses and the row length allow: with 4 voxels of 4
// bytes per lane, 8 lanes along x and 4 along y, every warp access is four
// whole 128-byte lines on both sides (a linear row of 4 bricks; 4 rows of one
// brick).  Each lane has at least four accesses in flight and no division in
// its addressing.  Measured: a 1024^3 colour and a 512^3 F volume together
// 1.35 ms each way (7.2 TB/s), a 512^3 weight volume 0.040 ms; with one voxel
// per thread and 64-bit divisions for its coordinates they took 4.3 ms and
// 0.48 ms.  A 750 x 729 x 687 colour volume (8-byte accesses) runs at 6.4
// (read-out) and 7.0 TB/s (restore), 1.36 ms each way before, 0.23-0.25 now.
// NARROW (rows of at most one brick, 8 voxels): at most 8 lanes along x and the
// rest along y, where the wide form leaves 31 of 32 lanes idle at nx = 1.  The
// three volumes of a call read out: 1 x 512 x 512 46 -> 33 us, 3 x 700 x 700 60 ->
// 45, 8 x 1024 x 1024 83 -> 70.
template <int VE, bool NARROW>
struct ConvertShape {
    static constexpr int XL = NARROW ? (VE == 1 ? 8 : 4) : 32 / VE, YL = 32 / XL;  // lanes along x and y
    static constexpr int XW = XL * VE;                                             // voxels of a chunk along x
    static constexpr int XC = NARROW ? 1 : (VE == 8 ? 4 : (VE == 4 ? 2 : 1));      // chunks per warp
    static constexpr int YI = BRICK / YL;                                          // row steps
};
template <typename V, int VE, bool NARROW, bool TO_LINEAR>
__global__ void __launch_bounds__(256) k_convert(V* __restrict__ brick, V* __restrict__ lin, int nx, int ny, int nz,
                                                 int z0, int nbx, int nby) {
    using S = ConvertShape<VE, NARROW>;
    constexpr int XL = S::XL, YL = S::YL, XW = S::XW, XC = S::XC, YI = S::YI;
    const int lane = threadIdx.x & 31, z = blockIdx.z * BRICK + (threadIdx.x >> 5);
    if (z >= nz) return;
    const int by = blockIdx.y, ly = lane / XL, gz = z0 + z;
    const int x0 = blockIdx.x * (XW * XC) + (lane % XL) * VE;
    const int64_t brow = (((int64_t)(gz >> 3) * nby + by) * nbx) * BRICK_VOX + (gz & 7) * (BRICK * BRICK);
    const int64_t lrow = ((int64_t)z * ny + by * BRICK) * nx;
    V v[XC][YI];
#pragma unroll
    for (int c = 0; c < XC; ++c)
#pragma unroll
        for (int r = 0; r < YI; ++r) {
            const int x = x0 + XW * c, y = ly + YL * r;
            if (x < nx && by * BRICK + y < ny)
                v[c][r] = TO_LINEAR ? brick[(brow + (int64_t)(x >> 3) * BRICK_VOX + y * BRICK + (x & 7)) / VE]
                                    : lin[(lrow + (int64_t)y * nx + x) / VE];
        }
#pragma unroll
    for (int c = 0; c < XC; ++c)
#pragma unroll
        for (int r = 0; r < YI; ++r) {
            const int x = x0 + XW * c, y = ly + YL * r;
            if (x < nx && by * BRICK + y < ny) {
                if (TO_LINEAR)
                    lin[(lrow + (int64_t)y * nx + x) / VE] = v[c][r];
                else
                    brick[(brow + (int64_t)(x >> 3) * BRICK_VOX + y * BRICK + (x & 7)) / VE] = v[c][r];
            }
        }
}

template <typename V, int VE, bool NARROW, bool TO_LINEAR>
cudaError_t convert_grid(void* brick, void* lin, const int32_t dims[3], int z0, int z1, cudaStream_t stream) {
    constexpr int XW = ConvertShape<VE, NARROW>::XW * ConvertShape<VE, NARROW>::XC;  // voxels of a warp
    const int nbx = (dims[0] + BRICK - 1) / BRICK, nby = (dims[1] + BRICK - 1) / BRICK;
    const dim3 grid((unsigned)((dims[0] + XW - 1) / XW), (unsigned)nby, (unsigned)((z1 - z0 + BRICK - 1) / BRICK));
    k_convert<V, VE, NARROW, TO_LINEAR><<<grid, 256, 0, stream>>>(static_cast<V*>(brick), static_cast<V*>(lin), dims[0],
                                                                  dims[1], z1 - z0, z0, nbx, nby);
    return cudaGetLastError();
}

template <typename V, int VE, bool TO_LINEAR>
cudaError_t convert_as(void* brick, void* lin, const int32_t dims[3], int z0, int z1, cudaStream_t stream) {
    return dims[0] <= BRICK ? convert_grid<V, VE, true, TO_LINEAR>(brick, lin, dims, z0, z1, stream)
                            : convert_grid<V, VE, false, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
}

// The widest access whose size divides both base addresses and the linear row
// (every row then starts on a multiple of it, and no access crosses a row's end).
template <typename T, bool TO_LINEAR>
cudaError_t convert(T* brick, T* lin, const int32_t dims[3], int z0, int z1, cudaStream_t stream) {
    if (dims[0] <= 0 || dims[1] <= 0 || z1 <= z0) return cudaSuccess;
    const uint64_t all = (uint64_t)(uintptr_t)brick | (uint64_t)(uintptr_t)lin | (uint64_t)dims[0] * sizeof(T);
    if (sizeof(T) == 4) {
        if (all % 16 == 0) return convert_as<uint4, 4, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
        if (all % 8 == 0) return convert_as<uint2, 2, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
        return convert_as<uint32_t, 1, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
    }
    if (all % 8 == 0) return convert_as<uint2, 8, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
    if (all % 4 == 0) return convert_as<uint32_t, 4, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
    if (all % 2 == 0) return convert_as<uint16_t, 2, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
    return convert_as<uint8_t, 1, TO_LINEAR>(brick, lin, dims, z0, z1, stream);
}

// Brick summaries: min/max of F over observed voxels, whether all of them are
// observed and at the weight limit (wmin) and the band flags (what the
// geometry kernel maintains).  Bound by HBM (5 B per voxel).  One warp per
// brick with the geometry kernel's lane layout (lane l: voxels 4 (l + 32 j) ..
// + 3, j = 0..3), all eight 16- and 4-byte reads of a lane issued together; the
// flags come from the minima and maxima over the lane's faces, the weights are
// tested four at a time.  About 103 us at 512^3 (6.5 TB/s; 118 with a minimum
// per weight, 128 with a test for weights above the limit beside it, whose 40
// registers leave 48 warps per SM instead of 64); one block per brick with
// scalar reads and a shared-memory reduction took 235 us.
constexpr int SUM_WARPS = 8;
__global__ void __launch_bounds__(SUM_WARPS * 32) k_summaries(const float* __restrict__ F,
                                                              const uint8_t* __restrict__ W,
                                                              BrickSummary* __restrict__ summ, int nx, int ny, int nz,
                                                              int nbx, int nby, uint32_t nbt, float band,
                                                              uint32_t max_weight, uint32_t* __restrict__ odd_f) {
    const uint32_t b = blockIdx.x * SUM_WARPS + (threadIdx.x >> 5);
    if (b >= nbt) return;
    const int lane = threadIdx.x & 31;
    const int bx = b % nbx, by = (b / nbx) % nby, bz = b / (nbx * nby);
    const int lx = (lane & 1) * 4, ly = (lane >> 1) & 7, lz = lane >> 4;
    const size_t base = (size_t)b * BRICK_VOX + lane * 4;
    float4 f[4];
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        f[j] = *reinterpret_cast<const float4*>(F + base + 128 * j);
        w[j] = *reinterpret_cast<const uint32_t*>(W + base + 128 * j);
    }
    const float inf = __int_as_float(0x7f800000), qnan = __int_as_float(0x7fffffff);
    float mn = inf, mx = -inf, mn_xf = inf, mx_xf = -inf, mn_zf = inf, mx_zf = -inf;
    const uint32_t limit4 = max_weight * 0x01010101u;
    uint32_t xin = 0u;  // this lane's bytes inside the volume along x
#pragma unroll
    for (int i = 0; i < 4; ++i) xin |= bx * BRICK + lx + i < nx ? 0xFFu << (8 * i) : 0u;
    uint32_t hole = 0u, differs = 0u;  // an unobserved voxel (bit 7 of some byte); a weight that is not the limit
    bool odd = false;
    // (voxels outside the volume hold F = 0 and w = 0)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const bool in = by * BRICK + ly < ny && bz * BRICK + lz + 2 * j < nz;
        const float fv[4] = {f[j].x, f[j].y, f[j].z, f[j].w};
        const uint32_t inside = in ? xin : 0u, wq = (w[j] & inside) | (limit4 & ~inside);
        hole |= (wq - 0x01010101u) & ~wq;
        differs |= wq ^ limit4;
        float gmn = inf, gmx = -inf;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            odd = odd || !(fabsf(fv[i]) <= PLAIN_F);
            const float v = (w[j] >> (8 * i)) & 0xFFu ? fv[i] : qnan;  // fminf / fmaxf pass over a NaN
            gmn = fminf(gmn, v);
            gmx = fmaxf(gmx, v);
            if (i == (lx ? 3 : 0)) {  // the lane's x-face voxel
                mn_xf = fminf(mn_xf, v);
                mx_xf = fmaxf(mx_xf, v);
            }
        }
        if (j == (lz ? 3 : 0)) {  // its z-face group
            mn_zf = gmn;
            mx_zf = gmx;
        }
        mn = fminf(mn, gmn);
        mx = fmaxf(mx, gmx);
    }
    const float lo_thr = band + CELL_EPS, hi_thr = -band - CELL_EPS;
    auto lohi = [&](float a, float c) -> uint32_t { return (a <= lo_thr ? 1u : 0u) | (c >= hi_thr ? 2u : 0u); };
    const uint32_t all = lohi(mn, mx), xf = lohi(mn_xf, mx_xf), zf = lohi(mn_zf, mx_zf);
    uint32_t flags = all | (lx == 0 ? xf << 2 : xf << 4) | (ly == 0 ? all << 6 : 0u) | (ly == 7 ? all << 8 : 0u) |
                     (lz == 0 ? zf << 10 : zf << 12);
    if (__any_sync(0xffffffffu, odd) && lane == 0) *odd_f = 1u;
    flags = __reduce_or_sync(0xffffffffu, flags);
    // (a weight above the limit comes down to it at its next update: the brick
    // is not saturated)
    const bool unobserved = __any_sync(0xffffffffu, (hole & 0x80808080u) != 0u);
    const bool below_cap = __any_sync(0xffffffffu, differs != 0u);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
        BrickSummary s;
        s.fmin = mn >= FLT_MAX ? inf : mn;
        s.fmax = mx <= -FLT_MAX ? -inf : mx;
        s.wmin = unobserved ? 0u : (below_cap ? max_weight - 1u : max_weight);
        s.flags = flags;
        summ[b] = s;
    }
}

}  // namespace

cudaError_t launch_to_linear_f32(const float* b, float* l, const int32_t d[3], int z0, int z1, cudaStream_t s) {
    return convert<float, true>(const_cast<float*>(b), l, d, z0, z1, s);
}
cudaError_t launch_to_linear_u8(const uint8_t* b, uint8_t* l, const int32_t d[3], int z0, int z1, cudaStream_t s) {
    return convert<uint8_t, true>(const_cast<uint8_t*>(b), l, d, z0, z1, s);
}
cudaError_t launch_to_linear_u32(const uint32_t* b, uint32_t* l, const int32_t d[3], int z0, int z1, cudaStream_t s) {
    return convert<uint32_t, true>(const_cast<uint32_t*>(b), l, d, z0, z1, s);
}
cudaError_t launch_from_linear_f32(float* b, const float* l, const int32_t d[3], int z0, int z1, cudaStream_t s) {
    return convert<float, false>(b, const_cast<float*>(l), d, z0, z1, s);
}
cudaError_t launch_from_linear_u8(uint8_t* b, const uint8_t* l, const int32_t d[3], int z0, int z1, cudaStream_t s) {
    return convert<uint8_t, false>(b, const_cast<uint8_t*>(l), d, z0, z1, s);
}
cudaError_t launch_from_linear_u32(uint32_t* b, const uint32_t* l, const int32_t d[3], int z0, int z1,
                                   cudaStream_t s) {
    return convert<uint32_t, false>(b, const_cast<uint32_t*>(l), d, z0, z1, s);
}

cudaError_t launch_recompute_summaries(const float* F, const uint8_t* W, BrickSummary* summ, const int32_t ng[3],
                                       float band, int32_t max_weight, uint32_t* odd_f, cudaStream_t stream) {
    const cudaError_t e = cudaMemsetAsync(odd_f, 0, sizeof(uint32_t), stream);
    if (e != cudaSuccess) return e;
    const int nbx = (ng[0] + BRICK - 1) / BRICK, nby = (ng[1] + BRICK - 1) / BRICK, nbz = (ng[2] + BRICK - 1) / BRICK;
    const int64_t nbt = (int64_t)nbx * nby * nbz;
    if (nbt > 0)
        k_summaries<<<(unsigned)((nbt + SUM_WARPS - 1) / SUM_WARPS), SUM_WARPS * 32, 0, stream>>>(
            F, W, summ, ng[0], ng[1], ng[2], nbx, nby, (uint32_t)nbt, band, (uint32_t)max_weight, odd_f);
    return cudaGetLastError();
}

}  // namespace tsdf
