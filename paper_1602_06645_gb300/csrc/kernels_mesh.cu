// Mesh extraction from the geometry volume (marching cubes, or marching
// tetrahedra as an option) and per-polygon texture maps from the colour
// volume (Section IV.C-D, Eq. 11-14).  Definitions (operation order, cases,
// orientation, map layout) as stated in tsdf.h; compiled with --fmad=false so
// only the written fmaf() fuse.
#include <cfloat>
#include <cstdint>

#include "common.cuh"
#include "device_math.cuh"

namespace tsdf {
namespace {

constexpr int MESH_THREADS = 128;  // 4 warps, one candidate brick per warp
constexpr int TILE_M = BRICK + 1;  // cells of a brick need one more voxel on the + sides
constexpr int TILE_M3 = TILE_M * TILE_M * TILE_M;
constexpr int CASE_BYTES = 16;     // a row of the marching-cubes case table (CubeCases)

// Corner orders of the six tetrahedra of a cell (main-diagonal split): for the
// axis orderings (x,y,z), (x,z,y), (y,x,z), (y,z,x), (z,x,y), (z,y,x) the path
// 0, 0 + a0, 0 + a0 + a1, 7.
__device__ __forceinline__ void tet_corners(int t, int c[4]) {
    const int a0 = t < 2 ? 0 : (t < 4 ? 1 : 2);
    const int a1 = (t == 0 || t == 5) ? 1 : ((t == 1 || t == 3) ? 2 : 0);
    c[0] = 0;
    c[1] = 1 << a0;
    c[2] = c[1] | (1 << a1);
    c[3] = 7;
}

// Lower and upper corner of cell edge e = 4 a + r: the lower corner is r with
// a zero bit inserted at position a.
__device__ __forceinline__ void cube_edge_corners(int e, int& p, int& q) {
    const int a = e >> 2, r = e & 3;
    p = a == 0 ? r << 1 : (a == 1 ? (r & 1) | ((r & 2) << 1) : r);
    q = p | (1 << a);
}

// ------------------------------------------------------- candidate bricks --
// A brick holds cells (min corner in the brick) whose corners span it and its
// +x/+y/+z neighbours; some cell can have triangles only if among those
// bricks' observed voxels there is one with F < 0 and one with F >= 0.
__global__ void __launch_bounds__(256) k_mesh_bricks(MeshConst c, const BrickSummary* __restrict__ summ,
                                                     uint32_t* __restrict__ list, uint32_t* __restrict__ n_list) {
    const uint32_t nbt = (uint32_t)c.nb[0] * c.nb[1] * c.nb[2];
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    bool cand = false;
    if (b < nbt) {
        const int bx = b % c.nb[0], by = (b / c.nb[0]) % c.nb[1], bz = b / (c.nb[0] * c.nb[1]);
        float mn = FLT_MAX, mx = -FLT_MAX;
        bool any = false;
        for (int k = 0; k < 8; ++k) {
            const int x = bx + (k & 1), y = by + ((k >> 1) & 1), z = bz + (k >> 2);
            if (x >= c.nb[0] || y >= c.nb[1] || z >= c.nb[2]) continue;
            const BrickSummary s = summ[((size_t)z * c.nb[1] + y) * c.nb[0] + x];
            if (!(s.fmin <= FLT_MAX)) continue;  // no observed voxel
            any = true;
            mn = fminf(mn, s.fmin);
            mx = fmaxf(mx, s.fmax);
        }
        cand = any && mn < 0.0f && mx >= 0.0f;
    }
    append(cand, b, n_list, list);
}

// One warp's working set: the F of its brick and of the next bricks' first
// layers, per tile row (z * 9 + y) a bit per voxel (x = observed, 9 + x = F <
// 0), and the cells (z, y, x of the lower corner) that the surface crosses.
struct MeshSlot {
    float F[TILE_M3];
    uint32_t row[TILE_M * TILE_M];
    uint16_t cells[BRICK_VOX];
};

__device__ __forceinline__ float centre_of(const MeshConst& c, int a, int i) {
    return fmaf((float)i + 0.5f, c.s_g, c.origin[a]);
}

// Vertex on the edge between cell corners a and b (p the lower corner index,
// which is the lower linear voxel index).
__device__ __forceinline__ void edge_vertex(const MeshConst& c, const int base[3], const float Fc[8], int a, int b,
                                            float out[3]) {
    const int p = min(a, b), q = max(a, b);
    const float t = __fdiv_rn(Fc[p], Fc[p] - Fc[q]);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const float Pp = centre_of(c, ax, base[ax] + ((p >> ax) & 1));
        const float Pq = centre_of(c, ax, base[ax] + ((q >> ax) & 1));
        out[ax] = fmaf(t, Pq - Pp, Pp);
    }
}

// Orient (normal toward the outside corner) and store one triangle.
__device__ __forceinline__ void emit(const MeshConst& c, const int base[3], const float v0[3], const float v1[3],
                                     const float v2[3], int cin, int cout, float* __restrict__ dst) {
    float e1[3], e2[3], d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        e1[a] = v1[a] - v0[a];
        e2[a] = v2[a] - v0[a];
        d[a] = centre_of(c, a, base[a] + ((cout >> a) & 1)) - centre_of(c, a, base[a] + ((cin >> a) & 1));
    }
    const float n0 = e1[1] * e2[2] - e1[2] * e2[1];
    const float n1 = e1[2] * e2[0] - e1[0] * e2[2];
    const float n2 = e1[0] * e2[1] - e1[1] * e2[0];
    const bool flip = fmaf(n0, d[0], fmaf(n1, d[1], n2 * d[2])) < 0.0f;
    const float* a1 = flip ? v2 : v1;
    const float* a2 = flip ? v1 : v2;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        dst[a] = v0[a];
        dst[3 + a] = a1[a];
        dst[6 + a] = a2[a];
    }
}

// Triangles of a cell by tetrahedra, from the mask of its inside corners.
__device__ __forceinline__ int tet_count(uint32_t m) {
    int n = 0;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
        int cc[4];
        tet_corners(t, cc);
        int ni = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) ni += (m >> cc[k]) & 1u;
        n += (ni == 0 || ni == 4) ? 0 : (ni == 2 ? 2 : 1);
    }
    return n;
}

// Write the triangles of one cell from slot `slot` on (those at or beyond cap
// are dropped).
__device__ void cell_emit(const MeshConst& c, const int base[3], const float Fc[8], float* __restrict__ out,
                          uint64_t slot, uint64_t cap) {
    for (int t = 0; t < 6; ++t) {
        int cc[4];
        tet_corners(t, cc);
        int ins[4], outs[4], ni = 0, no = 0;
        for (int k = 0; k < 4; ++k) {
            if (Fc[cc[k]] < 0.0f) ins[ni++] = cc[k];
            else outs[no++] = cc[k];
        }
        if (ni == 0 || no == 0) continue;
        if (ni == 1 || no == 1) {
            const int lone = ni == 1 ? ins[0] : outs[0];
            const int* others = ni == 1 ? outs : ins;
            float v[3][3];
            for (int e = 0; e < 3; ++e) edge_vertex(c, base, Fc, lone, others[e], v[e]);
            if (slot < cap) emit(c, base, v[0], v[1], v[2], ins[0], outs[0], out + 9 * slot);
            ++slot;
        } else {
            float q[4][3];
            edge_vertex(c, base, Fc, ins[0], outs[0], q[0]);
            edge_vertex(c, base, Fc, ins[0], outs[1], q[1]);
            edge_vertex(c, base, Fc, ins[1], outs[1], q[2]);
            edge_vertex(c, base, Fc, ins[1], outs[0], q[3]);
            if (slot < cap) emit(c, base, q[0], q[1], q[2], ins[0], outs[0], out + 9 * slot);
            ++slot;
            if (slot < cap) emit(c, base, q[0], q[2], q[3], ins[0], outs[0], out + 9 * slot);
            ++slot;
        }
    }
}

// Marching cubes: write the n triangles of one cell from its case row.
__device__ void cube_emit(const MeshConst& c, const int base[3], const float Fc[8], const uint8_t* row, int n,
                          float* __restrict__ out, uint64_t slot, uint64_t cap) {
    for (int t = 0; t < n; ++t, ++slot) {
        if (slot >= cap) continue;
        float* dst = out + 9 * slot;
        for (int k = 0; k < 3; ++k) {
            int p, q;
            cube_edge_corners(row[1 + 3 * t + k], p, q);
            edge_vertex(c, base, Fc, p, q, dst + 3 * k);
        }
    }
}

// Stage one tile voxel.
template <bool KEEP_F>
__device__ __forceinline__ void mesh_stage(MeshSlot& S, int tx, int ty, int tz, float f, bool observed) {
    const int r = tz * TILE_M + ty;
    if (KEEP_F) S.F[r * TILE_M + tx] = f;
    const uint32_t bits = (observed ? 1u : 0u) | (f < 0.0f ? 1u << 9 : 0u);
    if (bits) atomicOr(&S.row[r], bits << tx);
}

// Mask of the inside corners of cell (cx, cy, cz) (bit dx + 2 dy + 4 dz).
__device__ __forceinline__ uint32_t cell_mask(const MeshSlot& S, int cx, int cy, int cz) {
    const int r = cz * TILE_M + cy, sh = 9 + cx;
    return ((S.row[r] >> sh) & 3u) | ((S.row[r + 1] >> sh) & 3u) << 2 | ((S.row[r + TILE_M] >> sh) & 3u) << 4 |
           ((S.row[r + TILE_M + 1] >> sh) & 3u) << 6;
}

// One warp per candidate brick: the brick is staged with 16-byte reads and the
// 217 voxels of the next bricks' first layers by one read each, all issued
// together; the row bits give the cells that are wholly observed and have
// corners on both sides, 64 cells in a handful of bitwise steps; those are
// counted and their triangles written 32 at a time.  The warp claims its
// triangles' places with one atomic per brick (one per 32 cells, some 130,000
// on one address, bounded the kernel), and where nothing is written (cap 0)
// with one per block.  Counting and then writing the triangles of the fused
// 512^3 scan (24 frames, about 700,000): 2 x 169 -> 32 + 95 us.
// WRITE: false only counts (cap is 0), without keeping the F of the tile.
template <bool CUBES, bool WRITE>
__global__ void __launch_bounds__(MESH_THREADS) k_mesh(const __grid_constant__ CubeCases table, MeshConst c,
                                                      const float* __restrict__ F,
                                                      const uint8_t* __restrict__ W,
                                                      const uint32_t* __restrict__ list,
                                                      const uint32_t* __restrict__ n_list, float* __restrict__ out,
                                                      uint64_t cap, unsigned long long* __restrict__ count) {
    __shared__ MeshSlot slots[MESH_THREADS / 32];
    // the case table: lanes look up different rows, which the parameter space would serve one by one
    __shared__ __align__(16) uint8_t cases[CUBES ? 256 * CASE_BYTES : 16];
    __shared__ unsigned long long block_total;
    if (CUBES) {
        for (int i = threadIdx.x; i < 256; i += MESH_THREADS)
            reinterpret_cast<uint4*>(cases)[i] = reinterpret_cast<const uint4*>(table.t)[i];
    }
    if (threadIdx.x == 0) block_total = 0ull;
    __syncthreads();
    MeshSlot& S = slots[threadIdx.x >> 5];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n = *n_list;
    unsigned long long counted = 0;
    for (uint32_t item = warp; item < n; item += nwarps) {
        const uint32_t b = list[item];
        const int bb[3] = {(int)(b % c.nb[0]), (int)((b / c.nb[0]) % c.nb[1]), (int)(b / (c.nb[0] * c.nb[1]))};
        const int base0[3] = {bb[0] * BRICK, bb[1] * BRICK, bb[2] * BRICK};
        // reads: the brick's four groups of four voxels per lane, and the halo:
        // 3 faces x 64, 3 edges x 8, 1 corner
        float4 f[4];
        uint32_t w[4];
        {
            const size_t at = (size_t)b * BRICK_VOX + lane * 4;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                f[j] = *reinterpret_cast<const float4*>(F + at + 128 * j);
                w[j] = *reinterpret_cast<const uint32_t*>(W + at + 128 * j);
            }
        }
        int hx[7], hy[7], hz[7];
#pragma unroll
        for (int i = 0; i < 6; ++i) {  // faces: i = 2 * axis + half
            const int axis = i >> 1, q = lane + 32 * (i & 1), u = q & 7, v = q >> 3;
            hx[i] = axis == 0 ? BRICK : u;
            hy[i] = axis == 1 ? BRICK : (axis == 0 ? u : v);
            hz[i] = axis == 2 ? BRICK : v;
        }
        {  // edges (lanes 0..23, along axis lane / 8) and the corner (lane 24)
            const int e = lane >> 3, m = lane & 7;
            hx[6] = e == 0 ? m : BRICK;
            hy[6] = e == 1 ? m : BRICK;
            hz[6] = e == 2 ? m : BRICK;
        }
        float hf[7];
        bool ho[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            const int x = base0[0] + hx[i], y = base0[1] + hy[i], z = base0[2] + hz[i];
            const bool in = (i < 6 || lane < 25) && x < c.ng[0] && y < c.ng[1] && z < c.ng[2];
            const int64_t o = in ? brick_offset(x, y, z, c.nb) : 0;
            hf[i] = in ? F[o] : 0.0f;
            ho[i] = in && W[o] != 0;
        }
        for (int r = lane; r < TILE_M * TILE_M; r += 32) S.row[r] = 0u;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = lane + 32 * j, x0 = (q & 1) * 4, y = (q >> 1) & 7, z = q >> 4, r = z * TILE_M + y;
            const float fv[4] = {f[j].x, f[j].y, f[j].z, f[j].w};
            const bool yz = base0[1] + y < c.ng[1] && base0[2] + z < c.ng[2];
            uint32_t bits = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (WRITE) S.F[r * TILE_M + x0 + i] = fv[i];
                const bool seen = yz && base0[0] + x0 + i < c.ng[0] && ((w[j] >> (8 * i)) & 0xFFu) != 0u;
                bits |= ((seen ? 1u : 0u) | (fv[i] < 0.0f ? 1u << 9 : 0u)) << i;
            }
            if (bits) atomicOr(&S.row[r], bits << x0);
        }
#pragma unroll
        for (int i = 0; i < 7; ++i)
            if (i < 6 || lane < 25) mesh_stage<WRITE>(S, hx[i], hy[i], hz[i], hf[i], ho[i]);
        __syncwarp();
        // the crossed cells of two cell rows (y, z) per lane, compacted
        uint32_t act[2];
        int mine = 0;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int yz = lane + 32 * r, at = (yz >> 3) * TILE_M + (yz & 7);
            const uint32_t a = S.row[at], b1 = S.row[at + 1], c1 = S.row[at + TILE_M], d1 = S.row[at + TILE_M + 1];
            const uint32_t all = a & b1 & c1 & d1, any = a | b1 | c1 | d1;
            const uint32_t seen = all & (all >> 1);                                       // bits 0..7
            const uint32_t neg_all = (all >> 9) & (all >> 10), neg_any = (any >> 9) | (any >> 10);
            act[r] = seen & neg_any & ~neg_all & 0xFFu;
            mine += __popc(act[r]);
        }
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += v;
        }
        const int nact = __shfl_sync(full, incl, 31);
        int pos = incl - mine;
#pragma unroll
        for (int r = 0; r < 2; ++r)
            for (uint32_t a = act[r]; a; a &= a - 1u) S.cells[pos++] = (uint16_t)((lane + 32 * r) * BRICK + __ffs(a) - 1);
        __syncwarp();
        auto triangles = [&](int k, uint32_t& m, int& cell) -> uint32_t {
            cell = S.cells[k];
            m = cell_mask(S, cell & 7, (cell >> 3) & 7, cell >> 6);
            return CUBES ? cases[m * CASE_BYTES] : (uint32_t)tet_count(m);
        };
        uint32_t total = 0, m;
        int cell;
        for (int k = lane; k < nact; k += 32) total += triangles(k, m, cell);
        total = __reduce_add_sync(full, total);
        if (!WRITE) {
            counted += total;
            __syncwarp();
            continue;
        }
        unsigned long long at = 0;
        if (lane == 0 && total) at = atomicAdd(count, (unsigned long long)total);
        at = __shfl_sync(full, at, 0);
        for (int k0 = 0; k0 < nact && at < cap; k0 += 32) {
            const uint32_t tri = k0 + lane < nact ? triangles(k0 + lane, m, cell) : 0u;
            uint32_t sum = tri;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(full, sum, o);
                if (lane >= o) sum += v;
            }
            if (tri) {
                const int cx = cell & 7, cy = (cell >> 3) & 7, cz = cell >> 6;
                const int base[3] = {base0[0] + cx, base0[1] + cy, base0[2] + cz};
                float Fc[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    Fc[k] = S.F[((cz + (k >> 2)) * TILE_M + cy + ((k >> 1) & 1)) * TILE_M + cx + (k & 1)];
                if (CUBES) cube_emit(c, base, Fc, cases + m * CASE_BYTES, (int)tri, out, at + sum - tri, cap);
                else cell_emit(c, base, Fc, out, at + sum - tri, cap);
            }
            at += __shfl_sync(full, sum, 31);
        }
        __syncwarp();
    }
    if (!WRITE) {
        if (lane == 0 && counted) atomicAdd(&block_total, counted);
        __syncthreads();
        if (threadIdx.x == 0 && block_total) atomicAdd(count, block_total);
    }
}

// ------------------------------------------------------------ textures ----
constexpr int SCAN_THREADS = 1024;

__device__ __forceinline__ float length3(float x, float y, float z) {
    return __fsqrt_rn(fmaf(x, x, fmaf(y, y, z * z)));
}

__device__ __forceinline__ int map_side(float dist, float size_pixel, int max_side) {
    const float q = floorf(__fdiv_rn(dist, size_pixel) + 0.5f);
    if (!(q >= 2.0f)) return 2;
    if (q > (float)max_side) return max_side;
    return (int)q;
}

// Block-wide exclusive scan of one int64 per thread (the block total is the
// last thread's excl + v).
__device__ void block_scan(int64_t v, int64_t& excl) {
    __shared__ int64_t warp_sums[SCAN_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int64_t s = lane < SCAN_THREADS / 32 ? warp_sums[lane] : 0;
        int64_t si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += t;
        }
        if (lane < SCAN_THREADS / 32) warp_sums[lane] = si - s;  // exclusive warp offsets
    }
    __syncthreads();
    excl = warp_sums[wid] + incl - v;
    __syncthreads();
}

__global__ void __launch_bounds__(SCAN_THREADS) k_tex_sizes(const float* __restrict__ tris, int64_t n, float size_pixel,
                                                           int32_t max_side, int32_t* __restrict__ wh,
                                                           int64_t* __restrict__ off, int64_t* __restrict__ sums) {
    const int64_t i = (int64_t)blockIdx.x * SCAN_THREADS + threadIdx.x;
    int64_t texels = 0;
    if (i < n) {
        const float* T = tris + 9 * i;
        const int w = map_side(length3(T[3] - T[0], T[4] - T[1], T[5] - T[2]), size_pixel, max_side);
        const int h = map_side(length3(T[6] - T[0], T[7] - T[1], T[8] - T[2]), size_pixel, max_side);
        wh[2 * i] = w;
        wh[2 * i + 1] = h;
        texels = (int64_t)w * h;
    }
    int64_t excl;
    block_scan(texels, excl);
    if (i < n) off[i] = excl;
    if (threadIdx.x == SCAN_THREADS - 1) sums[blockIdx.x] = excl + texels;
}

// Exclusive scan of the block sums in one block; sums[nb] = grand total.
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_sums(int64_t* __restrict__ sums, int64_t nb) {
    int64_t carry = 0;
    for (int64_t base = 0; base < nb; base += SCAN_THREADS) {
        const int64_t i = base + threadIdx.x;
        const int64_t v = i < nb ? sums[i] : 0;
        int64_t excl;
        block_scan(v, excl);
        __shared__ int64_t chunk;
        if (threadIdx.x == SCAN_THREADS - 1) chunk = excl + v;
        __syncthreads();
        if (i < nb) sums[i] = carry + excl;
        carry += chunk;
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[nb] = carry;
}

__global__ void k_tex_offsets(int64_t* __restrict__ off, int64_t n, const int64_t* __restrict__ sums, int64_t nb) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) off[i] += sums[i / SCAN_THREADS];
    if (i == n) off[n] = sums[nb];
}

// Byte i of a packed colour as binary32 (the bits 0x4B0000bb are 2^23 + b).
template <int I>
__device__ __forceinline__ float colour_byte(uint32_t col) {
    return __uint_as_float(__byte_perm(col, 0x4B000000u, 0x7440u + I)) - 8388608.0f;
}

// Trilinear colour at a point over the observed colour voxels of its cell.  A
// corner that is unobserved or outside the volume has weight 0, which leaves
// the sums as they are.  The eight reads are addressed from the lower corner
// by one step per axis and issued together.
__device__ __forceinline__ uint32_t texel_colour(const ColourConst& c, const uint32_t* __restrict__ C, float px,
                                                 float py, float pz) {
    const float p[3] = {px, py, pz};
    float wgt[3][2];
    int i0[3];
    bool in[3][2];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float g = fmaf(p[a] - c.origin[a], c.inv_sc, -0.5f);
        const float fl = floorf(g);
        if (!(fl >= -1.0f) || !(fl <= (float)c.nc[a])) return 0u;
        const int i = (int)fl;
        const float f = g - fl;
        in[a][0] = i >= 0 && i < c.nc[a];
        in[a][1] = i + 1 < c.nc[a];
        wgt[a][0] = 1.0f - f;
        wgt[a][1] = f;
        i0[a] = i;
    }
    // the lower corner's offset, and the steps to the upper one (from local 7
    // into the next brick, which also takes -1, local 7 of brick -1, to 0)
    const int lx = i0[0] & 7, ly = i0[1] & 7, lz = i0[2] & 7;
    const int64_t base = (((int64_t)(i0[2] >> 3) * c.ncb[1] + (i0[1] >> 3)) * c.ncb[0] + (i0[0] >> 3)) * BRICK_VOX +
                         (lz * BRICK + ly) * BRICK + lx;
    const int dx = lx == 7 ? BRICK_VOX - 7 : 1;
    const int dy = ly == 7 ? c.ncb[0] * BRICK_VOX - 7 * BRICK : BRICK;
    const int dz = lz == 7 ? c.ncb[0] * c.ncb[1] * BRICK_VOX - 7 * BRICK * BRICK : BRICK * BRICK;
    uint32_t col[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const bool ok = in[0][k & 1] && in[1][(k >> 1) & 1] && in[2][k >> 2];
        col[k] = ok ? __ldg(C + base + ((k & 1) ? dx : 0) + ((k & 2) ? dy : 0) + ((k & 4) ? dz : 0)) : 0u;
    }
    float acc0 = 0.0f, acc1 = 0.0f, acc2 = 0.0f, wsum = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float w = wgt[0][k & 1] * wgt[1][(k >> 1) & 1];
        w = w * wgt[2][k >> 2];
        w = (col[k] >> 24) ? w : 0.0f;
        acc0 = fmaf(w, colour_byte<0>(col[k]), acc0);
        acc1 = fmaf(w, colour_byte<1>(col[k]), acc1);
        acc2 = fmaf(w, colour_byte<2>(col[k]), acc2);
        wsum = wsum + w;
    }
    if (!(wsum > 0.0f)) return 0u;
    const float acc[3] = {acc0, acc1, acc2};
    uint32_t out = 255u << 24;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        const float val = floorf(__fdiv_rn(acc[ch], wsum) + 0.5f);
        const uint32_t u = val <= 0.0f ? 0u : (val >= 255.0f ? 255u : (uint32_t)val);
        out |= u << (8 * ch);
    }
    return out;
}

// A triangle's map: its first texel's corner, the steps of a texel along its
// two sides (Eq. 13-14), the map's width and its offset.
struct TexMap {
    float p[3], green[3], blue[3];
    int32_t w;
    int64_t start;
};
__device__ __forceinline__ TexMap tex_map(const float* __restrict__ tris, const int32_t* __restrict__ wh,
                                          const int64_t* __restrict__ off, int64_t t) {
    TexMap m;
    m.start = off[t];
    m.w = wh[2 * t];
    const int h = wh[2 * t + 1];
    const float* T = tris + 9 * t;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        m.p[a] = T[a];
        m.green[a] = __fdiv_rn(T[3 + a] - T[a], (float)(m.w - 1));
        m.blue[a] = __fdiv_rn(T[6 + a] - T[a], (float)(h - 1));
    }
    return m;
}

// One thread per texel, a warp TEX_ITEM consecutive ones.  A texel's triangle is
// the last t with off[t] <= idx.  The warp finds the first one's by a search
// of 32 probes a step and then holds a window of 32 triangles, one per lane
// with its map's steps (their six divisions once per triangle), among which
// its texels find theirs by five shuffles; the window moves on when the texels
// leave it (maps from the layout have at least four texels, so it serves at
// least 128).  A texel beyond the window searches the rest alone.  What bounds
// it is instruction issue, then the colour gathers: 158 us for the 4 M texels
// of 700,000 triangles in no spatial order; 348 us with a binary search of
// twenty dependent reads, every division and eight full addresses per texel.
constexpr int TEX_ITEM = 256;
__global__ void __launch_bounds__(256) k_tex_fill(ColourConst c, const uint32_t* __restrict__ C,
                                                  const float* __restrict__ tris, int64_t n,
                                                  const int32_t* __restrict__ wh, const int64_t* __restrict__ off,
                                                  int64_t total, uint32_t* __restrict__ texels) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t first = warp * TEX_ITEM; first < total; first += nwarps * TEX_ITEM) {
        // the first texel's triangle: [lo, hi] holds it, off[lo] <= first
        int64_t lo = 0, hi = n - 1;
        while (lo < hi) {
            const int64_t step = (hi - lo + 31) / 32, probe = lo + step * (lane + 1);
            const bool le = probe <= hi && off[probe] <= first;
            const int up = __popc(__ballot_sync(full, le));  // offsets do not decrease: the lanes below `up`
            const int64_t l2 = lo + step * up;
            hi = min(hi, l2 + step - 1);
            lo = l2;
        }
        int64_t t0 = lo;
        TexMap mine;
        int edge;  // the next triangle's offset from `first`; beyond the last triangle and 2^31: a bound no texel reaches
        auto window = [&]() {
            const int64_t t = t0 + lane;
            mine = tex_map(tris, wh, off, min(t, n - 1));
            const int64_t e = t + 1 < n ? off[t + 1] - first : (int64_t)INT32_MAX;
            edge = (int)min(e, (int64_t)INT32_MAX);
        };
        window();
        for (int rel = 0; rel < TEX_ITEM && first + rel < total; rel += 32) {
            if (rel + 31 >= __shfl_sync(full, edge, 31)) {  // start the window at this item's first triangle
                t0 = min(t0 + __popc(__ballot_sync(full, edge <= rel)), n - 1);
                window();
            }
            const int at = rel + lane;
            int k = 0;  // offsets of the window that are <= the texel's
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(full, edge, k + o - 1) <= at) k += o;
            const bool beyond = __shfl_sync(full, edge, 31) <= at;
            TexMap m;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                m.p[a] = __shfl_sync(full, mine.p[a], k);
                m.green[a] = __shfl_sync(full, mine.green[a], k);
                m.blue[a] = __shfl_sync(full, mine.blue[a], k);
            }
            m.w = __shfl_sync(full, mine.w, k);
            m.start = __shfl_sync(full, mine.start, k);
            const int64_t idx = first + at;
            if (idx >= total) continue;
            if (beyond) {
                int64_t a = min(t0 + 32, n - 1), b = n - 1;
                while (a < b) {
                    const int64_t mid = (a + b + 1) >> 1;
                    if (off[mid] <= idx) a = mid;
                    else b = mid - 1;
                }
                m = tex_map(tris, wh, off, a);
            }
            const int64_t local = idx - m.start;
            int i, j;
            if ((uint64_t)local >> 32) {
                j = (int)(local / m.w);
                i = (int)(local % m.w);
            } else {
                j = (int)((uint32_t)local / (uint32_t)m.w);
                i = (int)((uint32_t)local - (uint32_t)j * (uint32_t)m.w);
            }
            float p[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) p[a] = fmaf((float)j, m.blue[a], fmaf((float)i, m.green[a], m.p[a]));
            texels[idx] = texel_colour(c, C, p[0], p[1], p[2]);
        }
    }
}

}  // namespace

cudaError_t launch_mesh(const MeshConst& c, const float* F, const uint8_t* W, const BrickSummary* summ,
                        uint32_t* list, uint32_t* n_list, float* out, uint64_t cap, unsigned long long* count,
                        bool cubes, const CubeCases& cases, cudaStream_t stream) {
    const uint32_t nbt = (uint32_t)c.nb[0] * c.nb[1] * c.nb[2];
    k_mesh_bricks<<<(nbt + 255) / 256, 256, 0, stream>>>(c, summ, list, n_list);
    int sms = 0, dev = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto k = cubes ? (cap ? k_mesh<true, true> : k_mesh<true, false>)
                   : (cap ? k_mesh<false, true> : k_mesh<false, false>);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, MESH_THREADS, 0);
    k<<<max(1, sms * max(1, per_sm)), MESH_THREADS, 0, stream>>>(cases, c, F, W, list, n_list, out, cap, count);
    return cudaGetLastError();
}

cudaError_t launch_texture_layout(const float* tris, int64_t n, float size_pixel, int32_t max_side, int32_t* wh,
                                  int64_t* off, int64_t* scratch, cudaStream_t stream) {
    const int64_t nb = (n + SCAN_THREADS - 1) / SCAN_THREADS;
    if (nb > 0) k_tex_sizes<<<(unsigned)nb, SCAN_THREADS, 0, stream>>>(tris, n, size_pixel, max_side, wh, off, scratch);
    k_scan_sums<<<1, SCAN_THREADS, 0, stream>>>(scratch, nb);
    k_tex_offsets<<<(unsigned)((n + 1 + 255) / 256), 256, 0, stream>>>(off, n, scratch, nb);
    return cudaGetLastError();
}

cudaError_t launch_texture_fill(const ColourConst& c, const uint32_t* C, const float* tris, int64_t n,
                                const int32_t* wh, const int64_t* off, int64_t total, uint32_t* texels,
                                cudaStream_t stream) {
    if (total <= 0 || n <= 0) return cudaSuccess;
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t per_block = (int64_t)TEX_ITEM * (256 / 32), want = (total + per_block - 1) / per_block;
    const unsigned grid = (unsigned)(want < (int64_t)sms * 8 ? want : (int64_t)sms * 8);
    k_tex_fill<<<grid, 256, 0, stream>>>(c, C, tris, n, wh, off, total, texels);
    return cudaGetLastError();
}

}  // namespace tsdf
