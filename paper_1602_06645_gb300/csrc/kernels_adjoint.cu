// Photometric colour loss of the fused colour volume and its adjoint, for
// refining the HD camera's calibration (intrinsics of Eq. 4, extrinsic of
// Eq. 3) from the colour consistency of the fused volume.
//
// For every colour voxel v recorded in the sets S_k (frames whose depth-side
// gates it passes), the forward pass is the mean of its binary32 bilinear HD
// samples over the frames where the 2x2 footprint lies inside the image:
//   C_v = (1/n_v) sum_k s_k(v),   s_k = bilinear(I_k, K_hd T P_vc)
// (Eq. 9 with W = 1, unrounded).  The backward pass takes dL/dC_v and returns
// dL/dI_k (scattered to the 4 footprint pixels with atomics), dL/dK_hd and the
// derivative with respect to a left se(3) perturbation of the extrinsic at the
// linearisation point: dP/drho = I, dP/dphi_j = e_j x P.
//
// One thread per voxel slot; a slot's frames are visited in ascending order,
// so the colours are deterministic.  Camera-parameter gradients are summed
// error-free per warp, then over warps and blocks in binary64 in a fixed order.
#include <cstdint>

#include "common.cuh"
#include "device_math.cuh"
#include "ffloat.cuh"

namespace tsdf {
namespace {

constexpr int ADJ_THREADS = 256;

// ------------------------------------------------------------ finalize ----
// Slots: the first pair of a voxel claims it (-1 -> -2) and takes the next
// slot number; the voxel map then holds the slot.
__global__ void k_slot_claim(AdjBuffers a, uint32_t* err) {
    const uint32_t n = min(a.counters[0], a.pair_cap);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t v = a.pair_vox[i];
        if (atomicCAS(&a.slot_of[v], -1, -2) == -1) {
            const uint32_t s = atomicAdd(&a.counters[1], 1u);
            if (s < a.slot_cap) {
                a.V[s] = v;
                a.slot_of[v] = (int32_t)s;
            } else {
                atomicOr(err, ERR_SLOT_OVERFLOW);
            }
        }
    }
}

__global__ void k_slot_fill(AdjBuffers a, uint32_t* err) {
    const uint32_t n = min(a.counters[0], a.pair_cap);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t s = a.slot_of[a.pair_vox[i]];
        if (s < 0) continue;
        const uint32_t j = atomicAdd(&a.slot_count[s], 1u);
        if (j < (uint32_t)a.max_frames)
            a.slot_frames[(size_t)s * a.max_frames + j] = a.pair_frame[i];
        else
            atomicOr(err, ERR_SLOT_OVERFLOW);
    }
}

// Insertion sort of each slot's frame ids (a frame appears at most once).
__global__ void k_slot_sort(AdjBuffers a) {
    const uint32_t n = min(a.counters[1], a.slot_cap);
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        uint8_t* f = a.slot_frames + (size_t)s * a.max_frames;
        const int m = min((int)a.slot_count[s], a.max_frames);
        for (int i = 1; i < m; ++i) {
            const uint8_t key = f[i];
            int j = i - 1;
            while (j >= 0 && f[j] > key) {
                f[j + 1] = f[j];
                --j;
            }
            f[j + 1] = key;
        }
    }
}

// ------------------------------------------------------------- sample -----
struct Sample {
    bool valid;
    int x0, y0;
    float ax, ay, X, Y, Z;
};

// HD sample position of voxel (centre p) in frame k at the linearisation
// point: P_vc = R_n p + t_n (Eq. 5), P = R P_vc + t (Eq. 3), (u, v) = K P / Z
// (Eq. 4) with the operations of the colour update's projection
// (xh = fmaf(fx, X, cx Z), u = xh * (1/Z)); the bilinear footprint
// (x0..x0+1, y0..y0+1), x0 = floor(u), must lie in the image.  The cell is an
// integer decision, taken exactly as the fusion's bilinear sampling takes it.
__device__ __forceinline__ Sample hd_sample(const AdjCamera& cam, const AdjFrame& fr, float px, float py, float pz) {
    Sample s;
    float Xc, Yc, Zc;
    rigid(fr.R, fr.t, px, py, pz, Xc, Yc, Zc);
    rigid(cam.R, cam.t, Xc, Yc, Zc, s.X, s.Y, s.Z);
    s.valid = false;
    if (!(s.Z > 0.0f)) return s;
    const float rz = __frcp_rn(s.Z);
    const float u = fmaf(cam.fx, s.X, cam.cx * s.Z) * rz, v = fmaf(cam.fy, s.Y, cam.cy * s.Z) * rz;
    const float fx0 = floorf(u), fy0 = floorf(v);
    if (!(fx0 >= 0.0f && fx0 + 1.0f <= (float)(cam.width - 1) && fy0 >= 0.0f && fy0 + 1.0f <= (float)(cam.height - 1)))
        return s;
    s.valid = true;
    s.x0 = (int)fx0;
    s.y0 = (int)fy0;
    return s;
}

// The frames' constants, staged by the block: lanes of a warp are at different
// frames, which shared memory serves faster than global memory.
constexpr int MAX_ADJ_FRAMES = 64;
__device__ __forceinline__ void stage_frames(AdjFrame* s, const AdjCamera& cam, const AdjBuffers& a) {
    static_assert(sizeof(AdjFrame) == 48, "three 16-byte words");
    for (int i = threadIdx.x; i < 3 * cam.n_frames; i += blockDim.x)
        reinterpret_cast<float4*>(s)[i] = reinterpret_cast<const float4*>(a.frames)[i];
    __syncthreads();
}

// The bilinear fractions (u - x0, v - y0) of a valid sample, from the sample
// position in float-float arithmetic: the voxel centre origin + (k + 1/2) s_c,
// both rigid motions and the projection carry ~48 bits, so the fractions are
// those of the exact position for the given binary32 constants to within a
// few binary32 roundings (binary32 throughout would be ~1e-4 pixel off at
// HD resolution, a visible colour error across a sharp image edge).
__device__ __forceinline__ void hd_fractions(const AdjCamera& cam, const AdjFrame& fr, const int k[3], Sample& s) {
    ff p[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) p[a] = ff_add(two_prod((float)k[a] + 0.5f, cam.s_c), cam.origin[a]);
    ff c[3], h[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) c[r] = ff_row(fr.R + 3 * r, fr.t[r], p);
#pragma unroll
    for (int r = 0; r < 3; ++r) h[r] = ff_row(cam.R + 3 * r, cam.t[r], c);
    const ff qx = ff_div(h[0], h[2]), qy = ff_div(h[1], h[2]);
    const ff u = ff_add(ff_mul(qx, cam.fx), cam.cx), v = ff_add(ff_mul(qy, cam.fy), cam.cy);
    s.ax = (u.hi - (float)s.x0) + u.lo;  // the difference of the high parts is exact (Sterbenz)
    s.ay = (v.hi - (float)s.y0) + v.lo;
}

__device__ __forceinline__ void voxel_index(const AdjCamera& cam, uint32_t lin, int k[3]) {
    const uint32_t nx = (uint32_t)cam.nc[0], ny = (uint32_t)cam.nc[1];
    k[0] = (int)(lin % nx);
    k[1] = (int)((lin / nx) % ny);
    k[2] = (int)(lin / (nx * ny));
}

__device__ __forceinline__ void voxel_centre(const AdjCamera& cam, const int k[3], float& px, float& py, float& pz) {
    px = fmaf((float)k[0] + 0.5f, cam.s_c, cam.origin[0]);
    py = fmaf((float)k[1] + 0.5f, cam.s_c, cam.origin[1]);
    pz = fmaf((float)k[2] + 0.5f, cam.s_c, cam.origin[2]);
}

// The six floats at o (two RGB pixels).  VEC: the image starts on a 16-byte
// boundary and holds a multiple of four floats, so the aligned window of two
// 16-byte words around them (and one float more at an offset of 3) can be
// read; the window is shifted into place.  Lanes read scattered pixels, so
// the accesses, not their width, count.
template <bool VEC>
__device__ __forceinline__ void load6(const float* __restrict__ p, size_t o, float v[6]) {
    if (!VEC) {
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = __ldg(p + o + k);
        return;
    }
    const unsigned a = (unsigned)o & 3u;
    const float4* q = reinterpret_cast<const float4*>(p + (o - a));
    const float4 q0 = __ldg(q), q1 = __ldg(q + 1);
    float w[9] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, 0.0f};
    if (a == 3u) w[8] = __ldg(p + o + 5);
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = (a & 1u) ? w[k + 1] : w[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = (a & 2u) ? w[k + 2] : w[k];
}

// Adds six floats at o.  VEC (as in load6): two 16-byte reductions, the
// floats around the six getting -0, which changes no value, and a float more
// at an offset of 3.
template <bool VEC>
__device__ __forceinline__ void add6(float* __restrict__ p, size_t o, const float v[6]) {
    if (!VEC) {
#pragma unroll
        for (int k = 0; k < 6; ++k) atomicAdd(p + o + k, v[k]);
        return;
    }
    const unsigned a = (unsigned)o & 3u;
    float w[9] = {v[0], v[1], v[2], v[3], v[4], v[5], -0.0f, -0.0f, -0.0f};
#pragma unroll
    for (int k = 8; k > 0; --k) w[k] = (a & 1u) ? w[k - 1] : w[k];
    w[0] = (a & 1u) ? -0.0f : w[0];
#pragma unroll
    for (int k = 8; k > 1; --k) w[k] = (a & 2u) ? w[k - 2] : w[k];
    w[1] = (a & 2u) ? -0.0f : w[1];
    w[0] = (a & 2u) ? -0.0f : w[0];
    float* q = p + (o - a);
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(q), "f"(w[0]), "f"(w[1]), "f"(w[2]), "f"(w[3])
                 : "memory");
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(q + 4), "f"(w[4]), "f"(w[5]), "f"(w[6]),
                 "f"(w[7])
                 : "memory");
    if (a == 3u) atomicAdd(q + 8, w[8]);
}

// ------------------------------------------------------------ forward -----
// Near the HBM rate of the images it touches: 100 us for 4.0 M pairs of 20
// full-HD images (498 MB; 110 us at the registers the compiler takes unasked).
template <bool VEC>
__global__ void __launch_bounds__(ADJ_THREADS, 4) k_adj_forward(AdjCamera cam, AdjBuffers a, uint32_t n_slots,
                                                             const float* __restrict__ images, float* __restrict__ C,
                                                             int32_t* __restrict__ n_out) {
    __shared__ __align__(16) AdjFrame frames[MAX_ADJ_FRAMES];
    stage_frames(frames, cam, a);
    const size_t plane = (size_t)cam.height * cam.width * 3;
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < n_slots; s += gridDim.x * blockDim.x) {
        int kv[3];
        float px, py, pz;
        voxel_index(cam, a.V[s], kv);
        voxel_centre(cam, kv, px, py, pz);
        const uint8_t* fl = a.slot_frames + (size_t)s * a.max_frames;
        const int m = min((int)a.slot_count[s], a.max_frames);
        float sum[3] = {0.0f, 0.0f, 0.0f};
        int n = 0;
        for (int j = 0; j < m; ++j) {
            const int k = fl[j];
            Sample smp = hd_sample(cam, frames[k], px, py, pz);
            if (!smp.valid) continue;
            const size_t o00 = k * plane + ((size_t)smp.y0 * cam.width + smp.x0) * 3;
            float r0[6], r1[6];
            load6<VEC>(images, o00, r0);
            load6<VEC>(images, o00 + (size_t)cam.width * 3, r1);
            hd_fractions(cam, frames[k], kv, smp);
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                const float top = fmaf(smp.ax, r0[3 + ch] - r0[ch], r0[ch]);
                const float bot = fmaf(smp.ax, r1[3 + ch] - r1[ch], r1[ch]);
                sum[ch] += fmaf(smp.ay, bot - top, top);
            }
            ++n;
        }
        const float inv = n ? 1.0f / (float)n : 0.0f;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) C[(size_t)s * 3 + ch] = sum[ch] * inv;
        n_out[s] = n;
        a.n_valid[s] = n;
    }
}

// ----------------------------------------------------------- backward -----
// Bound by the image gradient's atomics (four pixels per pair, scattered) and
// the sample arithmetic.  The two pixels of a footprint row are added as
// 16-byte reductions (2.25 per row instead of 6 scalar ones), and the ten
// camera sums are kept per thread as error-free triples (see fsum3), combined
// over the warp by halves and turned into binary64 once per warp; the last
// block to finish adds the blocks' sums in a fixed order.  Measured for 4.0 M
// pairs of 20 full-HD images: 264 us, of which the images and their gradient
// take 220 at the HBM rate; with scalar atomics, binary64 sums per
// pair, a thread per voxel and a one-block reduction 700 and 37 us.  Two
// blocks per SM (100 registers) beat three and four at fewer registers.
constexpr int ADJ_SLOTS = 16;  // the ten sums, padded
template <bool VEC>
__global__ void __launch_bounds__(ADJ_THREADS) k_adj_backward(AdjCamera cam, AdjBuffers a, uint32_t n_slots,
                                                              const float* __restrict__ images,
                                                              const float* __restrict__ grad_C,
                                                              float* __restrict__ grad_images) {
    constexpr int NW = ADJ_THREADS / 32;
    __shared__ __align__(16) AdjFrame frames[MAX_ADJ_FRAMES];
    __shared__ double red[NW][ADJ_SLOTS];
    __shared__ bool last;
    stage_frames(frames, cam, a);
    const size_t plane = (size_t)cam.height * cam.width * 3;
    fsum3 acc[ADJ_SLOTS];
#pragma unroll
    for (int j = 0; j < ADJ_SLOTS; ++j) acc[j] = {0.0f, 0.0f, 0.0f};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a warp takes 32 slots and spreads their pairs, which number from 1 to
    // the frames recorded, evenly over its lanes
    for (uint32_t base = (blockIdx.x * NW + warp) * 32u; base < n_slots; base += gridDim.x * NW * 32u) {
        const uint32_t s = base + lane;
        const int n = s < n_slots ? a.n_valid[s] : 0;
        float gs[3] = {0.0f, 0.0f, 0.0f};
        uint32_t lin = 0;
        int m = 0;
        if (n != 0) {
            const float inv = 1.0f / (float)n;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) gs[ch] = grad_C[(size_t)s * 3 + ch] * inv;
            if (!(gs[0] == 0.0f && gs[1] == 0.0f && gs[2] == 0.0f)) {
                lin = a.V[s];
                m = min((int)a.slot_count[s], a.max_frames);
            }
        }
        int kvs[3];
        voxel_index(cam, lin, kvs);
        int end = m;  // pairs of the lanes up to and including this one
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        const int total = __shfl_sync(0xffffffffu, end, 31);
        for (int first = 0; first < total; first += 32) {
            const int idx = first + lane;
            int own = 0;  // the lane whose slot the pair belongs to: the first with end > idx
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, end, own + o - 1) <= idx) own += o;
            own = min(own, 31);
            const int j = idx - (__shfl_sync(0xffffffffu, end, own) - __shfl_sync(0xffffffffu, m, own));
            const int kv[3] = {__shfl_sync(0xffffffffu, kvs[0], own), __shfl_sync(0xffffffffu, kvs[1], own),
                               __shfl_sync(0xffffffffu, kvs[2], own)};
            const float g[3] = {__shfl_sync(0xffffffffu, gs[0], own), __shfl_sync(0xffffffffu, gs[1], own),
                                __shfl_sync(0xffffffffu, gs[2], own)};
            if (idx >= total) continue;
            const int k = a.slot_frames[(size_t)(base + own) * a.max_frames + j];
            float px, py, pz;
            voxel_centre(cam, kv, px, py, pz);
            Sample smp = hd_sample(cam, frames[k], px, py, pz);
            if (!smp.valid) continue;
            const size_t o00 = k * plane + ((size_t)smp.y0 * cam.width + smp.x0) * 3;
            const size_t o01 = o00 + (size_t)cam.width * 3;
            float p00[6], p01[6];
            load6<VEC>(images, o00, p00);
            load6<VEC>(images, o01, p01);
            hd_fractions(cam, frames[k], kv, smp);
            float dsdu = 0.0f, dsdv = 0.0f;
            const float w00 = (1.0f - smp.ax) * (1.0f - smp.ay), w10 = smp.ax * (1.0f - smp.ay);
            const float w01 = (1.0f - smp.ax) * smp.ay, w11 = smp.ax * smp.ay;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                dsdu += g[ch] * ((1.0f - smp.ay) * (p00[3 + ch] - p00[ch]) + smp.ay * (p01[3 + ch] - p01[ch]));
                dsdv += g[ch] * ((1.0f - smp.ax) * (p01[ch] - p00[ch]) + smp.ax * (p01[3 + ch] - p00[3 + ch]));
            }
            const float d0[6] = {g[0] * w00, g[1] * w00, g[2] * w00, g[0] * w10, g[1] * w10, g[2] * w10};
            const float d1[6] = {g[0] * w01, g[1] * w01, g[2] * w01, g[0] * w11, g[1] * w11, g[2] * w11};
            add6<VEC>(grad_images, o00, d0);
            add6<VEC>(grad_images, o01, d1);
            const float rz = 1.0f / smp.Z;
            const float X = smp.X, Y = smp.Y, Z = smp.Z;
            const float dPx = dsdu * cam.fx * rz, dPy = dsdv * cam.fy * rz;
            const float dPz = -(dsdu * cam.fx * X + dsdv * cam.fy * Y) * rz * rz;
            const float term[10] = {dsdu * X * rz, dsdv * Y * rz, dsdu, dsdv, dPx, dPy, dPz,
                                    Y * dPz - Z * dPy, Z * dPx - X * dPz, X * dPy - Y * dPx};
#pragma unroll
            for (int q = 0; q < 10; ++q) fsum3_add(acc[q], term[q]);
        }
    }
    // warp: by halves, lane l then holds sum l & 15 of its half warp; both
    // halves; block and grid in binary64, fixed order
#pragma unroll
    for (int h = ADJ_SLOTS / 2; h >= 1; h >>= 1) {
        const bool up = (lane & h) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const fsum3 give = up ? acc[k] : acc[k + h], keep = up ? acc[k + h] : acc[k];
            acc[k] = fsum3_merge(keep, fsum3_shfl_xor(give, h));
        }
    }
    acc[0] = fsum3_merge(acc[0], fsum3_shfl_xor(acc[0], 16));
    if (lane < ADJ_SLOTS) red[warp][lane] = fsum3_value(acc[0]);
    __syncthreads();
    if (threadIdx.x < 10) {
        double v = 0.0;
        for (int w = 0; w < NW; ++w) v += red[w][threadIdx.x];
        a.partials[(size_t)blockIdx.x * 10 + threadIdx.x] = v;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&a.counters[3], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int q = warp; q < 10; q += NW) {  // lane l: blocks l, l + 32, ... in order, then the lanes
        double v = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) v += __ldcg(a.partials + (size_t)b * 10 + q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) a.grad[q] = v;
    }
    if (threadIdx.x == 0) a.counters[3] = 0u;
}

}  // namespace

cudaError_t launch_adjoint_finalize(const AdjBuffers& a, uint32_t n_pairs_max, cudaStream_t stream) {
    // a.counters[2] is used as the error word of this phase
    const unsigned blocks = n_pairs_max ? (unsigned)((n_pairs_max + 255) / 256 > 4096 ? 4096 : (n_pairs_max + 255) / 256) : 1u;
    k_slot_claim<<<blocks, 256, 0, stream>>>(a, a.counters + 2);
    k_slot_fill<<<blocks, 256, 0, stream>>>(a, a.counters + 2);
    k_slot_sort<<<blocks, 256, 0, stream>>>(a);
    return cudaGetLastError();
}

// The image stack holds a multiple of four floats (see load6).
static bool whole_words(const AdjCamera& cam) {
    return (int64_t)cam.n_frames * cam.height * cam.width * 3 % 4 == 0;
}

cudaError_t launch_adjoint_forward(const AdjCamera& cam, const AdjBuffers& a, uint32_t n_slots, const float* images,
                                   float* C, int32_t* n_out, cudaStream_t stream) {
    if (n_slots == 0) return cudaSuccess;
    unsigned blocks = (n_slots + ADJ_THREADS - 1) / ADJ_THREADS;
    if (blocks > 8192u) blocks = 8192u;
    const bool vec = whole_words(cam) && ((uintptr_t)images & 15u) == 0;
    (vec ? k_adj_forward<true> : k_adj_forward<false>)<<<blocks, ADJ_THREADS, 0, stream>>>(cam, a, n_slots, images, C,
                                                                                          n_out);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_backward(const AdjCamera& cam, const AdjBuffers& a, uint32_t n_slots, const float* images,
                                    const float* grad_C, float* grad_images, int blocks, cudaStream_t stream) {
    const bool vec = whole_words(cam) && (((uintptr_t)images | (uintptr_t)grad_images) & 15u) == 0;
    (vec ? k_adj_backward<true> : k_adj_backward<false>)<<<blocks, ADJ_THREADS, 0, stream>>>(cam, a, n_slots, images,
                                                                                            grad_C, grad_images);
    return cudaGetLastError();
}

}  // namespace tsdf
