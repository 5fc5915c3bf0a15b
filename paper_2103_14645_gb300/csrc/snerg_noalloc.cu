// snerg_noalloc.cu -- ray-list render that allocates nothing and needs no workspace.
//
// Some callers cannot allocate device memory: a plug-in living inside a host
// application that owns every byte of the GPU through its own pool (and forbids
// cudaMalloc), a real-time loop where the implicit device synchronisation of
// cudaMalloc/cudaFree would stall the frame, or a sandboxed caller granted only the
// buffers it was handed. snerg_render_rays_noalloc serves them: it renders straight from
// the caller's indirection grid and uint8 atlas (no padded copy, no voxel distance map),
// and keeps its only scratch -- a status word and the block-level empty-space distance
// map with its transform's temporary -- in one file-scope __device__ array of fixed
// size that every GPU loading the library holds until the process exits.
//
// The array's host-side name is only a stand-in; its device address is fetched with
// cudaGetSymbolAddress, and every kernel a call can launch is loaded, once per device (with
// that device current) on the first call made on that device, so that first call should
// happen before any stream capture. The address is kept for the life of the process: a
// device reset (cudaDeviceReset, or a reset of the primary context) reloads the module and
// may move the array, after which the kept address is stale, so this entry point must not be
// used across a reset.
// Every call shares the array: calls whose work overlaps on the GPU (two streams, or two
// host threads) race on it and must be serialised by the caller.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "snerg_internal.cuh"

namespace snerg {
namespace {

constexpr int kNoAllocMaxG = 64;                               // N / B <= 64
constexpr size_t kNoAllocG3 = (size_t)kNoAllocMaxG * kNoAllocMaxG * kNoAllocMaxG;
constexpr size_t kNoAllocHeader = 256;                         // status word at byte 0
constexpr size_t kNoAllocBytes = kNoAllocHeader + 2 * kNoAllocG3;   // 524,544 bytes
constexpr int kNoAllocMaxDevices = 64;

// [0, 256): status word | bdist [G^3] | the distance transform after its x and y passes [G^3]
__device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocBytes];

// ---------------------------------------------------------------------------------
// The two-sided block map in two launches: the x and y passes of one z slice per CTA in
// shared memory (the x distances from a row's bit mask), then the z pass. The first launch
// also clears the status word. 17 us for 48^3 blocks, bound by latency; the general passes took
// four launches and 27 us.
// ---------------------------------------------------------------------------------
constexpr int kMapCap = 32;

__global__ void __launch_bounds__(1024) noalloc_map_xy_kernel(const int32_t* __restrict__ ind, int G, int32_t* status,
                                                              uint8_t* __restrict__ xy) {
    __shared__ uint8_t s_x[kNoAllocMaxG][kNoAllocMaxG];
    const int z = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (z == 0 && threadIdx.x == 0) *status = 0;
    for (int y = warp; y < G; y += 32) {
        const int32_t* row = ind + ((int64_t)z * G + y) * G;
        const uint32_t lo = __ballot_sync(0xffffffffu, lane < G && __ldg(row + lane) >= 0);
        const uint32_t hi = __ballot_sync(0xffffffffu, lane + 32 < G && __ldg(row + lane + 32) >= 0);
        const uint64_t bits = lo | (uint64_t)hi << 32;
        for (int x = lane; x < G; x += 32) {
            const uint64_t up = bits >> x, down = bits << (63 - x);     // bit x lowest / highest
            const int d = min(up ? __ffsll((long long)up) - 1 : kMapCap, down ? __clzll((long long)down) : kMapCap);
            s_x[y][x] = (uint8_t)min(d, kMapCap);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G * G; i += 1024) {
        const int x = i % G, y = i / G;
        int best = s_x[y][x];
        for (int d = 1; d < best; ++d) {
            if (y - d < 0 && y + d >= G) break;
            if (y - d >= 0) best = min(best, max(d, (int)s_x[y - d][x]));
            if (y + d < G) best = min(best, max(d, (int)s_x[y + d][x]));
        }
        xy[(int64_t)z * G * G + i] = (uint8_t)best;
    }
}

__global__ void __launch_bounds__(256) noalloc_map_z_kernel(const uint8_t* __restrict__ xy, int G,
                                                            uint8_t* __restrict__ bdist) {
    const int64_t n = (int64_t)G * G;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * G) return;
    const int z = (int)(t / n);
    int best = xy[t];
    for (int d = 1; d < best; d += 2) {             // two distances' loads at a time
        if (z - d < 0 && z + d >= G) break;
        int v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = d + (i >> 1), q = (i & 1) ? z + e : z - e;
            v[i] = q >= 0 && q < G ? max(e, (int)__ldg(xy + t + (int64_t)((i & 1) ? e : -e) * n)) : kMapCap;
        }
        best = min(best, min(min(v[0], v[1]), min(v[2], v[3])));
    }
    bdist[t] = (uint8_t)best;
}

// value of channel 0..7 of voxel (x, y, z) of the virtual grid, clamped to the grid;
// 0 in empty blocks (Sec. 5.1)
template <class SC>
__device__ __forceinline__ uint2 raw_voxel(const SC& s, const uint2* atlas, int64_t nb, int x, int y, int z) {
    x = min(max(x, 0), s.N - 1);
    y = min(max(y, 0), s.N - 1);
    z = min(max(z, 0), s.N - 1);
    const int slot = __ldg(s.ind + (((z >> s.lgB) * s.G + (y >> s.lgB)) * s.G + (x >> s.lgB)));
    if (slot < 0 || slot >= nb) return make_uint2(0u, 0u);
    const int B = s.B;
    const int loc = ((z & (B - 1)) * B + (y & (B - 1))) * B + (x & (B - 1));
    return __ldg(atlas + (size_t)slot * B * B * B + loc);
}

constexpr int kProbes = 8;

// The march of snerg_internal.cuh on the caller's unpadded atlas: empty blocks are
// skipped through the block distance map, every lattice sample of an occupied block
// probes its nearest voxel's density code, and the 8 trilinear corners are fetched from the
// block itself, or through the indirection grid where the stencil leaves it. Same lattice,
// same binary32 control arithmetic (so the same composited samples and the same early exit),
// and the same colour accumulation (accumulate_colour).
//
// Without a voxel distance map a ray meets every sample of a block, and one probe after the
// other is a chain of memory latencies: kProbes samples' codes are loaded together, and those
// with density composited in order. 65,537 scattered rays of a 768^3 grid: 294 us one by one,
// 150 us for 8 together (the whole call 301 -> 169 us; 174 for 4, 192 for 16), 165 with the block
// edge as a constant. On edges of 2 and 4, whose runs are mostly shorter than 8 samples, fewer
// would do: whole calls of 200,000 rays 311 and 315 us with 8, 286 and 303 with 4, 276 and 308 with 1.
template <class SC>
__device__ __forceinline__ void march_raw(const SC& s, const uint2* atlas, int64_t nb, const Ray& r,
                                          MarchState& st) {
#pragma unroll
    for (int c = 0; c < 7; ++c) st.acc[c] = 0.0f;
    st.T = 1.0f;
    st.tau = 0.0f;
    st.steps = 0;
    st.active = 0;
    st.blocks = 0;
    st.limit = false;
    if (!r.hit) return;
    const int N = s.N, B = s.B;
    float inv_d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) inv_d[i] = __fdividef(1.0f, r.d[i] == 0.0f ? 0.0f : r.d[i]);   // +inf for -0 too
    const float exit_half = 0.5f - exit_margin(r, s.fN);
    float kh = 0.5f;                                   // k + 1/2
    for (;;) {
        if (kh >= (float)s.kmax) { st.limit = true; return; }
        const float t = __fadd_rn(r.t0, kh);
        if (!(t < r.t1)) return;
        int j[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) j[i] = nearest_voxel(lattice_u(r, t, i), N);
        const int bi = ((j[2] >> s.lgB) * s.G + (j[1] >> s.lgB)) * s.G + (j[0] >> s.lgB);
        const int slot = __ldg(s.ind + bi);
        const int D = __ldg(s.bdist + bi);             // 0 where occupied
        const float kx = march_exit(s, r, inv_d, kh, j, max(D, 1), exit_half);
        if (slot < 0 || slot >= nb) {
            // an entry outside the atlas is reported and read as empty
            if (slot >= nb) atomicCAS(s.status, 0, (int)SNERG_E_INVAL);
            kh = kx;
            continue;
        }
        const uint2* blk = atlas + (size_t)slot * B * B * B;
        const int m = B - 1, o3[3] = {j[0] & -B, j[1] & -B, j[2] & -B};
        for (; kh < kx; kh += (float)kProbes) {
            uint32_t set = 0;
#pragma unroll
            for (int i = 0; i < kProbes; ++i) {
                const float tk = __fadd_rn(r.t0, kh + (float)i);
                const int v0 = nearest_voxel(lattice_u(r, tk, 0), N) & m, v1 = nearest_voxel(lattice_u(r, tk, 1), N) & m,
                          v2 = nearest_voxel(lattice_u(r, tk, 2), N) & m;
                // beyond the run the index is some voxel of this block, and not read
                if (kh + (float)i < kx &&
                    __ldg(reinterpret_cast<const uint8_t*>(blk + ((v2 << s.lgB) + v1 << s.lgB) + v0)) != 0)
                    set |= 1u << i;
            }
            while (set) {
                const int i = __ffs(set) - 1;
                set &= set - 1;
                const float tk = __fadd_rn(r.t0, kh + (float)i);
                float u[3], f[3], g[3];
                int fi[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) u[a] = lattice_u(r, tk, a);
                stencil_weights(u, f, g, fi);
                st.active++;
                uint2 cv[8];   // index = z*4 + y*2 + x
                const int l0 = fi[0] - o3[0], l1 = fi[1] - o3[1], l2 = fi[2] - o3[2];
                if ((unsigned)l0 < (unsigned)m && (unsigned)l1 < (unsigned)m && (unsigned)l2 < (unsigned)m) {
                    const uint2* p0 = blk + ((l2 << s.lgB) + l1 << s.lgB) + l0;
#pragma unroll
                    for (int c = 0; c < 8; ++c) cv[c] = __ldg(p0 + ((c >> 2) * B + ((c >> 1) & 1)) * B + (c & 1));
                } else {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        cv[c] = raw_voxel(s, atlas, nb, fi[0] + (c & 1), fi[1] + ((c >> 1) & 1), fi[2] + (c >> 2));
                }
                bool saturated;
                const float wk = composite(s, cv, f, g, st.T, st.tau, saturated);
                accumulate_colour(st, cv, wk, f, g);
                if (saturated) return;
            }
        }
        kh = kx;
    }
}

// LGB: see BlockScene (density codes only); MINB and lanes as for render_rays_kernel
template <int LGB, int MINB>
__global__ void __launch_bounds__(128, MINB) render_rays_noalloc_kernel(const BlockScene<LGB, 0> s, const uint2* __restrict__ atlas,
                                                                        int64_t nb,
                                                                        const __grid_constant__ CamTable cams,
                                                                        int32_t n_cams, const int32_t* __restrict__ pix,
                                                                        int64_t n, const float* __restrict__ mlp,
                                                                        float* __restrict__ rgb, int lanes) {
    __shared__ __align__(16) float sW[kNParam + 1];
    load_mlp_smem_t(sW, mlp);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * 4 + (threadIdx.x >> 5)) * lanes + lane;
    if (lane >= lanes || i >= n) return;
    const int ci = __ldg(pix + 3 * i), px = __ldg(pix + 3 * i + 1), py = __ldg(pix + 3 * i + 2);
    Ray r;
    if (ci >= 0 && ci < n_cams && px >= 0 && py >= 0 && px < cams.c[ci].W && py < cams.c[ci].H) {
        r = make_ray(s, cams.c[ci], px, py);
    } else {
        r.hit = false;
        r.d[0] = r.d[1] = r.d[2] = 0.0f;
        atomicCAS(s.status, 0, (int)SNERG_E_INVAL);
    }
    MarchState st;
    march_raw(s, atlas, nb, r, st);
    record_status(s, st);
    float c[3], aux[kAuxCh];
    finish_ray(s, sW, r, st, c, aux);
    rgb[i * 3 + 0] = c[0];
    rgb[i * 3 + 1] = c[1];
    rgb[i * 3 + 2] = c[2];
}

std::mutex g_setup_mu;
void* g_scratch_dev[kNoAllocMaxDevices] = {};

// Every kernel that a call can launch, loaded on the current device: the runtime loads a kernel's
// code (device memory, and host time in the middle of a frame) at its first use otherwise, and
// which of the builds runs goes by the block edge and the number of rays.
cudaError_t load_kernels() {
    const void* const kernels[] = {
        (const void*)noalloc_map_xy_kernel,            (const void*)noalloc_map_z_kernel,
        (const void*)render_rays_noalloc_kernel<0, 4>, (const void*)render_rays_noalloc_kernel<0, 8>,
        (const void*)render_rays_noalloc_kernel<3, 4>, (const void*)render_rays_noalloc_kernel<3, 8>,
        (const void*)render_rays_noalloc_kernel<4, 4>, (const void*)render_rays_noalloc_kernel<4, 8>,
        (const void*)render_rays_noalloc_kernel<5, 4>, (const void*)render_rays_noalloc_kernel<5, 8>,
        (const void*)render_rays_noalloc_kernel<6, 4>, (const void*)render_rays_noalloc_kernel<6, 8>};
    for (const void* k : kernels) {
        cudaFuncAttributes a;
        const cudaError_t e = cudaFuncGetAttributes(&a, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// the current device's set-up, once per device: the kernels and the device address of
// g_noalloc_scratch
cudaError_t scratch_address(void** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_setup_mu);
    if (!g_scratch_dev[dev]) {
        void* p = nullptr;
        e = load_kernels();
        if (e == cudaSuccess) e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_dev[dev] = p;
    }
    *out = g_scratch_dev[dev];
    return cudaSuccess;
}

bool desc_ok_noalloc(const snerg_scene_desc* d) {
    if (!d || d->N < 1 || d->N > 16384 || d->B < 2 || d->B > 64 || (d->B & (d->B - 1)) || d->N % d->B) return false;
    if (d->max_steps < 0 || (d->flags & ~SNERG_FLAG_UNPREMULTIPLY)) return false;   // deferred model only
    if (!(d->extent > 0.0f) || !(d->extent < INFINITY) || !(d->sigma_max >= 0.0f) || !(d->sigma_max < INFINITY))
        return false;
    for (int i = 0; i < 3; ++i)
        if (!(d->bmin[i] > -INFINITY && d->bmin[i] < INFINITY && d->bg[i] > -INFINITY && d->bg[i] < INFINITY))
            return false;
    return true;
}

}  // namespace
}  // namespace snerg

using namespace snerg;

extern "C" snerg_status snerg_render_rays_noalloc(const snerg_scene_desc* desc, const int32_t* d_indirection,
                                                  const uint8_t* d_atlas, int64_t num_blocks,
                                                  const snerg_camera* cams, int32_t n_cams, const int32_t* d_pix,
                                                  int64_t n, const float* d_mlp, float* d_rgb, int32_t* d_status,
                                                  void* stream) {
    if (!desc_ok_noalloc(desc) || num_blocks < 0 || n < 0) return SNERG_E_INVAL;
    const int N = desc->N, B = desc->B, G = N / B;
    if (G > kNoAllocMaxG) return SNERG_E_UNSUPPORTED;
    if (!cams || n_cams < 1 || n_cams > kMaxCams) return SNERG_E_INVAL;
    if (!d_indirection || (num_blocks > 0 && (!d_atlas || ((uintptr_t)d_atlas & 7u)))) return SNERG_E_INVAL;
    CamTable table;                      // on the stack: this entry point allocates nothing
    std::memset(&table, 0, sizeof(table));
    for (int i = 0; i < n_cams; ++i) {
        const snerg_camera& c = cams[i];
        for (int k = 0; k < 12; ++k)
            if (!(c.c2w[k] > -INFINITY && c.c2w[k] < INFINITY)) return SNERG_E_INVAL;
        if (!(c.fx > -INFINITY && c.fx < INFINITY && c.fy > -INFINITY && c.fy < INFINITY) || c.fx == 0.0f ||
            c.fy == 0.0f || !(c.cx > -INFINITY && c.cx < INFINITY && c.cy > -INFINITY && c.cy < INFINITY) ||
            c.W < 0 || c.H < 0)
            return SNERG_E_INVAL;
        table.c[i] = c;
    }
    if (n > 0 && (!d_pix || !d_mlp || !d_rgb)) return SNERG_E_INVAL;
    cudaStream_t st = (cudaStream_t)stream;
    void* base = nullptr;
    if (scratch_address(&base) != cudaSuccess) return SNERG_E_CUDA;
    uint8_t* scratch = (uint8_t*)base;
    int32_t* status = (int32_t*)scratch;
    uint8_t* bdist = scratch + kNoAllocHeader;
    const size_t G3 = (size_t)G * G * G;
    // the status word is set to zero and the distance map rewritten in full
    uint8_t* xy = bdist + kNoAllocG3;
    noalloc_map_xy_kernel<<<(unsigned)G, 1024, 0, st>>>(d_indirection, G, status, xy);
    noalloc_map_z_kernel<<<(unsigned)((G3 + 255) / 256), 256, 0, st>>>(xy, G, bdist);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && n > 0) {
        DevScene s;
        std::memset(&s, 0, sizeof(s));
        s.ind = d_indirection;
        s.bdist = bdist;
        s.status = status;
        s.N = N;
        s.B = B;
        int lg = 0;
        while ((1 << lg) < B) ++lg;
        s.lgB = lg;
        s.G = G;
        s.P = B + 2;
        s.P3 = s.P * s.P * s.P;
        s.fN = (float)N;
        s.scale = (float)N / desc->extent;
        for (int i = 0; i < 3; ++i) {
            s.bmin[i] = desc->bmin[i];
            s.bg[i] = desc->bg[i];
        }
        s.kappa = (float)((double)desc->sigma_max * ((double)desc->extent / (double)N) / 255.0);
        s.taumax = (float)std::log(1000.0);
        s.tmin = (float)1e-3;
        s.inv255 = (float)(1.0 / 255.0);
        s.flags = desc->flags;
        s.kmax = desc->max_steps > 0 ? (desc->max_steps < 4 * N + 16 ? desc->max_steps : 4 * N + 16) : 4 * N + 16;
        int dev = 0, sms = 1;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        s.sms = sms;
        // one wave of 4 CTAs per SM: 10,000 rays of a 1024^3 grid 118 us with 32 rays per warp, 79 with 4;
        // 38,000 with 32 / 16 (16 warps per SM) 191 / 157, but of a 128^3 grid 84 / 89
        const int lanes = lanes_per_warp(n, sms, {by_side(s, 12, 12, 16), 16, 16, 16, 16});
        const int64_t ctas = (n + 4 * lanes - 1) / (4 * lanes);
        with_block_build(s, [&](auto build) {
            constexpr int L = decltype(build)::lgB;
            auto* kernel = ctas <= 4 * (int64_t)sms ? render_rays_noalloc_kernel<L, 4> : render_rays_noalloc_kernel<L, 8>;
            kernel<<<(unsigned)ctas, 128, 0, st>>>(BlockScene<L, 0>(s), reinterpret_cast<const uint2*>(d_atlas), num_blocks,
                                                   table, n_cams, d_pix, n, d_mlp, d_rgb, lanes);
        });
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && d_status) e = cudaMemcpyAsync(d_status, status, sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? SNERG_OK : SNERG_E_CUDA;
}
