// snerg_bake.cu -- baking an analytic radiance field into the sparse grid on the GPU
// (Sec. 5.3-5.4): alpha at voxel centres, macroblock culling at tau_alpha, packing of the
// kept blocks in raster order, and the anti-aliased content of each kept voxel (the field
// averaged over 16 Gaussian-jittered positions) stored as 8-bit codes.
//
// Three launches and one read-back:
//   alpha pass   persistent CTAs walk the macroblocks; each evaluates its block's voxel
//                centres some at a time and stops at the first lot holding alpha >= tau_alpha;
//   scan         numbers the flagged blocks (exclusive scan in raster order, one CTA per
//                4,096 of them) into the indirection grid and a slot -> block list;
//   fill pass    persistent CTAs walk the kept blocks' voxels and write 8 codes per voxel.
// Blocks of 8^3 and more have kernels that take one exponential per blob and axis, smaller
// blocks one per blob and voxel: their boxes have too few voxels to share the factors.
// Each unit of work (a block in the alpha pass, an item of it in the fill pass) first keeps
// only the density blobs that can matter over its box (jitter included): blob i is dropped
// where peak_i exp(-|x - c_i|^2 / (2 s_i^2)) < eps over the whole box, with
// eps = 2^-30 min(sigma_max, sigma_tau) and sigma_tau = -ln(1 - tau_alpha) / v the density
// at which alpha reaches tau_alpha. The dropped terms change sigma by less than
// 64 eps = 6e-8 of both the code step and the culling density.
// The colour channels use angle addition: the mean over the 16 samples of
// sin(a + b_s) with a = w . x_centre + phi and b_s = w . j_s v equals
// sin a * mean(cos b_s) + cos a * mean(sin b_s), and the two means depend only on the
// channel, so one sincos per voxel and channel replaces 16 sines.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#include "snerg.h"

namespace bake_gpu {

constexpr int kMaxBlobs = SNERG_BAKE_MAX_BLOBS;
constexpr int kThreads = 64;           // of the kernels for blocks below 8^3 (gather_blobs takes 64)
constexpr int kScanThreads = 1024;
constexpr int kMaxG = 256;
constexpr size_t kAlign = 256;

struct BakeParams {
    int32_t N, B, lgB, G;
    int32_t n_blob;
    int32_t alpha_codes;        // channel 0 = 1 - exp(-sigma v) instead of sigma / sigma_max
    float v, tau, inv_sigma_max;
    float sigma_reject;         // a block whose density is below this everywhere is not kept
    float bmin[3];
    float jit_lo[3], jit_hi[3]; // per-axis extremes of the jitter offsets (voxel units)
    float blob[kMaxBlobs][5];   // centre xyz, k = log2(e) / (2 s^2), peak
    float cull[kMaxBlobs];      // ln(peak / eps) / ln 2: the blob is dropped beyond this k |x - c|^2
    float color[7][4];          // w xyz, phi
    float cbar[7], sbar[7];     // mean over the samples of cos / sin (w_c . j_s v)
    float jv[16][3];            // jitter offsets times v (world units)
    float jq[16];               // |jv_s|^2
};

struct ItemBox {
    int32_t lo[3], hi[3];       // inclusive global voxel ranges of the item
};

// the voxels of block b
__device__ __forceinline__ ItemBox block_box(const BakeParams& P, int64_t b) {
    const int c[3] = {(int)(b % P.G), (int)((b / P.G) % P.G), (int)(b / ((int64_t)P.G * P.G))};
    ItemBox r;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        r.lo[a] = c[a] * P.B;
        r.hi[a] = r.lo[a] + P.B - 1;
    }
    return r;
}

// Threads 0..63 test one blob each against the item's box (voxel centres moved by the
// jitter extremes when `jittered`) and compact the blobs that may contribute into shared
// memory, in blob order. Returns their number after a barrier.
__device__ __forceinline__ int gather_blobs(const BakeParams& P, const ItemBox& box, bool jittered, float4* s_blob,
                                            float* s_peak, int* s_cnt) {
    const int t = threadIdx.x;
    bool rel = false;
    if (t < P.n_blob) {
        float a = 0.0f;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const float lo = P.bmin[ax] + ((float)box.lo[ax] + 0.5f + (jittered ? P.jit_lo[ax] : 0.0f)) * P.v;
            const float hi = P.bmin[ax] + ((float)box.hi[ax] + 0.5f + (jittered ? P.jit_hi[ax] : 0.0f)) * P.v;
            const float c = P.blob[t][ax];
            const float d = fmaxf(fmaxf(lo - c, c - hi), 0.0f);
            a = fmaf(d, d, a);
        }
        rel = a * P.blob[t][3] <= P.cull[t];
    }
    int pos = 0;
    if (t < 64) {
        const unsigned m = __ballot_sync(0xffffffffu, rel);
        pos = __popc(m & ((1u << (t & 31)) - 1u));
        if ((t & 31) == 0) s_cnt[t >> 5] = __popc(m);
    }
    __syncthreads();
    if (rel) {
        const int o = (t >= 32 ? s_cnt[0] : 0) + pos;
        s_blob[o] = make_float4(P.blob[t][0], P.blob[t][1], P.blob[t][2], P.blob[t][3]);
        s_peak[o] = P.blob[t][4];
    }
    __syncthreads();
    return s_cnt[0] + s_cnt[1];
}

// 2^x with the PTX approximate base-2 exponential (relative error about 2^-22 over the
// exponents used here, which are >= -cull > -64).
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float density_at(const float4* s_blob, const float* s_peak, int n, float x, float y,
                                            float z) {
    float acc = 0.0f;
    for (int i = 0; i < n; ++i) {
        const float4 b = s_blob[i];
        const float dx = x - b.x, dy = y - b.y, dz = z - b.z;
        const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        acc = fmaf(s_peak[i], ex2(-d2 * b.w), acc);
    }
    return acc;
}

__device__ __forceinline__ uint32_t code8(float x) {
    const float q = floorf(fmaf(x, 255.0f, 0.5f));
    return q > 0.0f ? (q < 255.0f ? (uint32_t)q : 255u) : 0u;   // NaN -> 0
}

// flags[b] bit 0: block b is kept; the first flag of a tile of kTile blocks counts the
// tile's kept blocks in the bits above
constexpr int kTile = 4096;
__device__ __forceinline__ void keep_block(int32_t* flags, int64_t b) {
    atomicAdd(flags + b, 1);
    atomicAdd(flags + b / kTile * kTile, 2);
}

// blocks below 8^3: one exponential per blob and voxel
__global__ void __launch_bounds__(kThreads) bake_alpha_kernel(const __grid_constant__ BakeParams P,
                                                              int32_t* __restrict__ flags, int64_t G3) {
    __shared__ float4 s_blob[kMaxBlobs];
    __shared__ float s_peak[kMaxBlobs];
    __shared__ int s_cnt[2];
    const int t = threadIdx.x, m = P.B - 1;
    for (int64_t b = blockIdx.x; b < G3; b += gridDim.x) {
        const ItemBox box = block_box(P, b);
        __syncthreads();                                   // the previous block's readers are done
        const int n = gather_blobs(P, box, false, s_blob, s_peak, s_cnt);
        if (n == 0) continue;                              // uniform: alpha = 0 < tau everywhere
        bool keep = false;
        if (t < 1 << (3 * P.lgB)) {
            const float x = P.bmin[0] + ((float)(box.lo[0] + (t & m)) + 0.5f) * P.v;
            const float y = P.bmin[1] + ((float)(box.lo[1] + ((t >> P.lgB) & m)) + 0.5f) * P.v;
            const float z = P.bmin[2] + ((float)(box.lo[2] + (t >> (2 * P.lgB))) + 0.5f) * P.v;
            const float sigma = density_at(s_blob, s_peak, n, x, y, z);
            keep = -expm1f(-sigma * P.v) >= P.tau;         // alpha = 1 - exp(-sigma v)
        }
        if (__syncthreads_or(keep) && t == 0) keep_block(flags, b);
    }
}

// ---------------------------------------------------------------------------------
// Blocks of 8^3 and more: a blob's term is a product of one factor per axis,
// 2^(-k |x - c|^2) = prod_a 2^(-k (x_a - c_a)^2), so a box of voxels needs one exponential
// per blob, axis and coordinate instead of one per blob and voxel, and the sums over the
// blobs (and over the 16 samples in the fill) become multiply-adds on register tiles.
// Each factor is as accurate as the direct exponential (its argument is the smaller one);
// the product of three adds two roundings.
// ---------------------------------------------------------------------------------
template <int LGB>
struct AlphaShape {
    static constexpr int B = 1 << LGB;
    static constexpr int LX = B < 32 ? B : 32;
    static constexpr int T = LGB == 3 ? 64 : 256;            // threads
    static constexpr int LY = T / LX;                        // rows of a sweep
    static constexpr int SX = B / LX, SY = B / LY, SZ = B / 8;   // sweeps along each axis (their strides in y and z)
    static constexpr int kSmem = 3 * kMaxBlobs * B * 4;
};

// Which blocks are kept. A block whose blobs cannot reach sigma_tau together even at their
// nearest points is dropped at once; otherwise the block is swept 8 z values per thread, a
// sweep being spread over the whole block so that a kept one is recognised in the first.
// Bound by the sweeps of the blocks around the threshold: 32,768 blocks of 32^3 with 64 blobs
// 2.41 ms with one exponential per blob and voxel -> 0.125 ms.
template <int LGB>
__global__ void __launch_bounds__(AlphaShape<LGB>::T) bake_alpha_sep_kernel(const __grid_constant__ BakeParams P,
                                                                            int32_t* __restrict__ flags, int64_t G3) {
    using S = AlphaShape<LGB>;
    constexpr int B = S::B;
    extern __shared__ __align__(16) float s_tab[];           // [3][blob][B]; z in sweep order
    __shared__ float4 s_blob[kMaxBlobs];
    __shared__ float s_peak[kMaxBlobs];
    __shared__ int s_cnt[2];
    __shared__ float s_top[2];
    float* tx = s_tab;
    float* ty = s_tab + kMaxBlobs * B;
    float* tz = s_tab + 2 * kMaxBlobs * B;
    const int t = threadIdx.x;
    for (int64_t b = blockIdx.x; b < G3; b += gridDim.x) {
        const int o[3] = {(int)(b % P.G) * B, (int)((b / P.G) % P.G) * B, (int)(b / ((int64_t)P.G * P.G)) * B};
        ItemBox box;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            box.lo[a] = o[a];
            box.hi[a] = o[a] + B - 1;
        }
        __syncthreads();                                     // the previous block's readers are done
        const int n = gather_blobs(P, box, false, s_blob, s_peak, s_cnt);
        if (n == 0) continue;                                // uniform: alpha = 0 < tau everywhere
        if (t < 64) {
            float top = 0.0f;                                // the blob's largest term over the block
            if (t < n) {
                const float4 q = s_blob[t];
                const float c[3] = {q.x, q.y, q.z};
                float d2 = 0.0f;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float lo = P.bmin[a] + ((float)box.lo[a] + 0.5f) * P.v;
                    const float hi = P.bmin[a] + ((float)box.hi[a] + 0.5f) * P.v;
                    const float d = fmaxf(fmaxf(lo - c[a], c[a] - hi), 0.0f);
                    d2 = fmaf(d, d, d2);
                }
                top = s_peak[t] * ex2(-d2 * q.w);
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) top += __shfl_xor_sync(0xffffffffu, top, s);
            if ((t & 31) == 0) s_top[t >> 5] = top;
        }
        for (int i = t; i < n * B; i += S::T) {
            const float4 q = s_blob[i / B];
            const int l = i % B;
            const float dx = P.bmin[0] + ((float)(o[0] + l) + 0.5f) * P.v - q.x;
            const float dy = P.bmin[1] + ((float)(o[1] + l) + 0.5f) * P.v - q.y;
            const float dz = P.bmin[2] + ((float)(o[2] + l) + 0.5f) * P.v - q.z;
            tx[i] = ex2(-q.w * dx * dx);
            ty[i] = ex2(-q.w * dy * dy);
            tz[i / B * B + (l % S::SZ) * 8 + l / S::SZ] = s_peak[i / B] * ex2(-q.w * dz * dz);
        }
        __syncthreads();
        if (s_top[0] + s_top[1] < P.sigma_reject) continue;  // uniform
        for (int sw = 0; sw < S::SX * S::SY * S::SZ; ++sw) {
            const int x = (sw % S::SX) * S::LX + t % S::LX;
            const int y = t / S::LX * S::SY + (sw / S::SX) % S::SY;
            const float* z8 = tz + sw / (S::SX * S::SY) * 8;
            float2 acc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] = make_float2(0.0f, 0.0f);
            for (int i = 0; i < n; ++i) {
                const float w = tx[i * B + x] * ty[i * B + y];
                const float2 ww = make_float2(w, w);
                const float4 a = *reinterpret_cast<const float4*>(z8 + i * B);
                const float4 c = *reinterpret_cast<const float4*>(z8 + i * B + 4);
                acc[0] = __ffma2_rn(ww, make_float2(a.x, a.y), acc[0]);
                acc[1] = __ffma2_rn(ww, make_float2(a.z, a.w), acc[1]);
                acc[2] = __ffma2_rn(ww, make_float2(c.x, c.y), acc[2]);
                acc[3] = __ffma2_rn(ww, make_float2(c.z, c.w), acc[3]);
            }
            float top = 0.0f;
#pragma unroll
            for (int j = 0; j < 4; ++j) top = fmaxf(top, fmaxf(acc[j].x, acc[j].y));
            if (__syncthreads_or(-expm1f(-top * P.v) >= P.tau)) {          // alpha = 1 - exp(-sigma v)
                if (t == 0) keep_block(flags, b);
                break;                                       // uniform
            }
        }
    }
}

// Slots of the kept blocks in raster order: ind[b] = slot or -1, list[slot] = b, *count =
// number of kept blocks. CTA i numbers the flags of tile i after summing the counts of the
// tiles before it (in the tiles' first flags). 32,768 blocks: 57 us as one CTA's scan over
// contiguous chunks -> 4 us; a grid of 256^3 blocks has 4,096 tiles.
__global__ void __launch_bounds__(kScanThreads) bake_scan_kernel(const int32_t* __restrict__ flags, int64_t G3,
                                                                 int32_t* __restrict__ ind,
                                                                 int32_t* __restrict__ list,
                                                                 int64_t* __restrict__ count) {
    __shared__ int s_warp[kScanThreads / 32];
    __shared__ int s_before;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t == 0) s_before = 0;
    __syncthreads();
    int before = 0;
    for (int64_t i = t; i < blockIdx.x; i += kScanThreads) before += flags[i * kTile] >> 1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (lane == 0 && before) atomicAdd(&s_before, before);
    // thread t: flags 4 t .. 4 t + 3 of the tile
    constexpr int kPer = kTile / kScanThreads;
    const int64_t first = (int64_t)blockIdx.x * kTile + (int64_t)t * kPer;
    int f[kPer], c = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        f[j] = first + j < G3 ? flags[first + j] & 1 : 0;
        c += f[j];
    }
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        int s = s_warp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        s_warp[lane] = s;                                  // inclusive over warps
    }
    __syncthreads();
    int off = s_before + incl - c + (w > 0 ? s_warp[w - 1] : 0);
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        if (first + j >= G3) break;
        ind[first + j] = f[j] ? off : -1;
        if (f[j]) list[off++] = (int32_t)(first + j);
    }
    if (blockIdx.x == gridDim.x - 1 && t == kScanThreads - 1) *count = off;
}

// blocks below 8^3: one exponential per blob, sample and voxel
__global__ void __launch_bounds__(kThreads) bake_fill_kernel(const __grid_constant__ BakeParams P,
                                                             const int32_t* __restrict__ list,
                                                             const int64_t* __restrict__ count, int64_t max_blocks,
                                                             uint2* __restrict__ atlas) {
    __shared__ float4 s_blob[kMaxBlobs];
    __shared__ float s_peak[kMaxBlobs];
    __shared__ int s_cnt[2];
    const int t = threadIdx.x, m = P.B - 1;
    const int64_t nb = min(*count, max_blocks);
    const int lg3 = 3 * P.lgB;
    for (int64_t slot = blockIdx.x; slot < nb; slot += gridDim.x) {
        const int64_t b = list[slot];
        const ItemBox box = block_box(P, b);
        __syncthreads();
        const int n = gather_blobs(P, box, true, s_blob, s_peak, s_cnt);
        if (t >= 1 << lg3) continue;
        const float fx = (float)(box.lo[0] + (t & m)) + 0.5f;
        const float fy = (float)(box.lo[1] + ((t >> P.lgB) & m)) + 0.5f;
        const float fz = (float)(box.lo[2] + (t >> (2 * P.lgB))) + 0.5f;
        const float cx = P.bmin[0] + fx * P.v, cy = P.bmin[1] + fy * P.v, cz = P.bmin[2] + fz * P.v;
        // sum over blobs of peak * sum over samples of 2^(-k |D + jv_s|^2), D = centre - c,
        // expanded as -k |D|^2 - 2k D . jv_s - k |jv_s|^2: four FMAs per blob and sample
        float sigma = 0.0f;
        for (int i = 0; i < n; ++i) {
            const float4 b = s_blob[i];
            const float dx = cx - b.x, dy = cy - b.y, dz = cz - b.z;
            const float a = -b.w * fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const float gx = -2.0f * b.w * dx, gy = -2.0f * b.w * dy, gz = -2.0f * b.w * dz;
            float part = 0.0f;
#pragma unroll
            for (int s = 0; s < 16; ++s)
                part += ex2(fmaf(gx, P.jv[s][0], fmaf(gy, P.jv[s][1], fmaf(gz, P.jv[s][2], fmaf(-b.w, P.jq[s], a)))));
            sigma = fmaf(s_peak[i], part, sigma);
        }
        uint32_t q[8];
        q[0] = P.alpha_codes ? code8(-expm1f(-sigma * 0.0625f * P.v)) : code8(sigma * 0.0625f * P.inv_sigma_max);
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            const float a = fmaf(P.color[c][0], cx, fmaf(P.color[c][1], cy, fmaf(P.color[c][2], cz, P.color[c][3])));
            float sa, ca;
            sincosf(a, &sa, &ca);
            q[1 + c] = code8(fmaf(0.5f, fmaf(sa, P.cbar[c], ca * P.sbar[c]), 0.5f));
        }
        atlas[(slot << lg3) + t] = make_uint2(q[0] | q[1] << 8 | q[2] << 16 | q[3] << 24,
                                              q[4] | q[5] << 8 | q[6] << 16 | q[7] << 24);
    }
}

// ---------------------------------------------------------------------------------
// The fill for blocks of 8^3 and more: an item is a box of IX x IY x IZ voxels, a thread's
// tile 8 (x) by TY (y) by TZ (z) voxels. The density is a product of matrices, sigma[x][yz] =
// sum over (blob, sample) X[.][x] (Y[.][y] Z[.][z]), with the factors of kChunk blobs at a
// time in shared memory (one exponential per blob, sample, axis and coordinate instead of one
// per blob, sample and voxel); FP32 FMAs in packed pairs, as the codes need the FP32 sums, each
// blob's 16 samples summed by themselves first (one running sum over all terms doubled the
// density codes that differ from 64 bits). The colour channels split their sine the same way: per voxel and channel two multiply-adds of a
// sine / cosine pair of x and one of (y, z) with the sample means folded in.
// Bound by issue (58 % of the slots, 12 warps of 168 registers per SM): 4,997 blocks of 32^3
// with 64 blobs 6.98 -> 1.50 ms; 4 x 4 x 2 tiles without the per-blob sums took 1.49 ms, bound
// by shared-memory returns, and 8 x 4 x 2 with every operand stored twice 1.85 ms.
// Three CTAs per SM with some spills: the whole bake takes 1.75 ms, with two and none 1.92; six
// blobs a chunk or no unrolling of the samples change it by 1 % at most. Edges of 8 and 16 take six,
// 504 bytes of spills at 16: a 512^3 grid of 16^3 blocks 476 us, with five 473, four 508, three 505;
// a 256^3 grid of 8^3 blocks 271, 262, 262, 267.
// ---------------------------------------------------------------------------------
template <int LGB>
struct FillShape {
    static constexpr int B = 1 << LGB;
    static constexpr int IX = B < 32 ? B : 32, IY = IX, IZ = B == 16 ? 16 : 8;
    static constexpr int TY = LGB == 3 ? 1 : 4, TZ = LGB == 3 ? 1 : 2;
    static constexpr int NX = IX / 8, NY = IY / TY, NZ = IZ / TZ;
    static constexpr int T = NX * NY * NZ;                   // threads: 64, 64, 128, 128
    static constexpr int PX = B / IX, PY = B / IY, PZ = B / IZ;   // items of a block along each axis
    static constexpr int kItems = PX * PY * PZ;
    static constexpr int kChunk = 3;
};

// 8-bit code of x, floor(255 x + 1/2) clamped (NaN -> 0), in the low byte: the floor is a
// directed add of 1.5 * 2^23
__device__ __forceinline__ uint32_t floor_bits(float q) {
    return (uint32_t)__float_as_int(__fadd_rd(fminf(fmaxf(q, 0.0f), 255.0f), 12582912.0f));
}
__device__ __forceinline__ uint32_t code_bits(float x) { return floor_bits(fmaf(x, 255.0f, 0.5f)); }
__device__ __forceinline__ uint32_t pack4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

// 2^(-k d^2) of the binary32 k and d, the rounding errors of the exponent carried into the
// result (three factors are multiplied where one exponential was). Where the exponential is 0
// its correction is not taken: an exponent beyond binary32 (blobs of s below 1e-19) has an
// infinite or undefined one.
__device__ __forceinline__ float gauss_factor(float k, float d) {
    const float p = k * d, e = p * d;
    const float low = fmaf(fmaf(k, d, -p), d, fmaf(p, d, -e));
    const float r = ex2(-e);
    return r > 0.0f ? fmaf(r * -0.69314718f, low, r) : r;
}

// the centre of voxel i along an axis, rounded, and what the rounding left
__device__ __forceinline__ float2 centre2(float bmin, float v, int i) {
    const float fx = (float)i + 0.5f, p = fx * v, pe = fmaf(fx, v, -p);
    const float s = bmin + p, bb = s - bmin, e = ((bmin - (s - bb)) + (p - bb)) + pe;
    const float c = s + e;
    return make_float2(c, e - (c - s));
}

template <int LGB>
__global__ void __launch_bounds__(FillShape<LGB>::T, LGB >= 5 ? 3 : 6) bake_fill_sep_kernel(
    const __grid_constant__ BakeParams P, const int32_t* __restrict__ list, const int64_t* __restrict__ count,
    int64_t max_blocks, uint2* __restrict__ atlas) {
    using S = FillShape<LGB>;
    constexpr int B = S::B, IX = S::IX, IY = S::IY, IZ = S::IZ, TY = S::TY, TZ = S::TZ;
    __shared__ float4 s_blob[kMaxBlobs];
    __shared__ float s_peak[kMaxBlobs];
    __shared__ int s_cnt[2];
    __shared__ float2 s_pos[IX + IY + IZ];                         // voxel centres along x, y, z
    __shared__ __align__(16) float s_x[S::kChunk * 16][IX];
    __shared__ __align__(16) float s_y[S::kChunk * 16][IY], s_z[S::kChunk * 16][IZ];
    __shared__ float2 s_cx[7][IX];                                 // sin, cos of w_x x
    __shared__ float2 s_cyz[7][IY * IZ];                           // their factors at (y, z)
    const int t = threadIdx.x;
    // a thread's x: xq, xq + NX, ..., so that a warp's stores of one of them fill whole sectors;
    // s_x holds them side by side
    const int xq = t % S::NX, yq = (t / S::NX) % S::NY, zq = t / (S::NX * S::NY);
    const int64_t nb = min(*count, max_blocks);
    const int64_t n_items = nb * S::kItems;
    for (int64_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const int64_t slot = it / S::kItems;
        const int part = (int)(it % S::kItems);
        const int lo[3] = {part % S::PX * IX, part / S::PX % S::PY * IY, part / (S::PX * S::PY) * IZ};   // in the block
        const int64_t b = list[slot];
        const int o[3] = {(int)(b % P.G) * B + lo[0], (int)((b / P.G) % P.G) * B + lo[1],
                          (int)(b / ((int64_t)P.G * P.G)) * B + lo[2]};
        ItemBox box;
        box.lo[0] = o[0];
        box.lo[1] = o[1];
        box.lo[2] = o[2];
        box.hi[0] = o[0] + IX - 1;
        box.hi[1] = o[1] + IY - 1;
        box.hi[2] = o[2] + IZ - 1;
        __syncthreads();                                     // the previous item's readers are done
        for (int i = t; i < IX + IY + IZ; i += S::T) {
            const int a = i < IX ? 0 : (i < IX + IY ? 1 : 2);
            s_pos[i] = centre2(P.bmin[a], P.v, o[a] + i - (a == 0 ? 0 : (a == 1 ? IX : IX + IY)));
        }
        const int n = gather_blobs(P, box, true, s_blob, s_peak, s_cnt);
        // the colours' sines: of x, and of (y, z) with the phase
        for (int i = t; i < 7 * IX; i += S::T) {
            const int c = i / IX, l = i % IX;
            float sv, cv;
            sincosf(P.color[c][0] * s_pos[l].x, &sv, &cv);
            s_cx[c][l] = make_float2(sv, cv);
        }
        for (int i = t; i < 7 * IY * IZ; i += S::T) {
            const int c = i / (IY * IZ), l = i % (IY * IZ);
            const float cy = s_pos[IX + l % IY].x, cz = s_pos[IX + IY + l / IY].x;
            float sv, cv;
            sincosf(fmaf(P.color[c][1], cy, fmaf(P.color[c][2], cz, P.color[c][3])), &sv, &cv);
            // 0.5 (sin(ax + ayz) cbar + cos(ax + ayz) sbar) = sin ax * a + cos ax * b
            s_cyz[c][l] = make_float2(0.5f * (cv * P.cbar[c] - sv * P.sbar[c]), 0.5f * (sv * P.cbar[c] + cv * P.sbar[c]));
        }
        float2 acc[TZ][TY][4];
#pragma unroll
        for (int z = 0; z < TZ; ++z)
#pragma unroll
            for (int y = 0; y < TY; ++y)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[z][y][j] = make_float2(0.0f, 0.0f);
        const int lxy = t % IX;
        const float2 cx = s_pos[lxy], cy = s_pos[IX + lxy];
        for (int i0 = 0; i0 < n; i0 += S::kChunk) {
            const int m = min(S::kChunk, n - i0) * 16;
            if (i0 > 0) __syncthreads();                     // the last chunk's factors are used up
            // a thread's coordinate along x and y is the same for all its factors (IX = IY divides T)
            for (int k = t / IX; k < m; k += S::T / IX) {
                const float4 q = s_blob[i0 + (k >> 4)];
                const int sm = k & 15;
                s_x[k][lxy % S::NX * 8 + lxy / S::NX] = gauss_factor(q.w, (cx.x - q.x) + (cx.y + P.jv[sm][0]));
                s_y[k][lxy] = gauss_factor(q.w, (cy.x - q.y) + (cy.y + P.jv[sm][1]));
            }
            for (int i = t; i < m * IZ; i += S::T) {
                const int k = i / IZ, l = i % IZ;
                const float4 q = s_blob[i0 + (k >> 4)];
                const float2 c = s_pos[IX + IY + l];
                s_z[k][l] = s_peak[i0 + (k >> 4)] * gauss_factor(q.w, (c.x - q.z) + (c.y + P.jv[k & 15][2]));
            }
            __syncthreads();
#pragma unroll 1
            for (int i = 0; i < m; i += 16) {
                float2 part[TZ][TY][4];                      // this blob's 16 samples
#pragma unroll
                for (int z = 0; z < TZ; ++z)
#pragma unroll
                    for (int y = 0; y < TY; ++y)
#pragma unroll
                        for (int j = 0; j < 4; ++j) part[z][y][j] = make_float2(0.0f, 0.0f);
#pragma unroll 2
                for (int k = i; k < i + 16; ++k) {
                    const float4 xa = *reinterpret_cast<const float4*>(&s_x[k][8 * xq]);
                    const float4 xb = *reinterpret_cast<const float4*>(&s_x[k][8 * xq + 4]);
                    float yy[TY], zz[TZ];
                    if constexpr (TY == 4) {
                        const float4 v = *reinterpret_cast<const float4*>(&s_y[k][4 * yq]);
                        const float2 u = *reinterpret_cast<const float2*>(&s_z[k][2 * zq]);
                        yy[0] = v.x;
                        yy[1] = v.y;
                        yy[2] = v.z;
                        yy[3] = v.w;
                        zz[0] = u.x;
                        zz[1] = u.y;
                    } else {
                        yy[0] = s_y[k][yq];
                        zz[0] = s_z[k][zq];
                    }
#pragma unroll
                    for (int z = 0; z < TZ; ++z)
#pragma unroll
                        for (int y = 0; y < TY; ++y) {
                            const float w1 = yy[y] * zz[z];
                            const float2 w = make_float2(w1, w1);
                            float2* a = part[z][y];
                            a[0] = __ffma2_rn(w, make_float2(xa.x, xa.y), a[0]);
                            a[1] = __ffma2_rn(w, make_float2(xa.z, xa.w), a[1]);
                            a[2] = __ffma2_rn(w, make_float2(xb.x, xb.y), a[2]);
                            a[3] = __ffma2_rn(w, make_float2(xb.z, xb.w), a[3]);
                        }
                }
#pragma unroll
                for (int z = 0; z < TZ; ++z)
#pragma unroll
                    for (int y = 0; y < TY; ++y)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[z][y][j] = __fadd2_rn(acc[z][y][j], part[z][y][j]);
            }
        }
        if (n == 0) __syncthreads();                         // the colour tables
        uint2* dst = atlas + slot * ((int64_t)B * B * B) + ((lo[2] + TZ * zq) * B + lo[1] + TY * yq) * B + lo[0];
        const float2 half = make_float2(0.5f, 0.5f), full = make_float2(255.0f, 255.0f);
        // two x at a time: their sines and cosines stay in registers over the tile's rows; a
        // rolled loop (its accumulators move down) keeps the kernel in the instruction cache
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
            const int xl = xq + S::NX * 2 * j, xh = xl + S::NX;
            float2 sn[7], cs[7];
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                const float2 l = s_cx[c][xl], h = s_cx[c][xh];
                sn[c] = make_float2(l.x, h.x);
                cs[c] = make_float2(l.y, h.y);
            }
#pragma unroll
            for (int z = 0; z < TZ; ++z)
#pragma unroll
                for (int y = 0; y < TY; ++y) {
                    const float2* f = &s_cyz[0][(TZ * zq + z) * IY + TY * yq + y];
                    const float2 s = make_float2(acc[z][y][0].x * 0.0625f, acc[z][y][0].y * 0.0625f);
                    uint32_t ql[8], qh[8];
                    if (P.alpha_codes) {
                        ql[0] = code_bits(-expm1f(-s.x * P.v));
                        qh[0] = code_bits(-expm1f(-s.y * P.v));
                    } else {
                        ql[0] = code_bits(s.x * P.inv_sigma_max);
                        qh[0] = code_bits(s.y * P.inv_sigma_max);
                    }
#pragma unroll
                    for (int c = 0; c < 7; ++c) {
                        const float2 ab = f[c * (IY * IZ)];
                        const float2 v = __ffma2_rn(sn[c], make_float2(ab.x, ab.x),
                                                    __ffma2_rn(cs[c], make_float2(ab.y, ab.y), half));
                        const float2 q = __ffma2_rn(v, full, half);
                        // at most 255.5 and a rounding: no upper clamp (the sample means' norm is at most 1)
                        ql[1 + c] = (uint32_t)__float_as_int(__fadd_rd(fmaxf(q.x, 0.0f), 12582912.0f));
                        qh[1 + c] = (uint32_t)__float_as_int(__fadd_rd(fmaxf(q.y, 0.0f), 12582912.0f));
                    }
                    uint2* d = dst + (z * B + y) * B;
                    d[xl] = make_uint2(pack4(ql[0], ql[1], ql[2], ql[3]), pack4(ql[4], ql[5], ql[6], ql[7]));
                    d[xh] = make_uint2(pack4(qh[0], qh[1], qh[2], qh[3]), pack4(qh[4], qh[5], qh[6], qh[7]));
#pragma unroll
                    for (int i = 0; i < 3; ++i) acc[z][y][i] = acc[z][y][i + 1];
                }
        }
    }
}

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

int ilog2_exact(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return (1 << l) == v ? l : -1;
}

bool desc_ok(const snerg_scene_desc* d) {
    if (!d) return false;
    if (d->N < 1 || d->N > 16384) return false;
    if (d->B < 2 || d->B > 64 || ilog2_exact(d->B) < 0 || d->N % d->B != 0) return false;
    if (d->N / d->B > kMaxG) return false;
    if (!(std::isfinite(d->extent) && d->extent > 0.0f)) return false;
    if (!(std::isfinite(d->sigma_max) && d->sigma_max > 0.0f)) return false;
    return std::isfinite(d->bmin[0]) && std::isfinite(d->bmin[1]) && std::isfinite(d->bmin[2]);
}

bool field_ok(const snerg_bake_field* f) {
    if (!f || f->n_blob < 0 || f->n_blob > kMaxBlobs) return false;
    if (!(f->tau_alpha > 0.0f && f->tau_alpha < 1.0f)) return false;
    for (int i = 0; i < f->n_blob; ++i) {
        for (int k = 0; k < 5; ++k)
            if (!std::isfinite(f->blob[i][k])) return false;
        if (!(f->blob[i][3] > 0.0f) || !(f->blob[i][4] >= 0.0f)) return false;
    }
    for (int c = 0; c < 7; ++c)
        for (int k = 0; k < 4; ++k)
            if (!std::isfinite(f->color[c][k])) return false;
    for (int s = 0; s < 16; ++s)
        for (int k = 0; k < 3; ++k)
            if (!(std::fabs(f->jitter[s][k]) <= 8.0f)) return false;
    return true;
}

struct WsLayout {
    size_t count, flags, list, total;
};

WsLayout ws_layout(int64_t G3) {
    WsLayout L;
    L.count = 0;
    L.flags = kAlign;
    L.list = align_up(L.flags + (size_t)G3 * 4);
    L.total = align_up(L.list + (size_t)G3 * 4);
    return L;
}

int grid_for(const void* fn, int threads, size_t smem, int64_t items) {
    int dev = 0, sms = 1, per = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem);
    const int64_t g = (int64_t)sms * (per > 0 ? per : 1);
    return (int)(items < g ? (items > 0 ? items : 1) : g);
}

template <int LGB>
cudaError_t alpha_sep(const BakeParams& P, int32_t* flags, int64_t G3, cudaStream_t st) {
    using S = AlphaShape<LGB>;
    auto* fn = bake_alpha_sep_kernel<LGB>;
    if (S::kSmem > 40 * 1024) {        // with the static arrays beyond the default 48 KB
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmem);
        if (e != cudaSuccess) return e;
    }
    fn<<<grid_for((const void*)fn, S::T, S::kSmem, G3), S::T, S::kSmem, st>>>(P, flags, G3);
    return cudaGetLastError();
}

cudaError_t launch_alpha(const BakeParams& P, int32_t* flags, int64_t G3, cudaStream_t st) {
    switch (P.lgB) {
        case 3: return alpha_sep<3>(P, flags, G3, st);
        case 4: return alpha_sep<4>(P, flags, G3, st);
        case 5: return alpha_sep<5>(P, flags, G3, st);
        case 6: return alpha_sep<6>(P, flags, G3, st);
    }
    bake_alpha_kernel<<<grid_for((const void*)bake_alpha_kernel, kThreads, 0, G3), kThreads, 0, st>>>(P, flags, G3);
    return cudaGetLastError();
}

template <int LGB>
cudaError_t fill_sep(const BakeParams& P, const int32_t* list, const int64_t* d_count, int64_t count,
                     int64_t max_blocks, uint2* atlas, cudaStream_t st) {
    using S = FillShape<LGB>;
    auto* fn = bake_fill_sep_kernel<LGB>;
    fn<<<grid_for((const void*)fn, S::T, 0, count * S::kItems), S::T, 0, st>>>(P, list, d_count, max_blocks, atlas);
    return cudaGetLastError();
}

cudaError_t launch_fill(const BakeParams& P, const int32_t* list, const int64_t* d_count, int64_t count,
                        int64_t max_blocks, uint2* atlas, cudaStream_t st) {
    switch (P.lgB) {
        case 3: return fill_sep<3>(P, list, d_count, count, max_blocks, atlas, st);
        case 4: return fill_sep<4>(P, list, d_count, count, max_blocks, atlas, st);
        case 5: return fill_sep<5>(P, list, d_count, count, max_blocks, atlas, st);
        case 6: return fill_sep<6>(P, list, d_count, count, max_blocks, atlas, st);
    }
    bake_fill_kernel<<<grid_for((const void*)bake_fill_kernel, kThreads, 0, count), kThreads, 0, st>>>(
        P, list, d_count, max_blocks, atlas);
    return cudaGetLastError();
}

}  // namespace bake_gpu

using namespace bake_gpu;

extern "C" size_t snerg_bake_workspace_bytes(const snerg_scene_desc* desc) {
    if (!desc_ok(desc)) return 0;
    const int64_t G = desc->N / desc->B;
    return ws_layout(G * G * G).total;
}

namespace bake_gpu {

BakeParams make_params(const snerg_scene_desc* desc, const snerg_bake_field* field) {
    BakeParams P;
    std::memset(&P, 0, sizeof(P));
    P.N = desc->N;
    P.B = desc->B;
    P.lgB = ilog2_exact(desc->B);
    P.G = desc->N / desc->B;
    P.n_blob = field->n_blob;
    P.alpha_codes = (desc->flags & SNERG_FLAG_ALPHA_ATLAS) ? 1 : 0;
    const double v = (double)desc->extent / (double)desc->N;
    P.v = (float)v;
    P.tau = field->tau_alpha;
    P.inv_sigma_max = (float)(1.0 / (double)desc->sigma_max);
    for (int k = 0; k < 3; ++k) {
        P.bmin[k] = desc->bmin[k];
        float lo = field->jitter[0][k], hi = lo;
        for (int s = 1; s < 16; ++s) {
            lo = std::fmin(lo, field->jitter[s][k]);
            hi = std::fmax(hi, field->jitter[s][k]);
        }
        P.jit_lo[k] = lo;
        P.jit_hi[k] = hi;
    }
    const double sigma_tau = -std::log1p(-(double)field->tau_alpha) / v;
    P.sigma_reject = (float)(sigma_tau * (1.0 - 1e-3));      // well beyond the rounding of the sum of terms
    const double eps = std::ldexp(std::fmin((double)desc->sigma_max, sigma_tau), -30);
    for (int i = 0; i < field->n_blob; ++i) {
        for (int k = 0; k < 3; ++k) P.blob[i][k] = field->blob[i][k];
        const double s = field->blob[i][3], peak = field->blob[i][4];
        P.blob[i][3] = (float)(1.0 / (2.0 * s * s * std::log(2.0)));
        P.blob[i][4] = (float)peak;
        P.cull[i] = peak > eps ? (float)(std::log(peak / eps) / std::log(2.0)) : -1.0f;
    }
    std::memcpy(P.color, field->color, sizeof(P.color));
    for (int j = 0; j < 16; ++j) {
        double q = 0.0;
        for (int k = 0; k < 3; ++k) {
            const double o = (double)field->jitter[j][k] * v;
            P.jv[j][k] = (float)o;
            q += o * o;
        }
        P.jq[j] = (float)q;
    }
    for (int c = 0; c < 7; ++c) {
        double cs = 0.0, sn = 0.0;
        for (int s = 0; s < 16; ++s) {
            const double b = ((double)field->color[c][0] * field->jitter[s][0] +
                              (double)field->color[c][1] * field->jitter[s][1] +
                              (double)field->color[c][2] * field->jitter[s][2]) * v;
            cs += std::cos(b);
            sn += std::sin(b);
        }
        P.cbar[c] = (float)(cs / 16.0);
        P.sbar[c] = (float)(sn / 16.0);
    }
    return P;
}

}  // namespace bake_gpu

extern "C" snerg_status snerg_bake(const snerg_scene_desc* desc, const snerg_bake_field* field,
                                   int32_t* d_indirection, uint8_t* d_atlas, int64_t max_blocks, void* d_workspace,
                                   size_t ws_bytes, int64_t* num_blocks, void* stream) {
    if (!desc_ok(desc) || !field_ok(field) || !d_indirection || !num_blocks || max_blocks < 0) return SNERG_E_INVAL;
    if (max_blocks > 0 && (!d_atlas || ((uintptr_t)d_atlas & 7u))) return SNERG_E_INVAL;
    if (!d_workspace || ((uintptr_t)d_workspace & (kAlign - 1))) return SNERG_E_INVAL;
    const int64_t G = desc->N / desc->B, G3 = G * G * G;
    const WsLayout L = ws_layout(G3);
    if (ws_bytes < L.total) return SNERG_E_NOMEM;
    *num_blocks = 0;

    const BakeParams P = make_params(desc, field);
    cudaStream_t st = (cudaStream_t)stream;
    uint8_t* ws = (uint8_t*)d_workspace;
    int64_t* d_count = (int64_t*)(ws + L.count);
    int32_t* d_flags = (int32_t*)(ws + L.flags);
    int32_t* d_list = (int32_t*)(ws + L.list);
    cudaError_t e = cudaMemsetAsync(d_flags, 0, (size_t)G3 * 4, st);
    if (e == cudaSuccess) {
        e = launch_alpha(P, d_flags, G3, st);
    }
    if (e == cudaSuccess) {
        bake_scan_kernel<<<(unsigned)((G3 + kTile - 1) / kTile), kScanThreads, 0, st>>>(d_flags, G3, d_indirection, d_list,
                                                                                      d_count);
        e = cudaGetLastError();
    }
    int64_t count = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&count, d_count, sizeof(count), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return SNERG_E_CUDA;
    *num_blocks = count;
    if (count > max_blocks) return SNERG_E_NOMEM;
    if (count > 0) {
        e = launch_fill(P, d_list, d_count, count, max_blocks, (uint2*)d_atlas, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return SNERG_E_CUDA;
    }
    return SNERG_OK;
}

extern "C" snerg_status snerg_bake_atlas(const snerg_scene_desc* desc, const snerg_bake_field* field, uint8_t* d_atlas,
                                         int64_t num_blocks, const void* d_workspace, size_t ws_bytes, void* stream) {
    if (!desc_ok(desc) || !field_ok(field) || num_blocks < 0) return SNERG_E_INVAL;
    if (num_blocks > 0 && (!d_atlas || ((uintptr_t)d_atlas & 7u))) return SNERG_E_INVAL;
    if (!d_workspace || ((uintptr_t)d_workspace & (kAlign - 1))) return SNERG_E_INVAL;
    const int64_t G = desc->N / desc->B;
    const WsLayout L = ws_layout(G * G * G);
    if (ws_bytes < L.total) return SNERG_E_NOMEM;
    if (num_blocks == 0) return SNERG_OK;
    if (num_blocks > G * G * G) return SNERG_E_INVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const uint8_t* ws = (const uint8_t*)d_workspace;
    cudaError_t e = launch_fill(make_params(desc, field), (const int32_t*)(ws + L.list), (const int64_t*)(ws + L.count),
                                num_blocks, num_blocks, (uint2*)d_atlas, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? SNERG_OK : SNERG_E_CUDA;
}
