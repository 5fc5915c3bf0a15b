// snerg_prep.cu -- scene set-up kernels: validate the indirection grid (Sec. 5.1),
// build the device layout of the atlas (apron-padded blocks) and the two Chebyshev
// distance maps the march uses to skip empty space; requantise fine-tuned values.
//
// The paper's viewer keeps density in its own 8-bit texture so that empty space inside
// occupied blocks costs one byte per sample (App. A); the voxel distance plane here
// plays that role and, being a distance rather than a code, also says how many of the
// following samples are certainly empty. The 1-voxel apron makes every trilinear
// stencil of a sample a fetch from one block: atlas neighbours are not spatial neighbours (Sec. 5.1), so without it a sample
// near a block face would need up to 8 indirection lookups.
#include <type_traits>

#include "snerg_internal.cuh"

namespace snerg {

// err bit 1: entry outside [-1, nb); bit 2: a slot referenced twice.
__global__ void validate_kernel(const int32_t* __restrict__ ind, int64_t n_ind, int64_t nb,
                                int32_t* __restrict__ blk_of_slot, int32_t* __restrict__ err) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_ind; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = ind[i];
        if (v < -1 || (int64_t)v >= nb) {
            atomicOr(err, 1);
        } else if (v >= 0) {
            if (atomicCAS(blk_of_slot + v, -1, (int32_t)i) != -1) atomicOr(err, 2);
        }
    }
}

// Requantisation of fine-tuned colour/feature values into the padded atlas (Sec. 5.4
// codes): every stored voxel takes channels 1..7 from floor(255 x + 1/2) of its values
// (binary32, clamped) and keeps its density byte, so the empty-space maps built from the
// densities stay valid; atlas_out (nullable) receives the codes in the unpadded layout.
//
// By itself: one thread per padded entry, whose source it gathers, so that every store is
// part of a row. Bound by memory: 70 M voxels 0.87 ms, whether codes change or not; by voxels,
// as in the optimiser's pass below, 0.86 ms if none does and 1.42 if all do (the apron copies
// are scattered 4-byte stores).
__device__ __forceinline__ uint32_t quant8(float x) {
    const float q = floorf(__fmaf_rn(x, 255.0f, 0.5f));
    return q > 0.0f ? (q < 255.0f ? (uint32_t)q : 255u) : 0u;   // NaN -> 0
}

__global__ void requantize_padded_kernel(const int32_t* __restrict__ ind, const int32_t* __restrict__ blk_of_slot,
                                         const float4* __restrict__ values, int64_t nb, int N, int B, int lgB,
                                         uint2* __restrict__ patlas, uint2* __restrict__ atlas_out) {
    const int P = B + 2, P3 = P * P * P, G = N >> lgB;
    const int64_t total = nb * (int64_t)P3, B3 = (int64_t)B * B * B;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t slot = t / P3;
        const int r = (int)(t - slot * P3);
        const int px = r % P, py = (r / P) % P, pz = r / (P * P);
        const int blk = blk_of_slot[slot];
        if (blk < 0) continue;                                 // an unreferenced slot has no codes to keep
        const int bx = blk % G, by = (blk / G) % G, bz = blk / (G * G);
        const int gx = min(max(bx * B + px - 1, 0), N - 1);
        const int gy = min(max(by * B + py - 1, 0), N - 1);
        const int gz = min(max(bz * B + pz - 1, 0), N - 1);
        const int owner = ind[((gz >> lgB) * G + (gy >> lgB)) * G + (gx >> lgB)];
        if (owner < 0) continue;                               // apron of an empty block: stays 0
        const int loc = ((gz & (B - 1)) * B + (gy & (B - 1))) * B + (gx & (B - 1));
        const int64_t src = (int64_t)owner * B3 + loc;
        const float4 a = values[2 * src], b = values[2 * src + 1];
        const uint2 old = patlas[t];
        uint2 v;
        v.x = (old.x & 0xffu) | quant8(a.y) << 8 | quant8(a.z) << 16 | quant8(a.w) << 24;
        v.y = quant8(b.x) | quant8(b.y) << 8 | quant8(b.z) << 16 | quant8(b.w) << 24;
        patlas[t] = v;
        if (atlas_out && px >= 1 && px <= B && py >= 1 && py <= B && pz >= 1 && pz <= B) atlas_out[src] = v;
    }
}

// The end of a fine-tuning step: one optimiser step on the values and their codes, so that
// the values are read once.
//
// One thread per 4 channels (16-byte loads of consecutive lanes, 4-byte code words). A voxel's
// copies in the aprons are found from the voxel: along each axis it is also in the apron of
// the block before (if it is the first of its block) or after (the last), or beside itself at
// the grid's border, so at most 2 x 2 x 2 entries. A code word that does not change is not
// stored (its copies hold the same word).
// Bound by memory: a step on 125 M values, most of them untouched, reads 16 bytes of each (and
// the codes) at 5.7 TB/s, 0.41 ms; an Adam pass over all of them and a requantisation by
// themselves took 0.74 + 0.19 ms. With every value's gradient set and every code changing,
// 561 M values take 2.50 ms and the two calls 2.61.
__global__ void __launch_bounds__(256) adam_requantize_kernel(const int32_t* __restrict__ ind,
                                                              const int32_t* __restrict__ blk_of_slot, float4* values,
                                                              float4* __restrict__ m, float4* __restrict__ v,
                                                              const float4* __restrict__ g, int64_t nb, int N, int B,
                                                              int lgB, uint32_t* __restrict__ patlas,
                                                              uint32_t* __restrict__ atlas_out, const AdamArgs a) {
    const int P = B + 2, G = N >> lgB;
    const int64_t P3 = (int64_t)P * P * P, total = nb << (3 * lgB + 1);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t slot = t >> (3 * lgB + 1);
        const int h = (int)(t & 1), l = (int)(t >> 1) & ((1 << (3 * lgB)) - 1);
        const int c[3] = {l & (B - 1), (l >> lgB) & (B - 1), l >> (2 * lgB)};
        uint32_t* own = patlas + 2 * (slot * P3 + ((c[2] + 1) * P + c[1] + 1) * P + c[0] + 1) + h;
        // all loads before the first is used
        float4 x = values[t], mi = m[t], vi = v[t];
        const float4 gi = __ldcs(g + t);
        const uint32_t old = *own;
        const int blk = __ldg(blk_of_slot + slot);
        // three exact divisions and a root per parameter: a pass over mostly untouched values would
        // be bound by them
        if (!adam_untouched(a, gi, mi, vi)) {
            adam_quad(a, gi, mi, vi, x);
            m[t] = mi;
            v[t] = vi;
            values[t] = x;
        }
        if (blk < 0) continue;                                 // an unreferenced slot has no codes to keep
        const uint32_t w = (h ? quant8(x.x) : old & 0xffu) | quant8(x.y) << 8 | quant8(x.z) << 16 | quant8(x.w) << 24;
        if (atlas_out) __stcs(atlas_out + t, w);
        if (w == old) continue;
        *own = w;
        // per axis: the other block's offset and the padded coordinate there (-1: none)
        const int b[3] = {blk % G, (blk / G) % G, blk / (G * G)};
        int db[3], q[3], some = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            db[i] = 0;
            q[i] = -1;
            if (c[i] == 0) {
                q[i] = b[i] > 0 ? P - 1 : 0;
                db[i] = b[i] > 0 ? -1 : 0;
            } else if (c[i] == B - 1) {
                q[i] = b[i] < G - 1 ? 0 : P - 1;
                db[i] = b[i] < G - 1 ? 1 : 0;
            }
            some |= q[i] >= 0 ? 1 << i : 0;
        }
        for (int k = 1; k < 8; ++k) {
            if (k & ~some) continue;
            const int64_t n = ((int64_t)(b[2] + (k & 4 ? db[2] : 0)) * G + b[1] + (k & 2 ? db[1] : 0)) * G + b[0] +
                              (k & 1 ? db[0] : 0);
            const int s = __ldg(ind + n);
            if (s < 0) continue;
            patlas[2 * (s * P3 + ((k & 4 ? q[2] : c[2] + 1) * P + (k & 2 ? q[1] : c[1] + 1)) * P +
                        (k & 1 ? q[0] : c[0] + 1)) + h] = w;
        }
    }
}

// ---------------------------------------------------------------------------------
// Chebyshev (L-infinity) distance transform of a cube of side n, in three separable
// passes: along one axis, out(p) = min over q on p's line of max(|q - p|, in(q)),
// capped at `cap`. Starting from in = 0 on occupied cells and cap elsewhere, after the
// x, y and z passes out(p) = min over occupied q of max_i |q_i - p_i| (max distributes
// over min, so the passes compose). The scan walks outwards from p and stops once the
// offset reaches the best value found, so its cost is the distance itself.
//
// `side` restricts q to one half-line (bit 0: q <= p, bit 1: q >= p). With one side per
// axis the result is the distance to the nearest occupied cell in the
// octant cone {q : q_i - p_i of the chosen sign}: the cone is a product of half-lines,
// so the one-sided passes compose the same way.
// ---------------------------------------------------------------------------------
constexpr int kSideLow = 1, kSideHigh = 2;

__device__ __forceinline__ int dt_line(const uint8_t* __restrict__ in, int64_t base, int64_t stride, int pos, int n,
                                       int cap, int side) {
    int best = min((int)in[base + pos * stride], cap);
    const int a_end = (side & kSideLow) ? -1 : pos, b_end = (side & kSideHigh) ? n : pos;
    for (int d = 1; d < best; ++d) {
        const int a = pos - d, b = pos + d;
        if (a <= a_end && b >= b_end) break;
        if (a > a_end) best = min(best, max(d, (int)in[base + a * stride]));
        if (b < b_end) best = min(best, max(d, (int)in[base + b * stride]));
    }
    return best;
}

// the side of axis i for octant o (bit i of o set: the ray runs towards -i)
__host__ __device__ __forceinline__ int octant_side(int o, int i) { return ((o >> i) & 1) ? kSideLow : kSideHigh; }

// axis: 0 = x (stride 1), 1 = y (stride n), 2 = z (stride n^2)
__global__ void dt_pass_kernel(const uint8_t* __restrict__ in, uint8_t* __restrict__ out, int n, int axis, int cap,
                               int side) {
    const int64_t total = (int64_t)n * n * n;
    const int64_t stride = axis == 0 ? 1 : (axis == 1 ? n : (int64_t)n * n);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)t;                                  // n <= 1024
        const int c[3] = {r % n, (r / n) % n, r / (n * n)};
        const int pos = c[axis];
        const int64_t base = t - (int64_t)pos * stride;
        out[t] = (uint8_t)dt_line(in, base, stride, pos, n, cap, side);
    }
}

// 0 where the block is occupied, cap elsewhere
__global__ void block_seed_kernel(const int32_t* __restrict__ ind, int64_t n, int cap, uint8_t* __restrict__ out) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        out[t] = ind[t] >= 0 ? 0 : (uint8_t)cap;
}

// dst[i] = src[i] for an occupied block, -bdist[i] (>= 1) for an empty one: the march
// reads one word per block.
__global__ void encode_distance_kernel(const int32_t* __restrict__ src, const uint8_t* __restrict__ bdist, int32_t* __restrict__ dst,
                                       int64_t n) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = src[t];
        dst[t] = v >= 0 ? v : -(int32_t)max((int)bdist[t], 1);
    }
}

// ---------------------------------------------------------------------------------
// The device layout of the stored blocks, one CTA for one block (B >= 32) or for 32 / B blocks
// side by side in a warp's lanes:
//   1. the padded copy row by row, and each of the block's own rows' non-zero density codes as a
//      bit mask in shared memory: padded coordinate p in [0, B+2) is the global voxel
//      block_origin + p - 1, clamped to the grid (clamp-to-edge); its owner block supplies the
//      value, 0 if empty (one owner for a row, two more for its ends);
//   2. the warps compute the octants' voxel distances from the masks, with no pass over memory
//      but the store of the result. The distance to the nearest set voxel in the cone obeys
//          D(p) = 0 if p is set, else 1 + min over the 7 neighbours p + {0, 1}^3 \ 0
//      (steps in the cone's directions). Along x, D(x) <= 1 + D(x + 1) in the rows already
//      done, so all of a row's candidates but two reduce to the distance to the row's own next
//      set bit: D = min(bits, 1 + m(x), 1 + m(x + 1)), m the minimum over the three rows behind
//      at y + 1 and z + 1. Lanes hold x in the order that puts the cone's next voxel into the
//      lane before, the z + 1 slice stays in registers, and a row costs about 14 instructions
//      without any barrier.
// Apron cells of the distance planes hold 255, or, outside the grid, the value of the voxel
// that they clamp to, so that a sample which rounding puts a hair outside the grid finds its
// clamped nearest voxel's value without a clamp.
// 2,144 blocks of 32^3 take 0.53 ms: the first part 0.22, bound by memory (1.35 GB at 6 TB/s), the
// second 0.30, bound by issue. Separate seed, x, y, z, apron and border passes with a scan per
// voxel took 25.4 ms; one octant per warp and the apron gathered voxel by voxel 0.77 ms.
// ---------------------------------------------------------------------------------
template <int LGB>
struct PrepShape {
    static constexpr int B = 1 << LGB, P = B + 2, P2 = P * P, P3 = P2 * P, B2 = B * B, B3 = B2 * B;
    static constexpr int LX = B < 32 ? B : 32;      // lanes along x
    static constexpr int NB = 32 / LX;              // blocks per CTA
    static constexpr int VPL = B / LX;              // voxels per lane along x (2 for B = 64)
    static constexpr int OPW = VPL == 2 ? 1 : 2;    // octants per warp: the two sides along y
    static constexpr int kWarps = 8 / OPW, kThreads = 32 * kWarps;
    static constexpr int kMinCtas = VPL == 2 ? 2 : 8;
    static constexpr int kSmem = 2 * VPL * B2 * 4 + 8 * NB * P2;    // row masks, the octants' slices
};

// The cone distance of one row: prev / pprev the z + 1 slice's rows y and y + 1, cur the row
// y + 1, all as 16-bit pairs. VPL 1: the row y of the octant with the cone towards lower y and
// the row B - 1 - y of the other, wa and wb their masks in lane order. VPL 2: the lane's two
// voxels of one octant's row, wa and wb the masks of the first and of the second.
template <int VPL>
__device__ __forceinline__ uint32_t prep_row(uint32_t cur, uint32_t prev, uint32_t pprev, uint32_t wa, uint32_t wb,
                                             int lane, uint32_t le, uint32_t lt, int lx) {
    const uint32_t m = __vimin3_u16x2(cur, prev, pprev);
    // x + 1: the lane before's (the first lane of a block gets its own m back), or for VPL 2
    // (low: the lane before's high; high: own low)
    uint32_t mx = __shfl_up_sync(0xffffffffu, m, 1, lx);
    if (VPL == 2) mx = __byte_perm(m, lane == 0 ? 0x00ff00ffu : mx, 0x1076);
    uint32_t D = __viaddmin_u16x2(__vminu2(m, mx), 0x00010001u, 0x00ff00ffu);
    if (wa | wb) {                                                // the same for all lanes
        const uint32_t ta = wa & le, tb = wb & le;
        const int la = 31 - __clz(ta), lb = 31 - __clz(tb);
        int da, db;
        if (VPL == 1) {
            da = ta ? lane - la : 255;
            db = tb ? lane - lb : 255;
        } else {
            const uint32_t ua = wb & lt;
            const int lu = 31 - __clz(ua);
            da = min(ta ? 2 * (lane - la) : 255, ua ? 2 * (lane - lu) - 1 : 255);
            db = min(tb ? 2 * (lane - lb) : 255, ta ? 2 * (lane - la) + 1 : 255);
        }
        D = __vminu2(D, (uint32_t)da | ((uint32_t)db << 16));
    }
    return D;
}

// One slice (z) into shared memory: VPL 1 of both octants of a pair (out_a, out_b), VPL 2 of one
// (SY: the cone's side along y), its voxels at out_a and out_b.
template <int LGB, bool SY>
__device__ __forceinline__ void prep_slice(uint32_t (&prev)[1 << LGB], const uint32_t* ma, const uint32_t* mb,
                                           uint8_t* out_a, uint8_t* out_b, int lane, uint32_t le, uint32_t lt) {
    using S = PrepShape<LGB>;
    uint32_t cur = 0x00ff00ffu, pprev = cur;
#pragma unroll
    for (int yi = 0; yi < S::B; ++yi) {
        const int ya = SY ? yi : S::B - 1 - yi, yb = S::VPL == 2 ? ya : S::B - 1 - ya;
        cur = prep_row<S::VPL>(cur, prev[yi], pprev, ma[ya], mb[yb], lane, le, lt, S::LX);
        pprev = prev[yi];
        prev[yi] = cur;
        out_a[(ya + 1) * S::P] = (uint8_t)cur;
        out_b[(yb + 1) * S::P] = (uint8_t)(cur >> 16);
    }
}

template <int LGB>
__global__ void __launch_bounds__(PrepShape<LGB>::kThreads, PrepShape<LGB>::kMinCtas) prep_blocks_kernel(
    const int32_t* __restrict__ ind, const int32_t* __restrict__ blk_of_slot, const int32_t* __restrict__ err,
    const uint2* __restrict__ atlas, int64_t nb, int G, uint2* __restrict__ patlas, uint8_t* __restrict__ vskip) {
    using S = PrepShape<LGB>;
    constexpr int B = S::B, P = S::P, LX = S::LX;
    extern __shared__ __align__(16) uint32_t s_mem[];
    // a row's mask: bit g * LX + x (VPL 2: one word for even, one for odd x), and bit-reversed
    uint32_t(*s_mask)[S::VPL][S::B2] = reinterpret_cast<uint32_t(*)[S::VPL][S::B2]>(s_mem);
    // the octants' slices
    uint8_t(*s_slice)[S::NB][S::P2] = reinterpret_cast<uint8_t(*)[S::NB][S::P2]>(s_mem + 2 * S::VPL * S::B2);
    __shared__ int s_own[S::NB][27];             // slots of the 3^3 blocks around, -1 empty
    __shared__ int s_edge[S::NB];                // bit 2 a (+ 1): first (last) block along axis a
    if (*err) return;                            // an invalid indirection grid: the host reports it
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t slot0 = (int64_t)blockIdx.x * S::NB;
    for (int i = tid; i < S::NB * 27; i += S::kThreads) {
        const int g = i / 27, k = i % 27;
        const int blk = slot0 + g < nb ? blk_of_slot[slot0 + g] : -1;
        int own = -1;
        if (blk >= 0) {
            const int bx = blk % G, by = (blk / G) % G, bz = blk / (G * G);
            const int x = min(max(bx + k % 3 - 1, 0), G - 1), y = min(max(by + (k / 3) % 3 - 1, 0), G - 1),
                      z = min(max(bz + k / 9 - 1, 0), G - 1);
            own = ind[((int64_t)z * G + y) * G + x];
            if (k == 0)
                s_edge[g] = (bx == 0 ? 1 : 0) | (bx == G - 1 ? 2 : 0) | (by == 0 ? 4 : 0) | (by == G - 1 ? 8 : 0) |
                            (bz == 0 ? 16 : 0) | (bz == G - 1 ? 32 : 0);
        } else if (k == 0) {
            s_edge[g] = 0;
        }
        s_own[g][k] = own;
    }
    __syncthreads();

    // 1. the padded copy, a z slice per warp, kRows rows' loads in flight (the votes keep them from
    // being moved up); an unreferenced slot is stored as zeros
    {
        const int g = lane / LX, x = lane % LX;
        const int64_t slot = slot0 + g;
        const bool in = slot < nb, first = x == 0, last = x == LX - 1;
        const int edge = s_edge[g];
        // the x apron's voxel beside a block's first and last: of the neighbour, or the clamped one
        const int side = first ? 0 : 2;
        const int side_x = first ? (edge & 1 ? 0 : B - 1) : (edge & 2 ? B - 1 : 0);
        const int side_px = first ? 0 : P - 1;
        uint2* dst = patlas + slot * S::P3 + 1 + S::VPL * x;
        constexpr int kRows = B < 8 / S::VPL ? B : 8 / S::VPL;
        for (int pz = warp; pz < P; pz += S::kWarps) {
            const int nz = pz == 0 ? 0 : (pz == P - 1 ? 2 : 1);
            const int lz = nz == 1 ? pz - 1 : (nz == 0 ? (edge & 16 ? 0 : B - 1) : (edge & 32 ? B - 1 : 0));
            // n rows from py on, of the neighbours ny along y, from their row ly on
            auto rows = [&](auto n, int ny, int ly, int py) {
                constexpr int kN = decltype(n)::value;
                const int* own = s_own[g] + (nz * 3 + ny) * 3;
                const int mid = in ? own[1] : -1, beside = in && (first || last) ? own[side] : -1;
                const int64_t line = (int64_t)(lz * B + ly) * B;
                const uint2* src = atlas + (int64_t)mid * S::B3 + line + S::VPL * x;
                const uint2* end = atlas + (int64_t)beside * S::B3 + line + side_x;
                uint2* d = dst + (pz * P + py) * P;
                uint2 v[kN][S::VPL], e[kN];
#pragma unroll
                for (int u = 0; u < kN; ++u) {
#pragma unroll
                    for (int q = 0; q < S::VPL; ++q)  // 8-byte loads: the atlas need not be aligned to more
                        v[u][q] = mid >= 0 ? __ldg(src + u * B + q) : make_uint2(0u, 0u);
                    e[u] = beside >= 0 ? __ldg(end + u * B) : make_uint2(0u, 0u);
                }
#pragma unroll
                for (int u = 0; u < kN; ++u) {
#pragma unroll
                    for (int q = 0; q < S::VPL; ++q) {
                        if (in) d[u * P + q] = v[u][q];
                        if (nz == 1 && ny == 1) {
                            const uint32_t m = __ballot_sync(0xffffffffu, (v[u][q].x & 0xffu) != 0u);
                            if (lane == 0) {
                                s_mask[0][S::VPL - 1 - q][lz * B + ly + u] = __brev(m);
                                s_mask[1][q][lz * B + ly + u] = m;
                            }
                        }
                    }
                    if (in && (first || last)) d[u * P + side_px - 1 - S::VPL * x] = e[u];
                }
            };
            rows(std::integral_constant<int, 1>{}, 0, edge & 4 ? 0 : B - 1, 0);
            for (int y = 0; y < B; y += kRows) rows(std::integral_constant<int, kRows>{}, 1, y, y + 1);
            rows(std::integral_constant<int, 1>{}, 2, edge & 8 ? B - 1 : 0, P - 1);
        }
    }
    __syncthreads();

    // 2. the octants' distance planes, two per warp (B = 64: one): o0 and, with VPL 1, the octant
    // o0 + 2 whose cone runs towards lower y
    const int o0 = S::OPW == 2 ? (warp & 1) | (warp & 2) << 1 : warp;
    const bool sx = o0 & 1, sy = S::OPW == 2 || (o0 & 2), sz = o0 & 4;    // set: the cone runs towards lower coordinates
    const int bit = sx ? lane : 31 - lane;                // this lane's bit in a row's mask
    const int g = S::VPL == 1 ? bit / LX : 0;
    const uint32_t le = (2u << lane) - 1u, lt = le >> 1;
    const uint32_t own_le = S::VPL == 1 ? le & ~((1u << (lane / LX * LX)) - 1u) : le;
    // this lane's voxel(s) along x: xa (whose cone neighbour is in the lane before) and xb
    const int xa = S::VPL == 1 ? bit % LX : 2 * bit + (sx ? 0 : 1);
    const int xb = S::VPL == 1 ? xa : xa ^ 1;
    uint32_t prev[B];
#pragma unroll
    for (int y = 0; y < B; ++y) prev[y] = 0x00ff00ffu;
    const uint32_t* mask_a = s_mask[sx][0];
    const uint32_t* mask_b = s_mask[sx][S::VPL - 1];
    const int oa = S::OPW == 2 ? o0 + 2 : o0;
    uint8_t* out_a = s_slice[oa][g] + 1 + xa;
    uint8_t* out_b = s_slice[o0][g] + 1 + xb;
#pragma unroll 1
    for (int zi = 0; zi < B; ++zi) {
        const int z = sz ? zi : B - 1 - zi;
        if (sy) prep_slice<LGB, true>(prev, mask_a + z * B, mask_b + z * B, out_a, out_b, lane, own_le, lt);
        else prep_slice<LGB, false>(prev, mask_a + z * B, mask_b + z * B, out_a, out_b, lane, own_le, lt);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < S::OPW; ++p) {
            const int o = o0 + 2 * p;
            uint32_t* plane = reinterpret_cast<uint32_t*>(vskip + ((int64_t)o * nb + slot0) * S::P3) + (z + 1) * (S::P2 / 4);
            if constexpr (S::NB == 1) {
                // the x and then the y apron: 255, or outside the grid the voxel that they clamp to
                const int edge = s_edge[0];
                uint8_t* sl = s_slice[o][0];
#pragma unroll
                for (int q = 0; q < S::VPL; ++q) {
                    uint8_t* row = sl + (1 + lane + 32 * q) * P;
                    row[0] = (edge & 1) ? row[1] : (uint8_t)255;
                    row[P - 1] = (edge & 2) ? row[B] : (uint8_t)255;
                }
                __syncwarp();
                for (int px = lane; px < P; px += 32) {
                    sl[px] = (edge & 4) ? sl[P + px] : (uint8_t)255;
                    sl[(P - 1) * P + px] = (edge & 8) ? sl[B * P + px] : (uint8_t)255;
                }
                __syncwarp();
                // the slice goes out in words (P^2 and P^3 are multiples of 4), and once more where
                // it is beside the z apron: there as 255, or outside the grid as it is
                const uint32_t* w = reinterpret_cast<const uint32_t*>(sl);
#pragma unroll
                for (int i = 0; i < S::P2 / 4 / 32; ++i) plane[lane + 32 * i] = w[lane + 32 * i];
                if (lane < S::P2 / 4 % 32) plane[lane + S::P2 / 4 / 32 * 32] = w[lane + S::P2 / 4 / 32 * 32];
                if (z == 0 || z == B - 1)
                    for (int i = lane; i < S::P2 / 4; i += 32) {
                        if (z == 0) plane[i - S::P2 / 4] = (edge & 16) ? w[i] : 0xffffffffu;
                        if (z == B - 1) plane[i + S::P2 / 4] = (edge & 32) ? w[i] : 0xffffffffu;
                    }
            } else {
                // the same for the blocks beside one another
                for (int i = lane; i < S::NB * 2 * B; i += 32) {
                    const int gi = i / (2 * B), hi = i & 1, py = 1 + ((i % (2 * B)) >> 1);
                    uint8_t* sl = s_slice[o][gi] + py * P;
                    sl[hi ? P - 1 : 0] = (s_edge[gi] >> hi) & 1 ? sl[hi ? B : 1] : (uint8_t)255;
                }
                __syncwarp();
                for (int i = lane; i < S::NB * 2 * P; i += 32) {
                    const int gi = i / (2 * P), q = i % (2 * P), hi = q >= P, px = hi ? q - P : q;
                    uint8_t* sl = s_slice[o][gi];
                    sl[(hi ? P - 1 : 0) * P + px] = (s_edge[gi] >> (2 + hi)) & 1 ? sl[(hi ? B : 1) * P + px] : (uint8_t)255;
                }
                __syncwarp();
                for (int i = lane; i < S::NB * (S::P2 / 4); i += 32) {
                    const int gi = i / (S::P2 / 4), q = i % (S::P2 / 4);
                    if (slot0 + gi >= nb) break;
                    const uint32_t w = reinterpret_cast<const uint32_t*>(s_slice[o][gi])[q];
                    uint32_t* d = plane + (int64_t)gi * (S::P3 / 4) + q;
                    *d = w;
                    if (z == 0) d[-(S::P2 / 4)] = (s_edge[gi] & 16) ? w : 0xffffffffu;
                    if (z == B - 1) d[S::P2 / 4] = (s_edge[gi] & 32) ? w : 0xffffffffu;
                }
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------
// The block-level maps of grids of up to 64 blocks a side, one CTA per octant o:
// ind_oct[o] = the indirection grid with every empty entry replaced by -D, D >= 1 the
// Chebyshev distance (capped) to the nearest occupied block of o's cone, by the same
// recurrence as the voxel maps. Rows on one anti-diagonal y + z = s depend only on the two
// diagonals before and go to the CTA's warps side by side. A grid of 32^3 blocks takes 33 us;
// separate seed, x, y, z and encode passes were 40 launches and 240 us.
// ---------------------------------------------------------------------------------
constexpr int kMapThreads = 1024, kMapMaxG = 64;

// W: 32-block words per row
template <int W>
__global__ void __launch_bounds__(kMapThreads) block_maps_kernel(const int32_t* __restrict__ ind, int G, int cap,
                                                                 int32_t* __restrict__ ind_oct) {
    constexpr int M = 32 * W;
    __shared__ uint32_t s_bits[M * M][W];              // occupied blocks of a row in the cone's order along x
    // distances of the last three diagonals by row y + 1; rows that a diagonal does not have
    // (y = -1, z = -1) keep the cap
    __shared__ uint8_t s_diag[3][M + 1][M];
    const int o = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool sx = o & 1, sy = o & 2, sz = o & 4;
    int32_t* out = ind_oct + (int64_t)o * G * G * G;
    for (int i = threadIdx.x; i < 3 * (M + 1) * M; i += kMapThreads) (&s_diag[0][0][0])[i] = (uint8_t)cap;
    // occupied blocks keep their slot; the diagonals below write the empty ones
#pragma unroll 4
    for (int row = warp; row < G * G; row += kMapThreads / 32) {
#pragma unroll
        for (int h = 0; h < W; ++h) {
            const int c = 32 * h + lane, i = row * G + (sx ? c : G - 1 - c);
            const int32_t v = c < G ? __ldg(ind + i) : -1;
            if (v >= 0) out[i] = v;
            const uint32_t m = __ballot_sync(0xffffffffu, v >= 0);
            if (lane == 0) s_bits[row][h] = m;
        }
    }
    __syncthreads();
    const uint32_t le = (2u << lane) - 1u;
    int b0 = 0, b1 = 2, b2 = 1;                        // this diagonal's buffer and the two before
    for (int s = 0; s <= 2 * (G - 1); ++s) {
        for (int yi = max(0, s - G + 1) + warp; yi <= min(s, G - 1); yi += kMapThreads / 32) {
            const int zi = s - yi;
            const int row = (sz ? zi : G - 1 - zi) * G + (sy ? yi : G - 1 - yi);
            int carry_m = cap, carry_d = cap;          // of the voxel before the word
#pragma unroll
            for (int h = 0; h < W; ++h) {
                const int c = 32 * h + lane;
                const int m = min(min((int)s_diag[b1][yi][c], (int)s_diag[b1][yi + 1][c]), (int)s_diag[b2][yi][c]);
                int mx = __shfl_up_sync(0xffffffffu, m, 1);
                if (h > 0 && lane == 0) mx = carry_m;
                const uint32_t t = s_bits[row][h] & le;
                const int dist = t ? lane - (31 - __clz(t)) : min(cap, carry_d + 1 + lane);
                const int D = min(min(min(m, mx) + 1, dist), cap);
                if (h + 1 < W) {
                    carry_m = __shfl_sync(0xffffffffu, m, 31);
                    carry_d = __shfl_sync(0xffffffffu, dist, 31);
                }
                if (c < G) {
                    s_diag[b0][yi + 1][c] = (uint8_t)D;
                    if (D > 0) out[row * G + (sx ? c : G - 1 - c)] = -D;
                }
            }
        }
        __syncthreads();
        const int t = b2;
        b2 = b1;
        b1 = b0;
        b0 = t;
    }
}

static unsigned grid_for(int64_t n) {
    const int64_t b = (n + 255) / 256;
    return (unsigned)(b < 1048576 ? (b > 0 ? b : 1) : 1048576);
}

static void block_distance(const int32_t* ind, int G, int cap, uint8_t* tmp0, uint8_t* tmp1, uint8_t* bdist,
                           const int side[3], cudaStream_t st) {
    const int64_t n = (int64_t)G * G * G;
    block_seed_kernel<<<grid_for(n), 256, 0, st>>>(ind, n, cap, tmp0);
    dt_pass_kernel<<<grid_for(n), 256, 0, st>>>(tmp0, tmp1, G, 0, cap, side[0]);
    dt_pass_kernel<<<grid_for(n), 256, 0, st>>>(tmp1, tmp0, G, 1, cap, side[1]);
    dt_pass_kernel<<<grid_for(n), 256, 0, st>>>(tmp0, bdist, G, 2, cap, side[2]);
}

// For each octant o, ind_oct[o] = the indirection grid `ind` with every empty entry replaced by
// -D_o, D_o >= 1 the Chebyshev distance (in blocks, capped) to the nearest occupied block
// in o's cone. Grids beyond block_maps_kernel's shared memory run one pass per axis and
// octant over tmp0, tmp1 and bdist (G^3 bytes each). Adds the launches to *launches.
cudaError_t launch_block_distance_octants(const int32_t* ind, int G, int cap, uint8_t* tmp0, uint8_t* tmp1,
                                          uint8_t* bdist, int32_t* ind_oct, int64_t* launches, cudaStream_t st) {
    const int64_t n = (int64_t)G * G * G;
    if (G <= kMapMaxG) {
        if (G <= 32) block_maps_kernel<1><<<8, kMapThreads, 0, st>>>(ind, G, cap, ind_oct);
        else block_maps_kernel<2><<<8, kMapThreads, 0, st>>>(ind, G, cap, ind_oct);
        *launches += 1;
        return cudaGetLastError();
    }
    for (int o = 0; o < 8; ++o) {
        const int side[3] = {octant_side(o, 0), octant_side(o, 1), octant_side(o, 2)};
        block_distance(ind, G, cap, tmp0, tmp1, bdist, side, st);
        encode_distance_kernel<<<grid_for(n), 256, 0, st>>>(ind, bdist, ind_oct + (size_t)o * n, n);
    }
    *launches += 8 * 5;
    return cudaGetLastError();
}

cudaError_t launch_validate(const int32_t* ind, int64_t n_ind, int64_t nb, int32_t* blk_of_slot, int32_t* err,
                            cudaStream_t st) {
    if (n_ind <= 0) return cudaSuccess;
    const int64_t blocks = (n_ind + 255) / 256;
    validate_kernel<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, st>>>(ind, n_ind, nb, blk_of_slot, err);
    return cudaGetLastError();
}

template <int LGB>
static cudaError_t prep_blocks(const int32_t* ind, const int32_t* blk_of_slot, const int32_t* err,
                               const uint8_t* atlas, int64_t nb, int G, uint2* patlas, uint8_t* vskip, cudaStream_t st) {
    constexpr int n = PrepShape<LGB>::NB, smem = PrepShape<LGB>::kSmem;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(prep_blocks_kernel<LGB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   smem);
        if (e != cudaSuccess) return e;
    }
    prep_blocks_kernel<LGB><<<(unsigned)((nb + n - 1) / n), PrepShape<LGB>::kThreads, smem, st>>>(
        ind, blk_of_slot, err, reinterpret_cast<const uint2*>(atlas), nb, G, patlas, vskip);
    return cudaGetLastError();
}

cudaError_t launch_prep_blocks(const int32_t* ind, const int32_t* blk_of_slot, const int32_t* err, const uint8_t* atlas,
                               int64_t nb, int G, int lgB, uint2* patlas, uint8_t* vskip, cudaStream_t st) {
    if (nb <= 0) return cudaSuccess;
    switch (lgB) {
        case 1: return prep_blocks<1>(ind, blk_of_slot, err, atlas, nb, G, patlas, vskip, st);
        case 2: return prep_blocks<2>(ind, blk_of_slot, err, atlas, nb, G, patlas, vskip, st);
        case 3: return prep_blocks<3>(ind, blk_of_slot, err, atlas, nb, G, patlas, vskip, st);
        case 4: return prep_blocks<4>(ind, blk_of_slot, err, atlas, nb, G, patlas, vskip, st);
        case 5: return prep_blocks<5>(ind, blk_of_slot, err, atlas, nb, G, patlas, vskip, st);
        case 6: return prep_blocks<6>(ind, blk_of_slot, err, atlas, nb, G, patlas, vskip, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_requantize(const int32_t* ind, const int32_t* blk_of_slot, const float* values, int64_t nb, int N,
                              int B, int lgB, uint2* patlas, uint8_t* atlas_out, cudaStream_t st) {
    if (nb <= 0) return cudaSuccess;
    const int64_t total = nb * (int64_t)(B + 2) * (B + 2) * (B + 2);
    requantize_padded_kernel<<<grid_for(total), 256, 0, st>>>(ind, blk_of_slot, reinterpret_cast<const float4*>(values),
                                                              nb, N, B, lgB, patlas, reinterpret_cast<uint2*>(atlas_out));
    return cudaGetLastError();
}

cudaError_t launch_adam_requantize(const int32_t* ind, const int32_t* blk_of_slot, float* values, float* m, float* v,
                                   const float* g, const AdamArgs& adam, int64_t nb, int N, int B, int lgB,
                                   uint2* patlas, uint8_t* atlas_out, cudaStream_t st) {
    if (nb <= 0) return cudaSuccess;
    adam_requantize_kernel<<<grid_for(nb << (3 * lgB + 1)), 256, 0, st>>>(
        ind, blk_of_slot, reinterpret_cast<float4*>(values), reinterpret_cast<float4*>(m), reinterpret_cast<float4*>(v),
        reinterpret_cast<const float4*>(g), nb, N, B, lgB, reinterpret_cast<uint32_t*>(patlas),
        reinterpret_cast<uint32_t*>(atlas_out), adam);
    return cudaGetLastError();
}
}  // namespace snerg
