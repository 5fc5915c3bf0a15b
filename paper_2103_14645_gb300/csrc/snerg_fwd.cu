// snerg_fwd.cu -- forward render kernels: one camera per launch, ray lists, and the
// persistent multi-camera kernel that drains a (camera, tile) work queue.
// The per-ray arithmetic is in snerg_internal.cuh (Sec. 5.2, App. A; Eqs. 2, 5-7).
//
// Every kernel comes in two flavours for the view-dependence MLP (Eq. 7): PW = true
// reads the weights from the kernel parameter `pw` (constant-bank operands; set with
// snerg_set_mlp), PW = false stages them from device memory into shared memory (the
// form the autograd path uses, where the weights live in a tensor).
//
// Compiled once per block build (BlockScene): SNERG_LGB and SNERG_ALPHA are the build's LGB and A. Debug outputs and
// the per-sample model are in build 0 only.
#include "snerg_internal.cuh"

#if !defined(SNERG_LGB) || !defined(SNERG_ALPHA)
#error "SNERG_LGB: log2 of the block edge of this build, 0 for any; SNERG_ALPHA: 0, 1 or 2 for any"
#endif

namespace snerg {

// Each warp covers an 8x4 pixel packet, so its 32 rays are neighbours on screen and walk
// neighbouring voxels together. A CTA holds NW warps (1: 8x4, 2: 16x4, 4: 16x8 pixels);
// small CTAs free their SM slot as soon as their own packets are done, which matters
// because packets on the object take several times longer than background packets.
//
// With fewer rays per warp (lanes, see lanes_per_warp) the packet shrinks to 4x4, 4x2, 2x2, 2x1
// or one pixel, and the CTA's tile with it.
template <int NW>
struct ImageTile {
    static constexpr int WX = NW >= 2 ? 2 : 1;      // warps across
    static constexpr int WY = NW >= 4 ? 2 : 1;      // warps down
    static constexpr int TW = 8 * WX, TH = 4 * WY;  // CTA tile in pixels
};
__host__ __device__ __forceinline__ int packet_width_log2(int lanes) {
    return lanes == 32 ? 3 : (lanes >= 8 ? 2 : (lanes >= 2 ? 1 : 0));
}

// SCHED: the launch's CTAs take the image's tiles in the order of the previous frame's
// cost buckets (slowest first). The slowest tiles -- those whose recorded cost is at least
// kSchedSparseFrac of the previous frame's time, at most smax of them -- are rendered
// sparsely: four CTAs per tile, each CTA two of its eight rows, 8 rays per warp, so that
// their long chains of dependent loads run with less divergence beside them. Launch index
// c < 4 smax: quarter c % 4 of sparse tile c / 4 (idle if there are fewer); c >= 4 smax:
// the next tile in order, rendered as usual. The pixels of every tile are rendered once,
// whatever the order and mapping. Each CTA records its duration when all its warps are
// done (a sparse tile by its last quarter to finish, as its slowest quarter times
// kSchedSparseGain: about its dense cost, so that it stays sparse while it stays slow) and
// the launch's start and end. The grid is nt + 4 smax CTAs: 4 smax sparse slots (S <= smax
// used), then nt dense slots for the tiles S .. nt - 1 of the order (the last S idle).
// A small image (lanes_per_warp) has `parts` CTAs per dense slot, each a band of the tile's rows
// with 32 / parts rays per warp, and no sparse slots; the first band's duration stands for the
// tile's.
struct SchedSlot {
    int tile;       // -1: idle
    int quarter;    // -1: dense
    int part;       // dense: band of the tile's rows
};

__device__ __forceinline__ SchedSlot sched_map(const SchedArgs& sch, int c, unsigned long long* t0) {
    __shared__ SchedSlot s_slot;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        if (lane == 0) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            *t0 = t;
        }
        int incl = 0, c_b = 0, S = 0;
        bool use = false;
        const int b = kSchedBuckets - 1 - lane;          // lane 0: the slowest bucket
        if (sch.rd_count) {
            c_b = __ldg(sch.rd_count + b);
            incl = c_b;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            // the buckets are used only when they hold exactly this launch's tiles
            use = __shfl_sync(0xffffffffu, incl, 31) == sch.nt;
            if (use && sch.smax > 0) {
                const unsigned long long* tw = reinterpret_cast<const unsigned long long*>(sch.rd_count + kSchedHdrTimes);
                const float T = (float)(__ldg(tw + 1) - ~__ldg(tw));        // the previous frame's time
                const int bthr = (int)ceilf(3.0f * __log2f(fmaxf(kSchedSparseFrac * T, 250.0f) * (1.0f / 250.0f)));
                if (bthr < kSchedBuckets)
                    S = min(sch.smax, __shfl_sync(0xffffffffu, incl, kSchedBuckets - 1 - max(bthr, 0)));
            }
        }
        int item = -1, q = -1;
        if (c < 4 * sch.smax) {
            if ((c >> 2) < S) {
                item = c >> 2;
                q = c & 3;
            }
        } else {
            item = S + (c - 4 * sch.smax) / sch.parts;
            if (item >= sch.nt) item = -1;
        }
        if (lane == 0) {
            s_slot = SchedSlot{use ? -1 : item, q, q < 0 ? (c - 4 * sch.smax) % sch.parts : 0};
            if (c == 0) {           // what this launch did, for snerg_schedule_stats
                sch.wr_count[kSchedHdrInfo] = S + 1;
                sch.wr_count[kSchedHdrInfo + 1] = use ? 1 : 0;
            }
        }
        __syncwarp();
        const int excl = incl - c_b;
        if (use && item >= 0 && item >= excl && item < incl && item - excl < sch.cap)
            s_slot.tile = __ldg(sch.rd_list + (size_t)b * sch.cap + (item - excl));
    }
    __syncthreads();
    return s_slot;
}

__device__ __forceinline__ void sched_record(const SchedArgs& sch, const SchedSlot& sl, const unsigned long long* t0) {
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t1;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
        unsigned long long* tw = reinterpret_cast<unsigned long long*>(sch.wr_count + kSchedHdrTimes);
        atomicMax(tw, ~*t0);
        atomicMax(tw + 1, t1);
        float ns = (float)(t1 - *t0);
        bool rec = sl.tile >= 0 && sl.quarter < 0 && sl.part == 0;
        if (sl.tile >= 0 && sl.quarter >= 0) {
            // sparse: the last of the tile's four quarters records the slowest one
            const int j = (int)(blockIdx.x >> 2);
            unsigned int* qmax = reinterpret_cast<unsigned int*>(sch.wr_count + kSchedHdrSlotMax);
            int* qcnt = sch.wr_count + kSchedHdrSlotCnt;
            atomicMax(qmax + j, (unsigned int)min(t1 - *t0, 0xffffffffull));
            __threadfence();
            if (atomicAdd(qcnt + j, 1) == 3) {
                ns = (float)atomicMax(qmax + j, 0u) * kSchedSparseGain;
                rec = true;
            }
        }
        if (rec) {
            const int b = min(max((int)(3.0f * __log2f(fmaxf(ns, 1.0f) * (1.0f / 250.0f))), 0), kSchedBuckets - 1);
            const int pos = atomicAdd(sch.wr_count + b, 1);
            if (pos < sch.cap) sch.wr_list[(size_t)b * sch.cap + pos] = sl.tile;
        }
    }
}

// one pixel of render_image_kernel: march, MLP, store (and the debug outputs)
template <bool DBG, bool PS, class SC>
__device__ __forceinline__ void image_pixel(const SC& s, const snerg_camera& cam, const float* sW,
                                            const MlpWeights* pwp, float* __restrict__ rgb, const DebugOut& dbg,
                                            int px, int py) {
    const Ray r = make_ray(s, cam, px, py);
    const int64_t pix = cam.out_offset + (int64_t)py * cam.W + px;
    MarchState st;
    int k_first = 0;
    if (DBG && dbg.trace)
        march<true, false, PS>(s, r, st, dbg.trace + pix * dbg.trace_cap, dbg.trace_cap, nullptr, nullptr, 0,
                               &k_first, pwp, sW);
    else
        march<false, false, PS>(s, r, st, nullptr, 0, nullptr, nullptr, 0, DBG ? &k_first : nullptr, pwp, sW);
    record_status(s, st);
    float c[3], aux[kAuxCh];
    finish_ray(s, sW, r, st, c, aux, pwp);
    rgb[pix * 3 + 0] = c[0];
    rgb[pix * 3 + 1] = c[1];
    rgb[pix * 3 + 2] = c[2];
    if (DBG) {
        if (dbg.aux)
            for (int k = 0; k < kAuxCh; ++k) dbg.aux[pix * kAuxCh + k] = aux[k];
        if (dbg.counts) {
            dbg.counts[pix * 4] = st.steps;
            dbg.counts[pix * 4 + 1] = st.active;
            dbg.counts[pix * 4 + 2] = st.blocks;
            dbg.counts[pix * 4 + 3] = st.active > 0 ? k_first : -1;
        }
    }
}

// 8 CTAs per SM leave 64 registers: the builds per block edge spill 8 bytes with the weights as
// parameters and 56 with the weights in device memory (the any-edge build, with more instructions,
// none), and are the faster all the same: a full-HD view with weights in device memory 833 -> 794 us.
template <int LGB, int A, bool DBG, bool PW, int NW, bool PS, bool SCHED = false>
__global__ void __launch_bounds__(32 * NW, 32 / NW) render_image_kernel(const BlockScene<LGB, A> s, const snerg_camera cam,
                                                                        const float* __restrict__ mlp,
                                                                        const __grid_constant__ MlpWeights pw,
                                                                        float* __restrict__ rgb, const DebugOut dbg,
                                                                        int row0, int row1, int lanes,
                                                                        const SchedArgs sch) {
    __shared__ __align__(16) float sW[PW ? 4 : kNParam + 1];
    if (!PW) {
        load_mlp_smem_t(sW, mlp);
        __syncthreads();
    }
    const MlpWeights* pwp = PW ? &pw : nullptr;
    using T = ImageTile<NW>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if constexpr (SCHED) {
        static_assert(NW == 4, "the sparse mapping assumes 16x8 tiles of four 8x4 warps");
        __shared__ unsigned long long s_t0;
        const SchedSlot sl = sched_map(sch, (int)blockIdx.x, &s_t0);
        if (sl.tile >= 0) {
            const int tx = sl.tile % sch.tiles_x, ty = sl.tile / sch.tiles_x;
            int px, py;
            bool on = true;
            if (sl.quarter < 0 && sch.parts > 1) {
                const int lanes = 32 / sch.parts, idx = warp * lanes + lane;     // 16 x (8 / parts) pixels
                on = lane < lanes;
                px = tx * T::TW + (idx & 15);
                py = ty * T::TH + sl.part * (T::TH / sch.parts) + (idx >> 4);
            } else if (sl.quarter < 0) {
                px = tx * T::TW + (warp % T::WX) * 8 + (lane & 7);
                py = ty * T::TH + (warp / T::WX) * 4 + (lane >> 3);
            } else {
                const int idx = warp * 8 + (lane & 7);            // 0..31: rows 2q, 2q + 1
                on = lane < 8;
                px = tx * T::TW + (idx & 15);
                py = ty * T::TH + 2 * sl.quarter + (idx >> 4);
            }
            if (on && px < cam.W && py < row1) image_pixel<DBG, PS>(s, cam, sW, pwp, rgb, dbg, px, py);
        }
        sched_record(sch, sl, &s_t0);
    } else {
        const int lgx = packet_width_log2(lanes), h = lanes >> lgx;      // a warp's packet: (1 << lgx) x h
        const int px = (((int)blockIdx.x * T::WX + warp % T::WX) << lgx) + (lane & ((1 << lgx) - 1));
        const int py = row0 + ((int)blockIdx.y * T::WY + warp / T::WX) * h + (lane >> lgx);
        if (lane >= lanes || px >= cam.W || py >= row1) return;
        image_pixel<DBG, PS>(s, cam, sW, pwp, rgb, dbg, px, py);
    }
}

// MINB: resident CTAs per SM the build is limited to (8: 64 registers; 7: 72; 4: up to 128);
// lanes: rays per warp (the other lanes idle); REC: each ray's composited samples go to
// record (entry j of ray i at record[j * n + i], see march) for the adjoint
template <int LGB, int A, bool DBG, bool PW, int MINB, bool REC = false>
__global__ void __launch_bounds__(128, MINB) render_rays_kernel(const BlockScene<LGB, A> s, const __grid_constant__ CamTable cams,
                                                                int32_t n_cams, const int32_t* __restrict__ pix,
                                                                int64_t n, const float* __restrict__ mlp,
                                                                const __grid_constant__ MlpWeights pw,
                                                                float* __restrict__ rgb, const DebugOut dbg,
                                                                float2* __restrict__ record, int lanes) {
    __shared__ __align__(16) float sW[PW ? 4 : kNParam + 1];
    if (!PW) {
        load_mlp_smem_t(sW, mlp);
        __syncthreads();
    }
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
    int k_first = 0;
    if (REC)
        march<false, false, false, true, true>(s, r, st, nullptr, 0, nullptr, nullptr, 0, &k_first, nullptr, nullptr,
                                               record + i, n);
    else if (DBG && dbg.trace)
        march<true, false>(s, r, st, dbg.trace + i * dbg.trace_cap, dbg.trace_cap, nullptr, nullptr, 0, &k_first);
    else
        march<false, false, false, true>(s, r, st, nullptr, 0, nullptr, nullptr, 0, DBG ? &k_first : nullptr);
    record_status(s, st);
    float c[3], aux[kAuxCh];
    finish_ray(s, sW, r, st, c, aux, PW ? &pw : nullptr);
    rgb[i * 3 + 0] = c[0];
    rgb[i * 3 + 1] = c[1];
    rgb[i * 3 + 2] = c[2];
    if (DBG) {
        if (dbg.aux)
            for (int k = 0; k < kAuxCh; ++k) dbg.aux[i * kAuxCh + k] = aux[k];
        if (dbg.counts) {
            dbg.counts[i * 4] = st.steps;
            dbg.counts[i * 4 + 1] = st.active;
            dbg.counts[i * 4 + 2] = st.blocks;
            dbg.counts[i * 4 + 3] = st.active > 0 ? k_first : -1;
        }
    }
}

// Persistent multi-camera render: gridDim = SMs x CTAs/SM. Each warp pulls work items
// (tile_w x tile_h pixels of one camera) from a global counter until the queue is empty,
// and renders each item in warp_w x warp_h packets of 32 rays. The counter is zeroed by
// the launch sequence (a memset node of the captured graph) before every launch.
// One pixel of the persistent launch: march, shade and store.
template <bool PW, class SC>
__device__ __forceinline__ void persistent_pixel(const SC& s, const snerg_camera& cam, const float* sW,
                                                 const MlpWeights& pw, float* rgb, int px, int py) {
    // the output row before the march, so that only it stays live across it
    float* out = rgb + (cam.out_offset + (int64_t)py * cam.W + px) * 3;
    const Ray r = make_ray(s, cam, px, py);
    MarchState st;
    march<false, false>(s, r, st, nullptr, 0, nullptr, nullptr);
    record_status(s, st);
    float c[3], aux[kAuxCh];
    finish_ray(s, sW, r, st, c, aux, PW ? &pw : nullptr);
    out[0] = c[0];
    out[1] = c[1];
    out[2] = c[2];
}

// MULTI: a work item is several warp passes (tile_w x tile_h larger than warp_w x
// warp_h); without it an item is exactly one warp pass and no pass loop stays live across
// the march.
template <int LGB, int A, bool PW, bool MULTI>
__global__ void __launch_bounds__(128, 8) render_persistent_kernel(const BlockScene<LGB, A> s,
                                                                   const __grid_constant__ PersistentParams p,
                                                                   const float* __restrict__ mlp,
                                                                   const __grid_constant__ MlpWeights pw,
                                                                   float* __restrict__ rgb,
                                                                   int32_t* __restrict__ queue) {
    __shared__ __align__(16) float sW[PW ? 4 : kNParam + 1];
    if (!PW) {
        load_mlp_smem_t(sW, mlp);
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(queue, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= p.total_items) break;
        int lo = 0, hi = p.n_cams;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (p.tile_start[mid] <= item) lo = mid; else hi = mid;
        }
        const snerg_camera& cam = p.cams[lo];
        const int rem = item - p.tile_start[lo];
        const int tx = rem % p.tiles_x[lo], ty = rem / p.tiles_x[lo];
        const int lx = lane % p.warp_w, ly = lane / p.warp_w;
        if (MULTI) {
            const int passes_x = p.tile_w / p.warp_w;
            const int passes = passes_x * (p.tile_h / p.warp_h);
            for (int ps = 0; ps < passes; ++ps) {
                const int px = tx * p.tile_w + (ps % passes_x) * p.warp_w + lx;
                const int py = ty * p.tile_h + (ps / passes_x) * p.warp_h + ly;
                if (px < cam.W && py < cam.H) persistent_pixel<PW>(s, cam, sW, pw, rgb, px, py);
            }
        } else {
            const int px = tx * p.warp_w + lx;
            const int py = ty * p.warp_h + ly;
            if (px < cam.W && py < cam.H) persistent_pixel<PW>(s, cam, sW, pw, rgb, px, py);
        }
    }
}

// rows [row0, row1) of the camera
template <int LGB, int A>
cudaError_t Forward<LGB, A>::image(const DevScene& ds, const snerg_camera& cam, const float* mlp, const MlpWeights* pw,
                                float* rgb, const DebugOut& dbg, cudaStream_t st, int row0, int row1,
                                const SchedArgs* sch, int share) {
    using T = ImageTile<kImageWarps>;
    const BlockScene<LGB, A> s(ds);
    const int nt = 32 * kImageWarps;
    const bool ps = (ds.flags & SNERG_FLAG_PER_SAMPLE_MLP) != 0, d = dbg.aux || dbg.counts || dbg.trace;
    const MlpWeights& w = pw ? *pw : no_weights();
    const SchedArgs none{nullptr, nullptr, nullptr, nullptr, 0, 0, 0, 0, 1};
    if (sch && !ps && !d) {
        // 4 smax sparse slots, then nt dense ones of `parts` CTAs
        auto* kernel = pw ? render_image_kernel<LGB, A, false, true, kImageWarps, false, true>
                          : render_image_kernel<LGB, A, false, false, kImageWarps, false, true>;
        kernel<<<(unsigned)(sch->nt * sch->parts + 4 * sch->smax), nt, 0, st>>>(s, cam, mlp, w, rgb, dbg, row0, row1, 32,
                                                                               *sch);
        return cudaGetLastError();
    }
    const int64_t pixels = (int64_t)cam.W * (row1 - row0);
    const int lanes = ps || d ? 32 : image_lanes(ds, row1 - row0 < cam.H ? pixels + pixels / 4 : pixels, share);
    const int tw = T::WX << packet_width_log2(lanes), th = T::WY * (lanes >> packet_width_log2(lanes));
    const dim3 grid((cam.W + tw - 1) / tw, (row1 - row0 + th - 1) / th);
    auto* kernel = pw ? render_image_kernel<LGB, A, false, true, kImageWarps, false>
                      : render_image_kernel<LGB, A, false, false, kImageWarps, false>;
    if (ps || d) {
        if constexpr (LGB == 0) {
            if (ps)
                kernel = pw ? (d ? render_image_kernel<LGB, A, true, true, kImageWarps, true>
                                 : render_image_kernel<LGB, A, false, true, kImageWarps, true>)
                            : (d ? render_image_kernel<LGB, A, true, false, kImageWarps, true>
                                 : render_image_kernel<LGB, A, false, false, kImageWarps, true>);
            else
                kernel = pw ? render_image_kernel<LGB, A, true, true, kImageWarps, false>
                            : render_image_kernel<LGB, A, true, false, kImageWarps, false>;
        } else {
            return cudaErrorInvalidValue;
        }
    }
    kernel<<<grid, nt, 0, st>>>(s, cam, mlp, w, rgb, dbg, row0, row1, lanes, none);
    return cudaGetLastError();
}

// A short list is spread over the warps of one wave of 7 CTAs per SM (28 warps), with debug outputs,
// which need more registers, of 4: 16,000 scattered rays of a 1024^3 grid take 76 us with 32 rays per
// warp and 53 with 8 or 4. With 16 and 8 the limits grow with the grid's side: 43,241 rays with 32 / 16
// (18 warps) 84 / 68 on a 768^3 grid, but 58 / 61 on a 256^3 one. If 4 CTAs per SM hold the list, it runs
// the build limited to 4 (the march keeps its state in registers, and a single wave gains nothing
// from more CTAs). Longer lists keep 7 CTAs per SM to hide the march's latencies (8 spill with the
// weights in device memory: 130,313 and 218,548 rays of a 1024^3 grid 149 and 229 us with 8, 141 and
// 222 with 7), or 8 where those hold the list in one or two waves and 7 need one more (154,825 and
// 308,499 rays 184 and 286 us with 7, 160 and 278 with 8; of a 256^3 grid 125 and 191, 123 and 192),
// and, from 1024^3 on, where they save any wave (1,030,921 rays of a 2048^3 grid 4 % less).
template <int LGB, int A>
cudaError_t Forward<LGB, A>::rays(const DevScene& s, const CamTable& cams, int32_t n_cams, const int32_t* pix, int64_t n,
                               const float* mlp, const MlpWeights* pw, float* rgb, const DebugOut& dbg, float2* record,
                               cudaStream_t st) {
    const bool d = dbg.aux || dbg.counts || dbg.trace;
    const int lanes = d ? lanes_per_warp(n, s.sms, {16, 16, 16, 16, 16})
                        : lanes_per_warp(n, s.sms, {by_side(s, 16, 16, 28), by_side(s, 16, 20, 28), 28, 28, 28});
    const int64_t ctas = (n + 4 * lanes - 1) / (4 * lanes), w7 = (ctas + 7 * s.sms - 1) / (7 * s.sms),
                  w8 = (ctas + 8 * s.sms - 1) / (8 * s.sms);
    const int per = ctas <= 4 * (int64_t)s.sms ? 4 : (w8 < w7 && (w8 <= 2 || s.N >= 1024) ? 8 : 7);
    // the build for `per` CTAs per SM
    auto* kernel = pw ? (per == 4   ? render_rays_kernel<LGB, A, false, true, 4>
                         : per == 7 ? render_rays_kernel<LGB, A, false, true, 7>
                                    : render_rays_kernel<LGB, A, false, true, 8>)
                      : (per == 4   ? render_rays_kernel<LGB, A, false, false, 4>
                         : per == 7 ? render_rays_kernel<LGB, A, false, false, 7>
                                    : render_rays_kernel<LGB, A, false, false, 8>);
    if (record) {                       // weights in device memory
        kernel = per == 4   ? render_rays_kernel<LGB, A, true, false, 4, true>
                 : per == 7 ? render_rays_kernel<LGB, A, true, false, 7, true>
                            : render_rays_kernel<LGB, A, true, false, 8, true>;
    } else if (d) {
        if constexpr (LGB == 0)
            kernel = pw ? (per == 4   ? render_rays_kernel<LGB, A, true, true, 4>
                           : per == 7 ? render_rays_kernel<LGB, A, true, true, 7>
                                      : render_rays_kernel<LGB, A, true, true, 8>)
                        : (per == 4   ? render_rays_kernel<LGB, A, true, false, 4>
                           : per == 7 ? render_rays_kernel<LGB, A, true, false, 7>
                                      : render_rays_kernel<LGB, A, true, false, 8>);
        else
            return cudaErrorInvalidValue;
    }
    kernel<<<(unsigned)ctas, 128, 0, st>>>(
        BlockScene<LGB, A>(s), cams, n_cams, pix, n, mlp, pw ? *pw : no_weights(), rgb, dbg, record, lanes);
    return cudaGetLastError();
}

template <int LGB, int A>
const void* Forward<LGB, A>::persistent_fn(bool param_weights, bool multi) {
    // the launches through this pointer pass a DevScene as the kernel's scene
    static_assert(sizeof(BlockScene<LGB, A>) == sizeof(DevScene), "a build's scene adds no member");
    if (param_weights)
        return multi ? (const void*)render_persistent_kernel<LGB, A, true, true>
                     : (const void*)render_persistent_kernel<LGB, A, true, false>;
    return multi ? (const void*)render_persistent_kernel<LGB, A, false, true>
                 : (const void*)render_persistent_kernel<LGB, A, false, false>;
}

template struct Forward<SNERG_LGB, SNERG_ALPHA>;

}  // namespace snerg
