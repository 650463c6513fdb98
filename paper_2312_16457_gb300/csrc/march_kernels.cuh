// march_kernels.cuh -- K1 ray marcher with in-register block compositor and the fused
// K3 deferred-MLP epilogue.
//
// Per pixel (Sec. 4.2 rendering stage):
//   for each selected block, near to far (App. D depth sort):
//     for each lattice sample of the ray inside the block (Eq. 4 membership)
//       skip it when its occupancy cell is empty (Sec. 4.1, Sec. 4.5)
//       f = trilinear(grid) + bilinear(xy) + bilinear(xz) + bilinear(yz)
//       sigma = exp(f0), alpha = 1 - exp(-sigma delta)            (Eq. 1)
//       C_d += T alpha sigmoid(f1..3), F += T alpha sigmoid(f4..7) (Eq. 2)
//       T *= 1 - alpha
//   Carrying T across blocks is Eq. 12 with Eq. 13 (1 - alpha^k equals the
//   product of the block's (1 - alpha_i)), so no per-block partials exist.
//   C = C_d + sigmoid(MLP(C_d, F, d))                                (Eq. 3)
#pragma once

#include "cow_common.cuh"
#include "cow_kernels.h"
#include "kernel_launch.h"
#include "march_core.cuh"
#include "march_warp.cuh"

#ifndef COW_MARCH_MIN_BLOCKS
#define COW_MARCH_MIN_BLOCKS 4
#endif
#ifndef COW_MARCH_MIN_BLOCKS_W
#define COW_MARCH_MIN_BLOCKS_W 4
#endif
#ifndef COW_RAYS_MIN_BLOCKS
#define COW_RAYS_MIN_BLOCKS COW_MARCH_MIN_BLOCKS  // 3 or 5 measured slower on random rays, FP32 and BF16
#endif
#ifndef COW_WARP_W
#define COW_WARP_W 8  // pixels per warp row (the warp covers COW_WARP_W x 32/COW_WARP_W pixels)
#endif

namespace cow {

namespace {

constexpr int kTileW = 16, kTileH = 8, kThreads = 128;
constexpr int kWarpW = COW_WARP_W, kWarpH = 32 / kWarpW;  // one ray per thread: a warp's pixel patch
static_assert(kTileW % kWarpW == 0 && kTileH % kWarpH == 0 && (kTileW / kWarpW) * (kTileH / kWarpH) == kThreads / 32,
              "the CTA tile is an exact grid of warp patches");
constexpr int kMinBlocks = COW_MARCH_MIN_BLOCKS;  // CTAs per SM the register budget is sized for
constexpr int kMinBlocksW = COW_MARCH_MIN_BLOCKS_W;
constexpr int kMaxSmemRecs = 96;                  // block records a CTA stages in shared memory
constexpr unsigned kWaitPolls = 1u << 24;         // bound on mbarrier polls

__device__ __forceinline__ void write_outputs(const MarchArgs &a, int64_t row, const RayState &s, const float d[3],
                                              const float *w_mlp) {
    float x[10] = {s.Cd[0], s.Cd[1], s.Cd[2], s.F[0], s.F[1], s.F[2], s.F[3], d[0], d[1], d[2]};
    float o[3];
    deferred_mlp(w_mlp, x, (a.flags & 1u) != 0, o);
    float *rgb = a.out_rgb + 3 * row;
    rgb[0] = s.Cd[0] + o[0];
    rgb[1] = s.Cd[1] + o[1];
    rgb[2] = s.Cd[2] + o[2];
    if (a.out_aux) {
        float4 *ap = reinterpret_cast<float4 *>(a.out_aux + 8 * row);
        ap[0] = make_float4(s.Cd[0], s.Cd[1], s.Cd[2], s.F[0]);
        ap[1] = make_float4(s.F[1], s.F[2], s.F[3], s.T);
    }
    if (a.out_nsamp) a.out_nsamp[row] = s.nsamp;
}

// View of a tile: views are ordered by tile_begin.
__device__ __forceinline__ int view_of_tile(const MarchArgs &a, int tile) {
    int lo = 0, hi = a.n_views - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.views[mid].tile_begin <= tile) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Per-block MLP form (Eq. 5 with Eq. 3 per block): every block is marched
// from an in-block transmittance of 1 (its C_d^k, F^k and 1 - alpha^k, Eq. 1-2
// / Eq. 11), a block with occupied samples adds T C^k with its own MLP, and
// T carries the product of the blocks' 1 - alpha^k.  Early termination uses
// the ray's total transmittance: inside block k it stops once
// T_k < ert_eps / T.  rec_at(k) / mlp_at(k): the k-th block's record and
// MLP weights in near-to-far order; state(k): where the k-th block's state
// goes (a.out_block_state, ray mode), or null.
template <int DT, class RecAt, class MlpAt, class StateAt>
__device__ __forceinline__ void blend_blocks(const MarchArgs &a, int n_blk, RecAt rec_at, MlpAt mlp_at,
                                             StateAt state, const float o[3], const float d[3],
                                             const float inv_d[3], float omax, int64_t row) {
    float C[3] = {0.f, 0.f, 0.f}, Cd[3] = {0.f, 0.f, 0.f}, F[4] = {0.f, 0.f, 0.f, 0.f}, T = 1.f;
    int nsamp = 0;
    for (int k = 0; k < n_blk; k++) {
        RayState sb = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, 1.f, 0, false};
        march_block<DT>(rec_at(k), o, d, inv_d, omax, a.ert_eps > 0.f ? a.ert_eps / T : 0.f, sb, a.err);
        if (float *e = state(k)) {
            const bool any = sb.nsamp > 0;
            float4 *e4 = reinterpret_cast<float4 *>(e);
            e4[0] = any ? make_float4(sb.Cd[0], sb.Cd[1], sb.Cd[2], sb.F[0]) : make_float4(0.f, 0.f, 0.f, 0.f);
            e4[1] = any ? make_float4(sb.F[1], sb.F[2], sb.F[3], T) : make_float4(0.f, 0.f, 0.f, -1.f);
        }
        if (sb.nsamp == 0) continue;
        float phi[3];
        block_mlp(mlp_at(k), a.n_freq, sb.Cd, sb.F, d, phi);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            C[c] = fmaf(T, sb.Cd[c] + phi[c], C[c]);
            Cd[c] = fmaf(T, sb.Cd[c], Cd[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; c++) F[c] = fmaf(T, sb.F[c], F[c]);
        T *= sb.T;
        nsamp += sb.nsamp;
        if (sb.done) break;
    }
    float *rgb = a.out_rgb + 3 * row;
    rgb[0] = C[0];
    rgb[1] = C[1];
    rgb[2] = C[2];
    if (a.out_aux) {
        float4 *ap = reinterpret_cast<float4 *>(a.out_aux + 8 * row);
        ap[0] = make_float4(Cd[0], Cd[1], Cd[2], F[0]);
        ap[1] = make_float4(F[1], F[2], F[3], T);
    }
    if (a.out_nsamp) a.out_nsamp[row] = nsamp;
}

template <int DT>
__device__ __forceinline__ void march_blocks_blend(const MarchArgs &a, const ViewRec &v, const BlockRec *recs,
                                                   const float o[3], const float d[3], const float inv_d[3],
                                                   float omax, int64_t row) {
    blend_blocks<DT>(
        a, v.ids_count, [&](int k) -> const BlockRec & { return recs[k]; },
        [&](int k) { return a.block_mlps[v.ids_begin + k]; }, [](int) -> float * { return nullptr; }, o, d, inv_d,
        omax, row);
}

// One ray per thread of the tile: march the view's near-to-far block list
// recs[0 .. ids_count) and write the pixel.
template <int DT, bool kBlockMlp>
__device__ __forceinline__ void march_tile_rays(const MarchArgs &a, const ViewRec &v, const BlockRec *recs, int tile,
                                                const float *s_mlp) {
    const int t = tile - v.tile_begin;
    int tx, ty;
    tile_xy(v, t, kTileH, tx, ty);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kWarpsX = kTileW / kWarpW;
    const int px = tx * kTileW + (warp % kWarpsX) * kWarpW + (lane % kWarpW);
    const int py = ty * kTileH + (warp / kWarpsX) * kWarpH + (lane / kWarpW);
    if (px >= v.W || py >= v.H) return;
    float o[3], d[3], inv_d[3], omax;
    pixel_ray(v, px, py, o, d);
    ray_setup(d, o, inv_d, omax);
    const int64_t row = v.pix_offset + (int64_t)py * v.W + px;
    if (kBlockMlp) {
        march_blocks_blend<DT>(a, v, recs, o, d, inv_d, omax, row);
        return;
    }
    RayState s = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, 1.f, 0, false};
    const int n_blk = v.ids_count;
    for (int k = 0; k < n_blk && !s.done; k++) march_block<DT>(recs[k], o, d, inv_d, omax, a.ert_eps, s, a.err);
    write_outputs(a, row, s, d, s_mlp);
}

// Thread schedule, block records in shared memory.
template <int DT, bool kBlockMlp>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_march_views(MarchArgs a) {
    __shared__ float s_mlp[kMlpParams + 1];
    extern __shared__ __align__(16) unsigned char s_dyn[];  // a.smem_recs block records
    BlockRec *s_rec = reinterpret_cast<BlockRec *>(s_dyn);
    __shared__ alignas(8) uint64_t s_bar;
    const int tile = blockIdx.x;
    const ViewRec &v = a.views[view_of_tile(a, tile)];
    const int n_blk = v.ids_count;
    const bool staged = n_blk > 0 && n_blk <= a.smem_recs;
    if (threadIdx.x == 0 && staged) mbar_init(&s_bar, 1);
    if (!kBlockMlp) load_mlp(a.mlp, s_mlp, (a.flags & 1u) != 0);
    __syncthreads();
    // the view's block records (near to far) go to shared memory by one TMA
    // bulk copy.  A wait that runs out records kErrTimeout and waits once more
    // (bounded) for the copy; if that also runs out the CTA leaves without
    // touching the records (the copy would then still be writing this CTA's
    // shared memory: two waits of 2^24 polls each, seconds, never seen short
    // of a stalled copy engine).
    if (staged) {
        const unsigned polls = a.wait_polls ? a.wait_polls : kWaitPolls;
        if (threadIdx.x == 0 && !(a.test_flags & kTestSkipRecordCopy))
            bulk_copy_g2s(s_rec, a.recs + v.ids_begin, (unsigned)(n_blk * sizeof(BlockRec)), &s_bar);
        if (!mbar_wait(&s_bar, 0, polls)) {
            atomicOr(a.err, kErrTimeout);
            if (!mbar_wait(&s_bar, 0, polls)) return;  // copy still in flight: leave without touching it
        }
    }
    march_tile_rays<DT, kBlockMlp>(a, v, staged ? s_rec : a.recs + v.ids_begin, tile, s_mlp);
}

// Thread schedule, block records in the launch's parameter buffer: the
// record fields the sample loop re-reads then come through the constant
// cache instead of taking shared-memory wavefronts from the L1 data pipe
// that the feature gathers are bound by.
template <int DT, bool kBlockMlp>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_march_views_c(const __grid_constant__ MarchArgs a, const __grid_constant__ ParamRecs pr) {
    __shared__ float s_mlp[kMlpParams + 1];
    const int tile = blockIdx.x;
    const ViewRec &v = a.views[view_of_tile(a, tile)];
    if (!kBlockMlp) {
        load_mlp(a.mlp, s_mlp, (a.flags & 1u) != 0);
        __syncthreads();
    }
    march_tile_rays<DT, kBlockMlp>(a, v, pr.r + v.ids_begin, tile, s_mlp);
}

// ---------------------------------------------------------------------------
// One ray per warp (march_warp.cuh).

// Outputs of the warp's ray: lane c < 7 holds channel c.
__device__ __forceinline__ void write_outputs_warp(const MarchArgs &a, int64_t row, float acc, float T, int nsamp,
                                                   float rgb) {
    const int lane = threadIdx.x & 31;
    if (lane < 3) a.out_rgb[3 * row + lane] = rgb;
    if (a.out_aux && lane < 8) a.out_aux[8 * row + lane] = lane < 7 ? acc : T;
    if (a.out_nsamp && lane == 0) a.out_nsamp[row] = nsamp;
}

__device__ __forceinline__ void shade_and_write(const MarchArgs &a, int64_t row, const WarpRay &s, const float d[3],
                                                const float *s_mlp) {
    float x[10];
#pragma unroll
    for (int c = 0; c < 7; c++) x[c] = __shfl_sync(kFullMask, s.acc, c);
#pragma unroll
    for (int c = 0; c < 3; c++) x[7 + c] = d[c];
    const float out = deferred_mlp_warp(s_mlp, x, (a.flags & 1u) != 0);
    write_outputs_warp(a, row, s.acc, s.T, s.nsamp, s.acc + out);
}

// blend_blocks for the warp's ray.  state(k): where the k-th block's state
// goes (written for the blocks that are marched), or null.
template <int DT, class RecAt, class MlpAt, class StateAt>
__device__ __forceinline__ void blend_blocks_warp(WarpScratch &ws, const MarchArgs &a, int n_blk, RecAt rec_at,
                                                  MlpAt mlp_at, StateAt state, const float o[3], const float d[3],
                                                  const float inv_d[3], float omax, int64_t row) {
    const int lane = threadIdx.x & 31;
    float C = 0.f, CF = 0.f, T = 1.f;
    int nsamp = 0;
    for_each_hit(n_blk, rec_at, o, d, inv_d, [&](int k) {
        WarpRay sb;
        march_block_warp<DT>(ws, rec_at(k), o, d, inv_d, omax, a.ert_eps > 0.f ? a.ert_eps / T : 0.f, sb, a.err);
        if (sb.nsamp == 0) return true;
        if (float *e = state(k))
            if (lane < 8) e[lane] = lane < 7 ? sb.acc : T;
        const float phi = block_mlp_warp(mlp_at(k), a.n_freq, sb.acc, d);
        C = fmaf(T, sb.acc + phi, C);
        CF = fmaf(T, sb.acc, CF);
        T *= sb.T;
        nsamp += sb.nsamp;
        return !sb.done;
    });
    write_outputs_warp(a, row, CF, T, nsamp, C);
}

// The ray form, one ray per thread, where that is the faster one (ray_form in
// cow_api.cu): the gathers of a camera's rays share lines in the given order, as
// the view marcher's do.
template <int DT, bool kBlockMlp>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_march_rays_t(const __grid_constant__ MarchArgs a,
                                                                       const __grid_constant__ RayRecs rr) {
    __shared__ float s_mlp[kMlpParams + 1];
    bool given;
    if (!thread_form(a, given)) return;
    if (!kBlockMlp) {
        load_mlp(a.mlp, s_mlp, (a.flags & 1u) != 0);
        __syncthreads();
    }
    float o[3], d[3];
    const int64_t r = load_ray(a, (int64_t)blockIdx.x * kThreads + threadIdx.x, given, o, d);
    if (r < 0) return;
    int order[kMaxRayIds];
    const int n = sort_blocks_for_ray(rr, o, order);
    float inv_d[3], omax;
    ray_setup(d, o, inv_d, omax);
    if (kBlockMlp) {
        blend_blocks<DT>(
            a, n, [&](int k) -> const BlockRec & { return rr.r[order[k]]; },
            [&](int k) { return a.block_mlp_base + (int64_t)rr.id[order[k]] * a.block_mlp_stride; },
            [&](int k) -> float * {
                return a.out_block_state ? a.out_block_state + 8 * (r * n + order[k]) : nullptr;
            },
            o, d, inv_d, omax, r);
        return;
    }
    RayState s = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, 1.f, 0, false};
    if (a.out_block_T) {  // no early termination (k_march_rays)
        float *bt = a.out_block_T + r * n;
        for (int k = 0; k < n; k++) {
            DepthSum tau;
            const int n0 = s.nsamp;
            march_block<DT>(rr.r[order[k]], o, d, inv_d, omax, a.ert_eps, s, a.err, &tau);
            bt[order[k]] = s.nsamp > n0 ? tau.transmittance() : -1.f;
        }
    } else {
        for (int k = 0; k < n && !s.done; k++)
            march_block<DT>(rr.r[order[k]], o, d, inv_d, omax, a.ert_eps, s, a.err);
    }
    write_outputs(a, r, s, d, s_mlp);
}

template <int DT, bool kBlockMlp>
__global__ void __launch_bounds__(kThreads, COW_RAYS_MIN_BLOCKS) k_march_rays(const __grid_constant__ MarchArgs a,
                                                                          const __grid_constant__ RayRecs rr) {
    __shared__ float s_mlp[kMlpParams + 1];
    __shared__ WarpScratch s_ws[kThreads / 32];
    if (rays_alike(a)) return;  // the thread form has them
    if (!kBlockMlp) {
        load_mlp(a.mlp, s_mlp, (a.flags & 1u) != 0);
        __syncthreads();
    }
    WarpScratch &ws = s_ws[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    float o[3], d[3], inv_d[3], omax;
    const int64_t r = load_ray_warp(a, first_ray(), o, d);
    if (r < 0) return;
    ray_setup(d, o, inv_d, omax);
    // per-ray depth order: xy distance of block centres to this origin (App. D)
    const int n = sort_blocks_warp(ws, rr, o);
    auto rec_at = [&](int k) -> const BlockRec & { return rr.r[ws.ord[k]]; };
    if (kBlockMlp) {  // Eq. 5 with block id's own MLP at block_mlp_base + id * block_mlp_stride
        float *bs = a.out_block_state ? a.out_block_state + 8 * r * n : nullptr;
        if (bs) {  // blocks without an occupied sample
            for (int k = lane; k < 8 * n; k += 32) bs[k] = (k & 7) == 7 ? -1.f : 0.f;
            __syncwarp();
        }
        blend_blocks_warp<DT>(
            ws, a, n, rec_at,
            [&](int k) { return a.block_mlp_base + (int64_t)rr.id[ws.ord[k]] * a.block_mlp_stride; },
            [&](int k) -> float * { return bs ? bs + 8 * ws.ord[k] : nullptr; }, o, d, inv_d, omax, r);
        return;
    }
    WarpRay s;
    if (a.out_block_T) {
        // also every block's own transmittance, at its position in ids; -1
        // for a block without occupied samples (the call has no early
        // termination, so every block is marched)
        float *bt = a.out_block_T + r * n;
        for (int k = lane; k < n; k += 32) bt[k] = -1.f;
        __syncwarp();
        for_each_hit(n, rec_at, o, d, inv_d, [&](int k) {
            float tb = 1.f;
            const int n0 = s.nsamp;
            march_block_warp<DT>(ws, rec_at(k), o, d, inv_d, omax, a.ert_eps, s, a.err, &tb);
            if (lane == 0 && s.nsamp > n0) bt[ws.ord[k]] = tb;
            return true;
        });
    } else {
        for_each_hit(n, rec_at, o, d, inv_d, [&](int k) {
            march_block_warp<DT>(ws, rec_at(k), o, d, inv_d, omax, a.ert_eps, s, a.err);
            return !s.done;
        });
    }
    shade_and_write(a, r, s, d, s_mlp);
}

// Block-parallel form, first half: every block of the call marched on its
// own from an in-block transmittance of 1 (Eq. 11: C_d^k, F^k and T^k =
// 1 - alpha^k of block k alone), written as 8 floats per (ray, block) in
// the order of the call's ids.  No early termination (a partial must not
// depend on the blocks in front of it).
template <int DT>
__global__ void __launch_bounds__(kThreads, COW_RAYS_MIN_BLOCKS) k_march_partials(const __grid_constant__ MarchArgs a,
                                                                              const __grid_constant__ RayRecs rr) {
    __shared__ WarpScratch s_ws[kThreads / 32];
    if (rays_alike(a)) return;
    WarpScratch &ws = s_ws[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    float o[3], d[3], inv_d[3], omax;
    const int64_t r = load_ray_warp(a, first_ray(), o, d);
    if (r < 0) return;
    ray_setup(d, o, inv_d, omax);
    float *pp = a.out_partials + 8 * r * rr.n;
    for (int k = lane; k < 8 * rr.n; k += 32) pp[k] = (k & 7) == 7 ? 1.f : 0.f;
    __syncwarp();
    for_each_hit(rr.n, [&](int k) -> const BlockRec & { return rr.r[k]; }, o, d, inv_d, [&](int k) {
        WarpRay s;
        march_block_warp<DT>(ws, rr.r[k], o, d, inv_d, omax, 0.f, s, a.err);
        if (lane < 8) pp[8 * k + lane] = lane < 7 ? s.acc : s.T;
        return true;
    });
}

// The same, one ray per thread.
template <int DT>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_march_partials_t(const __grid_constant__ MarchArgs a,
                                                                           const __grid_constant__ RayRecs rr) {
    bool given;
    if (!thread_form(a, given)) return;
    float o[3], d[3], inv_d[3], omax;
    const int64_t r = load_ray(a, (int64_t)blockIdx.x * kThreads + threadIdx.x, given, o, d);
    if (r < 0) return;
    ray_setup(d, o, inv_d, omax);
    for (int k = 0; k < rr.n; k++) {
        RayState s = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, 1.f, 0, false};
        march_block<DT>(rr.r[k], o, d, inv_d, omax, 0.f, s, a.err);
        float4 *pp = reinterpret_cast<float4 *>(a.out_partials + 8 * (r * rr.n + k));
        pp[0] = make_float4(s.Cd[0], s.Cd[1], s.Cd[2], s.F[0]);
        pp[1] = make_float4(s.F[1], s.F[2], s.F[3], s.T);
    }
}

// One ray per warp over a view's near-to-far block list.
template <int DT>
__device__ __forceinline__ WarpRay march_view_warp(WarpScratch &ws, const MarchArgs &a, int n_blk, const BlockRec *recs,
                                                   const float o[3], const float d[3], const float inv_d[3],
                                                   float omax) {
    WarpRay s;
    for_each_hit(n_blk, [&](int k) -> const BlockRec & { return recs[k]; }, o, d, inv_d, [&](int k) {
        march_block_warp<DT>(ws, recs[k], o, d, inv_d, omax, a.ert_eps, s, a.err);
        return !s.done;
    });
    return s;
}

template <int DT, bool kBlockMlp>
__device__ __forceinline__ void march_pixel_warp(WarpScratch &ws, const MarchArgs &a, const ViewRec &v,
                                                 const BlockRec *recs, int px, int py, const float *s_mlp) {
    if (px >= v.W || py >= v.H) return;  // uniform across the warp
    float o[3], d[3], inv_d[3], omax;
    pixel_ray(v, px, py, o, d);
    ray_setup(d, o, inv_d, omax);
    const int64_t row = v.pix_offset + (int64_t)py * v.W + px;
    if (kBlockMlp) {
        blend_blocks_warp<DT>(
            ws, a, v.ids_count, [&](int k) -> const BlockRec & { return recs[k]; }, [&](int k) { return a.block_mlps[v.ids_begin + k]; },
            [](int) -> float * { return nullptr; }, o, d, inv_d, omax, row);
        return;
    }
    const WarpRay s = march_view_warp<DT>(ws, a, v.ids_count, recs, o, d, inv_d, omax);
    shade_and_write(a, row, s, d, s_mlp);
}

// Small frames, records in the parameter buffer: a CTA takes a 2x2 patch of a
// 16x8 tile, one pixel per warp.
template <int DT, bool kBlockMlp>
__global__ void __launch_bounds__(kThreads, kMinBlocksW)
    k_march_views_cw(const __grid_constant__ MarchArgs a, const __grid_constant__ ParamRecs pr) {
    __shared__ float s_mlp[kMlpParams + 1];
    __shared__ WarpScratch s_ws[kThreads / 32];
    const int tile = blockIdx.x >> 5, sub = blockIdx.x & 31;
    const ViewRec &v = a.views[view_of_tile(a, tile)];
    int tx, ty;
    tile_xy(v, tile - v.tile_begin, kTileH, tx, ty);
    const int px0 = tx * kTileW + 2 * (sub & 7), py0 = ty * kTileH + 2 * (sub >> 3);
    if (px0 >= v.W || py0 >= v.H) return;
    if (!kBlockMlp) {
        load_mlp(a.mlp, s_mlp, (a.flags & 1u) != 0);
        __syncthreads();
    }
    const int warp = threadIdx.x >> 5;
    march_pixel_warp<DT, kBlockMlp>(s_ws[warp], a, v, pr.r + v.ids_begin, px0 + (warp & 1), py0 + (warp >> 1), s_mlp);
}

// COW_SCHED_WARP: the tile's rays one after another, 32 per warp, records in
// shared memory.  The MLPs run at the end, one ray a lane: an MLP on the whole warp
// after every ray took 3390 us for 1024x768 pixels of one block of 64^3 FP32, this
// 3168; 320x240 of 16 blocks of 128^3 3330 -> 3279 (BF16 2503 -> 2458), 720p 18.86 ->
// 18.57 ms (BF16 14.28 -> 13.97).
template <int DT>
__global__ void __launch_bounds__(kThreads, kMinBlocksW) k_march_views_w(MarchArgs a) {
    __shared__ float s_mlp[kMlpParams + 1];
    __shared__ WarpScratch s_ws[kThreads / 32];
    __shared__ float s_sum[kThreads / 32][32][9];  // odd stride: no bank conflicts
    __shared__ alignas(16) BlockRec s_rec[kMaxSmemRecs];
    __shared__ alignas(8) uint64_t s_bar;
    const int tile = blockIdx.x;
    const ViewRec &v = a.views[view_of_tile(a, tile)];
    const int n_blk = v.ids_count;
    const bool staged = n_blk > 0 && n_blk <= kMaxSmemRecs;
    if (threadIdx.x == 0 && staged) mbar_init(&s_bar, 1);
    load_mlp(a.mlp, s_mlp, (a.flags & 1u) != 0);
    __syncthreads();
    if (staged) {  // as in k_march_views
        const unsigned polls = a.wait_polls ? a.wait_polls : kWaitPolls;
        if (threadIdx.x == 0 && !(a.test_flags & kTestSkipRecordCopy))
            bulk_copy_g2s(s_rec, a.recs + v.ids_begin, (unsigned)(n_blk * sizeof(BlockRec)), &s_bar);
        if (!mbar_wait(&s_bar, 0, polls)) {
            atomicOr(a.err, kErrTimeout);
            if (!mbar_wait(&s_bar, 0, polls)) return;
        }
        __syncwarp();
    }
    const BlockRec *recs = staged ? s_rec : a.recs + v.ids_begin;
    int tx, ty;
    tile_xy(v, tile - v.tile_begin, kTileH, tx, ty);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int px0 = tx * kTileW + (warp & 1) * 8, py0 = ty * kTileH + (warp >> 1) * 4;
    WarpScratch &ws = s_ws[warp];
    float o[3], d[3];
    for (int q = 0; q < 32; q++) {
        const int px = px0 + (q & 7), py = py0 + (q >> 3);
        if (px >= v.W || py >= v.H) continue;  // uniform across the warp
        float inv_d[3], omax;
        pixel_ray(v, px, py, o, d);
        ray_setup(d, o, inv_d, omax);
        const WarpRay s = march_view_warp<DT>(ws, a, v.ids_count, recs, o, d, inv_d, omax);
        if (lane < 9) s_sum[warp][q][lane] = lane < 7 ? s.acc : lane == 7 ? s.T : __int_as_float(s.nsamp);
    }
    __syncwarp();
    const int px = px0 + (lane & 7), py = py0 + (lane >> 3);
    if (px >= v.W || py >= v.H) return;
    pixel_ray(v, px, py, o, d);
    const float *m = s_sum[warp][lane];
    const RayState s = {{m[0], m[1], m[2]}, {m[3], m[4], m[5], m[6]}, m[7], __float_as_int(m[8]), false};
    write_outputs(a, v.pix_offset + (int64_t)py * v.W + px, s, d, s_mlp);
}

template <int DT, bool kBlockMlp>
cudaError_t launch_thread(const MarchArgs &a, int n_tiles, bool in_params, cudaStream_t st, const ParamRecs *pr) {
    if (in_params) {
        k_march_views_c<DT, kBlockMlp><<<n_tiles, kThreads, 0, st>>>(a, *pr);
    } else {
        // records staged in dynamic shared memory sized to the largest view's
        // list (the driver then sizes the shared-memory carveout for full
        // occupancy and leaves the rest of the SM's 256 KB to L1)
        const size_t smem = (size_t)a.smem_recs * sizeof(BlockRec);
        k_march_views<DT, kBlockMlp><<<n_tiles, kThreads, smem, st>>>(a);
    }
    return cudaGetLastError();
}

}  // namespace

// Per-dtype launchers (explicitly instantiated by march.cu for the dense
// grids and by march_bricks.cu for the brick-sparse ones).
template <int DT>
cudaError_t launch_views_dt(const MarchArgs &a, int n_tiles, int schedule, cudaStream_t st, const ParamRecs *pr) {
    const bool block_mlp = a.block_mlps != nullptr;
    if (schedule == kSchedWarp && !block_mlp) {
        k_march_views_w<DT><<<n_tiles, kThreads, 0, st>>>(a);
        return cudaGetLastError();
    }
    const bool in_params = schedule == kSchedThreadConst;
    if (in_params && !pr) return cudaErrorInvalidValue;
    if (in_params && a.form == kFormWarp) {
        if (block_mlp) k_march_views_cw<DT, true><<<n_tiles * 32, kThreads, 0, st>>>(a, *pr);
        else k_march_views_cw<DT, false><<<n_tiles * 32, kThreads, 0, st>>>(a, *pr);
        return cudaGetLastError();
    }
    return block_mlp ? launch_thread<DT, true>(a, n_tiles, in_params, st, pr)
                     : launch_thread<DT, false>(a, n_tiles, in_params, st, pr);
}

// kFormWarp with a count of alike rays: both forms are launched, and the count
// decides on the device which of them returns at once.
template <int DT>
cudaError_t launch_rays_dt(const MarchArgs &a, const RayRecs &rr, cudaStream_t st) {
    const unsigned nw = (unsigned)((a.n_rays + kThreads / 32 - 1) / (kThreads / 32));
    const unsigned nt = (unsigned)((a.n_rays + kThreads - 1) / kThreads);
    if (a.form == kFormThread || a.ray_alike) {
        if (a.block_mlp_base) k_march_rays_t<DT, true><<<nt, kThreads, 0, st>>>(a, rr);
        else k_march_rays_t<DT, false><<<nt, kThreads, 0, st>>>(a, rr);
    }
    if (a.form == kFormThread) return cudaGetLastError();
    if (a.block_mlp_base) k_march_rays<DT, true><<<nw, kThreads, 0, st>>>(a, rr);
    else k_march_rays<DT, false><<<nw, kThreads, 0, st>>>(a, rr);
    return cudaGetLastError();
}

template <int DT>
cudaError_t launch_partials_dt(const MarchArgs &a, const RayRecs &rr, cudaStream_t st) {
    const unsigned nw = (unsigned)((a.n_rays + kThreads / 32 - 1) / (kThreads / 32));
    const unsigned nt = (unsigned)((a.n_rays + kThreads - 1) / kThreads);
    if (a.form == kFormThread || a.ray_alike) k_march_partials_t<DT><<<nt, kThreads, 0, st>>>(a, rr);
    if (a.form == kFormWarp) k_march_partials<DT><<<nw, kThreads, 0, st>>>(a, rr);
    return cudaGetLastError();
}

#define COW_INST_MARCH(D)                                                                                           \
    template cudaError_t launch_views_dt<(D)>(const MarchArgs &, int, int, cudaStream_t, const ParamRecs *);       \
    template cudaError_t launch_rays_dt<(D)>(const MarchArgs &, const RayRecs &, cudaStream_t);                    \
    template cudaError_t launch_partials_dt<(D)>(const MarchArgs &, const RayRecs &, cudaStream_t);

}  // namespace cow
