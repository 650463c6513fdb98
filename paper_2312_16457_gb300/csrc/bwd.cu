// bwd.cu -- K6 / K7: gradients of the rendered colour with respect to every
// grid, plane and deferred-MLP parameter, for the ray-batch form.
//
// Per ray, given g = dL/dC:
//   K7  recompute the deferred MLP (Eq. 3) from the forward's saved C_d, F and
//       back-propagate it: dL/dC_d = g + dPhi/dC_d^T g, dL/dF, and the ray's
//       contribution to dL/dW (outer products kept in shared memory).
//   K6  (one ray per warp, march_warp.cuh) re-march the ray over exactly the
//       forward's samples (same sequence code) with the transmittance T and the running prefix sums P_C, P_F;
//       the contribution of the samples after i is the saved total minus the
//       prefix, so no sample is stored.  With e = 1 - alpha = exp(-sigma delta)
//       and the weights of Eq. 1 (w_i = T_i alpha_i):
//         dL/dc_i  = w_i gC,   dL/ds_i = w_i gF
//         dL/dalpha_i = T_i (gC.c_i + gF.s_i) - (gC.S_C + gF.S_F) / e_i
//         dL/df0  = dL/dalpha_i * sigma delta e_i
//                 = sigma delta (T_i e_i (gC.c_i + gF.s_i) - (gC.S_C + gF.S_F))
//       (no division), then dL/df = dL/df0, c(1-c) dL/dc, s(1-s) dL/ds is
//       scattered with the interpolation weights to the 8 grid vertices and
//       12 plane texels (float4 reductions into FP32 gradient arrays in the
//       natural layout).
// K6's bound was the L2's rate of scattered reductions, 40 float4 a sample (one
// ray per thread: 130 ms for 2^20 random rays over 2x2 blocks of 128^3 FP32,
// 5.6e8 samples).  With a voxel's or texel's contributions added up before they
// are reduced (25.5 float4 a sample, counted) and the reductions in 64-byte groups
// it takes 65 ms, of which 35 are the reductions (timed without them); the rest
// is latency at 20 warps per SM (100000 of the rays: issue slots 42 % busy, L1 data
// pipe 73 %, L2 60 %).
// The CTA's MLP weight gradient (499 sums over its 128 rays) goes to a
// per-CTA scratch row; a second kernel adds the rows in a fixed order, so the
// MLP gradient does not depend on scheduling.
#include <algorithm>

#include "cow_common.cuh"
#include "cow_kernels.h"
#include "march_core.cuh"
#include "march_warp.cuh"

namespace cow {

namespace {

#ifndef COW_BWD_MIN_BLOCKS
// CTAs per SM the re-march's register budget is sized for: the 2^20-ray step
// took 142 ms at 2, 120 at 3, 107 at 4; with the present ray order 97.0 at 4 and
// 96.2 at 5, though that spills 16 to 40 bytes (100003 rays of the per-block MLP
// form 10.8 and 10.6 ms, 65537 BF16 rays 8.85 and 8.66 ms); 6 was slower
#define COW_BWD_MIN_BLOCKS 5
#endif

#ifndef COW_REG_MIN_BLOCKS
#define COW_REG_MIN_BLOCKS 4  // 6 and 8 measured the same
#endif

constexpr int kBwdThreads = kBwdCtaThreads;
constexpr int kBwdWarps = kBwdThreads / 32;
constexpr int kVec = 77;  // x (10), dz1 (16), h1 (16), dz2 (16), h2 (16), dz3 (3)

// Vector reduction without a returned value (red, not atom: a float4
// atomicAdd compiles to an atomic that returns the old value through L1, and
// those returns kept the backward's L1 pipe saturated).  16-byte aligned.
__device__ __forceinline__ void red_add4(float *dst, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

__device__ __forceinline__ void red_add1(float *dst, float a) {
    asm volatile("red.global.add.f32 [%0], %1;" ::"l"(dst), "f"(a) : "memory");
}

// One sample's feature gradient and where it goes, in shared memory while the
// warp scatters a chunk.
struct alignas(16) TapRec {
    float fr[3];        // place inside the voxel
    uint32_t base_lo;   // the voxel's first vertex
    float hf[3];        // places inside the texel cells along x, y, z
    uint32_t base_hi;
    uint32_t texel[3];  // first texel of the xy, xz, yz footprints
    float g0;           // gradient of channel 0
    float gf[8];        // of all eight
};

// Shared scratch of one warp of the re-march.
struct alignas(16) BwdScratch {
    WarpScratch w;
    float T[kRowPad];  // transmittance in front of the chunk's samples
    TapRec tap[32];
};

// Bits j of a chunk's first n samples after which a run of equal keys ends.
// `same`: this lane's key equals the previous lane's.
__device__ __forceinline__ unsigned run_ends(bool same, int n) {
    const unsigned starts = __ballot_sync(kFullMask, !same);
    return ((starts >> 1) | (1u << (n - 1))) & (kFullMask >> (32 - n));
}

// acc += w v over the four channels of a half
__device__ __forceinline__ void add_half(float2 acc[2], float w, const float4 &v) {
    const float2 w2 = make_float2(w, w);
    acc[0] = __ffma2_rn(w2, make_float2(v.x, v.y), acc[0]);
    acc[1] = __ffma2_rn(w2, make_float2(v.z, v.w), acc[1]);
}

__device__ __forceinline__ void flush_half(float *dst, float2 acc[2]) {
    red_add4(dst, acc[0].x, acc[0].y, acc[1].x, acc[1].y);
    acc[0] = acc[1] = make_float2(0.f, 0.f);
}

// Put lane j's sample (j < n; lookup coordinates rel and g, gradient gf) into
// tap[j]; ends: where the chunk's runs of samples in one voxel end, pends[k]:
// in one texel cell of plane k.
template <int NCH>
__device__ __forceinline__ void make_taps(const BlockRec &b, TapRec *tap, int n, const float rel[3], const float g[3],
                                          const float gf[NCH], unsigned &ends, unsigned pends[3]) {
    const int lane = threadIdx.x & 31;
    uint64_t base = 0;
    uint32_t tx[3] = {0, 0, 0};
    if (lane < n) {
        int c0[3], h0[3];
        float fr[3], hf[3];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            c0[a] = lookup_cell(g[a], b.R, fr[a]);
            h0[a] = lookup_cell(__fmul_rn(rel[a], b.kp[a]), b.P, hf[a]);
        }
        base = ((uint64_t)c0[2] * b.R + c0[1]) * b.R + c0[0];
        // below 2^32: a plane of more texels, with its gradient, exceeds the device
        tx[0] = (uint32_t)h0[1] * b.P + h0[0];
        tx[1] = (uint32_t)h0[2] * b.P + h0[0];
        tx[2] = (uint32_t)h0[2] * b.P + h0[1];
        float4 *o = reinterpret_cast<float4 *>(tap + lane);
        o[0] = make_float4(fr[0], fr[1], fr[2], __uint_as_float((uint32_t)base));
        o[1] = make_float4(hf[0], hf[1], hf[2], __uint_as_float((uint32_t)(base >> 32)));
        o[2] = make_float4(__uint_as_float(tx[0]), __uint_as_float(tx[1]), __uint_as_float(tx[2]), gf[0]);
        if constexpr (NCH == 8) {
            o[3] = make_float4(gf[0], gf[1], gf[2], gf[3]);
            o[4] = make_float4(gf[4], gf[5], gf[6], gf[7]);
        }
    }
    const uint64_t pbase = __shfl_up_sync(kFullMask, base, 1);
    ends = run_ends(pbase == base && lane > 0, n);
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const uint32_t ptx = __shfl_up_sync(kFullMask, tx[k], 1);
        pends[k] = run_ends(ptx == tx[k] && lane > 0, n);
    }
    __syncwarp();
}

// Scatter a chunk of n samples (lane j < n holds sample j's lookup coordinates
// and gradient gf) to the taps of their lookups, as a warp: a lane has one tap and one half
// of its eight channels, so the lanes of one reduction cover whole 64-byte
// vertex or texel pairs (the L2 takes 64-byte groups of float4 reductions 1.6
// times as fast as scattered ones: 330 against 205 G/s into 32 MiB, 147 against
// 46 G/s into 256 MiB), and it walks its samples in ray order, adding up what
// goes to one voxel or texel cell before it issues the reduction (a lattice
// step is about a quarter of a voxel, so a voxel takes some 2.5 samples).
__device__ __forceinline__ void scatter_chunk(const BlockRec &b, TapRec *tap, int n, const float rel[3],
                                              const float g[3], const float gf[8], float *gg, float *const gp[3]) {
    const int lane = threadIdx.x & 31;
    unsigned ends, pends[3];
    make_taps<8>(b, tap, n, rel, g, gf, ends, pends);
    // place q (0 or 1) of an axis: weight 1 - f or f, as s f + c
    const float s1 = (lane & 2) ? 1.f : -1.f, c1 = (lane & 2) ? 0.f : 1.f;
    const float s2 = (lane & 4) ? 1.f : -1.f, c2 = (lane & 4) ? 0.f : 1.f;
    const int half = 4 * (lane & 1);
    const bool a1 = lane & 2, a2 = lane & 4;
    if (gg) {  // two runs of samples, 16 lanes each: 8 vertices x 2 halves
        const float s3 = (lane & 8) ? 1.f : -1.f, c3 = (lane & 8) ? 0.f : 1.f;
        const int64_t R = b.R;
        float *const dst = gg + 8 * (((lane & 8 ? R : 0) + (a2 ? 1 : 0)) * R + (a1 ? 1 : 0)) + half;
        const int len = (n + 1) >> 1, j0 = (lane >> 4) * len;
        ends |= 1u << (len - 1);
        const unsigned mine = ends >> j0;
        const TapRec *t = tap + j0;
        float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 2
        for (int j = 0; j < len; j++) {
            const float4 f = *reinterpret_cast<const float4 *>(t[j].fr);
            const float4 v = *reinterpret_cast<const float4 *>(t[j].gf + half);
            add_half(acc, (fmaf(f.y, s2, c2) * fmaf(f.z, s3, c3)) * fmaf(f.x, s1, c1), v);
            if ((mine >> j) & 1u)
                flush_half(dst + 8 * ((uint64_t)t[j].base_hi << 32 | __float_as_uint(f.w)), acc);
        }
    }
    // four runs, 8 lanes each: per plane 4 texels x 2 halves
    const int len = (n + 3) >> 2, j0 = (lane >> 3) * len;
    const unsigned cuts = ((1u << (len - 1)) | (1u << (2 * len - 1)) | (1u << (3 * len - 1))) & (kFullMask >> (32 - n));
    const TapRec *t = tap + j0;
    const uint32_t off = (a2 ? b.P : 0) + (a1 ? 1 : 0);
    float2 acc[3][2];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        acc[k][0] = acc[k][1] = make_float2(0.f, 0.f);
        pends[k] = gp[k] ? (pends[k] | cuts) >> j0 : 0u;
    }
    for (int j = 0; j < len; j++) {
        const float4 h = *reinterpret_cast<const float4 *>(t[j].hf);
        const uint4 x = *reinterpret_cast<const uint4 *>(t[j].texel);
        const float4 v = *reinterpret_cast<const float4 *>(t[j].gf + half);
        const float u0 = fmaf(h.x, s1, c1), u1 = fmaf(h.y, s1, c1), v1 = fmaf(h.y, s2, c2), v2 = fmaf(h.z, s2, c2);
        add_half(acc[0], v1 * u0, v);
        add_half(acc[1], v2 * u0, v);
        add_half(acc[2], v2 * u1, v);
        if ((pends[0] >> j) & 1u) flush_half(gp[0] + 8 * (uint64_t)(x.x + off) + half, acc[0]);
        if ((pends[1] >> j) & 1u) flush_half(gp[1] + 8 * (uint64_t)(x.y + off) + half, acc[1]);
        if ((pends[2] >> j) & 1u) flush_half(gp[2] + 8 * (uint64_t)(x.z + off) + half, acc[2]);
    }
    __syncwarp();
}

// The same for the density channel alone: 8 lanes a run, one vertex each, then
// one texel of the xy and xz planes each; 4 lanes a run for the yz plane.
__device__ __forceinline__ void scatter_density_chunk(const BlockRec &b, TapRec *tap, int n, const float rel[3],
                                                      const float g[3], float g0, float *gg, float *const gp[3]) {
    const int lane = threadIdx.x & 31;
    unsigned ends, pends[3];
    make_taps<1>(b, tap, n, rel, g, &g0, ends, pends);
    const bool a0 = lane & 1, a1 = lane & 2, a2 = lane & 4;
    const float s0 = a0 ? 1.f : -1.f, c0 = a0 ? 0.f : 1.f, s1 = a1 ? 1.f : -1.f, c1 = a1 ? 0.f : 1.f;
    const unsigned all = kFullMask >> (32 - n);
    {
        const int len = (n + 3) >> 2, j0 = (lane >> 3) * len;
        const unsigned cuts = ((1u << (len - 1)) | (1u << (2 * len - 1)) | (1u << (3 * len - 1))) & all;
        const TapRec *t = tap + j0;
        if (gg) {
            const float s2 = a2 ? 1.f : -1.f, c2 = a2 ? 0.f : 1.f;
            const int64_t R = b.R;
            float *const dst = gg + 8 * (((a2 ? R : 0) + (a1 ? 1 : 0)) * R + (a0 ? 1 : 0));
            const unsigned mine = (ends | cuts) >> j0;
            float acc = 0.f;
#pragma unroll 2
            for (int j = 0; j < len; j++) {
                const float4 f = *reinterpret_cast<const float4 *>(t[j].fr);
                acc = fmaf((fmaf(f.y, s1, c1) * fmaf(f.z, s2, c2)) * fmaf(f.x, s0, c0), t[j].g0, acc);
                if ((mine >> j) & 1u) {
                    red_add1(dst + 8 * ((uint64_t)t[j].base_hi << 32 | __float_as_uint(f.w)), acc);
                    acc = 0.f;
                }
            }
        }
        // lanes with bit 2: the xz plane, the others: the xy plane
        if (float *const gq = a2 ? gp[1] : gp[0]) {
            const unsigned mine = ((a2 ? pends[1] : pends[0]) | cuts) >> j0;
            const uint32_t off = (a1 ? b.P : 0) + (a0 ? 1 : 0);
            float acc = 0.f;
#pragma unroll 2
            for (int j = 0; j < len; j++) {
                const float4 h = *reinterpret_cast<const float4 *>(t[j].hf);
                const float4 x = *reinterpret_cast<const float4 *>(t[j].texel);
                acc = fmaf(fmaf(a2 ? h.z : h.y, s1, c1) * fmaf(h.x, s0, c0), x.w, acc);
                if ((mine >> j) & 1u) {
                    red_add1(gq + 8 * (uint64_t)(__float_as_uint(a2 ? x.y : x.x) + off), acc);
                    acc = 0.f;
                }
            }
        }
    }
    if (gp[2]) {
        const int len = (n + 7) >> 3, j0 = (lane >> 2) * len;
        unsigned cuts = 0;
        for (int k = 1; k < 8; k++) cuts |= 1u << (k * len - 1);
        const unsigned mine = j0 < n ? (pends[2] | (cuts & all)) >> j0 : 0u;
        const TapRec *t = tap + min(j0, n - 1);
        const uint32_t off = (a1 ? b.P : 0) + (a0 ? 1 : 0);
        float acc = 0.f;
        for (int j = 0; j < len; j++) {
            if (j0 + j >= n) break;
            const float4 h = *reinterpret_cast<const float4 *>(t[j].hf);
            const float4 x = *reinterpret_cast<const float4 *>(t[j].texel);
            acc = fmaf(fmaf(h.z, s1, c1) * fmaf(h.y, s0, c0), x.w, acc);
            if ((mine >> j) & 1u) {
                red_add1(gp[2] + 8 * (uint64_t)(__float_as_uint(x.z) + off), acc);
                acc = 0.f;
            }
        }
    }
    __syncwarp();
}

// What the re-march of a ray carries from sample to sample: the transmittance
// (uniform) and, in lane q < 7, the prefix sum of channel q of (C_d, F).
struct BwdRay {
    float T = 1.f, pre = 0.f;
};

// Re-march the warp's ray through one block and scatter its feature gradients.
// gcf: dL/dC_d, dL/dF (uniform); total: the ray's (or the block's) final sum
// of lane q's channel; Q: what else depends on the samples' transmittance.
// Prefix and transmittance are taken in lattice order with the forward's
// operations, so total - prefix is exactly what the forward added after the
// sample.  Returns false when the ray ended early.
template <int DT>
__device__ __forceinline__ bool remarch_block(BwdScratch &bs, const BlockRec &b, const float o[3], const float d[3],
                                              const float inv_d[3], float omax, const float gcf[7], float total,
                                              float Q, float ert_eps, BwdRay &s, float *gg, float *const gp[3],
                                              unsigned *err) {
    const int lane = threadIdx.x & 31;
    WarpScratch &ws = bs.w;
    BrickCache bc;
    return for_each_chunk(ws, b, o, d, inv_d, omax, err, [&](bool active, int n, const float rel[3], const float g[3],
                                                             float delta) {
        float e = 1.f, sigma = 0.f, gdot = 0.f, c[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (active) {
            float2 f2[4];
            accumulate_sample<DT>(b, rel, g, f2, &bc);
            const float f[8] = {f2[0].x, f2[0].y, f2[1].x, f2[1].y, f2[2].x, f2[2].y, f2[3].x, f2[3].y};
            sigma = __expf(f[0]);
            e = __expf(-sigma * delta);
#pragma unroll
            for (int q = 0; q < 7; q++) {
                c[q] = sigmoidf_fast(f[1 + q]);
                gdot = fmaf(gcf[q], c[q], gdot);
            }
        }
#pragma unroll
        for (int q = 0; q < 7; q++) ws.row[q][lane] = c[q];
        ws.row[7][lane] = e;
        __syncwarp();
        float T = s.T;
        if (lane < 8) {  // lane q < 7: total - prefix after every sample, in place; lane 7: T in front of it
            float4 *x4 = reinterpret_cast<float4 *>(lane < 7 ? ws.row[lane] : bs.T);
            const float4 *e4 = reinterpret_cast<const float4 *>(ws.row[7]);
            float pre = s.pre;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                if (4 * k >= n) break;
                const float4 ee = e4[k], xx = lane < 7 ? x4[k] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float Ts[4] = {T, T * ee.x, (T * ee.x) * ee.y, ((T * ee.x) * ee.y) * ee.z};
                const float xv[4] = {xx.x, xx.y, xx.z, xx.w};
                float w[4], out[4];
                chunk_weights(ee, T, w);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    pre = fmaf(w[j], xv[j], pre);
                    out[j] = lane < 7 ? total - pre : Ts[j];
                }
                x4[k] = make_float4(out[0], out[1], out[2], out[3]);
            }
            s.pre = pre;
        }
        T = __shfl_sync(kFullMask, T, 0);
        bool more = true;
        int used = n;
        if (!(T >= ert_eps)) {  // the ray ends in this chunk, perhaps in front of a NaN
            float Ts = s.T;
            for (used = 0; used < n && more;) {
                Ts *= ws.row[7][used++];
                more = !(Ts < ert_eps);
            }
        }
        s.T = T;
        __syncwarp();
        float gf[8];
        {
            const float Tb = bs.T[lane], wt = Tb * (1.f - e);
            float sdot = Q;
#pragma unroll
            for (int q = 0; q < 7; q++) sdot = fmaf(gcf[q], ws.row[q][lane], sdot);
            gf[0] = sigma * delta * (Tb * e * gdot - sdot);
#pragma unroll
            for (int q = 0; q < 7; q++) gf[1 + q] = wt * gcf[q] * c[q] * (1.f - c[q]);
        }
        scatter_chunk(b, bs.tap, used, rel, g, gf, gg, gp);
        return more;
    });
}

// K7: deferred-MLP backward per ray; writes (dL/dC_d, dL/dF) of the ray to
// a.gcf (8 floats per ray) and the CTA's 499 weight-gradient sums to its row.
__global__ void __launch_bounds__(kBwdThreads) k_mlp_backward(BwdArgs a) {
    __shared__ float s_w[kMlpParams + 1];
    __shared__ float s_vec[kBwdThreads][kVec];
    for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) s_w[i] = __ldg(a.mlp + i);
    __syncthreads();
    const int64_t r = (int64_t)blockIdx.x * kBwdThreads + threadIdx.x;
    float *vec = s_vec[threadIdx.x];
    if (r >= a.n_rays) {
        for (int k = 0; k < kVec; k++) vec[k] = 0.f;
    } else {
        const float *w = s_w;
        float x[10], gC[3], gF[4];
#pragma unroll
        for (int c = 0; c < 7; c++) x[c] = __ldg(a.aux + 8 * r + c);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            x[7 + c] = __ldg(a.ray_d + 3 * r + c);
            gC[c] = __ldg(a.dL_drgb + 3 * r + c);
        }
        float dz3[3];
#pragma unroll 1
        for (int j = 0; j < 16; j++) {
            float s = w[kOffB1 + j];
#pragma unroll
            for (int i = 0; i < 10; i++) s = fmaf(x[i], w[kOffW1 + i * 16 + j], s);
            vec[26 + j] = fmaxf(s, 0.f);  // h1
        }
#pragma unroll 1
        for (int j = 0; j < 16; j++) {
            float s = w[kOffB2 + j];
#pragma unroll
            for (int i = 0; i < 16; i++) s = fmaf(vec[26 + i], w[kOffW2 + i * 16 + j], s);
            vec[58 + j] = fmaxf(s, 0.f);  // h2
        }
#pragma unroll
        for (int j = 0; j < 3; j++) {
            float s = w[kOffB3 + j];
#pragma unroll
            for (int i = 0; i < 16; i++) s = fmaf(vec[58 + i], w[kOffW3 + i * 3 + j], s);
            const float sg = 1.f / (1.f + expf(-s));
            dz3[j] = gC[j] * sg * (1.f - sg);
            vec[74 + j] = dz3[j];
        }
#pragma unroll 1
        for (int i = 0; i < 16; i++) {
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < 3; j++) s = fmaf(w[kOffW3 + i * 3 + j], dz3[j], s);
            vec[42 + i] = vec[58 + i] > 0.f ? s : 0.f;  // dz2 (h2 > 0 iff z2 > 0)
        }
#pragma unroll 1
        for (int i = 0; i < 16; i++) {
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < 16; j++) s = fmaf(w[kOffW2 + i * 16 + j], vec[42 + j], s);
            vec[10 + i] = vec[26 + i] > 0.f ? s : 0.f;  // dz1 (h1 > 0 iff z1 > 0)
        }
#pragma unroll 1
        for (int i = 0; i < 7; i++) {
            float s = 0.f;
#pragma unroll
            for (int j = 0; j < 16; j++) s = fmaf(w[kOffW1 + i * 16 + j], vec[10 + j], s);
            if (i < 3) gC[i] += s;
            else gF[i - 3] = s;
        }
#pragma unroll
        for (int k = 0; k < 10; k++) vec[k] = x[k];
        float4 *out = reinterpret_cast<float4 *>(a.gcf + 8 * r);
        out[0] = make_float4(gC[0], gC[1], gC[2], gF[0]);
        out[1] = make_float4(gF[1], gF[2], gF[3], 0.f);
    }
    __syncthreads();
    // MLP weight gradient of this CTA's rays -> its scratch row
    float *row = a.partials + (int64_t)blockIdx.x * kMlpParams;
    for (int t = threadIdx.x; t < kMlpParams; t += blockDim.x) {
        int ia, ib;  // vec offsets of the two factors; ia < 0: bias (single factor)
        if (t < kOffB1) { ia = t / 16; ib = 10 + t % 16; }
        else if (t < kOffW2) { ia = -1; ib = 10 + (t - kOffB1); }
        else if (t < kOffB2) { ia = 26 + (t - kOffW2) / 16; ib = 42 + (t - kOffW2) % 16; }
        else if (t < kOffW3) { ia = -1; ib = 42 + (t - kOffB2); }
        else if (t < kOffB3) { ia = 58 + (t - kOffW3) / 3; ib = 74 + (t - kOffW3) % 3; }
        else { ia = -1; ib = 74 + (t - kOffB3); }
        float s = 0.f;
        for (int q = 0; q < kBwdThreads; q++) s = fmaf(ia >= 0 ? s_vec[q][ia] : 1.f, s_vec[q][ib], s);
        row[t] = s;
    }
}

// K6: re-march and scatter the feature gradients, one ray per warp.
template <int DT>
__global__ void __launch_bounds__(kBwdThreads, COW_BWD_MIN_BLOCKS) k_remarch_backward(
    const __grid_constant__ BwdArgs a, const __grid_constant__ RayRecs rr) {
    __shared__ BwdScratch s_bs[kBwdWarps];
    BwdScratch &bs = s_bs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    float o[3], d[3], inv_d[3], omax;
    const int64_t r = load_ray_warp(a, first_ray(), o, d);
    if (r < 0) return;
    ray_setup(d, o, inv_d, omax);
    float gcf[7];
#pragma unroll
    for (int q = 0; q < 7; q++) gcf[q] = __ldg(a.gcf + 8 * r + q);
    const float total = __ldg(a.aux + 8 * r + (lane & 7));
    const int n = sort_blocks_warp(bs.w, rr, o);
    BwdRay s;
    for_each_hit(n, [&](int k) -> const BlockRec & { return rr.r[bs.w.ord[k]]; }, o, d, inv_d, [&](int k) {
        const int id = rr.id[bs.w.ord[k]];
        float *const gp[3] = {a.grad_planes[3 * id], a.grad_planes[3 * id + 1], a.grad_planes[3 * id + 2]};
        return remarch_block<DT>(bs, rr.r[bs.w.ord[k]], o, d, inv_d, omax, gcf, total, 0.f, a.ert_eps, s,
                                 a.grad_grid[id], gp, a.err);
    });
}

// ---------------------------------------------------------------------------
// Training-stage regularisers (Sec. 4.3).
//   Sparsity (Eq. 7): alpha(p) = 1 - exp(-sigma(p) delta_b) at given points,
//     in the block containing p (Eq. 4, first in ids); loss += weight/n alpha,
//     d alpha / d f0 = sigma delta (1 - alpha).
//   Opacity (Eq. 8): per ray and block with occupied samples, alpha^k =
//     1 - prod (1 - alpha_i); loss += weight/n H(clamp(alpha^k)) with H the
//     binary entropy and the clamp to [1e-6, 1 - 1e-6];
//     d alpha^k / d f0_i = sigma_i delta (1 - alpha^k).  The block is marched
//     once for alpha^k -- or alpha^k comes from the forward's in-block
//     transmittance -- and once to scatter.
// Gradients reach the density channel only: 20 scalar reductions per point or
// sample (8 grid vertices, 4 texels of each plane), in the opacity term added
// up per voxel and texel cell first.

__device__ __forceinline__ void scatter_ch0(const BlockRec &b, float *gg, float *const gp[3], const float rel[3],
                                            const float g[3], float g0) {
    if (gg) {
        float fr[3];
        int c0[3];
#pragma unroll
        for (int a = 0; a < 3; a++) c0[a] = lookup_cell(g[a], b.R, fr[a]);
        const int64_t R = b.R;
        const int64_t base = (c0[2] * R + c0[1]) * R + c0[0];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
            const float w = (dy ? fr[1] : 1.f - fr[1]) * (dz ? fr[2] : 1.f - fr[2]) * (dx ? fr[0] : 1.f - fr[0]);
            red_add1(gg + 8 * (base + (dz * R + dy) * R + dx), w * g0);
        }
    }
    float hf[3];
    int h0[3];
#pragma unroll
    for (int a = 0; a < 3; a++) h0[a] = lookup_cell(__fmul_rn(rel[a], b.kp[a]), b.P, hf[a]);
    const int64_t P = b.P;
#pragma unroll
    for (int pl = 0; pl < 3; pl++) {
        if (!gp[pl]) continue;
        const int ua = pl == 2 ? 1 : 0, va = pl == 0 ? 1 : 2;
        const int64_t tb = (int64_t)h0[va] * P + h0[ua];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int du = q & 1, dv = q >> 1;
            const float w = (dv ? hf[va] : 1.f - hf[va]) * (du ? hf[ua] : 1.f - hf[ua]);
            red_add1(gp[pl] + 8 * (tb + dv * P + du), w * g0);
        }
    }
}

// sum of v over the CTA, in thread 0
__device__ __forceinline__ float cta_sum(float v) {
    __shared__ float s_part[32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = threadIdx.x < (blockDim.x >> 5) ? s_part[threadIdx.x] : 0.f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    }
    return v;
}

template <int DT>
__global__ void __launch_bounds__(kBwdThreads) k_sparsity(RegArgs a, const __grid_constant__ RayRecs rr) {
    const int64_t r = (int64_t)blockIdx.x * kBwdThreads + threadIdx.x;
    float term = 0.f;
    if (r < a.n_rays) {
        const float p[3] = {__ldg(a.pts + 3 * r), __ldg(a.pts + 3 * r + 1), __ldg(a.pts + 3 * r + 2)};
        int pos = -1;
        for (int k = 0; k < rr.n && pos < 0; k++) {
            const BlockRec &bc = rr.r[k];
            if ((bc.unb & kUnbContracted) ? owned_unbounded(bc, p) : inside_block(bc, p)) pos = k;
        }
        if (pos >= 0) {
            const int id = rr.id[pos];
            const BlockRec &b = rr.r[pos];
            float q[3], g[3];
            lookup_coords(b, p, q, g);
            float2 f2[4];
            accumulate_sample<DT>(b, q, g, f2);
            const float sigma = expf(f2[0].x);
            const float alpha = -expm1f(-sigma * b.delta);
            const float scale = a.weight / (float)a.n_rays;
            term = scale * alpha;
            if (a.grad_grid) {
                float *const gp[3] = {a.grad_planes[3 * id], a.grad_planes[3 * id + 1], a.grad_planes[3 * id + 2]};
                scatter_ch0(b, a.grad_grid[id], gp, q, g, scale * sigma * b.delta * (1.f - alpha));
            }
        }
    }
    term = cta_sum(term);
    if (threadIdx.x == 0 && a.loss) atomicAdd(a.loss, term);
}

// One (ray, block)'s share of the loss, from alpha^k.
constexpr float kAlphaEps = 1e-6f;
__device__ __forceinline__ float opacity_term(const RegArgs &a, float a_raw) {
    const float al = fminf(fmaxf(a_raw, kAlphaEps), 1.f - kAlphaEps);
    return -(a.weight / (float)a.n_rays) * (al * logf(al) + (1.f - al) * log1pf(-al));
}

// Opacity, one ray per warp: 9.9 scalar reductions a sample instead of 20 (65537
// BF16 rays: a training step of 8.4 ms, 12.1 ms with one ray per thread), then
// bound by latency (issue slots 26 % busy, L1 data pipe 56 %, L2 42 %).
template <int DT>
__global__ void __launch_bounds__(kBwdThreads, COW_REG_MIN_BLOCKS) k_opacity(const __grid_constant__ RegArgs a,
                                                                          const __grid_constant__ RayRecs rr) {
    __shared__ BwdScratch s_bs[kBwdWarps];
    BwdScratch &bs = s_bs[threadIdx.x >> 5];
    WarpScratch &ws = bs.w;
    const int lane = threadIdx.x & 31;
    float term = 0.f;
    const float scale = a.weight / (float)a.n_rays, eps = kAlphaEps;
    bool given;
    const bool marched = thread_form(a, given);  // by k_opacity_t: into out_T, or to the term itself
    const int64_t n_rays = marched && !a.out_T ? 0 : a.n_rays;
    const float *block_T = marched ? a.out_T : a.block_T;
    for (int64_t ray = first_ray(); ray < n_rays; ray += (int64_t)gridDim.x * kBwdWarps) {
        float o[3], d[3], inv_d[3], omax;
        const int64_t r = load_ray_warp(a, ray, o, d);
        ray_setup(d, o, inv_d, omax);
        __syncwarp();
        const int n = sort_blocks_warp(ws, rr, o);
        for_each_hit(n, [&](int k) -> const BlockRec & { return rr.r[ws.ord[k]]; }, o, d, inv_d, [&](int k) {
            const int pos = ws.ord[k], id = rr.id[pos];
            const BlockRec &b = rr.r[pos];
            float T = 1.f;
            if (block_T) {  // the forward's in-block transmittance, or k_opacity_t's
                T = __ldg(block_T + r * rr.n + pos);
                if (T < 0.f) return true;  // no occupied sample
            } else {
                int nk = 0;
                float tau = 0.f;  // this lane's samples (march_block_warp)
                BrickCache bc;
                for_each_chunk(ws, b, o, d, inv_d, omax, a.err,
                               [&](bool active, int m, const float rel[3], const float g[3], float delta) {
                    if (active) {
                        float2 f2[4];
                        accumulate_sample<DT>(b, rel, g, f2, &bc);
                        tau += expf(f2[0].x) * delta;
                    }
                    nk += m;
                    return true;
                });
                T = expf(-warp_sum(tau));
                if (nk == 0) return true;
            }
            const float a_raw = 1.f - T;
            const float al = fminf(fmaxf(a_raw, eps), 1.f - eps);
            term += opacity_term(a, a_raw);
            if (!a.grad_grid || !(a_raw > eps && a_raw < 1.f - eps)) return true;
            const float ga = -scale * (logf(al) - log1pf(-al));  // d loss / d alpha^k
            float *const gp[3] = {a.grad_planes[3 * id], a.grad_planes[3 * id + 1], a.grad_planes[3 * id + 2]};
            BrickCache bc;
            for_each_chunk(ws, b, o, d, inv_d, omax, a.err,
                           [&](bool active, int m, const float rel[3], const float g[3], float delta) {
                float g0 = 0.f;
                if (active) {
                    float2 f2[4];
                    accumulate_sample<DT>(b, rel, g, f2, &bc);
                    g0 = ga * expf(f2[0].x) * delta * T;
                }
                scatter_density_chunk(b, bs.tap, m, rel, g, g0, a.grad_grid[id], gp);
                return true;
            });
            return true;
        });
    }
    term = cta_sum(lane == 0 ? term : 0.f);
    if (threadIdx.x == 0) a.loss_parts[blockIdx.x] = term;
}

// Its first march, one ray per thread (ray_form in cow_api.cu): the blocks' own
// transmittances go to out_T, for k_opacity to scatter from, or, without a
// gradient, the term is taken at once, its parts behind k_opacity's.
template <int DT>
__global__ void __launch_bounds__(kBwdThreads, COW_REG_MIN_BLOCKS) k_opacity_t(const __grid_constant__ RegArgs a,
                                                                            const __grid_constant__ RayRecs rr) {
    float term = 0.f;
    bool given;
    const int64_t n_rays = thread_form(a, given) ? a.n_rays : 0;
    for (int64_t ray = (int64_t)blockIdx.x * kBwdThreads + threadIdx.x; ray < n_rays;
         ray += (int64_t)gridDim.x * kBwdThreads) {
        float o[3], d[3], inv_d[3], omax;
        const int64_t r = load_ray(a, ray, given, o, d);
        ray_setup(d, o, inv_d, omax);
        for (int k = 0; k < rr.n; k++) {
            const BlockRec &b = rr.r[k];
            int nk = 0;
            DepthSum tau;
            BrickCache bc;
            for_each_sample(b, o, d, inv_d, omax, a.err,
                            [&](const float *, const float rel[3], const float g[3], float delta) {
                float2 f2[4];
                accumulate_sample<DT>(b, rel, g, f2, &bc);
                tau.add(expf(f2[0].x) * delta);
                nk++;
                return true;
            });
            const float T = nk ? tau.transmittance() : -1.f;
            if (a.out_T) a.out_T[r * rr.n + k] = T;
            else if (nk) term += opacity_term(a, 1.f - T);
        }
    }
    if (a.out_T) return;
    term = cta_sum(term);
    if (threadIdx.x == 0) a.loss_parts[kOpacityMaxCtas + blockIdx.x] = term;
}

// *loss += the CTAs' sums (in a fixed order: thousands of additions to one
// float would cost its last bits)
__global__ void __launch_bounds__(1024) k_add_parts(const float *__restrict__ parts, int nw, int nt, float *loss) {
    float v = 0.f;
    for (int k = threadIdx.x; k < nw; k += 1024) v += parts[k];
    for (int k = threadIdx.x; k < nt; k += 1024) v += parts[kOpacityMaxCtas + k];
    v = cta_sum(v);
    if (threadIdx.x == 0) atomicAdd(loss, v);
}

// grad_mlp[t] += sum over the CTAs' rows, in a fixed order: a CTA has 32 columns
// and 32 row streams, whose sums it adds in order (8192 rows: one thread a
// column took 318 us).
__global__ void __launch_bounds__(1024) k_reduce_rows(const float *__restrict__ partials, int n_rows, float *grad_mlp) {
    __shared__ float s_sum[32][33];
    const int c = threadIdx.x & 31, y = threadIdx.x >> 5, t = blockIdx.x * 32 + c;
    float s = 0.f;
    if (t < kMlpParams) {
#pragma unroll 8
        for (int k = y; k < n_rows; k += 32) s += __ldg(partials + (int64_t)k * kMlpParams + t);
    }
    s_sum[y][c] = s;
    __syncthreads();
    if (y == 0 && t < kMlpParams) {
        for (int k = 1; k < 32; k++) s += s_sum[k][c];
        grad_mlp[t] += s;
    }
}

struct AdamArgs {
    float lr, b1, b2, eps, bc1, bc2;
};

__device__ __forceinline__ void adam_one(float &p, float gi, float &m, float &v, const AdamArgs &a) {
    const float mi = a.b1 * m + (1.f - a.b1) * gi;
    const float vi = a.b2 * v + (1.f - a.b2) * gi * gi;
    m = mi;
    v = vi;
    p -= a.lr * (mi / a.bc1) / (sqrtf(vi / a.bc2) + a.eps);
}

// Bound by HBM, 28 bytes a value; with one value a thread at a time the four
// loads in flight a thread were too few (16.8 M values: 88 us, 5.3 TB/s).  vec:
// the arrays are 16-byte aligned, n4 = n / 4 groups.
__global__ void __launch_bounds__(256) k_adam(float *__restrict__ p, const float *__restrict__ g,
                                              float *__restrict__ m, float *__restrict__ v, int64_t n, int64_t n4,
                                              AdamArgs a) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = t; i < n4; i += step) {
        float4 P = reinterpret_cast<float4 *>(p)[i], M = reinterpret_cast<float4 *>(m)[i],
               V = reinterpret_cast<float4 *>(v)[i];
        const float4 G = reinterpret_cast<const float4 *>(g)[i];
        adam_one(P.x, G.x, M.x, V.x, a);
        adam_one(P.y, G.y, M.y, V.y, a);
        adam_one(P.z, G.z, M.z, V.z, a);
        adam_one(P.w, G.w, M.w, V.w, a);
        reinterpret_cast<float4 *>(p)[i] = P;
        reinterpret_cast<float4 *>(m)[i] = M;
        reinterpret_cast<float4 *>(v)[i] = V;
    }
    for (int64_t i = 4 * n4 + t; i < n; i += step) adam_one(p[i], g[i], m[i], v[i], a);
}

__global__ void __launch_bounds__(1024) k_mse_grad(const float *__restrict__ rgb, const float *__restrict__ tgt, int64_t n, float scale,
                           float *__restrict__ grad, float *loss) {
    __shared__ float s_part[32];
    float acc = 0.f;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float e = rgb[i] - tgt[i];
        grad[i] = 2.f * scale * e;
        acc = fmaf(e, e, acc);
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        float v = threadIdx.x < (blockDim.x >> 5) ? s_part[threadIdx.x] : 0.f;
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (threadIdx.x == 0 && loss) atomicAdd(loss, v * scale);
    }
}

// ---------------------------------------------------------------------------
// Per-block MLP form (Eq. 5 with Eq. 3 per block):
//   C = sum_k B_k X_k,  X_k = C^k + Phi^k(C^k, F^k, PE(d)),  B_{k+1} = B_k (1 - alpha^k)
// over the blocks with occupied samples.  Three passes, ray by ray:
//   P1  march every block once: C^k, F^k and B_k to scratch S;
//   P2  per (ray, block): Phi^k backward with u = B_k dL/dC gives
//       dL/dC^k = u + J_C^T u, dL/dF^k = J_F^T u and dL/dC . X_k (scratch G),
//       and adds u's weight gradient to block k's MLP gradient;
//   P3  march every block again and scatter the feature gradients: with
//       Q_k = sum_{j>k} B_j dL/dC . X_j (the later blocks' dependence on
//       1 - alpha^k), the Eq. 11 backward of the global form gives
//         dL/df0 = sigma delta (T_i e_i (gC.c_i + gF.s_i) - (gC.S_C + gF.S_F) - Q_k)
//       with in-block T_i and the block's own totals and upstreams.
// No early termination (the ray form's training calls use none).

// The per-block MLP input i: C^k (3), F^k (4), d (3), then sin / cos(2^l d).
__device__ __forceinline__ float bm_input(int i, const float ck[7], const float d[3]) {
    if (i < 7) return ck[i];
    if (i < 10) return d[i - 7];
    const int j = i - 10, l = j / 6, q = j % 6;
    const float v = ldexpf(d[q % 3], l);
    return q < 3 ? sinf(v) : cosf(v);
}

// P1
template <int DT>
__global__ void __launch_bounds__(kBwdThreads) k_bm_pass1(const __grid_constant__ BmBwdArgs a,
                                                          const __grid_constant__ RayRecs rr) {
    __shared__ WarpScratch s_ws[kBwdWarps];
    WarpScratch &ws = s_ws[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    float o[3], d[3], inv_d[3], omax;
    const int64_t r = load_ray_warp(a, first_ray(), o, d);
    if (r < 0) return;
    ray_setup(d, o, inv_d, omax);
    const int n = sort_blocks_warp(ws, rr, o);
    float *S = a.S + 8 * r * a.n_ids;
    for (int k = lane; k < n; k += 32) S[8 * k + 7] = -1.f;  // no occupied sample
    __syncwarp();
    float B = 1.f;
    for_each_hit(n, [&](int k) -> const BlockRec & { return rr.r[ws.ord[k]]; }, o, d, inv_d, [&](int k) {
        WarpRay sb;
        march_block_warp<DT>(ws, rr.r[ws.ord[k]], o, d, inv_d, omax, 0.f, sb, a.err);
        if (sb.nsamp == 0) return true;
        if (lane < 8) S[8 * ws.ord[k] + lane] = lane < 7 ? sb.acc : B;
        B *= sb.T;
        return true;
    });
}

// A weight-gradient term summed over the warp's 32 rays, then one reduction.
__device__ __forceinline__ void warp_red(float *dst, float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red_add1(dst, v);
}

// Sixteen weight-gradient terms (dst[0 .. 15]) summed over the warp's 32 rays
// at once: the two half-warps are folded, then at each of the four remaining
// lane bits every lane keeps one half of its values and adds the partner's
// copy of that half, so lane l ends with the warp sum of term l & 15 -- 31
// shuffles for the sixteen sums instead of 80 -- and lanes 0-15 reduce one
// term each.  v is overwritten.
__device__ __forceinline__ void warp_red16(float *dst, float v[16]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 16; j++) v[j] += __shfl_xor_sync(0xffffffffu, v[j], 16);
#pragma unroll
    for (int s = 8; s >= 1; s >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int j = 0; j < s; j++) {
            const float send = up ? v[j] : v[j + s];
            const float keep = up ? v[j + s] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
    if (lane < 16) red_add1(dst + lane, v[0]);
}

// P2: one thread per (ray, block) pair.  The pairs are laid out block-major
// with each block's rays padded to a multiple of 32, so a warp holds one
// block for 32 rays and sums that block's weight gradients before reducing;
// padding lanes and blocks a ray has no sample in take part with zeros.
__global__ void __launch_bounds__(kBwdThreads) k_bm_mlp(BmBwdArgs a, const __grid_constant__ RayRecs rr) {
    const int64_t t = (int64_t)blockIdx.x * kBwdThreads + threadIdx.x;
    const int64_t rows = (a.n_rays + 31) & ~(int64_t)31;
    const int k = (int)min(t / rows, (int64_t)a.n_ids - 1);  // warp-uniform
    const int64_t r = t - (int64_t)k * rows;
    const bool ray = t < rows * a.n_ids && r < a.n_rays;
    const int64_t pe = r * a.n_ids + k;  // the pair's scratch entry
    float4 e0 = make_float4(0.f, 0.f, 0.f, 0.f), e1 = make_float4(0.f, 0.f, 0.f, -1.f);
    if (ray) {
        const float4 *e = reinterpret_cast<const float4 *>(a.S + 8 * pe);
        e0 = e[0];
        e1 = e[1];
    }
    const bool act = ray && e1.w >= 0.f;
    if (!act) {  // the scratch of a block without samples holds no C^k, F^k: zeros, not stale values
        e0 = make_float4(0.f, 0.f, 0.f, 0.f);
        e1 = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float ck[7] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z};
    const float B = act ? e1.w : 0.f;
    float d[3], g[3], u[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        d[c] = ray ? __ldg(a.ray_d + 3 * r + c) : 0.f;
        g[c] = ray ? __ldg(a.dL_drgb + 3 * r + c) : 0.f;
        u[c] = B * g[c];
    }
    const int id = rr.id[k];
    const int n_in = 10 + 6 * a.n_freq;
    const float *W1 = a.mlps + (int64_t)id * a.mlp_stride;
    const float *b1 = W1 + n_in * 16, *W2 = b1 + 16, *b2 = W2 + 256, *W3 = b2 + 16, *b3 = W3 + 48;
    float *gW1 = a.grad_mlps + (int64_t)id * a.grad_stride;
    float *gb1 = gW1 + n_in * 16, *gW2 = gb1 + 16, *gb2 = gW2 + 256, *gW3 = gb2 + 16, *gb3 = gW3 + 48;
    float h1[16], h2[16];
#pragma unroll
    for (int j = 0; j < 16; j++) h1[j] = __ldg(b1 + j);
    for (int i = 0; i < n_in; i++) {
        const float xi = bm_input(i, ck, d);
#pragma unroll
        for (int j = 0; j < 16; j++) h1[j] = fmaf(xi, __ldg(W1 + i * 16 + j), h1[j]);
    }
#pragma unroll
    for (int j = 0; j < 16; j++) h1[j] = fmaxf(h1[j], 0.f);  // h1 > 0 iff z1 > 0
#pragma unroll
    for (int j = 0; j < 16; j++) {
        float z = __ldg(b2 + j);
#pragma unroll
        for (int i = 0; i < 16; i++) z = fmaf(h1[i], __ldg(W2 + i * 16 + j), z);
        h2[j] = fmaxf(z, 0.f);
    }
    float phi[3], dz3[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        float z = __ldg(b3 + j);
#pragma unroll
        for (int i = 0; i < 16; i++) z = fmaf(h2[i], __ldg(W3 + i * 3 + j), z);
        phi[j] = 1.f / (1.f + expf(-z));
        dz3[j] = u[j] * phi[j] * (1.f - phi[j]);
        warp_red(gb3 + j, dz3[j]);
    }
    float dz2[16];
#pragma unroll
    for (int i = 0; i < 16; i++) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            s = fmaf(__ldg(W3 + i * 3 + j), dz3[j], s);
            warp_red(gW3 + i * 3 + j, h2[i] * dz3[j]);
        }
        dz2[i] = h2[i] > 0.f ? s : 0.f;
    }
    float dz1[16], gv[16];
#pragma unroll
    for (int j = 0; j < 16; j++) gv[j] = dz2[j];
    warp_red16(gb2, gv);
#pragma unroll
    for (int i = 0; i < 16; i++) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 16; j++) {
            s = fmaf(__ldg(W2 + i * 16 + j), dz2[j], s);
            gv[j] = h1[i] * dz2[j];
        }
        warp_red16(gW2 + i * 16, gv);
        dz1[i] = h1[i] > 0.f ? s : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 16; j++) gv[j] = dz1[j];
    warp_red16(gb1, gv);
    float gx[7];
    for (int i = 0; i < n_in; i++) {
        const float xi = bm_input(i, ck, d);
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 16; j++) {
            s = fmaf(__ldg(W1 + i * 16 + j), dz1[j], s);
            gv[j] = xi * dz1[j];
        }
        warp_red16(gW1 + i * 16, gv);
        if (i < 7) gx[i] = s;
    }
    if (!ray) return;
    float4 *go = reinterpret_cast<float4 *>(a.G + 8 * pe);
    if (!act) {
        go[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        go[1] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    float xg = 0.f;
#pragma unroll
    for (int c = 0; c < 3; c++) xg = fmaf(g[c], ck[c] + phi[c], xg);
    go[0] = make_float4(u[0] + gx[0], u[1] + gx[1], u[2] + gx[2], gx[3]);
    go[1] = make_float4(gx[4], gx[5], gx[6], xg);
}

// P3, one ray per warp
template <int DT>
__global__ void __launch_bounds__(kBwdThreads, COW_BWD_MIN_BLOCKS) k_bm_remarch(const __grid_constant__ BmBwdArgs a,
                                                                          const __grid_constant__ RayRecs rr) {
    __shared__ BwdScratch s_bs[kBwdWarps];
    BwdScratch &bs = s_bs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    float o[3], d[3], inv_d[3], omax;
    const int64_t r = load_ray_warp(a, first_ray(), o, d);
    if (r < 0) return;
    ray_setup(d, o, inv_d, omax);
    const float *S = a.S + 8 * r * a.n_ids, *G = a.G + 8 * r * a.n_ids;
    float Qtot = 0.f;  // sum_k B_k dL/dC . X_k
    for (int k = 0; k < a.n_ids; k++) {
        const float B = __ldg(S + 8 * k + 7);
        if (B >= 0.f) Qtot = fmaf(B, __ldg(G + 8 * k + 7), Qtot);
    }
    const int n = sort_blocks_warp(bs.w, rr, o);
    float P = 0.f;
    for (int k = 0; k < n; k++) {
        const int idx = bs.w.ord[k];
        const float B = __ldg(S + 8 * idx + 7);
        if (B < 0.f) continue;  // no occupied sample: no part in Eq. 5
        float gcf[7];
#pragma unroll
        for (int q = 0; q < 7; q++) gcf[q] = __ldg(G + 8 * idx + q);
        P = fmaf(B, __ldg(G + 8 * idx + 7), P);
        const int id = rr.id[idx];
        float *const gp[3] = {a.grad_planes[3 * id], a.grad_planes[3 * id + 1], a.grad_planes[3 * id + 2]};
        BwdRay s;
        // Q: the blocks behind this one
        remarch_block<DT>(bs, rr.r[idx], o, d, inv_d, omax, gcf, __ldg(S + 8 * idx + (lane & 7)), Qtot - P, 0.f, s,
                          a.grad_grid[id], gp, a.err);
    }
}

}  // namespace

int backward_rows(int64_t n_rays) { return (int)((n_rays + kBwdThreads - 1) / kBwdThreads); }

cudaError_t launch_backward_rays(const BwdArgs &a, const RayRecs &rr, cudaStream_t st) {
    if (a.n_rays <= 0) return cudaSuccess;
    const int nb = backward_rows(a.n_rays);
    const unsigned nw = (unsigned)((a.n_rays + kBwdWarps - 1) / kBwdWarps);  // one ray per warp
    k_mlp_backward<<<nb, kBwdThreads, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_reduce_rows<<<(kMlpParams + 31) / 32, 1024, 0, st>>>(a.partials, nb, a.grad_mlp);
    {
        const cudaError_t e_ = dispatch_dt(a.dtype, [&](auto D) {
            k_remarch_backward<decltype(D)::value><<<nw, kBwdThreads, 0, st>>>(a, rr);
            return cudaSuccess;
        });
        if (e_ != cudaSuccess) return e_;
    }
    return cudaGetLastError();
}

cudaError_t launch_backward_block_mlps(const BmBwdArgs &a, const RayRecs &rr, cudaStream_t st) {
    if (a.n_rays <= 0) return cudaSuccess;
    const unsigned nw = (unsigned)((a.n_rays + kBwdWarps - 1) / kBwdWarps);  // one ray per warp
    const int64_t padded = ((a.n_rays + 31) & ~(int64_t)31) * a.n_ids;  // k_bm_mlp's threads
    if (!a.have_state) {
        const cudaError_t e_ = dispatch_dt(a.dtype, [&](auto D) {
            k_bm_pass1<decltype(D)::value><<<nw, kBwdThreads, 0, st>>>(a, rr);
            return cudaSuccess;
        });
        if (e_ != cudaSuccess) return e_;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_bm_mlp<<<(unsigned)((padded + kBwdThreads - 1) / kBwdThreads), kBwdThreads, 0, st>>>(a, rr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    {
        const cudaError_t e_ = dispatch_dt(a.dtype, [&](auto D) {
            k_bm_remarch<decltype(D)::value><<<nw, kBwdThreads, 0, st>>>(a, rr);
            return cudaSuccess;
        });
        if (e_ != cudaSuccess) return e_;
    }
    return cudaGetLastError();
}

cudaError_t launch_sparsity(const RegArgs &a, const RayRecs &rr, cudaStream_t st) {
    if (a.n_rays <= 0) return cudaSuccess;
    const int nb = (int)((a.n_rays + kBwdThreads - 1) / kBwdThreads);
    {
        const cudaError_t e_ = dispatch_dt(a.dtype, [&](auto D) {
            k_sparsity<decltype(D)::value><<<nb, kBwdThreads, 0, st>>>(a, rr);
            return cudaSuccess;
        });
        if (e_ != cudaSuccess) return e_;
    }
    return cudaGetLastError();
}

cudaError_t launch_opacity(const RegArgs &a, const RayRecs &rr, cudaStream_t st) {
    if (a.n_rays <= 0) return cudaSuccess;
    // a ray per warp or per thread; beyond kOpacityMaxCtas CTAs (8 waves) one ray after another
    const auto ctas = [&](int rays) {
        return (unsigned)std::min<int64_t>((a.n_rays + rays - 1) / rays, kOpacityMaxCtas);
    };
    // as launch_rays_dt: with a count of alike rays the device decides
    const unsigned nt = a.form == kFormThread || a.ray_alike ? ctas(kBwdThreads) : 0;
    const unsigned nw = a.form == kFormWarp || a.out_T ? ctas(kBwdWarps) : 0;
    const cudaError_t e_ = dispatch_dt(a.dtype, [&](auto D) {
        if (nt) k_opacity_t<decltype(D)::value><<<nt, kBwdThreads, 0, st>>>(a, rr);
        if (nw) k_opacity<decltype(D)::value><<<nw, kBwdThreads, 0, st>>>(a, rr);
        return cudaSuccess;
    });
    if (e_ != cudaSuccess) return e_;
    if (a.loss) k_add_parts<<<1, 1024, 0, st>>>(a.loss_parts, (int)nw, a.out_T ? 0 : (int)nt, a.loss);
    return cudaGetLastError();
}

cudaError_t launch_adam(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                        float eps, int step, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
    const bool vec = !(((uintptr_t)p | (uintptr_t)g | (uintptr_t)m | (uintptr_t)v) & 15u);
    const int64_t n4 = vec ? n / 4 : 0;
    int64_t blocks = ((vec ? n4 : n) + 255) / 256;
    if (blocks > kSms * 32) blocks = kSms * 32;
    if (blocks < 1) blocks = 1;
    k_adam<<<(int)blocks, 256, 0, st>>>(p, g, m, v, n, n4, AdamArgs{lr, b1, b2, eps, bc1, bc2});
    return cudaGetLastError();
}

cudaError_t launch_mse_grad(const float *rgb, const float *tgt, int64_t n, float *grad, float *loss, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (loss) {
        cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(float), st);
        if (e != cudaSuccess) return e;
    }
    // one CTA of 32 warps per SM at most: every CTA adds its part to the loss, and
    // the 2432 additions of 3.1 M values at 256 threads a CTA cost it 1.5e-6
    int64_t blocks = (n + 1023) / 1024;
    if (blocks > kSms) blocks = kSms;
    k_mse_grad<<<(int)blocks, 1024, 0, st>>>(rgb, tgt, n, 1.0f / (float)n, grad, loss);
    return cudaGetLastError();
}

}  // namespace cow
