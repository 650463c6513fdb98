// march_warp.cuh -- one ray per warp: the 32 lanes take the ray's next 32
// occupied lattice samples, and the composite runs over them in order.
//
// A ray's samples are independent up to the composite (Eq. 1-2): lookups and
// activations, almost all of the work, need no transmittance.  With one ray
// per thread a batch of a few thousand rays leaves most of the chip idle and
// takes as long as its longest ray's chain of dependent gathers; here the
// chain is 32 times shorter and the gathers of one instruction read
// neighbouring texels of one ray.  The composite takes the samples' alphas and
// colours from shared memory and adds them in lattice order with the
// operations of march_block, so every output, sample count and early
// termination is that of the one-ray-per-thread march, bit for bit.
#pragma once

#include "march_core.cuh"

namespace cow {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kRowPad = 36;  // row stride: the float4 reads of 8 rows fall into distinct banks

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(kFullMask, x, off);
    return x;
}

// Shared scratch of one warp.
struct alignas(16) WarpScratch {
    float row[8][kRowPad];   // channels 0-6 of the chunk's samples, then exp(-sigma delta)
    int32_t q[64];           // occupied samples found and not yet taken: lattice index, or t when unbounded
    int32_t ord[kMaxRayIds]; // ray form: the call's blocks in the ray's order
};

// Occupied lattice samples of the warp's ray inside block b, in order, 32 at a
// time: fn(active, n, rel, g, s) is called with lanes 0 .. n-1 holding one sample
// each (n = 32 except for the block's last call); it returns false (uniformly)
// to stop the ray.  The lattice is scanned 32 points at a step, occupied points
// are queued, and a chunk is handed out when 32 are there, so empty space costs
// only the scan.  The jump out of empty cells is for_each_sample's, taken from
// the scan's last point.
template <typename Fn>
__device__ __forceinline__ bool for_each_chunk(WarpScratch &ws, const BlockRec &b, const float o[3], const float d[3],
                                               const float inv_d[3], float omax, unsigned *err, Fn &&fn) {
    const int lane = threadIdx.x & 31;
    const bool unb = (b.unb & kUnbContracted) != 0;
    const float delta = b.delta, inv_delta = 1.0f / b.delta;
    const int Nc = b.Nc, C = b.C, R = b.R;
    int base, last;
    float m = 0.f, t_next = 0.f;
    if (unb) {
        base = first_owned_index(b, o, d);
        if (base < 0) return true;
        t_next = __fmul_rn(__fadd_rn(__int2float_rn(base), 0.5f), delta);
        base = 0;
        last = kContractSteps - 1;
    } else {
        float tfar;
        if (!candidate_range(b, o, d, inv_d, base, last, tfar)) return true;
        if (last - base > kMaxSpan) {
            if (lane == 0) atomicOr(err, kErrRange);
            last = base + kMaxSpan;
        }
        m = 4e-6f * (omax + tfar + b.bmax);
    }
    int qn = 0;
    do {
        while (qn < 32 && base <= last) {
            bool occ = false;
            int item, jump = -1;
            if (unb) {
                // t advances by each point's own step: every lane walks the
                // scan's points and keeps its own
                bool end = false;
                float tl = 0.f;
                int k = 0;
                for (; k < 32 && base + k <= last; k++) {
                    float p[3], x[3];
#pragma unroll
                    for (int a = 0; a < 3; a++) p[a] = __fadd_rn(o[a], __fmul_rn(t_next, d[a]));
                    end = !owned_unbounded(b, p);
                    if (end) break;
                    const float mm = unbounded_x(b, p, x);
                    end = mm > kContractMax;
                    if (end) break;
                    if (k == lane) tl = t_next;
                    const float m1 = fmaxf(mm, 1.f);
                    t_next = __fadd_rn(t_next, __fmul_rn(__fmul_rn(delta, m1), m1));
                }
                if (lane < k) {
                    float p[3], x[3], u[3], rel[3], g[3];
#pragma unroll
                    for (int a = 0; a < 3; a++) p[a] = __fadd_rn(o[a], __fmul_rn(tl, d[a]));
                    contract_u(x, unbounded_x(b, p, x), u);
                    lookup_u(b, u, rel, g);
                    int cell[3];
#pragma unroll
                    for (int a = 0; a < 3; a++) {
                        const int v = min(__float2int_rd(g[a]), R - 2);
                        cell[a] = C == 1 ? v : (int)__umulhi((unsigned)v, b.cdiv);
                    }
                    const int ci = (cell[2] * Nc + cell[1]) * Nc + cell[0];
                    occ = (__ldg(b.occ + (ci >> 5)) >> (ci & 31)) & 1u;
                }
                item = __float_as_int(tl);
                base = end ? last + 1 : base + 32;
            } else {
                item = base + lane;
                if (item <= last) {
                    float p[3];
                    lattice_point(o, d, delta, item, p);
                    if (inside_block(b, p)) {
                        float rel[3], g[3];
                        lookup_p(b, p, rel, g);
                        int cell[3];
#pragma unroll
                        for (int a = 0; a < 3; a++) {
                            const int v = min(__float2int_rd(g[a]), R - 2);
                            cell[a] = C == 1 ? v : (int)__umulhi((unsigned)v, b.cdiv);
                        }
                        const int ci = (cell[2] * Nc + cell[1]) * Nc + cell[0];
                        occ = (__ldg(b.occ + (ci >> 5)) >> (ci & 31)) & 1u;
                        if (!occ && lane == 31) jump = empty_exit(b, cell, o, d, inv_d, m, inv_delta);
                    }
                }
            }
            const unsigned occm = __ballot_sync(kFullMask, occ);
            if (occ) ws.q[qn + __popc(occm & ((1u << lane) - 1u))] = item;
            qn += __popc(occm);
            if (!unb) {
                base += 32;
                if (!(occm >> 31)) base = max(base, __shfl_sync(kFullMask, jump, 31) + 1);
            }
        }
        if (qn == 0) break;
        __syncwarp();
        const int n = min(qn, 32);
        const bool active = lane < n;
        const int item = ws.q[active ? lane : 0];
        const int rest = ws.q[32 + lane];
        __syncwarp();
        if (32 + lane < qn) ws.q[lane] = rest;
        qn -= n;
        float p[3], rel[3], g[3], s = delta;
        if (unb) {
            const float t = __int_as_float(item);
            float q[3], x[3];
#pragma unroll
            for (int a = 0; a < 3; a++) q[a] = __fadd_rn(o[a], __fmul_rn(t, d[a]));
            const float mm = unbounded_x(b, q, x), m1 = fmaxf(mm, 1.f);
            s = __fmul_rn(__fmul_rn(delta, m1), m1);
            contract_u(x, mm, p);
            lookup_u(b, p, rel, g);
        } else {
            lattice_point(o, d, delta, item, p);
            lookup_p(b, p, rel, g);
        }
        if (!fn(active, n, rel, g, s)) return false;
    } while (qn > 0 || base <= last);
    return true;
}

// The composite of one ray, carried by its warp: lane c < 7 holds channel c
// of (C_d, F); the rest is uniform.
struct WarpRay {
    float acc = 0.f, T = 1.f;
    int nsamp = 0;
    bool done = false;
};

// Weights T_i (1 - e_i) of four successive samples; T moves past them.
__device__ __forceinline__ void chunk_weights(const float4 &e, float &T, float w[4]) {
    const float2 one = make_float2(1.f, 1.f), neg = make_float2(-1.f, -1.f);
    const float T1 = T * e.x, T2 = T1 * e.y, T3 = T2 * e.z;
    const float2 a = __fmul2_rn(make_float2(T, T1), __ffma2_rn(make_float2(e.x, e.y), neg, one));
    const float2 b = __fmul2_rn(make_float2(T2, T3), __ffma2_rn(make_float2(e.z, e.w), neg, one));
    T = T3 * e.w;
    w[0] = a.x, w[1] = a.y, w[2] = b.x, w[3] = b.y;
}

// Composite a chunk of n samples (Eq. 1-2) in order: each lane brings its
// sample's e = exp(-sigma s) and seven colours (e = 1, colours 0 beyond n,
// which leave T and the sums as they are).  Returns false once T < ert_eps, with the samples after it unused.
__device__ __forceinline__ bool composite_chunk(WarpScratch &ws, int n, float e, const float c[7], float ert_eps,
                                                WarpRay &s) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < 7; q++) ws.row[q][lane] = c[q];
    ws.row[7][lane] = e;
    __syncwarp();
    const float4 *x4 = reinterpret_cast<const float4 *>(ws.row[lane & 7]);
    const float4 *e4 = reinterpret_cast<const float4 *>(ws.row[7]);
    float T = s.T, acc = s.acc;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if (4 * k >= n) break;
        const float4 ee = e4[k], xx = x4[k];
        float w[4];
        chunk_weights(ee, T, w);
        acc = fmaf(w[3], xx.w, fmaf(w[2], xx.z, fmaf(w[1], xx.y, fmaf(w[0], xx.x, acc))));
    }
    bool more = true;
    int used = n;
    if (!(T >= ert_eps)) {  // the ray ends in this chunk, perhaps in front of a NaN: again, up to there
        T = s.T;
        acc = s.acc;
        const float *er = ws.row[7], *xr = ws.row[lane & 7];
        for (used = 0; used < n;) {
            const float ev = er[used];
            acc = fmaf(T * (1.f - ev), xr[used], acc);
            T *= ev;
            used++;
            if (T < ert_eps) {
                more = false;
                break;
            }
        }
    }
    __syncwarp();
    s.acc = acc;
    s.T = T;
    s.nsamp += used;
    return more;
}

// March the warp's ray through one block, updating its composite (march_block
// of the one-ray-per-thread form).  tb, when given, receives the block's own
// transmittance (Eq. 11) as exp(-sum of sigma s): the product of the rounded
// 1 - alpha loses what thin samples take (the opacity term of 65537 rays: 5e-6
// off in the product's form).
template <int DT>
__device__ __forceinline__ void march_block_warp(WarpScratch &ws, const BlockRec &b, const float o[3],
                                                 const float d[3], const float inv_d[3], float omax, float ert_eps,
                                                 WarpRay &s, unsigned *err, float *tb = nullptr) {
    BrickCache bc;
    float tau = 0.f;  // this lane's samples
    const bool more = for_each_chunk(ws, b, o, d, inv_d, omax, err,
                                     [&](bool active, int n, const float rel[3], const float g[3], float dt) {
        float e = 1.f, c[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (active) {
            float2 f2[4];
            accumulate_sample<DT>(b, rel, g, f2, &bc);
            const float f[8] = {f2[0].x, f2[0].y, f2[1].x, f2[1].y, f2[2].x, f2[2].y, f2[3].x, f2[3].y};
            const float sd = __expf(f[0]) * dt;
            e = __expf(-sd);
            tau += sd;
#pragma unroll
            for (int q = 0; q < 7; q++) c[q] = sigmoidf_fast(f[1 + q]);
        }
        return composite_chunk(ws, n, e, c, ert_eps, s);
    });
    if (!more) s.done = true;
    if (tb) *tb = expf(-warp_sum(tau));
}

// The call's blocks in the order of sort_blocks_for_ray (FP32 key, ties by id,
// then position): each lane ranks the blocks l and l + 32 against all others.
// ws.ord[k] receives the position in rr of the k-th block.
__device__ __forceinline__ int sort_blocks_warp(WarpScratch &ws, const RayRecs &rr, const float o[3]) {
    const int lane = threadIdx.x & 31, n = rr.n;
    for (int h = 0; h < n; h += 32) {
        const int i = h + lane;
        float key = 0.f;
        int id = 0;
        if (i < n) {
            const float dx = __fsub_rn(rr.r[i].cx, o[0]), dy = __fsub_rn(rr.r[i].cy, o[1]);
            key = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
            id = rr.id[i];
        }
        int rank = 0;
        for (int j = 0; j < n; j++) {  // uniform: block j's key
            const float dx = __fsub_rn(rr.r[j].cx, o[0]), dy = __fsub_rn(rr.r[j].cy, o[1]);
            const float kj = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
            const int idj = rr.id[j];
            const bool before = kj < key || (!(key < kj) && (idj < id || (idj == id && j < i)));
            rank += before ? 1 : 0;
        }
        if (i < n) ws.ord[rank] = i;
    }
    __syncwarp();
    return n;
}

// f(k) for every k < n, in order, whose block the ray's candidate range
// reaches: 32 blocks are tested at a time, one per lane.  rec_at(k): the k-th
// block's record.  f returns false to stop.
template <class RecAt, class F>
__device__ __forceinline__ void for_each_hit(int n, RecAt rec_at, const float o[3], const float d[3],
                                             const float inv_d[3], F &&f) {
    const int lane = threadIdx.x & 31;
    for (int h = 0; h < n; h += 32) {
        bool hit = false;
        if (h + lane < n) {
            const BlockRec &b = rec_at(h + lane);
            int i0, i1;
            float tfar;
            hit = (b.unb & kUnbContracted) || candidate_range(b, o, d, inv_d, i0, i1, tfar);
        }
        for (unsigned left = __ballot_sync(kFullMask, hit); left; left &= left - 1)
            if (!f(h + __ffs(left) - 1)) return;
    }
}

// Ray t in the call's order (a: the ray arrays and the order of a ray-batch
// call; given: the order is the given one): its index, or -1 beyond the last.
template <class Args>
__device__ __forceinline__ int64_t load_ray(const Args &a, int64_t t, bool given, float o[3], float d[3]) {
    if (t >= a.n_rays) return -1;
    const int64_t r = a.ray_perm && !given ? (int64_t)__ldg(a.ray_perm + t) : t;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        o[c] = __ldg(a.ray_o + 3 * r + c);
        d[c] = __ldg(a.ray_d + 3 * r + c);
    }
    return r;
}

template <class Args>
__device__ __forceinline__ int64_t load_ray_warp(const Args &a, int64_t t, float o[3], float d[3]) {
    return load_ray(a, t, false, o, d);
}

// The warp's ray in the call's order.
__device__ __forceinline__ int64_t first_ray() { return (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); }

// A camera's rays given as a ray batch: three quarters of them enter and leave
// the blocks' box where the next ray does (32 consecutive rays can have 31 such).
template <class Args>
__device__ __forceinline__ bool rays_alike(const Args &a) {
    return a.ray_alike && mostly_alike(__ldg(a.ray_alike), a.n_rays);
}

// Whether the thread form has the call, and whether in the given order.
template <class Args>
__device__ __forceinline__ bool thread_form(const Args &a, bool &given) {
    given = rays_alike(a);
    return given || a.form == kFormThread;
}

// deferred_mlp with lane j < 16 on hidden unit j (the same sums in the same
// order); x is uniform.  Lane j < 3 returns output j.
__device__ __forceinline__ float deferred_mlp_warp(const float *w, const float x_in[10], bool bf16) {
    const int lane = threadIdx.x & 31, u = lane & 15, q = min(lane, 2);
    float h = w[kOffB1 + u];
#pragma unroll
    for (int i = 0; i < 10; i++) h = fmaf(bf16 ? bf16r(x_in[i]) : x_in[i], w[kOffW1 + i * 16 + u], h);
    h = fmaxf(h, 0.f);
    if (bf16) h = bf16r(h);
    float h2 = w[kOffB2 + u];
#pragma unroll
    for (int i = 0; i < 16; i++) h2 = fmaf(__shfl_sync(kFullMask, h, i), w[kOffW2 + i * 16 + u], h2);
    h2 = fmaxf(h2, 0.f);
    if (bf16) h2 = bf16r(h2);
    float a = w[kOffB3 + q];
#pragma unroll
    for (int i = 0; i < 16; i++) a = fmaf(__shfl_sync(kFullMask, h2, i), w[kOffW3 + i * 3 + q], a);
    return sigmoidf_fast(a);
}

// block_mlp in the same way: cd and f come as lane c's channel `acc`.
__device__ __forceinline__ float block_mlp_warp(const float *__restrict__ w, int n_freq, float acc, const float d[3]) {
    const int lane = threadIdx.x & 31, u = lane & 15, q = min(lane, 2);
    const float *b1 = w + (10 + 6 * n_freq) * 16, *W2 = b1 + 16, *b2 = W2 + 256, *W3 = b2 + 16, *b3 = W3 + 48;
    float h = __ldg(b1 + u);
#pragma unroll
    for (int i = 0; i < 7; i++) h = fmaf(__shfl_sync(kFullMask, acc, i), __ldg(w + i * 16 + u), h);
#pragma unroll
    for (int i = 0; i < 3; i++) h = fmaf(d[i], __ldg(w + (7 + i) * 16 + u), h);
    float sc = 1.0f;
#pragma unroll 1
    for (int l = 0; l < n_freq; l++) {
        const float *rows = w + (10 + 6 * l) * 16 + u;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            float sn, cs;
            sincosf(sc * d[a], &sn, &cs);
            h = fmaf(sn, __ldg(rows + a * 16), h);
            h = fmaf(cs, __ldg(rows + (3 + a) * 16), h);
        }
        sc *= 2.0f;
    }
    h = fmaxf(h, 0.f);
    float h2 = __ldg(b2 + u);
#pragma unroll
    for (int i = 0; i < 16; i++) h2 = fmaf(__shfl_sync(kFullMask, h, i), __ldg(W2 + i * 16 + u), h2);
    h2 = fmaxf(h2, 0.f);
    float a = __ldg(b3 + q);
#pragma unroll
    for (int i = 0; i < 16; i++) a = fmaf(__shfl_sync(kFullMask, h2, i), __ldg(W3 + i * 3 + q), a);
    return sigmoidf_fast(a);
}

}  // namespace cow
