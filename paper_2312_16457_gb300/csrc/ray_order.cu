// ray_order.cu -- a coherent processing order for ray batches.
//
// The ray-batch form (training rays: origins and directions in any order)
// marches one ray per warp; when the warps on the chip hold unrelated rays,
// they share few lines in L2 (2^20 random rays, 2x2 blocks of 128^3 FP32: the
// forward takes 39.9 ms in the given order, 28.3 ms in this one).  The order
// groups rays that cross the call's blocks along nearly the same segment: the
// key interleaves the bits of the cells in which a ray enters and leaves the
// blocks' bounding box (10 halvings of the box, each of its longest cell edge),
// and a counting sort of the keys gives the permutation the ray kernels read
// (warp t marches ray perm[t]; every output stays at its ray's own index, so the
// results per ray do not depend on the order).  Keys tried, ms a training step
// of those rays / 65537 BF16 rays / 30001 rays forward through 16 blocks: entry
// cell (8^3), then direction cell (8^3) 106.8 / 12.7 / 0.96; the same bits
// interleaved 102.7 / 12.8 / 0.94; entry and exit cell (8^3 each) interleaved
// 98.0 / 12.3 / 0.93; with 2^20 bins 16 x 16 x 4 cells 97.8 / 11.8 / 0.86, near
// cubic ones (which fit a box of any shape) 97.7 / 12.1 / 0.87.
// The key pass also counts the rays whose key is that of the next ray: a
// camera's rays, for which one ray per thread in the given order is the faster
// form (launch_march_rays).
#include <algorithm>

#include "cow_common.cuh"
#include "cow_kernels.h"

namespace cow {

namespace {

// One key step halves the cells of one axis: a bit of the entry cell and the
// same bit of the exit cell.
constexpr int kSteps = kRayOrderKeyBits / 2;

__device__ __forceinline__ uint32_t cell_of(float x, float lo, float inv_ext, int bits) {
    const float n = (float)(1 << bits);
    const float q = fminf(fmaxf((x - lo) * inv_ext * n, 0.f), n - 1.f);  // NaN -> 0
    return (uint32_t)q;
}

// What the keys are made of: the box, the axis of every step (two bits each,
// first step lowest) and the steps of each axis.
struct KeyGrid {
    float3 lo, hi;
    uint32_t axes;
    int3 bits;
    int alike_drop;  // low bits of the key that alike rays may differ in
};

// kSort: the keys and their histogram for the order; the count either way.
template <bool kSort>
__global__ void k_ray_keys(const float *__restrict__ o, const float *__restrict__ d, int64_t n, KeyGrid kg,
                           uint32_t *__restrict__ keys, uint32_t *__restrict__ hist, uint32_t *__restrict__ n_alike) {
    const float3 lo = kg.lo, hi = kg.hi;
    const float3 inv = make_float3(1.f / fmaxf(hi.x - lo.x, 1e-30f), 1.f / fmaxf(hi.y - lo.y, 1e-30f),
                                   1.f / fmaxf(hi.z - lo.z, 1e-30f));
    unsigned same = 0;  // of this warp's rays: those whose key is the next ray's
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + threadIdx.x;
        uint32_t key = 0xffffffffu;
        if (i < n) {
            const float oo[3] = {o[3 * i], o[3 * i + 1], o[3 * i + 2]};
            const float dd[3] = {d[3 * i], d[3 * i + 1], d[3 * i + 2]};
            const float l[3] = {lo.x, lo.y, lo.z}, h[3] = {hi.x, hi.y, hi.z};
            // entry into and exit out of the box (the origin itself when it is inside or behind)
            float tn = 0.f, tf = 3.0e38f;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                if (dd[a] == 0.f) continue;
                const float t1 = (l[a] - oo[a]) / dd[a], t2 = (h[a] - oo[a]) / dd[a];
                tn = fmaxf(tn, fminf(t1, t2));
                tf = fminf(tf, fmaxf(t1, t2));
            }
            tf = fmaxf(tf, tn);
            const float iv[3] = {inv.x, inv.y, inv.z};
            const int nb[3] = {kg.bits.x, kg.bits.y, kg.bits.z};
            uint32_t in[3], out[3];  // the axis' cells, the next bit on top
#pragma unroll
            for (int a = 0; a < 3; a++) {
                in[a] = cell_of(oo[a] + tn * dd[a], l[a], iv[a], nb[a]) << (32 - kSteps) << (kSteps - nb[a]);
                out[a] = cell_of(oo[a] + tf * dd[a], l[a], iv[a], nb[a]) << (32 - kSteps) << (kSteps - nb[a]);
            }
            key = 0;
#pragma unroll
            for (int s = 0; s < kSteps; s++) {
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    if ((int)((kg.axes >> (2 * s)) & 3u) != a) continue;  // uniform
                    key = (key << 2) | (in[a] >> 31 << 1) | (out[a] >> 31);
                    in[a] <<= 1;
                    out[a] <<= 1;
                }
            }
            if (kSort) {
                keys[i] = key;
                atomicAdd(hist + key, 1u);
            }
        }
        const uint32_t next = __shfl_down_sync(0xffffffffu, key, 1);
        const bool pair = i + 1 < n && (threadIdx.x & 31) != 31 && ((next ^ key) >> kg.alike_drop) == 0;
        same += __popc(__ballot_sync(0xffffffffu, pair));
    }
    if ((threadIdx.x & 31) == 0 && same) atomicAdd(n_alike, same);
}

// Exclusive prefix sum of the kRayOrderBins counts in two levels: every CTA
// scans its kScanThreads bins in place and writes its total to sums[]; one
// CTA then scans the totals, which the scatter adds back.
constexpr int kScanThreads = 1024;
constexpr int kScanBlocks = kRayOrderBins / kScanThreads;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *s_warp, uint32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        uint32_t w = lane < nw ? s_warp[lane] : 0u;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        if (lane < nw) s_warp[lane] = w;  // inclusive warp totals
    }
    __syncthreads();
    if (total) *total = s_warp[(blockDim.x >> 5) - 1];
    return x - v + (warp > 0 ? s_warp[warp - 1] : 0u);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_local(uint32_t *hist, uint32_t *sums) {
    __shared__ uint32_t s_warp[32];
    const int64_t i = (int64_t)blockIdx.x * kScanThreads + threadIdx.x;
    uint32_t total;
    const uint32_t ex = block_exclusive_scan(hist[i], s_warp, &total);
    hist[i] = ex;
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanBlocks) k_scan_sums(uint32_t *sums) {
    __shared__ uint32_t s_warp[32];
    sums[threadIdx.x] = block_exclusive_scan(sums[threadIdx.x], s_warp, nullptr);
}

__global__ void k_ray_scatter(const uint32_t *__restrict__ keys, int64_t n, uint32_t *__restrict__ offs,
                              const uint32_t *__restrict__ sums, int32_t *__restrict__ perm,
                              uint32_t *n_alike) {
    if (n_alike && blockIdx.x == 0 && threadIdx.x == 0) *n_alike = offs[kRayOrderAlike];  // behind the bins
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = keys[i];
        perm[sums[k / kScanThreads] + atomicAdd(offs + k, 1u)] = (int32_t)i;
    }
}

// Every step halves the longest edge of the cells: near cubic cells.
KeyGrid key_grid(const float lo[3], const float hi[3], int64_t n) {
    uint32_t axes = 0;
    int nb[3] = {0, 0, 0};
    float ext[3];
    for (int a = 0; a < 3; a++) ext[a] = hi[a] - lo[a];
    for (int s = 0; s < kSteps; s++) {
        int a = 0;
        for (int k = 1; k < 3; k++)
            if (ext[k] > ext[a]) a = k;
        axes |= (uint32_t)a << (2 * s);
        nb[a]++;
        ext[a] *= 0.5f;
    }
    // a camera of 2^17 rays has some eleven to a cell's edge; for fewer rays the
    // cells that count as the same grow with their spacing
    int drop = 0;
    for (int64_t m = n; m < kRaysAlikeMin && drop < 8; m *= 2) drop += 2;
    return {make_float3(lo[0], lo[1], lo[2]), make_float3(hi[0], hi[1], hi[2]), axes, make_int3(nb[0], nb[1], nb[2]),
            drop};
}

int key_blocks(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, kSms * 16); }

}  // namespace

cudaError_t launch_ray_order(const float *o, const float *d, int64_t n, const float lo[3], const float hi[3],
                             uint32_t *keys, uint32_t *hist, int32_t *perm, uint32_t *n_alike, cudaStream_t st) {
    static_assert(kRayOrderBins == kScanBlocks * kScanThreads && kScanBlocks <= 1024 && kScanBlocks % 32 == 0,
                  "two-level scan shape");
    static_assert(kRayOrderHistWords == kRayOrderBins + 32 + kScanBlocks && kRayOrderAlike == kRayOrderBins,
                  "histogram scratch: bins, the count of alike neighbours, block totals");
    if (n <= 0 || n > 0x7fffffff) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(hist, 0, (kRayOrderAlike + 1) * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    uint32_t *sums = hist + kRayOrderBins + 32;
    const int grid = key_blocks(n);
    k_ray_keys<true><<<grid, 256, 0, st>>>(o, d, n, key_grid(lo, hi, n), keys, hist, hist + kRayOrderAlike);
    k_scan_local<<<kScanBlocks, kScanThreads, 0, st>>>(hist, sums);
    k_scan_sums<<<1, kScanBlocks, 0, st>>>(sums);
    k_ray_scatter<<<grid, 256, 0, st>>>(keys, n, hist, sums, perm, n_alike);
    return cudaGetLastError();
}

cudaError_t launch_count_alike(const float *o, const float *d, int64_t n, const float lo[3], const float hi[3],
                               uint32_t *n_alike, cudaStream_t st) {
    if (n <= 0 || n > 0x7fffffff) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(n_alike, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    k_ray_keys<false><<<key_blocks(n), 256, 0, st>>>(o, d, n, key_grid(lo, hi, n), nullptr, nullptr, n_alike);
    return cudaGetLastError();
}

}  // namespace cow
