// The batch's default kernel: packets of rays (ss_packet.cuh) from one queue over
// all instances.
//
// The queue hands out strips of packets (consecutive strips of one
// instance are neighbours on its tile).  A warp keeps a copy of its instance's
// descriptor in shared memory and walks its strip as the single-tile kernel
// does; all its lanes work on one packet at a time, so nothing of another
// instance is ever in flight in the warp.  Penumbra rays are left pending and
// re-evaluated by a second kernel over the same strips, with full warps.
//
// Bound by instruction issue, as ss_packet.cuh.  16 tiles of 512^2 to 4096^2 (89 M
// rays, a sun each) take 32.6 ms against 89.9 ms with batch_task_kernel; 16 tiles of
// 512^2 1.69 against 11.7 ms, 4 tiles of 256^2 0.17 against 7.3 ms (its chunks of
// 4,096 texels leave most of the GPU's warps without one).
#include "ss_batch.h"
#include "ss_packet.cuh"

namespace ss {

namespace {

// instance that owns strip q: prefix[i] <= q < prefix[i + 1]
__device__ __forceinline__ int32_t strip_owner(const int64_t* prefix, int32_t n, int64_t q) {
    int32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (__ldg(prefix + mid) <= q) lo = mid; else hi = mid;
    }
    return lo;
}

template <bool kCount, bool kPoly, bool kLight>
__global__ void __launch_bounds__(kPkThreads, SS_PK_MIN_BLOCKS) batch_packet_kernel(const BatchArgs a) {
    __shared__ BatchItemDesc s_d[kPkThreads / 32];
    __shared__ PkWarp<kCount, true, kLight, false> s_w[kPkThreads / 32];
    const int lane = threadIdx.x & 31;
    BatchItemDesc& D = s_d[threadIdx.x >> 5];
    const Rays grid_rays = { 0, 0, nullptr, nullptr, nullptr };
    int32_t cur = -1;
    float span = 0.0f;
    while (true) {
        unsigned long long got = 0;
        if (lane == 0) got = atomicAdd(a.counter, 1ULL);
        const int64_t q = (int64_t)__shfl_sync(kFull, got, 0);
        if (q >= a.total_chunks) break;
        const int32_t item = strip_owner(a.chunk_prefix, a.n_items, q);
        if (item != cur) {
            __syncwarp();
            const uint32_t* src = reinterpret_cast<const uint32_t*>(a.items + item);
            uint32_t* dst = reinterpret_cast<uint32_t*>(&D);
            for (int i = lane; i < (int)(sizeof(BatchItemDesc) / 4); i += 32) dst[i] = __ldg(src + i);
            __syncwarp();
            cur = item;
            span = __ldg(D.stats) - __ldg(D.stats + 1);
            if (lane == 0) report_nonfinite_heights(D.stats, D.O.status);
        }
        pk_grid_strip<kCount, kPoly, kLight, false>(D.T, D.L, D.levels, grid_rays, D.O,
                                                    (uint32_t)(q - __ldg(a.chunk_prefix + item)),
                                                    a.pk, span, s_w[threadIdx.x >> 5], lane);
    }
}

// Re-evaluation of the rays left pending (refine_kernel over the strips): a
// block gathers the pending rays of kBatchRefineStrips strips, then every thread
// takes one.
constexpr int kBatchRefineStrips = 4;

__global__ void __launch_bounds__(256) batch_refine_kernel(const BatchArgs a) {
    __shared__ int64_t s_ray[kBatchRefineStrips * kPkMaxLen * kPkRows * kPkCols];
    __shared__ int32_t s_item[kBatchRefineStrips * kPkMaxLen * kPkRows * kPkCols];
    __shared__ int32_t s_cnt;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const int64_t q0 = (int64_t)blockIdx.x * kBatchRefineStrips;
    for (int64_t q = q0 + (threadIdx.x >> 5); q < min(q0 + kBatchRefineStrips, a.total_chunks);
         q += 8) {
        const int32_t item = strip_owner(a.chunk_prefix, a.n_items, q);
        const BatchItemDesc& D = a.items[item];
        const int32_t nx = D.T.nx, ny = D.T.ny;
        const uint32_t nbx = (uint32_t)(nx + kPkCols - 1) / kPkCols;
        const uint32_t strip = (uint32_t)(q - __ldg(a.chunk_prefix + item)), band = strip / nbx;
        const int32_t x = (int32_t)(strip - band * nbx) * kPkCols + (threadIdx.x & (kPkCols - 1));
        const int32_t rows = a.pk.rays / kPkCols * a.pk.len;
        for (int32_t k = (threadIdx.x & 31) / kPkCols; k < rows; k += kPkRows) {
            const int64_t y = (int64_t)band * rows + k;
            if (x >= nx || y >= ny) break;
            const int64_t r = y * nx + x;
            if (D.O.light[r] == kLightPending) {
                const int32_t i = atomicAdd(&s_cnt, 1);
                s_ray[i] = r;
                s_item[i] = item;
            }
        }
    }
    __syncthreads();
    const Rays grid_rays = { 0, 0, nullptr, nullptr, nullptr };
    for (int i = threadIdx.x; i < s_cnt; i += 256) {
        const BatchItemDesc& D = a.items[s_item[i]];
        const int64_t r = s_ray[i];
        float light, cost;
        refine_ray(D.T, grid_rays, r, D.O.argmin[r], false, light, cost);
        D.O.light[r] = light;
        if (D.O.cost) D.O.cost[r] = cost;
    }
}

template <bool C, bool P, bool L>
cudaError_t go(const BatchArgs& a, cudaStream_t s) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, batch_packet_kernel<C, P, L>, kPkThreads, 0);
    if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    const int64_t warps = a.total_chunks, cap = (int64_t)per_sm * device_sm_count();
    const int64_t want = (warps + kPkThreads / 32 - 1) / (kPkThreads / 32);
    batch_packet_kernel<C, P, L><<<(unsigned)(want < cap ? want : cap), kPkThreads, 0, s>>>(a);
    const int64_t blocks = (a.total_chunks + kBatchRefineStrips - 1) / kBatchRefineStrips;
    batch_refine_kernel<<<(unsigned)blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_batch_packets(const BatchArgs& a, bool count, cudaStream_t s) {
    const int k = (count ? 4 : 0) | (a.poly ? 2 : 0) | (a.light_only ? 1 : 0);
    switch (k) {
        case 0: return go<false, false, false>(a, s);
        case 1: return go<false, false, true>(a, s);
        case 2: return go<false, true, false>(a, s);
        case 3: return go<false, true, true>(a, s);
        case 4: return go<true, false, false>(a, s);
        case 5: return go<true, false, true>(a, s);
        case 6: return go<true, true, false>(a, s);
        default: return go<true, true, true>(a, s);
    }
}

}  // namespace ss
