// Exclusive prefix sums (no spin waits).  Up to kScanOne elements: one CTA, one
// launch.  Up to kScanTiles tiles: two launches, the tile sums and the tiles,
// every tile adding up the sums before its own (at most 16 loads a thread).
// Beyond: three launches, the sums scanned by one CTA in between.  A launch
// costs about 3 us in the chain of a small plan, which has five scans.
// Used for the rank of required columns, the gathered column pointers, the
// heavy-slab item lists and the column pointers of C.
#include "spg_internal.cuh"

namespace spg {

constexpr int kScanThreads = 256;
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;

// What is scanned: an array, or the population counts of H & D (D's W words
// again for every block of H).
template <typename T>
struct ScanArray {
    const T *in;
    __device__ __forceinline__ long long operator()(int64_t i) const { return (long long)in[i]; }
};
struct ScanBits {
    const uint32_t *H, *D;
    int64_t W;
    __device__ __forceinline__ long long operator()(int64_t i) const {
        const int64_t w = (i | W) >> 32 ? i % W : (int64_t)((uint32_t)i % (uint32_t)W);
        return __popc(H[i] & D[w]);
    }
};

template <typename T>
__global__ void k_scan_reduce(const T in, int64_t n, long long *__restrict__ part) {
    __shared__ long long red[kScanThreads / 32];
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    long long s = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; i++) {
        int64_t idx = base + (int64_t)i * kScanThreads + threadIdx.x;
        if (idx < n) s += in(idx);
    }
    s = warp_sum_ll(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        long long v = threadIdx.x < kScanThreads / 32 ? red[threadIdx.x] : 0;
        v = warp_sum_ll(v);
        if (threadIdx.x == 0) part[blockIdx.x] = v;
    }
}

// One block scans the per-tile partial sums in place (exclusive).
__global__ void k_scan_partials(long long *part, int64_t ntiles) {
    __shared__ long long carry_sh;
    __shared__ long long wsum[32];
    if (threadIdx.x == 0) carry_sh = 0;
    __syncthreads();
    for (int64_t base = 0; base < ntiles; base += blockDim.x) {
        int64_t idx = base + threadIdx.x;
        long long v = idx < ntiles ? part[idx] : 0;
        int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        long long incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            int nw = blockDim.x >> 5;
            long long w = lane < nw ? wsum[lane] : 0;
            long long wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                long long t = __shfl_up_sync(kFull, wi, o);
                if (lane >= o) wi += t;
            }
            if (lane < nw) wsum[lane] = wi - w;
        }
        __syncthreads();
        long long carry = carry_sh;
        if (idx < ntiles) part[idx] = carry + wsum[wid] + incl - v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry_sh = carry + wsum[wid] + incl;
        __syncthreads();
    }
}

constexpr int64_t kScanOne = 1024 * kScanPer, kScanTiles = 4096;

// SUM: part holds the tiles' sums (this tile adds up those before it), else
// their scanned prefixes.
template <bool SUM, typename T>
__global__ void __launch_bounds__(kScanThreads)
    k_scan_tiles(const T in, int64_t n, const long long *__restrict__ part, int64_t *__restrict__ out) {
    __shared__ long long wsum[kScanThreads / 32], psum[kScanThreads / 32];
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    // each thread owns kScanPer consecutive elements
    long long v[kScanPer];
    long long run = 0;
    int64_t my = base + (int64_t)threadIdx.x * kScanPer;
#pragma unroll
    for (int i = 0; i < kScanPer; i++) {
        v[i] = (my + i < n) ? in(my + i) : 0;
        run += v[i];
    }
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[wid] = incl;
    if (SUM) {
        long long p = 0;
        for (int t = threadIdx.x; t < (int)blockIdx.x; t += kScanThreads) p += part[t];
        p = warp_sum_ll(p);
        if (lane == 0) psum[wid] = p;
    }
    __syncthreads();
    long long acc = (SUM ? 0 : part[blockIdx.x]) + incl - run;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; w++) {
        if (SUM) acc += psum[w];
        if (w < wid) acc += wsum[w];
    }
#pragma unroll
    for (int i = 0; i < kScanPer; i++) {
        if (my + i < n) out[my + i] = acc;
        acc += v[i];
        if (my + i == n - 1) out[n] = acc;
    }
}

// The whole scan, of up to kScanOne elements, by one CTA (7 us: as much as two
// launches, so that a second pass would not pay).
template <typename T>
__global__ void __launch_bounds__(1024) k_scan_one(const T in, int64_t n, int64_t *__restrict__ out) {
    __shared__ long long wsum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t my = (int64_t)threadIdx.x * kScanPer;
    long long v[kScanPer], run = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; i++) {
        v[i] = my + i < n ? in(my + i) : 0;
        run += v[i];
    }
    long long incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    const long long w = wsum[lane];
    long long acc = warp_sum_ll(lane < wid ? w : 0) + incl - run;
    const long long total = warp_sum_ll(w);
#pragma unroll
    for (int i = 0; i < kScanPer; i++) {
        if (my + i < n) out[my + i] = acc;
        acc += v[i];
    }
    if (threadIdx.x == 0) out[n] = total;
}

template <typename T>
static spg_status scan_impl(spg_plan *p, const T in, int64_t *out, int64_t n) {
    if (n == 0) {
        return cuda_check(cudaMemsetAsync(out, 0, sizeof(int64_t), p->st), "scan memset");
    }
    if (n <= kScanOne) {
        launch(p, k_scan_one<T>, 1, 1024, 0, in, n, out);
        return cuda_check(cudaGetLastError(), "scan launch");
    }
    int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    long long *part = (long long *)ws_alloc(p, sizeof(long long) * (size_t)(ntiles + 1));
    if (!part) return SPG_OUT_OF_MEMORY;
    launch(p, k_scan_reduce<T>, (unsigned)ntiles, kScanThreads, 0, in, n, part);
    if (ntiles <= kScanTiles) {
        launch(p, k_scan_tiles<true, T>, (unsigned)ntiles, kScanThreads, 0, in, n, part, out);
    } else {
        launch(p, k_scan_partials, 1, 1024, 0, part, ntiles);
        launch(p, k_scan_tiles<false, T>, (unsigned)ntiles, kScanThreads, 0, in, n, part, out);
    }
    return cuda_check(cudaGetLastError(), "scan launch");
}

spg_status scan_exclusive_i32(spg_plan *p, const int32_t *in, int64_t *out, int64_t n) {
    return scan_impl(p, ScanArray<int32_t>{in}, out, n);
}
spg_status scan_exclusive_i64(spg_plan *p, const int64_t *in, int64_t *out, int64_t n) {
    return scan_impl(p, ScanArray<int64_t>{in}, out, n);
}

spg_status scan_exclusive_bits(spg_plan *p, const uint32_t *H, const uint32_t *D, int64_t W, int64_t *out, int64_t n) {
    return scan_impl(p, ScanBits{H, D, W}, out, n);
}

}  // namespace spg
