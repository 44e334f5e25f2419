// CTA-level helpers shared by the numeric, learned and batched kernels: scans,
// accumulators, rank tables.
#pragma once

#include "spg_internal.cuh"

namespace spg {

// Exclusive scan of popc(bits[w]) over n words by the whole CTA: writes
// pre[0..n) and returns the total to every thread.  One barrier: pre[] is
// complete for every thread only after the caller's next barrier, and wsum must
// not be written again before that barrier.
__device__ __forceinline__ int cta_scan_popc1(const uint32_t *bits, int *pre, int n, int *wsum) {
    const int nt = blockDim.x, tid = threadIdx.x;
    const int per = (n + nt - 1) / nt;
    const int w0 = tid * per;
    int local = 0;
    for (int w = w0; w < min(n, w0 + per); w++) local += __popc(bits[w]);
    const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    int incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    const int wt = lane < nw ? wsum[lane] : 0;
    const int before = __reduce_add_sync(kFull, lane < wid ? wt : 0);
    const int total = __reduce_add_sync(kFull, wt);
    int run = before + incl - local;
    for (int w = w0; w < min(n, w0 + per); w++) {
        pre[w] = run;
        run += __popc(bits[w]);
    }
    return total;
}

// Shared-memory accumulator of a heavy item (slots addressed by rank or by
// row).
//
// Doubles.  The FP64 pipe retires 1.6 multiplies, adds or fused multiply-adds
// per clock per SM on this GPU (20 clocks a warp instruction), and a shared
// atomicAdd(double) is a loop around a 64-bit compare-and-swap (0.81 per
// clock per SM), so a product as DMUL + atomicAdd takes about 55 clocks a
// warp.  add_products instead takes the slot by a 64-bit exchange (6.0 per
// clock per SM) that leaves a marker in it, and stores fma(a, b, old) back:
// one FP64 instruction per product, rounded once.  A lane that finds the
// marker (another lane or warp holds the slot) keeps the product and tries
// again after the step's other products, so that the retries of one step share
// their instructions.  The marker is a signalling NaN: no arithmetic
// instruction returns one, so no sum is taken for it.
//
// Where products crowd on few slots, that is slow: k lanes that want one slot
// cost k rounds, and a 64-bit exchange of k lanes on a slot takes k passes, which
// the holder's store waits for.  There add_crowded sums a warp's products of one
// slot in registers first and adds the sum once (the walks find out by sampling a
// window, see window_crowds).  100,000 products a column, 99% of them on one row:
// exchanges alone 14.7 ms, DMUL + atomicAdd 10.0, combined 1.2; all of a light
// column's products on four rows 0.76, 0.37 and 0.31 ms.  Combining inside
// add_products (after a few tries, without sampling) made squaring an R-MAT graph
// 12% slower: its registers and votes count in every step.
//
// Wrapping int64 sums are kept as two 32-bit halves in separate arrays: a
// 64-bit add is a 32-bit atomic add on the low half that returns the old low
// word, from which the carry out of the low half follows exactly; the high
// half then receives the value's high word plus that carry (skipped when zero,
// the common case for small non-negative values).  Every update is thus exact
// modulo 2^64 in any order, and 32-bit shared atomics run several times faster
// than 64-bit ones on this GPU.
constexpr unsigned long long kSlotTaken = 0x7ff4a5c300000000ull;  // signalling NaN
constexpr int kSlotTries = 1 << 22;  // bound of one lane's retries

__device__ __forceinline__ uint32_t shared_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long shared_exch64(uint32_t addr, unsigned long long v) {
    unsigned long long o;
    asm volatile("atom.shared.exch.b64 %0, [%1], %2;" : "=l"(o) : "r"(addr), "l"(v) : "memory");
    return o;
}
__device__ __forceinline__ void shared_st64(uint32_t addr, double v) {
    asm volatile("st.volatile.shared.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ uint32_t shared_add32(uint32_t addr, uint32_t v) {
    uint32_t o;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(o) : "r"(addr), "r"(v) : "memory");
    return o;
}
__device__ __forceinline__ void shared_red32(uint32_t addr, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}


// The sum of v over the lanes of `peers` (a group of lanes that this one belongs
// to; the whole warp calls it), in the lowest lane of the group.  In every step
// the group's lanes of odd rank hand their sums to the lane before them and drop
// out, and the ranks of the others halve.
__device__ __forceinline__ double warp_sum_peers(unsigned peers, int lane, double v) {
    unsigned rank = __popc(peers & ((1u << lane) - 1u));
    unsigned above = peers & (~1u << lane);  // lanes of the group above this one that still hold a sum
    bool live = true;
    while (__any_sync(kFull, above != 0u)) {
        const double t = __shfl_sync(kFull, v, above ? __ffs((int)above) - 1 : 0);
        live = live && !(rank & 1u);
        const unsigned hold = __ballot_sync(kFull, live);
        if (live && above) v += t;
        above = live ? above & hold : 0u;
        rank >>= 1;
    }
    return v;
}

template <typename Acc>
struct HeavyAcc;
template <>
struct HeavyAcc<double> {
    static constexpr bool crowds = true;  // many products on one slot want add_crowded
    double *a;
    uint32_t sa;  // its shared-memory address
    static constexpr size_t bytes_per_slot = 8;
    static constexpr int slot_shift = 3;  // slot i is at byte addr(0) + (i << slot_shift)
    __device__ __forceinline__ HeavyAcc(void *base, int) : a((double *)base), sa(shared_addr(base)) {}
    __device__ __forceinline__ uint32_t addr(int i) const { return sa + ((uint32_t)i << slot_shift); }
    __device__ __forceinline__ void zero(int i) const { a[i] = 0.0; }
    // the whole CTA: clear slots [0, n) (and up to 3 more, inside the array)
    __device__ __forceinline__ void zero_all(int n) const {
        uint4 *p = (uint4 *)a;
        for (int i = threadIdx.x; 2 * i < n; i += blockDim.x) p[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    __device__ __forceinline__ void add(int i, double v) const { atomicAdd(a + i, v); }
    __device__ __forceinline__ double get(int i) const { return a[i]; }
    __device__ __forceinline__ void set(int i, double v) const { a[i] = v; }
    __device__ __forceinline__ int32_t *scratch32() const { return (int32_t *)a; }
    static __device__ __forceinline__ bool try_add(uint32_t ad, double x, double y) {
        const unsigned long long o = shared_exch64(ad, kSlotTaken);
        if ((uint32_t)(o >> 32) == (uint32_t)(kSlotTaken >> 32)) return false;
        shared_st64(ad, __fma_rn(x, y, __longlong_as_double((long long)o)));
        return true;
    }
    // slot at address ad[u] += x[u] * y[u] wherever ok[u]; false if a slot
    // stayed taken (never expected: a holder stores within a few instructions)
    template <int N>
    __device__ __forceinline__ bool add_products(const uint32_t (&ad)[N], const double (&x)[N], const double (&y)[N],
                                                 const bool (&ok)[N]) const {
        uint32_t pend = 0;
#pragma unroll
        for (int u = 0; u < N; u++)
            if (ok[u] && !try_add(ad[u], x[u], y[u])) pend |= 1u << u;
        for (int t = 0; pend; t++) {
            if (t == kSlotTries) return false;
            const int q = __ffs((int)pend) - 1;
            uint32_t aq = ad[0];
            double xq = x[0], yq = y[0];
#pragma unroll
            for (int u = 1; u < N; u++)
                if (q == u) {
                    aq = ad[u];
                    xq = x[u];
                    yq = y[u];
                }
            if (try_add(aq, xq, yq)) pend &= pend - 1u;
        }
        return true;
    }
    // slot at address ad += x * y wherever ok, one product a lane (the whole warp
    // calls it); false as above
    __device__ __forceinline__ bool add_crowded(uint32_t ad, double x, double y, bool ok) const {
        const int lane = threadIdx.x & 31;
        const unsigned peers = __match_any_sync(kFull, ok ? ad : ~(uint32_t)lane);
        const double v = warp_sum_peers(peers, lane, x * y);
        if (!ok || lane != __ffs((int)peers) - 1) return true;
        for (int t = 0; t < kSlotTries; t++)
            if (try_add(ad, v, 1.0)) return true;
        return false;
    }
};
template <>
struct HeavyAcc<long long> {
    static constexpr bool crowds = false;
    uint32_t *lo, *hi;
    uint32_t sa, hoff;  // address of lo, distance of hi from lo in bytes
    static constexpr size_t bytes_per_slot = 8;
    static constexpr int slot_shift = 2;
    __device__ __forceinline__ HeavyAcc(void *base, int slots)
        : lo((uint32_t *)base), hi((uint32_t *)base + slots), sa(shared_addr(base)), hoff((uint32_t)slots * 4u) {}
    __device__ __forceinline__ uint32_t addr(int i) const { return sa + ((uint32_t)i << slot_shift); }
    __device__ __forceinline__ void zero(int i) const {
        lo[i] = 0u;
        hi[i] = 0u;
    }
    __device__ __forceinline__ void zero_all(int n) const {
        uint4 *p = (uint4 *)lo, *q = (uint4 *)hi;  // (a multiple of 4 slots: both are 16-byte aligned)
        for (int i = threadIdx.x; 4 * i < n; i += blockDim.x) p[i] = q[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    __device__ __forceinline__ void add(int i, long long v) const {
        const unsigned long long u = (unsigned long long)v;
        const uint32_t vlo = (uint32_t)u, vhi = (uint32_t)(u >> 32);
        const uint32_t old = atomicAdd(lo + i, vlo);
        const uint32_t h = vhi + ((uint32_t)(old + vlo) < old ? 1u : 0u);
        if (h) atomicAdd(hi + i, h);
    }
    __device__ __forceinline__ long long get(int i) const {
        return (long long)(((unsigned long long)hi[i] << 32) | (unsigned long long)lo[i]);
    }
    __device__ __forceinline__ void set(int i, long long v) const {
        lo[i] = (uint32_t)v;
        hi[i] = (uint32_t)((unsigned long long)v >> 32);
    }
    __device__ __forceinline__ int32_t *scratch32() const { return (int32_t *)lo; }
    template <int N>
    __device__ __forceinline__ bool add_products(const uint32_t (&ad)[N], const long long (&x)[N],
                                                 const long long (&y)[N], const bool (&ok)[N]) const {
#pragma unroll
        for (int u = 0; u < N; u++)
            if (ok[u]) {
                const unsigned long long v = (unsigned long long)x[u] * (unsigned long long)y[u];
                const uint32_t vlo = (uint32_t)v;
                const uint32_t old = shared_add32(ad[u], vlo);
                const uint32_t h = (uint32_t)(v >> 32) + ((uint32_t)(old + vlo) < old ? 1u : 0u);
                if (h) shared_red32(ad[u] + hoff, h);
            }
        return true;
    }
};

// The products of a walk's step into their slots, in the walk's form.
template <bool CROWDED, typename Acc, int N>
__device__ __forceinline__ bool add_to(const HeavyAcc<Acc> &acc, const uint32_t (&ad)[N], const Acc (&x)[N],
                                       const Acc (&y)[N], const bool (&ok)[N]) {
    if constexpr (CROWDED) {
        static_assert(N == 1, "a crowded walk takes one window at a time");
        return acc.add_crowded(ad[0], x[0], y[0], ok[0]);
    } else {
        return acc.add_products(ad, x, y, ok);
    }
}

// Rank table of a heavy item: one 32-bit entry per 16 rows, the rows' bits in
// the low half, the number of set bits before them (at most 65,535) in the
// high half, so that a look-up is one 4-byte shared load (an 8-byte pair of
// word and prefix took twice the shared-memory wavefronts: in the numeric
// kernel these are what the walk is short of).  The two entries of a bitmap
// word are one uint2.
__device__ __forceinline__ uint32_t rank_word(uint2 e) { return (e.x & 0xffffu) | (e.y << 16); }
__device__ __forceinline__ int rank_before(uint2 e) { return (int)(e.x >> 16); }
// The bits of an entry up to row r's own, moved to the top (r's own is the
// sign bit), and the rank of a present row counted from 1.
__device__ __forceinline__ uint32_t rank_upto(uint32_t e, int r) { return __funnelshift_l(0u, e, ~(uint32_t)r | 16u); }
__device__ __forceinline__ int rank1(uint32_t e, uint32_t upto) { return (int)(e >> 16) + __popc(upto); }

// Load a heavy item's bitmap words and build their rank table, returning the
// number of set bits.
// Warp w takes 128-word chunks w, w + nw, ... (at most MAXC of them): a lane
// loads four consecutive words at once and scans their counts with the warp's
// shuffles; the chunk totals cross one barrier and the entries are written
// once, with their final prefix.  ctot holds one int per chunk; src is 16-byte
// aligned, nwords is a multiple of 4 and at most 128 * MAXC * nw.  Ends with a
// barrier.
template <int MAXC, int NT>
__device__ __forceinline__ int cta_load_rank_table(const uint32_t *__restrict__ src, uint2 *tab, int nwords,
                                                   int *ctot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int nw = NT / 32;
    const int nch = (nwords + 127) >> 7;
    uint4 x[MAXC];
    int pre[MAXC];  // entries of the chunk before this lane's words
#pragma unroll
    for (int i = 0; i < MAXC; i++) {
        const int c = wid + i * nw, w = (c << 7) + 4 * lane;
        x[i] = w < nwords ? ld_stream((const uint4 *)(src + w)) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < MAXC; i++) {
        const int c = wid + i * nw;
        if (c < nch) {
            const int pc = __popc(x[i].x) + __popc(x[i].y) + __popc(x[i].z) + __popc(x[i].w);
            int inc = pc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += t;
            }
            pre[i] = inc - pc;
            if (lane == 31) ctot[c] = inc;
        }
    }
    __syncthreads();
    int total = 0, before[MAXC];
#pragma unroll
    for (int i = 0; i < MAXC; i++) before[i] = 0;
    for (int c0 = 0; c0 < nch; c0 += 32) {
        const int t = c0 + lane < nch ? ctot[c0 + lane] : 0;
        total += __reduce_add_sync(kFull, t);
#pragma unroll
        for (int i = 0; i < MAXC; i++)
            before[i] += __reduce_add_sync(kFull, c0 + lane < wid + i * nw ? t : 0);
    }
#pragma unroll
    for (int i = 0; i < MAXC; i++) {
        const int w = ((wid + i * nw) << 7) + 4 * lane;
        if (w < nwords) {
            const uint32_t word[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
            uint32_t e[8];
            int run = before[i] + pre[i];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const uint32_t lo = word[q] & 0xffffu;
                const int mid = run + __popc(lo);
                e[2 * q] = ((uint32_t)run << 16) | lo;
                e[2 * q + 1] = ((uint32_t)mid << 16) | (word[q] >> 16);
                run += __popc(word[q]);
            }
            uint4 *dst = (uint4 *)(tab + w);
            dst[0] = make_uint4(e[0], e[1], e[2], e[3]);
            dst[1] = make_uint4(e[4], e[5], e[6], e[7]);
        }
    }
    __syncthreads();
    return total;
}

// Load bitmap words, from any word on and any number of them, into bp[].x and
// their exclusive popcount prefix into bp[].y, returning the total (a batch's
// windows begin anywhere).  Warp w takes 32-word chunks w, w + nw, ...: lanes
// load consecutive words (coalesced, one word per bank pair) and scan them
// with shuffles; a second pass adds the chunk offsets (every warp scans the
// chunk totals itself).  ctot holds one int per chunk
// (nwords <= 32 * 64).  Ends with a barrier.
__device__ __forceinline__ int cta_load_scan_words(const uint32_t *__restrict__ src, uint2 *bp, int nwords,
                                                    int *ctot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nch = (nwords + 31) >> 5;
    for (int c = wid; c < nch; c += nw) {
        const int w = (c << 5) + lane;
        const uint32_t x = w < nwords ? ld_stream(src + w) : 0u;
        const int pc = __popc(x);
        int inc = pc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += t;
        }
        if (w < nwords) bp[w] = make_uint2(x, (uint32_t)(inc - pc));
        if (lane == 31) ctot[c] = inc;
    }
    __syncthreads();
    // exclusive prefix of the chunk totals, each warp for itself (<= 64 chunks)
    const int t0 = lane < nch ? ctot[lane] : 0, t1 = lane + 32 < nch ? ctot[lane + 32] : 0;
    int i0 = t0, i1 = t1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(kFull, i0, o), b = __shfl_up_sync(kFull, i1, o);
        if (lane >= o) {
            i0 += a;
            i1 += b;
        }
    }
    const int half = __shfl_sync(kFull, i0, 31);
    const int total = half + __shfl_sync(kFull, i1, 31);
    for (int c = wid; c < nch; c += nw) {
        // offset of chunk c = exclusive prefix at c
        const int src_lane = c & 31;
        const int e0 = __shfl_sync(kFull, i0 - t0, src_lane), e1 = __shfl_sync(kFull, i1 - t1, src_lane);
        const int off = c < 32 ? e0 : half + e1;
        const int w = (c << 5) + lane;
        if (w < nwords) bp[w].y += (uint32_t)off;
    }
    __syncthreads();
    return total;
}

}  // namespace spg
