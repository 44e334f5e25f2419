// CTA-wide walk over the products of one heavy output column (used by the
// heavy symbolic and numeric kernels).
#pragma once

#include <type_traits>

#include "spg_internal.cuh"

namespace spg {

// Staging area of cta_products for one batch of NT B' entries (NT threads): the
// non-empty A~ segments they multiply.  Window segments sit at [0, ns), long
// ones at [ns, ns + nl); each part numbers its products consecutively, and
// start holds a segment's first A~ entry minus its first product's number
// (product f of it is entry start + f).  pref holds the long segments' first
// products.  win describes every window of 32 consecutive products of the
// window part: .x has a bit for each product that begins a segment, and .y is
// one more than the segment that reaches into the window from the one before,
// or the segment that begins with the window: a product belongs to segment
// .y - 1 plus the number of bits up to its own.
template <typename Acc, int NT = kBatch>
struct CtaBatch {
    static constexpr int kShortWindows = short_windows(NT), kMidSeg = mid_seg(NT);
    static_assert(kLongSeg >= 32, "a 32-product window must meet at most two long segments");
    static_assert(NT * (kLongSeg - 1) <= 32 * kShortWindows, "segments below kLongSeg always fit the windows");
    static_assert(NT < 1024 && NT * (kMidSeg - 1) < 65536 && NT * (kLongSeg - 1) < 32768,
                  "the packed scan counters hold a batch");
    long long start[NT];
    int pref[NT + 2];
    Acc bv[NT];
    int wsum[3][33];
    uint2 win[kShortWindows];
    int cut[2];  // window segments and products of the middle class, if not all of it fits
    int next;    // next window to claim
    bool crowded;  // the products of the last sampled batch crowd on few rows
    // all threads, once, before the first cta_products (which leaves the bits
    // clear again); a barrier must follow
    __device__ __forceinline__ void clear() {
        for (int w = threadIdx.x; w < kShortWindows; w += NT) win[w].x = 0u;
    }
};

// Exclusive CTA scan of three counters at once; every thread gets the totals
// in tot[0..2].  One barrier: every warp reads all warp sums and takes its own
// offsets, so wsum must not be written again before the caller's next barrier.
template <int NT>
__device__ __forceinline__ void cta_scan3(const int v[3], int ex[3], int (*wsum)[33], int tot[3]) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int nw = NT / 32;
    int in[3];
#pragma unroll
    for (int q = 0; q < 3; q++) in[q] = v[q];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int q = 0; q < 3; q++) {
            int t = __shfl_up_sync(kFull, in[q], o);
            if (lane >= o) in[q] += t;
        }
    }
    if (lane == 31) {
#pragma unroll
        for (int q = 0; q < 3; q++) wsum[q][wid] = in[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; q++) {
        const int wt = lane < nw ? wsum[q][lane] : 0;
        ex[q] = __reduce_add_sync(kFull, lane < wid ? wt : 0) + in[q] - v[q];
        tot[q] = __reduce_add_sync(kFull, wt);
    }
}

// One thread's B' entry of a batch: its A~ segment and its value.
template <typename Acc>
struct SegReg {
    long long st = 0;
    int len = 0;
    Acc bv = Acc(0);
};

// The segment of this thread's entry in the first batch of [p0, p1); callers
// fetch it early so that its loads overlap their own set-up.
template <typename Acc, typename SegFn>
__device__ __forceinline__ SegReg<Acc> cta_first_seg(int64_t p0, int64_t p1, SegFn seg) {
    SegReg<Acc> r;
    if (p0 + threadIdx.x < p1) seg(p0 + threadIdx.x, r.st, r.len, r.bv);
    return r;
}

// A body that is called once per product, for the walks that need no more:
// each_product([&](int r, Acc v) { ... }).
template <typename F>
struct EachProduct {
    F f;
    template <int N, typename Acc, typename Crowded>
    __device__ __forceinline__ void operator()(const int (&r)[N], const Acc (&a)[N], const Acc (&b)[N],
                                               const bool (&ok)[N], Crowded) const {
#pragma unroll
        for (int u = 0; u < N; u++)
            if (ok[u]) f(r[u], mul_acc<Acc>(a[u], b[u]));
    }
};
template <typename F>
__device__ __forceinline__ EachProduct<F> each_product(F f) {
    return EachProduct<F>{f};
}

// Walk every product of the B' entries [p0, p1) of one output column with the
// whole CTA (all threads must call it; blockDim.x == NT); `first` is
// cta_first_seg(p0, p1, seg), and sb.clear() must have run once.
// seg(p, start, len, bv) gives the A~ positions [start, start+len) that B'
// entry p multiplies and its value; body(r, a, b, ok, crowded) takes this lane's
// next N products: rows r[u], the factors a[u] (from A~) and b[u] (from B'), and
// whether each exists; the whole warp calls it.  The segments of the next batch are fetched before the
// current batch is walked.
// Long segments (>= kMidSeg entries): a warp takes steps of 32 x U products,
// lanes reading consecutive entries, U loads per lane in flight.  A step inside
// one segment reads one base address, with the U windows at fixed offsets from
// it, and one B' value; a step that meets segment boundaries places every
// window by itself.
// Window segments (< kMidSeg entries, in order as far as they fit the windows;
// those below kLongSeg always do): U windows of 32 products in flight, every
// lane finding its segment from its window's bits, with no search and no chain
// from one window to the next.
// The long steps are shared evenly by the warps, the windows are claimed (few of
// them: shared by number).
// CROWD: body has a form for products that crowd on few rows (crowded is a true
// type, N is 1).  Warp 0 looks at the first window of every eighth batch that
// has a next one, and the batches after it take that form where it crowds
// (segments of 32 entries or more cannot: their rows are distinct).
// One batch must hold < 2^31 products (heavy items bound their segments to the
// item's row range).  Ends with a barrier.
template <bool NEED_VAL, int U, typename Acc, bool CROWD = false, int NT, typename SegFn, typename Body>
__device__ __forceinline__ void cta_products(int64_t p0, int64_t p1, CtaBatch<Acc, NT> &sb,
                                             const int32_t *__restrict__ At_row, const Acc *__restrict__ At_val,
                                             SegReg<Acc> first, SegFn seg, Body body) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int nw = NT / 32;
    constexpr int kShortWindows = CtaBatch<Acc, NT>::kShortWindows, kMidSeg = CtaBatch<Acc, NT>::kMidSeg;
    SegReg<Acc> cur = first;
    for (int64_t b0 = p0; b0 < p1; b0 += NT) {
        const long long st = cur.st;
        const int len = cur.len;
        const Acc bv = cur.bv;
        const bool crowd = CROWD && b0 > p0 && sb.crowded;  // (written between the barriers below)
        // the shortest class numbers its products from 0 (windows), the middle
        // one from there on (windows, as far as they go), the longest after
        // the middle class's own products (long part); counts packed in one
        // counter, products of the two shorter classes in another
        const int cls = len >= kMidSeg ? 0 : len >= kLongSeg ? 1 : 2;
        const int v[3] = {len > 0 ? 1 << (10 * cls) : 0, cls == 0 ? len : 0,
                          cls == 1 ? len : cls == 2 ? len << 16 : 0};
        int ex[3], tot[3];
        cta_scan3<NT>(v, ex, sb.wsum, tot);
        const int n0 = tot[0] & 1023, n1 = (tot[0] >> 10) & 1023, n2 = tot[0] >> 20;
        const int m1 = tot[2] & 0xffff, m2 = (int)((uint32_t)tot[2] >> 16);
        const bool all_mid = m1 + m2 <= 32 * kShortWindows;
        if (threadIdx.x == 0) sb.next = 0;
        if (len > 0) {
            const int e1 = ex[2] & 0xffff, e2 = (int)((uint32_t)ex[2] >> 16);
            const int i = cls == 0 ? n2 + n1 + (ex[0] & 1023)
                                   : cls == 1 ? n2 + ((ex[0] >> 10) & 1023) : (int)((uint32_t)ex[0] >> 20);
            if (cls == 0 || (cls == 1 && m2 + e1 + len > 32 * kShortWindows)) {
                const int f = cls == 0 ? m1 + ex[1] : e1;
                sb.start[i] = st - f;
                sb.pref[i] = f;
                if (cls == 1 && m2 + e1 <= 32 * kShortWindows) {  // the first of its class that does not fit
                    sb.cut[0] = i - n2;
                    sb.cut[1] = e1;
                }
            } else {
                const int f = cls == 1 ? m2 + e1 : e2;
                sb.start[i] = st - f;
                atomicOr(&sb.win[f >> 5].x, 1u << (f & 31));
                if ((f & 31) == 0) sb.win[f >> 5].y = (uint32_t)i;
                for (int w = (f >> 5) + 1; w <= (f + len - 1) >> 5; w++) sb.win[w].y = (uint32_t)i + 1u;
            }
            if (NEED_VAL) sb.bv[i] = bv;
        }
        __syncthreads();
        if constexpr (CROWD) {
            if (wid == 0 && b0 + NT < p1 && ((b0 - p0) / NT & 7) == 0) {
                // the first window is made of this warp's own short segments:
                // lane l's product belongs to the last one that begins by then
                const bool mine = cls == 2 && len > 0;
                const int e2 = (int)((uint32_t)ex[2] >> 16);
                const uint32_t M = __reduce_or_sync(kFull, mine && e2 < 32 ? 1u << e2 : 0u);
                const uint32_t segs = __ballot_sync(kFull, mine);
                const bool ok = lane < __shfl_sync(kFull, mine ? e2 + len : e2, 31);
                const int src = ok ? (int)__fns(segs, 0, __popc(M & (kFull >> (31 - lane)))) : 0;
                const long long at = __shfl_sync(kFull, st - e2, src) + lane;
                const bool crowds = window_crowds(ok ? __ldg(At_row + at) : ~lane);
                if (lane == 0) sb.crowded = crowds;
            }
        }
        if (b0 + NT < p1) cur = cta_first_seg<Acc>(b0 + NT, p1, seg);
        // window segments [0, ns) with products [0, nsp), long segments
        // [ns, n) with products [lp0, lp1)
        const int kmid = all_mid ? n1 : sb.cut[0];
        const int lp0 = all_mid ? m1 : sb.cut[1], lp1 = m1 + tot[1];
        const int n = n2 + n1 + n0, ns = n2 + kmid, nsp = m2 + lp0;
        const int nsteps = (lp1 - lp0 + 32 * U - 1) / (32 * U), nwin = (nsp + 31) >> 5;
        const int sper = nsteps / nw, srem = nsteps - sper * nw;

        // long segments: products [f0, f1) of this warp in the long
        // segments' own numbering (no padding between segments).  A long
        // segment holds >= 32 products, so a window of 32 consecutive products
        // meets at most two segments (the current one, A, and the next, B) and
        // crosses at most one boundary.
        {
            const int f0 = lp0 + (wid * sper + min(wid, srem)) * 32 * U;
            const int f1 = min(lp1, f0 + (sper + (wid < srem ? 1 : 0)) * 32 * U);
            if (f0 < f1) {
                int s = ns;
                for (int stp = NT >> 1; stp > 0; stp >>= 1)
                    if (s + stp < n && sb.pref[s + stp] <= f0) s += stp;
                long long baseA = sb.start[s];
                Acc bvA = NEED_VAL ? sb.bv[s] : Acc(0);
                int nB = s + 1 < n ? sb.pref[s + 1] : lp1;  // first product of B
                long long baseB = 0;
                Acc bvB = Acc(0);
                if (s + 1 < n) {
                    baseB = sb.start[s + 1];
                    if (NEED_VAL) bvB = sb.bv[s + 1];
                }
                auto advance = [&]() {  // B becomes A
                    s++;
                    baseA = baseB;
                    bvA = bvB;
                    nB = s + 1 < n ? sb.pref[s + 1] : lp1;
                    if (s + 1 < n) {
                        baseB = sb.start[s + 1];
                        if (NEED_VAL) bvB = sb.bv[s + 1];
                    }
                };
                // one step of N windows over segment boundaries: located and
                // loaded, then used
                auto step = [&](const int f, auto windows, auto full, auto crowded) {
                    constexpr int N = decltype(windows)::value;
                    constexpr bool FULL = decltype(full)::value;  // no lane past the warp's range
                    int r[N];
                    Acc a[N], bu[N];
                    bool ok[N];
#pragma unroll
                    for (int u = 0; u < N; u++) {
                        const int fb = f + 32 * u;
                        if (fb >= nB) advance();  // the window starts in B
                        const int fi = fb + lane;
                        const bool inB = fi >= nB;
                        const long long e = (inB ? baseB : baseA) + fi;
                        bu[u] = inB ? bvB : bvA;
                        ok[u] = FULL || fi < f1;
                        r[u] = 0;
                        a[u] = Acc(0);
                        if (ok[u]) {
                            r[u] = __ldg(At_row + e);
                            if (NEED_VAL) a[u] = __ldg(At_val + e);
                        }
                    }
                    body(r, a, bu, ok, crowded);
                };
                using One = std::integral_constant<int, 1>;
                using All = std::integral_constant<int, U>;
                int f = f0;
                if constexpr (CROWD) {
                    if (crowd)
                        for (; f < f1; f += 32) step(f, One{}, std::false_type{}, std::true_type{});
                }
                while (f < f1) {
                    if (f >= nB) advance();
                    const int lim = min(nB, f1);
                    if (f + 32 * U <= lim) {
                        const int32_t *rp = At_row + (baseA + f + lane);
                        const Acc *vp = At_val + (NEED_VAL ? baseA + f + lane : 0);
                        do {
                            int r[U];
                            Acc a[U], bu[U];
                            bool ok[U];
#pragma unroll
                            for (int u = 0; u < U; u++) {
                                r[u] = __ldg(rp + 32 * u);
                                a[u] = NEED_VAL ? __ldg(vp + 32 * u) : Acc(0);
                                bu[u] = bvA;
                                ok[u] = true;
                            }
                            body(r, a, bu, ok, std::false_type{});
                            f += 32 * U;
                            rp += 32 * U;
                            if (NEED_VAL) vp += 32 * U;
                        } while (f + 32 * U <= lim);
                    } else if (f + 32 * U <= f1) {
                        step(f, All{}, std::true_type{}, std::false_type{});
                        f += 32 * U;
                    } else {
                        step(f, One{}, std::false_type{}, std::false_type{});
                        f += 32;
                    }
                }
            }
        }
        // window segments: U windows at a time, claimed from a shared counter
        // (the next claim is made before the current windows are walked), so
        // that the warps finish together whatever their long steps took.  Up to
        // one window a warp they are shared by number, and so are U a warp where
        // there are no long steps: a batch of short segments waits for its claims
        // and leaves most warps idle otherwise (columns of 100,000 entries of B'
        // whose segments hold one row, int64: one slab 0.88 -> 0.81 ms, ten slabs
        // 2.72 -> 1.92, the fused learned pass 8.2 -> 5.4; with long steps the
        // claims are the better share: the betweenness batch 43.5 ms, 44.4 by number)
        {
            const uint32_t upto = kFull >> (31 - lane);
            auto step = [&](const int w, auto windows, auto full, auto crowded) {
                constexpr int N = decltype(windows)::value;
                constexpr bool FULL = decltype(full)::value;
                int r[N];
                Acc a[N], bu[N];
                bool ok[N];
#pragma unroll
                for (int u = 0; u < N; u++) {
                    const int fi = (w + u) * 32 + lane;
                    ok[u] = FULL || fi < nsp;
                    r[u] = 0;
                    a[u] = Acc(0);
                    bu[u] = Acc(0);
                    const uint2 x = sb.win[w + u];
                    if (ok[u]) {
                        const int k = (int)x.y + __popc(x.x & upto) - 1;
                        const long long e = sb.start[k] + fi;
                        r[u] = __ldg(At_row + e);
                        if (NEED_VAL) {
                            a[u] = __ldg(At_val + e);
                            bu[u] = sb.bv[k];
                        }
                    }
                }
                __syncwarp();
                if (lane < N) sb.win[w + lane].x = 0u;
                body(r, a, bu, ok, crowded);
            };
            auto claim = [&]() {
                int c = 0;
                if (lane == 0) c = atomicAdd(&sb.next, U);
                return __shfl_sync(kFull, c, 0);
            };
            using One = std::integral_constant<int, 1>;
            if (CROWD && crowd) {
                if constexpr (CROWD)
                    for (int w = wid; w < nwin; w += nw) step(w, One{}, std::false_type{}, std::true_type{});
            } else if (nwin <= nw) {
                if (wid < nwin) step(wid, One{}, std::false_type{}, std::false_type{});
            } else {
                const bool few = nsteps == 0 && nwin <= nw * U;  // one claim a warp: its own number
                for (int w = few ? wid * U : claim(); w < nwin;) {
                    const int wnext = few ? nwin : claim();
                    if ((w + U) * 32 <= nsp) {
                        step(w, std::integral_constant<int, U>{}, std::true_type{}, std::false_type{});
                    } else {
                        for (; w < nwin; w++) step(w, One{}, std::false_type{}, std::false_type{});
                    }
                    w = wnext;
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace spg
