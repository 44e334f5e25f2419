// A whole warp on one output column: the walk over its products, the
// open-addressing table of its rows, and its entries in row order (the light
// columns of the symbolic, numeric, learned, batched and one-launch kernels).
#pragma once

#include "block_ops.cuh"
#include "spg_internal.cuh"

namespace spg {

// Staging of up to 32 non-empty A~ segments: start is the segment's first entry
// minus its first product's number.
template <typename Acc>
struct WarpSeg {
    long long start[32];
    Acc bv[32];
};

// Stage the segments of the B' entries p0 + at .. p0 + at + 31 (below p0 + n): the
// number of their products; `first` is this lane's first one (INT32_MAX for an
// empty one).
template <bool NEED_VAL, typename Acc, typename SegFn>
__device__ __forceinline__ int warp_stage(int64_t p0, int at, int n, int lane, WarpSeg<Acc> &ws, SegFn &seg,
                                          int &first) {
    long long st = 0;
    int len = 0;
    Acc bv = Acc(0);
    if (at + lane < n) seg(p0 + at + lane, st, len, bv);
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    const int total = __shfl_sync(kFull, incl, 31);
    first = len > 0 ? incl - len : INT32_MAX;
    const uint32_t some = __ballot_sync(kFull, len > 0);
    if (len > 0) {
        const int i = __popc(some & ((1u << lane) - 1u));
        ws.start[i] = st - first;
        if (NEED_VAL) ws.bv[i] = bv;
    }
    __syncwarp();
    return total;
}

// The windows of a staged batch.
template <bool NEED_VAL, int U, bool CROWDED, typename Acc, typename ValFn, typename Body>
__device__ __forceinline__ void warp_windows(int total, int first, int lane, const WarpSeg<Acc> &ws,
                                             const int32_t *__restrict__ At_row, ValFn &aval, Body &body) {
    const uint32_t upto = kFull >> (31 - lane);
    int begun = -1;  // last segment begun before the window
    for (int f0 = 0; f0 < total; f0 += 32 * U) {
        int r[U];
        Acc a[U], b[U];
        bool ok[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int f = f0 + 32 * u;
            ok[u] = f + lane < total;
            r[u] = 0;
            a[u] = Acc(0);
            b[u] = Acc(0);
            if (f < total) {
                const uint32_t d = (uint32_t)(first - f);
                const uint32_t M = __reduce_or_sync(kFull, d < 32u ? 1u << d : 0u);
                const int k = begun + __popc(M & upto);
                begun += __popc(M);
                if (ok[u]) {
                    const long long e = ws.start[k] + (f + lane);
                    r[u] = __ldg(At_row + e);
                    if (NEED_VAL) {
                        a[u] = aval(e);
                        b[u] = ws.bv[k];
                    }
                }
            }
        }
        body(r, a, b, ok, min(U, (total - f0 + 31) >> 5), std::integral_constant<bool, CROWDED>{});
    }
    __syncwarp();
}

// Walk every product of the B' entries [p0, p1) of one output column with a
// whole warp.  seg(p, start, len, bv) gives the A~ positions [start, start+len)
// that B' entry p multiplies and its value; aval(e) loads A~'s value e.  The
// products of 32 consecutive entries are numbered consecutively; a window of 32
// products finds its segments from one bit per segment start (an OR over the
// lanes), so all 32 lanes stay busy however short the segments are.  U windows
// are located and loaded before any of them is used.  body(r, a, b, ok, windows,
// crowded) is called by the whole warp for a step's windows at once: `windows` of
// them hold products, one per lane where ok[u].  (Called for every window by
// itself: 32,000 products of 1000 rows a column 1.05 ms in doubles and 0.95 in int64,
// 0.95 and 0.83 so; columns of few products take the same time.)
// CROWD: the body has a form for products that crowd on few rows (crowded is a
// true type); a column of more than 32 entries takes it for 256 entries at a time
// whose first window of products crowds (fewer entries bring at most as many
// products of one row: not worth the look).
template <bool NEED_VAL, int U, typename Acc, bool CROWD = false, typename SegFn, typename ValFn, typename Body>
__device__ __forceinline__ void warp_walk(int64_t p0, int64_t p1, int lane, WarpSeg<Acc> &ws,
                                          const int32_t *__restrict__ At_row, SegFn seg, ValFn aval, Body body) {
    const int n = (int)(p1 - p0);  // (at most k < 2^31 - 1)
    bool crowds = false;
    for (int at = 0; at < n; at += 32) {
        int first;
        const int total = warp_stage<NEED_VAL>(p0, at, n, lane, ws, seg, first);
        if constexpr (CROWD) {
            if (n > 32 && (at & 255) == 0) {
                const uint32_t M = __reduce_or_sync(kFull, first < 32 ? 1u << first : 0u);
                const int k = __popc(M & (kFull >> (31 - lane))) - 1;
                crowds = window_crowds(lane < total ? __ldg(At_row + ws.start[k] + lane) : ~lane);
            }
            if (crowds) {
                warp_windows<NEED_VAL, 1, true>(total, first, lane, ws, At_row, aval, body);
                continue;
            }
        }
        warp_windows<NEED_VAL, U, false>(total, first, lane, ws, At_row, aval, body);
    }
}

// Slot of row r (where ok) in this warp's table of 2^logS row ids, inserting it
// if absent; the whole warp calls it.  A lane that finds its slot free stores
// its row there and reads it back: one of several stores to a slot stays, and
// the lanes that stored another row go on probing.  (The table belongs to one
// warp, so no compare-and-swap is needed: it retires 0.8 lanes per clock per SM
// on this GPU, a store and a load 8 or more.)  A lane that finds a row reads
// once: where nearly every product's row is in the table already and few warps
// are resident, the second read was waited for in every probe (32,000 int64
// products of 1000 rows a column: 0.98 -> 0.95 ms, learned 0.85 -> 0.82; the
// batch of 20 products 12.9 -> 12.7).  -1 where the table is full.
__device__ __forceinline__ int warp_hash_slot(int *keys, int logS, int r, bool ok) {
    const unsigned mask = (1u << logS) - 1u;
    const unsigned x = (unsigned)r * 0x9E3779B1u;
    unsigned h = x >> (32 - logS);
    const unsigned step = (x >> 3) | 1u;  // odd: visits every slot
    volatile int *vk = keys;
    bool pend = ok;
    for (unsigned probe = 0; probe <= mask; probe++) {
        int k = pend ? vk[h] : r;
        const bool empty = k == kEmptyKey;
        if (empty) vk[h] = r;
        __syncwarp();
        if (empty) k = vk[h];
        pend = k != r;
        if (!__any_sync(kFull, pend)) return (int)h;
        if (pend) h = (h + step) & mask;
    }
    return pend ? -1 : (int)h;
}

// Rows of a step's windows into a table, without values; false if it is full.
template <int N>
__device__ __forceinline__ bool warp_hash_rows(int *keys, int logS, const int (&r)[N], const bool (&ok)[N],
                                               int windows) {
    bool there = true;
#pragma unroll
    for (int u = 0; u < N; u++)
        if (u < windows && warp_hash_slot(keys, logS, r[u], ok[u]) < 0 && ok[u]) there = false;
    return there;
}

// Clear `ok` where an output mask drops the product.
template <int N>
__device__ __forceinline__ void mask_products(const OutMask &mask, int j, const int (&r)[N], bool (&ok)[N]) {
    if (mask.bits) {
#pragma unroll
        for (int u = 0; u < N; u++)
            if (ok[u] && !mask_keeps(mask, j, r[u])) ok[u] = false;
    }
}

// Fill the 2^logS (>= 32) entries of a table, 16-byte aligned, with empty keys.
__device__ __forceinline__ void warp_clear_keys(int *keys, int logS, int lane) {
    int4 *k4 = (int4 *)keys;
    for (int s = lane; s < (1 << logS) / 4; s += 32) k4[s] = make_int4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey);
}
// Zero `bytes` (a multiple of 16) of shared memory.
__device__ __forceinline__ void warp_zero(void *p, int bytes, int lane) {
    uint4 *q = (uint4 *)p;
    for (int s = lane; s < bytes / 16; s += 32) q[s] = make_uint4(0u, 0u, 0u, 0u);
}
// Occupied slots of a table.
__device__ __forceinline__ int warp_count_keys(const int *keys, int logS, int lane) {
    const int4 *k4 = (const int4 *)keys;
    int c = 0;
    for (int s = lane; s < (1 << logS) / 4; s += 32) {
        const int4 k = k4[s];
        c += (k.x != kEmptyKey) + (k.y != kEmptyKey) + (k.z != kEmptyKey) + (k.w != kEmptyKey);
    }
    return warp_sum_i(c);
}

// Sort rows[0..n) ascending with the positions they came from (idx[i] = i to
// begin with): LSD radix by the fewest passes of at most 8 bits that cover the
// largest row, ping-pong with rows[half..half + n) and idx[half..half + n); a
// pass is stable because 32 entries at a time are scattered in order and lanes
// of one digit are ranked by __match_any_sync.  hist: 256 (512) 16-bit counters.
// Returns the offset (0 or half) of the sorted lists.
__device__ __forceinline__ int warp_sort_rows(int *rows, uint16_t *idx, int n, int half, uint16_t *hist, int lane) {
    int kmax = 0;
    for (int s = lane; s < n; s += 32) {
        kmax = max(kmax, rows[s]);
        idx[s] = (uint16_t)s;
    }
    kmax = __reduce_max_sync(kFull, kmax);
    const int most = half >= 256 ? 9 : 8;
    const int bits = max(1, 32 - __clz(kmax)), passes = (bits + most - 1) / most, width = (bits + passes - 1) / passes;
    const int groups = width == 9 ? 2 : 1;  // of 8 counters per lane
    const unsigned dmask = (1u << width) - 1u, below = (1u << lane) - 1u;
    uint4 *h4 = (uint4 *)hist;
    unsigned *h1 = (unsigned *)hist;
    int from = 0;
    for (int shift = 0; shift < bits; shift += width) {
        for (int g = 0; g < groups; g++) h4[32 * g + lane] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        for (int s = lane; s < n; s += 32) {
            const unsigned d = ((unsigned)rows[from + s] >> shift) & dmask;
            atomicAdd(h1 + (d >> 1), 1u << (16 * (d & 1)));
        }
        __syncwarp();
        // exclusive scan of the counts, 256 at a time, 8 consecutive per lane
        unsigned before = 0;
        for (int g = 0; g < groups; g++) {
            const uint4 c = h4[32 * g + lane];
            const unsigned w[4] = {c.x, c.y, c.z, c.w};
            unsigned tot = 0, e[4];
#pragma unroll
            for (int u = 0; u < 4; u++) tot += (w[u] & 0xffffu) + (w[u] >> 16);
            unsigned incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned x = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += x;
            }
            unsigned run = before + incl - tot;
            before += __shfl_sync(kFull, incl, 31);
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const unsigned lo = w[u] & 0xffffu;
                e[u] = run | ((run + lo) << 16);
                run += lo + (w[u] >> 16);
            }
            h4[32 * g + lane] = make_uint4(e[0], e[1], e[2], e[3]);
        }
        __syncwarp();
        const int to = from ^ half;
        for (int c0 = 0; c0 < n; c0 += 32) {
            const int s = c0 + lane;
            const bool valid = s < n;
            const int k = valid ? rows[from + s] : 0;
            const uint16_t q = valid ? idx[from + s] : (uint16_t)0;
            const unsigned d = valid ? ((unsigned)k >> shift) & dmask : 512u + lane;
            const unsigned peers = __match_any_sync(kFull, d);
            const int rank = __popc(peers & below);
            const int pos = valid ? (int)hist[d] + rank : 0;
            __syncwarp();
            if (valid) {
                rows[to + pos] = k;
                idx[to + pos] = q;
                if (rank == 0) hist[d] = (uint16_t)(pos + __popc(peers));
            }
            __syncwarp();
        }
        from = to;
    }
    return from;
}

// One warp's numeric table of 2^logS slots: 8 bytes of value and 4 of row a
// slot.  Once its n <= 2^(logS - 1) entries are compacted to the front of both
// arrays, the upper halves of the values (of both 32-bit planes for int64) hold
// the sort's position lists and counters, so the table needs no more room: its
// size is what limits the warps resident on an SM.
template <typename Acc>
struct WarpTable {
    unsigned char *base;
    int logS;
    static constexpr __host__ __device__ size_t bytes(int logS) { return (size_t)12 << logS; }
    __device__ __forceinline__ WarpTable(unsigned char *b, int l) : base(b), logS(l) {}
    __device__ __forceinline__ HeavyAcc<Acc> acc() const { return HeavyAcc<Acc>(base, 1 << logS); }
    __device__ __forceinline__ int *keys() const { return (int *)(base + ((size_t)8 << logS)); }
    __device__ __forceinline__ void clear(int lane) const {
        warp_zero(base, 8 << logS, lane);
        warp_clear_keys(keys(), logS, lane);
        __syncwarp();
    }
    // body of warp_walk: the products of a step's windows into their slots; false if
    // the table is full
    template <bool CROWDED, int N>
    __device__ __forceinline__ bool add(const HeavyAcc<Acc> &acc, const int (&r)[N], const Acc (&a)[N],
                                        const Acc (&b)[N], const bool (&ok)[N], int windows) const {
        bool good = true;
#pragma unroll
        for (int u = 0; u < N; u++)
            if (u < windows) {
                const int slot = warp_hash_slot(keys(), logS, r[u], ok[u]);
                const uint32_t ad[1] = {acc.addr(max(slot, 0))};
                const Acc x[1] = {a[u]}, y[1] = {b[u]};
                const bool o[1] = {ok[u] && slot >= 0};
                if (!(add_to<CROWDED>(acc, ad, x, y, o) && (slot >= 0 || !ok[u]))) good = false;
            }
        return good;
    }
    // Move the occupied slots' rows and values to the front; returns their
    // number.  (A write never reaches a slot of a later, still unread chunk.)
    __device__ __forceinline__ int compact(const HeavyAcc<Acc> &acc, int lane) const {
        int *k_ = keys();
        int n = 0;
        for (int c0 = 0; c0 < (1 << logS); c0 += 32) {
            const int k = k_[c0 + lane];
            const Acc v = acc.get(c0 + lane);
            const unsigned bal = __ballot_sync(kFull, k != kEmptyKey);
            __syncwarp();
            if (k != kEmptyKey) {
                const int pos = n + __popc(bal & ((1u << lane) - 1u));
                k_[pos] = k;
                acc.set(pos, v);
            }
            n += __popc(bal);
            __syncwarp();
        }
        return n;
    }
    // Call out(position, row, value) for the n <= 2^(logS - 1) compacted
    // entries, the position being the row's rank.  Up to 64 entries a lane
    // counts the smaller rows of its one or two (broadcast 16-byte loads, no
    // chain: a bitonic network's 15 or 21 dependent exchanges wait longer than
    // they compute); above, a radix sort.
    template <typename Out>
    __device__ __forceinline__ void emit(const HeavyAcc<Acc> &acc, int n, int lane, Out out) const {
        int *k_ = keys();
        if (n <= 64) {
            if (lane < 4 && n + lane < (1 << logS)) k_[n + lane] = INT32_MAX;  // whole groups of four
            __syncwarp();
            const int a = lane < n ? k_[lane] : INT32_MAX, b = lane + 32 < n ? k_[lane + 32] : INT32_MAX;
            int ra = 0, rb = 0;
            const int4 *k4 = (const int4 *)k_;
            for (int i = 0; i < (n + 3) / 4; i++) {
                const int4 k = k4[i];
                ra += (k.x < a) + (k.y < a) + (k.z < a) + (k.w < a);
                if (n > 32) rb += (k.x < b) + (k.y < b) + (k.z < b) + (k.w < b);
            }
            if (lane < n) out(ra, a, acc.get(lane));
            if (lane + 32 < n) out(rb, b, acc.get(lane + 32));
        } else {
            uint16_t *idx = (uint16_t *)(base + ((size_t)(HeavyAcc<Acc>::slot_shift == 3 ? 4 : 2) << logS));
            uint16_t *hist = (uint16_t *)(base + ((size_t)6 << logS));
            const int at = warp_sort_rows(k_, idx, n, 1 << (logS - 1), hist, lane);
            for (int s = lane; s < n; s += 32) out(s, k_[at + s], acc.get(idx[at + s]));
        }
        __syncwarp();
    }
};

}  // namespace spg
