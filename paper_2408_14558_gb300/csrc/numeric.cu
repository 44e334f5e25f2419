// Numeric pass: the rows and values of C (Algorithm 1, local multiply
// C_i = A~_i * B_i, Gustavson column by column), written at the column
// pointers produced by the symbolic pass.
//   light bins: one warp per column, shared open-addressing table of
//               (row, value) sized >= 2 x nnz_j; afterwards the rows are
//               compacted and put in order (warp_hash.cuh)
//   heavy bin:  one CTA per (column, row slab): the symbolic bitmap of the
//               slab gives every present row its rank, products accumulate at
//               acc[rank] in shared memory, and the slab is written out in row
//               order with no sort
#include <algorithm>
#include <type_traits>

#include "block_ops.cuh"
#include "cta_products.cuh"
#include "spg_internal.cuh"
#include "warp_hash.cuh"

namespace spg {

// Small tables (up to 256 slots): 32 registers a thread and two windows in
// flight (one, see below) keep up to 64 warps on an SM.  Kernel time for 200,003 columns of doubles,
// so | without the bound and with four windows: 36 products a column (128 slots)
// 253 | 286 us, 64 products 323 | 356, 100 products (256 slots, of which shared
// memory holds seven CTAs) 686 | 746; int64 the same within 2%.  Six CTAs of
// 256-slot tables instead were 4% faster for int64 and 8% slower for doubles.
// Doubles in 64-slot tables take one window at a time (what two keep in registers
// spills): 9 products a column 151 -> 142 us, 25 products 189 -> 179, the refresh of
// A * P_agg on a 128^3 grid 342 -> 332 us; in int64 25 products would take 175 ->
// 178 us, in 128 slots both are the same, in 256 slots one is 5% slower.
// Tables of four times the entries instead of two made no difference.
template <int LOGS, typename Acc>
constexpr int kLightWindows = LOGS <= 6 && std::is_same<Acc, double>::value ? 1 : LOGS <= 8 ? 2 : 4;
template <int LOGS, int WARPS, typename Acc, typename OutIdx>
__global__ void __launch_bounds__(WARPS * 32, LOGS <= 8 ? 8 : 1)
    k_num_light(const int32_t *__restrict__ list, int64_t ncols, const void *Bcolptr, int p64,
                const int32_t *__restrict__ Bq, const Acc *__restrict__ Bv, const int64_t *__restrict__ At_colptr,
                const int32_t *__restrict__ At_row, const Acc *__restrict__ At_val,
                const int64_t *__restrict__ Ccolptr, OutIdx *__restrict__ Crow, Acc *__restrict__ Cval, int *err,
                OutMask mask) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WarpSeg<Acc> *segs = (WarpSeg<Acc> *)smem_raw;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const WarpTable<Acc> tab((unsigned char *)(segs + WARPS) + wid * WarpTable<Acc>::bytes(LOGS), LOGS);
    const HeavyAcc<Acc> acc = tab.acc();
    for (int64_t c = (int64_t)blockIdx.x * WARPS + wid; c < ncols; c += (int64_t)gridDim.x * WARPS) {
        const int j = list[c];
        const int64_t p0 = ld_ptr(Bcolptr, p64, j), p1 = ld_ptr(Bcolptr, p64, j + 1);
        const int64_t base = Ccolptr[j], want = Ccolptr[j + 1] - base;
        tab.clear(lane);
        bool full = false;
        warp_walk<true, kLightWindows<LOGS, Acc>, Acc, HeavyAcc<Acc>::crowds>(
            p0, p1, lane, segs[wid], At_row,
            [&](int64_t p, long long &st, int &len, Acc &bv) {
                int q = Bq[p];
                if (q >= 0) {
                    st = At_colptr[q];
                    len = (int)(At_colptr[q + 1] - st);
                    bv = Bv[p];
                }
            },
            [&](long long e) { return __ldg(At_val + e); },
            [&](const auto &r, const auto &a, const auto &b, auto &ok, int windows, auto crowded) {
                mask_products(mask, j, r, ok);
                if (!tab.template add<decltype(crowded)::value>(acc, r, a, b, ok, windows)) full = true;
            });
        __syncwarp();
        const int nout = tab.compact(acc, lane);
        if (nout != want) {
            full = true;
        } else {
            tab.emit(acc, nout, lane, [&](int pos, int row, Acc v) {
                st_stream(Crow + base + pos, (OutIdx)row);
                st_stream(Cval + base + pos, v);
            });
        }
        if (__any_sync(kFull, full) && lane == 0) atomicOr(err, kDevErrInternal);
        __syncwarp();
    }
}

// Slots of a numeric item's accumulator beyond its capacity: the guard slot,
// and room to clear it 16 bytes at a time.
constexpr int kAccPad = 4;
// Rows of a direct item at most: its row list (2 bytes a row) sits in the rank
// table's area behind the item's own words (8 bytes per 32 rows).
constexpr int kDirectRows = kNumMaxWords * 8 * 4 / 9;

// Everything a numeric item needs before its first product, in one record.
struct NumItem {
    int32_t j, t0, nr, cnt, r0, pad;
    long long cbase, p0, p1;  // first entry of the item in C; B(:, j) = [p0, p1)
};

__global__ void k_num_headers(int64_t nitems, const int32_t *__restrict__ num_rec0,
                              const int32_t *__restrict__ num_nrec, const int32_t *__restrict__ rec_col,
                              const int32_t *__restrict__ rec_slab, const int32_t *__restrict__ rec_cnt,
                              const int64_t *__restrict__ rec_off, const void *Bcolptr, int p64,
                              const int64_t *__restrict__ Ccolptr, NumItem *__restrict__ items) {
    for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < nitems;
         it += (int64_t)gridDim.x * blockDim.x) {
        NumItem h;
        h.r0 = num_rec0[it];
        h.nr = num_nrec[it];
        h.j = rec_col[h.r0];
        h.t0 = rec_slab[h.r0];
        int cnt = 0;
        for (int rr = 0; rr < h.nr; rr++) cnt += rec_cnt[h.r0 + rr];
        h.cnt = cnt;
        h.pad = 0;
        h.cbase = Ccolptr[h.j] + rec_off[h.r0];
        h.p0 = ld_ptr(Bcolptr, p64, h.j);
        h.p1 = ld_ptr(Bcolptr, p64, h.j + 1);
        items[it] = h;
    }
}

// One CTA per numeric item: records [r0, r0 + nr) of one heavy column (base
// slabs t0 .. t0 + nr - 1) holding cnt <= cap entries of C.  The symbolic
// bitmaps of the records give every present row its rank; products accumulate
// in shared memory and the item is then written at its final place in C.
//   rank items: a row's slot is its rank (cta_load_rank_table).  Slot 0 is a
//     guard: the rank of a row counts its own bit, so entry i sits in slot
//     i + 1, and a row missing from a bitmap (never expected) still lands
//     inside the accumulator.  Values and rows are written each as one
//     coalesced run.
//   direct items: the item's rows all have a slot (nr * R <= cap and
//     kDirectRows, the dense items, whose 4096 entries span one slab): a row's
//     slot is its offset,
//     with no table look-up per product (and no conflicting look-ups: a
//     segment's rows are distinct).
// Thread 0 claims the next item when the current one starts and fetches its
// header while the current one is written out.  MASKED: the bitmaps hold only
// the rows an output mask admits, and a product whose row is absent is dropped
// (rank items) or accumulated into a slot that is not written (direct items).
// What bounds it: the shared-memory pipe in the walk (l1tex wavefronts 66% of
// the whole kernel for int64, 73% for doubles on a 50,000-vertex R-MAT graph,
// of which 8 + 9 a window are the doubles' exchange and store) and, on sparse
// items, the barriers and latencies between an item's phases (about half of its
// time; issue slots 53-63% busy).  Measured against the walk that placed every
// window across segments, with 8-byte look-ups and atomicAdd(double): squaring
// an R-MAT graph of 262,144 vertices in doubles 65.6 -> 49.3 ms, of 100,003 in
// int64 5.4 -> 4.4 ms, one 25,000-column chunk of the similarity product (dense
// items) 39.6 -> 26.0 ms.
template <typename Acc, typename OutIdx, bool MASKED, int NT>
__global__ void __launch_bounds__(NT, SPG_NUM_MINB * kBatch / NT)
    k_num_heavy(int64_t nitems, const NumItem *__restrict__ items, const uint32_t *__restrict__ hbits,
                const int32_t *__restrict__ Bq, const Acc *__restrict__ Bv, const int64_t *__restrict__ At_colptr,
                const int32_t *__restrict__ At_row, const Acc *__restrict__ At_val,
                const int32_t *__restrict__ split, int T, int R, int cap, OutIdx *__restrict__ Crow,
                Acc *__restrict__ Cval, int *err, unsigned long long *next) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int RW = R >> 5;
    constexpr int kSlotShift = HeavyAcc<Acc>::slot_shift;
    CtaBatch<Acc, NT> &sb = *(CtaBatch<Acc, NT> *)smem_raw;
    unsigned char *acc_raw = smem_raw + ((sizeof(CtaBatch<Acc, NT>) + 15) & ~(size_t)15);
    const HeavyAcc<Acc> acc(acc_raw, cap + kAccPad);
    uint2 *tab = (uint2 *)(acc_raw + HeavyAcc<Acc>::bytes_per_slot * (size_t)(cap + kAccPad));  // rank table
    __shared__ int ctot[kNumMaxWords / 128];
    __shared__ int bad_sh;
    __shared__ long long claim;
    __shared__ NumItem hdr;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int nw = NT / 32;
    const uint32_t slot0 = acc.addr(0);
    sb.clear();
    if (tid == 0) {
        bad_sh = 0;
        const long long it = (long long)atomicAdd(next, 1ull);
        claim = it;
        if (it < nitems) hdr = items[it];
    }
    __syncthreads();
    for (;;) {
        const int64_t it = claim;
        if (it >= nitems) break;
        const NumItem h = hdr;
        unsigned long long nxt = 0;
        if (tid == 0) nxt = atomicAdd(next, 1ull);
        const int t0 = h.t0, nr = h.nr;
        const int nwords = nr * RW;
        auto seg = [&](int64_t p, long long &st, int &len, Acc &bv) {
            int q = Bq[p];
            if (q >= 0) {
                const int32_t *sp = split + (int64_t)q * (T + 1);
                int a = sp[t0], b = sp[t0 + nr];
                st = At_colptr[q] + a;
                len = b - a;
                bv = Bv[p];
            }
        };
        const SegReg<Acc> first = cta_first_seg<Acc>(h.p0, h.p1, seg);
        const uint32_t *src = hbits + (int64_t)h.r0 * RW;
        const bool direct = nr * R <= min(cap, kDirectRows);
        const int cnt = cta_load_rank_table<kNumMaxWords / (4 * NT), NT>(src, tab, nwords, ctot);
        const int64_t rbase = (int64_t)t0 * R;
        NumItem nh;
        if (cnt == h.cnt && cnt <= cap) {
            // (the first barrier of cta_products orders the zeroing before
            // every product)
            acc.zero_all(direct ? nr * R : cnt + 1);
            bool miss = false;
            if (direct) {
                const uint32_t base = slot0 - ((uint32_t)rbase << kSlotShift);
                cta_products<true, SPG_NUM_UNROLL, Acc, HeavyAcc<Acc>::crowds>(
                    h.p0, h.p1, sb, At_row, At_val, first, seg,
                    [&](const auto &r, const auto &a, const auto &b, const auto &ok, auto crowded) {
                        constexpr int N = sizeof(r) / sizeof(r[0]);
                        uint32_t ad[N];
#pragma unroll
                        for (int u = 0; u < N; u++) {
                            ad[u] = base + ((uint32_t)r[u] << kSlotShift);
#if SPG_CHECK_MEMBERSHIP
                            if (ok[u]) miss |= !MASKED && !((rank_word(tab[(r[u] - (int)rbase) >> 5]) >> (r[u] & 31)) & 1u);
#endif
                        }
                        if (!add_to<decltype(crowded)::value>(acc, ad, a, b, ok)) miss = true;
                    });
            } else {
                const uint32_t *ranks = (const uint32_t *)tab - 2 * t0 * RW;
                cta_products<true, SPG_NUM_UNROLL, Acc, HeavyAcc<Acc>::crowds>(
                    h.p0, h.p1, sb, At_row, At_val, first, seg,
                    [&](const auto &r, const auto &a, const auto &b, const auto &ok, auto crowded) {
                        constexpr int N = sizeof(r) / sizeof(r[0]);
                        uint32_t ad[N];
                        bool keep[N];
#pragma unroll
                        for (int u = 0; u < N; u++) {
                            ad[u] = slot0;
                            keep[u] = ok[u];
                            if (ok[u]) {
                                const uint32_t e = ranks[r[u] >> 4];
                                const uint32_t upto = rank_upto(e, r[u]);
                                ad[u] = acc.addr(rank1(e, upto));
                                if constexpr (MASKED) {
                                    keep[u] = (int)upto < 0;  // the row's own bit
                                } else {
#if SPG_CHECK_MEMBERSHIP
                                    // a row missing from the symbolic bitmap
                                    // goes to the guard slot and is reported
                                    if ((int)upto >= 0) {
                                        miss = true;
                                        ad[u] = slot0;
                                    }
#endif
                                }
                            }
                        }
                        if (!add_to<decltype(crowded)::value>(acc, ad, a, b, keep)) miss = true;
                    });
            }
            if (miss) bad_sh = 1;
            if (tid == 0 && (long long)nxt < nitems) nh = items[nxt];
            // cta_products ends with a barrier: acc is complete.  The writing
            // threads start so that every warp writes whole aligned lines of C
            // (a warp's 32 row ids are one 128-byte line, its values two): over
            // the CPU-GPU link a line written in parts crosses in parts.
            Acc *cval = Cval + h.cbase;
            OutIdx *crow = Crow + h.cbase;
            const int v0 = tid - (int)(((uintptr_t)cval / sizeof(Acc)) & 31);
            const int r0 = tid - (int)(((uintptr_t)crow / sizeof(OutIdx)) & 31);
            if (direct) {
                // the rows by rank (16-bit offsets behind the item's words),
                // then values and rows as coalesced runs
                uint16_t *srow = (uint16_t *)(tab + nwords);
                for (int w = wid; w < nwords; w += nw) {
                    const uint2 e = tab[w];
                    const uint32_t word = rank_word(e);
                    if ((word >> lane) & 1u)
                        srow[rank_before(e) + __popc(word & ((1u << lane) - 1u))] = (uint16_t)(w * 32 + lane);
                }
                __syncthreads();
                for (int i = v0; i < cnt; i += NT)
                    if (i >= 0) st_stream(cval + i, acc.get(srow[i]));
                for (int i = r0; i < cnt; i += NT)
                    if (i >= 0) st_stream(crow + i, (OutIdx)(rbase + srow[i]));
            } else {
                for (int i = v0; i < cnt; i += NT)
                    if (i >= 0) st_stream(cval + i, acc.get(i + 1));
                __syncthreads();
                // the row ids go to shared memory by rank first (over the
                // consumed values: cnt ints fit in the first cnt slots), then
                // to C in one coalesced run
                int32_t *srow = acc.scratch32();
                for (int w = tid; w < nwords; w += NT) {
                    const uint2 e = tab[w];
                    uint32_t word = rank_word(e);
                    int pos = rank_before(e);
                    while (word) {
                        int bb = __ffs(word) - 1;
                        srow[pos++] = w * 32 + bb;
                        word &= word - 1u;
                    }
                }
                __syncthreads();
                for (int i = r0; i < cnt; i += NT)
                    if (i >= 0) st_stream(crow + i, (OutIdx)(rbase + srow[i]));
            }
        } else {
            // the item's room in C was sized from the record counts: never
            // write past it
            if (tid == 0) {
                bad_sh = 1;
                if ((long long)nxt < nitems) nh = items[nxt];
            }
        }
        if (tid == 0) {
            claim = (long long)nxt;
            if ((long long)nxt < nitems) hdr = nh;
        }
        __syncthreads();
    }
    if (tid == 0 && bad_sh) atomicOr(err, kDevErrInternal);
}

template <int LOGS, int WARPS, typename Acc, typename OutIdx>
static spg_status launch_num_light(spg_plan *p, const int32_t *list, int64_t cnt, spg_csc *C) {
    size_t smem = (sizeof(WarpSeg<Acc>) + WarpTable<Acc>::bytes(LOGS)) * WARPS;
    auto kern = k_num_light<LOGS, WARPS, Acc, OutIdx>;
    struct Tag {};
    int g = grid_for(cnt, WARPS, p->sm_count * resident_ctas<Tag>(p, kern, WARPS * 32, smem));
    launch(p, kern, g, WARPS * 32, smem, list, cnt, p->B.colptr, p->B.ptr_type == SPG_IDX_I64, p->Bq,
                                         (const Acc *)p->Bv, p->At_colptr, p->At_row, (const Acc *)p->At_val,
                                         p->Ccolptr, (OutIdx *)C->rowidx, (Acc *)C->vals, p->d_err, p->omask);
    return cuda_check(cudaGetLastError(), "numeric light");
}

template <typename Acc, typename OutIdx>
static spg_status numeric_typed(spg_plan *p, spg_csc *C) {
    spg_status s = SPG_OK;
    const bool any_light = p->nbin_off[kMaxLightBin + 1] > p->nbin_off[1];
    if (any_light) group_begin(p, kKNumLight);
    for (int bin = 1; bin <= kMaxLightBin && !s; bin++) {
        int64_t cnt = p->nbin_off[bin + 1] - p->nbin_off[bin];
        if (cnt == 0) continue;
        const int32_t *list = p->nbinlist + p->nbin_off[bin];
        switch (bin) {
            case 1: s = launch_num_light<6, 8, Acc, OutIdx>(p, list, cnt, C); break;
            case 2: s = launch_num_light<7, 8, Acc, OutIdx>(p, list, cnt, C); break;
            case 3: s = launch_num_light<8, 8, Acc, OutIdx>(p, list, cnt, C); break;
            case 4: s = launch_num_light<9, 8, Acc, OutIdx>(p, list, cnt, C); break;
            case 5: s = launch_num_light<10, 8, Acc, OutIdx>(p, list, cnt, C); break;
            default: s = launch_num_light<11, 4, Acc, OutIdx>(p, list, cnt, C); break;
        }
    }
    if (any_light) group_end(p, kKNumLight);
    if (s) return s;
    if (p->nnum > 0) {
        const bool wide = p->num_wide;
        const int threads = wide ? kWideBatch : kBatch;
        const size_t staging = wide ? sizeof(CtaBatch<Acc, kWideBatch>) : sizeof(CtaBatch<Acc>);
        size_t smem = ((staging + 15) & ~(size_t)15) + sizeof(Acc) * (size_t)(p->num_cap + kAccPad) +
                      sizeof(uint2) * (size_t)kNumMaxWords;
        auto kern = wide            ? k_num_heavy<Acc, OutIdx, true, kWideBatch>
                    : p->omask.bits ? k_num_heavy<Acc, OutIdx, true, kBatch>
                                    : k_num_heavy<Acc, OutIdx, false, kBatch>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int occ = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
        if (occ < 1) occ = 1;
        // C in host memory: as many CTAs per SM as keep up with the link (one
        // per four products of an entry of C); more of them write over a wider
        // range at once, which the link answers with less bandwidth (40,009
        // vertices, 1.6 GB of C, four groups: 15.4 ms at four CTAs per SM,
        // 14.6 at two, 14.3 at one, 14.8 at 3/4).  Over eleven products of 5,003
        // to 100,003 columns with 1 to 4 products an entry, all the CTAs that fit
        // were 0 to 9% slower (12,011 vertices, four groups: 4.42 -> 4.84 ms), one
        // per two or eight products the same; at 8.6 products an entry one per
        // eight was 8% faster (8.54 -> 7.84 ms)
        if (p->c_on_host)
            occ = (int)std::max<int64_t>(1, std::min<int64_t>(occ, p->stats.products / 4 / std::max<int64_t>(p->nnzC, 1)));
        int g = grid_for(p->nnum, 1, p->sm_count * occ);
        if (!p->num_items) p->num_items = ws_alloc(p, sizeof(NumItem) * (size_t)p->nnum);
        NumItem *items = (NumItem *)p->num_items;
        if (!items) return SPG_OUT_OF_MEMORY;
        s = cuda_check(cudaMemsetAsync(p->d_cnt + kCntNumNextSlot, 0, sizeof(int64_t), p->st), "memset");
        if (s) return s;
        group_begin(p, kKNumHeavy);
        launch(p, k_num_headers, grid_for(p->nnum, 256, p->sm_count * 8), 256, 0, p->nnum, p->num_rec0, p->num_nrec,
               p->rec_col, p->rec_slab, p->rec_cnt, p->rec_off, p->B.colptr, p->B.ptr_type == SPG_IDX_I64,
               p->Ccolptr, items);
        launch(p, kern, g, threads, smem, p->nnum, items, p->hbits, p->Bq, (const Acc *)p->Bv, p->At_colptr,
               p->At_row, (const Acc *)p->At_val, p->split, p->T, p->R, p->num_cap, (OutIdx *)C->rowidx,
               (Acc *)C->vals, p->d_err, (unsigned long long *)(p->d_cnt + kCntNumNextSlot));
        group_end(p, kKNumHeavy);
        s = cuda_check(cudaGetLastError(), "numeric heavy");
    }
    return s;
}

// The light columns' numeric bins (by their exact counts): launched by the
// symbolic pass, whose read-back brings their sizes; a symbolic pass that is
// called again after a failed one makes them anew.
spg_status queue_numeric_bins(spg_plan *p) {
    const int64_t n = p->n;
    if (n == 0) return SPG_OK;
    int8_t *bn = (int8_t *)ws_alloc(p, (size_t)(n + 1));
    if (!p->nbinlist) p->nbinlist = (int32_t *)ws_alloc(p, sizeof(int32_t) * (size_t)(n + 1));
    if (!bn || !p->nbinlist) return SPG_OUT_OF_MEMORY;
    return bin_columns_queue(p, bn, p->nbinlist, 2);
}
void read_numeric_bins(spg_plan *p) {
    if (p->n > 0) bin_offsets(p, p->nbin_off);
}

spg_status run_numeric(spg_plan *p, spg_csc *C) {
    spg::PhaseRange nvtx_range("numeric");
    cudaStream_t st = p->st;
    const int64_t n = p->n;
    if (C->colptr && C->colptr != (void *)p->Ccolptr) {
        spg_status s = cuda_check(cudaMemcpyAsync(C->colptr, p->Ccolptr, sizeof(int64_t) * (size_t)(n + 1),
                                                  cudaMemcpyDeviceToDevice, st),
                                  "colptr copy");
        if (s) return s;
    }
    cudaEventRecord(p->ev[4], st);
    spg_status s;
    if (p->acc_f64)
        s = p->out_idx64 ? numeric_typed<double, long long>(p, C) : numeric_typed<double, int>(p, C);
    else
        s = p->out_idx64 ? numeric_typed<long long, long long>(p, C) : numeric_typed<long long, int>(p, C);
    cudaEventRecord(p->ev[5], st);
    p->ev_numeric = true;
    return s;
}

}  // namespace spg
