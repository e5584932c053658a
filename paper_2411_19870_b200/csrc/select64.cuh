// Exact top-k of a 64 x 64 chunk by its 64 threads (Section 2.1 "Top-k Sparsification"), thread t holding row t of the
// coefficients: shared by the kernels with chunk size 64 (kernels_fast64.cu, kernels_tc.cu).
#pragma once

#include <type_traits>

#include "demo_internal.h"
#include "fast_common.cuh"
#include "fast_dct.cuh"

namespace sel64 {

using namespace fastk;

constexpr int S = 64;
constexpr int XS = S + 4;     // row stride of the transpose tile: conflict-free column access, 128-bit row access
constexpr int LOG2S = 6;
constexpr int CAP = 128;      // candidate capacity of the fast top-k (two lists of 64)
constexpr int CAPW = CAP / 2;
constexpr int CAPWP = CAPW + 4;
constexpr int WCAP = 512;     // capacity of the wide candidate list (out-of-line path)
// Up to this k the k-th largest of the 64 row maxima bounds the top-k well enough (k = 48: about 90 candidates in a dense
// tile, k = 64: about 260) and the row stage of the inverse is cheaper from the list of records; above it the kernel
// variant with a bound from 256 quarter rows and a dense row stage takes over.  Measured, 4096 x 4096, one compress call:
// k = 40 / 48 from the list 53.7 / 57.2 us, k = 49 / 64 / 96 / 128 with the dense row stage 56.9 / 57.4 / 58.5 / 59.5 us
// (59 / 80 / 102 / 120 us from a list with the selection out of line); 8192 x 8192, k = 128: 430 -> 205 us.
constexpr int MAX_K_LISTED = 48;

// Shared memory of one slot.
struct SlotMem {
    unsigned char *raw;
    float *X;            // [S*XS] transpose / coefficient / row-stage tile (aliases the staged tiles)
    float *tmax;         // [S]
    int *cand_idx;       // [CAP + 8]
    float *cand_val;     // [CAP + 8]
    unsigned *cand_key;  // [CAP + 8]
    int4 *recs4;         // [65] kept records, pre-decoded for the row stage; entry 64 is always padding
    unsigned *misc;      // [16]
    unsigned *wkey;      // [WCAP + 4] wide list, behind the tile
    unsigned *widx;      // [WCAP + 4]
};

// How the selection leaves the kept coefficients besides the records: as the list of the sparse row stage, in the
// coefficient tile as q - alpha q (momentum in the transform domain), or as the tile itself with alpha q at the kept
// places and zero elsewhere.
enum { SELECT_LISTED, SELECT_QDOM, SELECT_DENSE };

// ------------------------------------------------------------------------------------------------
// Exact selection over the coefficient tile in X (row t complete for thread t), any k: the last resort of both variants below (tied or
// degenerate chunks, non-finite values, k above the bounds of the lists).  Row t goes into registers; a threshold with exactly k keys
// at or above it is searched bit by bit from the highest that any key has, one barrier per bit; if the bits run out, equal keys
// straddle the k-th place and the first ones are kept.  (A radix select over histograms in shared memory, where most keys meet in a few
// bins: 4096 x 4096, k = 193 / 256 / 512 196 us instead of 119, all-zero tiles 399 instead of 82; 1024 x 1024 under a caller's basis,
// k = 256 65 instead of 43.)
// ------------------------------------------------------------------------------------------------
static __device__ __noinline__ void select_search(const SlotMem sm, int k_eff, DemoRecord *rec, float alpha, int t, int bar_id, int mode)
{
    const SlotBarrier<S> sb{bar_id};
    const int lane = t & 31, warp = t >> 5;
    float *row = sm.X + t * XS;
    unsigned *misc = sm.misc;  // [2][2]: the warps' values, by turns
    float q[S];
#pragma unroll
    for (int v4 = 0; v4 < S / 4; ++v4) {
        const float4 f = reinterpret_cast<const float4 *>(row)[v4];
        q[4 * v4] = f.x;
        q[4 * v4 + 1] = f.y;
        q[4 * v4 + 2] = f.z;
        q[4 * v4 + 3] = f.w;
    }
    sb.sync();  // earlier readers of misc are done
    int turn = 0;
    auto both = [&](unsigned v, auto join) {  // v of this warp and of the other
        if (lane == 0) misc[2 * turn + warp] = v;
        sb.sync();
        const unsigned r = join(misc[2 * turn], misc[2 * turn + 1]);
        turn ^= 1;
        return r;
    };
    auto sum = [](unsigned x, unsigned y) { return x + y; };
    unsigned top = 0u;
#pragma unroll
    for (int v = 0; v < S; ++v) top = max(top, mag_key(q[v]));
    top = both(__reduce_max_sync(0xffffffffu, top), [](unsigned x, unsigned y) { return max(x, y); });
    unsigned thr = 0u, n_ge = (unsigned)(S * S);
#pragma unroll 1
    for (int b = 31 - __clz(top | 1u); b >= 0 && n_ge != (unsigned)k_eff; --b) {
        const unsigned cand = thr | (1u << b);
        unsigned n = 0u;
#pragma unroll
        for (int v = 0; v < S; ++v) n += mag_key(q[v]) >= cand;
        n = both(__reduce_add_sync(0xffffffffu, n), sum);
        if (n >= (unsigned)k_eff) {
            thr = cand;
            n_ge = n;
        }
    }
    // (n_ge = k: all at or above the threshold are kept, whatever lies between equal keys)
    unsigned gt = 0u, eq = 0u;
#pragma unroll
    for (int v = 0; v < S; ++v) {
        gt += mag_key(q[v]) > thr;
        eq += mag_key(q[v]) == thr;
    }
    const unsigned packed = gt | (eq << 16), inc = warp_inclusive_scan(packed, lane);
    const unsigned last = __shfl_sync(0xffffffffu, inc, 31);
    if (lane == 0) misc[2 * turn + warp] = last;
    sb.sync();
    const unsigned first_warp = misc[2 * turn], need_eq = (unsigned)k_eff - ((first_warp + misc[2 * turn + 1]) & 0xffffu);
    const unsigned before = inc - packed + (warp ? first_warp : 0u);
    unsigned gb = before & 0xffffu, eb = before >> 16;
#pragma unroll 1
    for (int v = 0; v < S; ++v) {
        const float val = row[v];
        const unsigned key = mag_key(val);
        const bool s = key > thr || (key == thr && eb < need_eq);
        if (s) {
            const unsigned pos = gb + min(eb, need_eq);
            DemoRecord r;
            r.idx = t * S + v;
            r.val = val;
            rec[pos] = r;
            if (mode == SELECT_QDOM)
                row[v] = fmaf(-alpha, val, val);
            else if (mode == SELECT_LISTED)
                sm.recs4[pos] = make_int4(t * XS, v * S, __float_as_int(alpha * val), 0);
        }
        if (mode == SELECT_DENSE) row[v] = s ? alpha * val : 0.f;
        gb += key > thr;
        eb += key == thr;
    }
}

// ------------------------------------------------------------------------------------------------
// Out-of-line selection (k <= MAX_K_LISTED) for the chunks the in-line path does not take: more than 64 candidates in
// a warp's list (tiles of low rank or with a concentrated spectrum, tied or degenerate chunks) or fewer
// candidates than k (NaN coefficients).  Works from the coefficient tile in X (row t is
// this thread's), writes the records to `rec` and the pre-decoded list for the row stage.
//   1. wide list: up to WCAP candidates under the bound `lmin` (the k-th largest of the 64 row maxima),
//      every warp takes the whole list into registers and finds the exact k-th largest key by a
//      bit-by-bit ballot search;
//   2. if the list overflows: a tighter bound from the 256 quarter-row and the 256 quarter-column
//      maxima, then 1. again;
//   3. otherwise select_search over the whole tile.
// ------------------------------------------------------------------------------------------------
static __device__ __noinline__ void select_slow(const SlotMem sm, int k_eff, DemoRecord *rec, float alpha, int t, int bar_id,
                                         unsigned lmin_w, bool qdom)
{
    const SlotBarrier<S> sb{bar_id};
    const int lane = t & 31, warp = t >> 5;
    float *X = sm.X;
    unsigned *misc = sm.misc;
    int4 *recs4 = sm.recs4;
    sb.sync();  // the coefficient tile is complete; the in-line path is done with its lists

    bool done = false;
    {
        unsigned long long mask = 0ull;
        unsigned off = 0, n_all = 0xffffffffu;
        auto count_under = [&](unsigned bound) {
            mask = 0ull;
#pragma unroll 4
            for (int v = 0; v < S; ++v) mask |= (unsigned long long)(mag_key(X[t * XS + v]) >= bound) << v;
            const unsigned cnt = (unsigned)__popcll(mask);
            const unsigned inc = warp_inclusive_scan(cnt, lane);
            sb.sync();  // earlier readers of misc are done
            if (lane == 31) misc[warp] = inc;
            sb.sync();
            const unsigned n0 = misc[0];
            n_all = n0 + misc[1];
            off = inc - cnt + (warp ? n0 : 0u);
        };
        count_under(lmin_w);
        if (n_all > (unsigned)WCAP) {
            // tighter bound: the k_eff-th largest of the 256 quarter-row maxima and of the 256 quarter-column maxima
            unsigned rk[4], ck[4];
            const float4 *row4 = reinterpret_cast<const float4 *>(X + t * XS);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                unsigned m = 0u;
#pragma unroll
                for (int v4 = 0; v4 < 4; ++v4) {
                    const float4 f = row4[4 * g + v4];
                    m = max(max(m, mag_key(f.x)), max(mag_key(f.y), max(mag_key(f.z), mag_key(f.w))));
                }
                rk[g] = m;
            }
            // (the quarter-column maxima matter for tiles with a few active columns)
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                unsigned m = 0u;
#pragma unroll 4
                for (int u = 0; u < 16; ++u) m = max(m, mag_key(X[(16 * g + u) * XS + t]));
                ck[g] = m;
            }
            unsigned *gq = sm.wkey;  // [8][64], behind the tile
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                gq[g * 64 + t] = rk[g];
                gq[(4 + g) * 64 + t] = ck[g];
            }
            sb.sync();
            unsigned prk[4], pck[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                prk[g] = gq[g * 64 + (t ^ 32)];
                pck[g] = gq[(4 + g) * 64 + (t ^ 32)];
            }
            auto kth_of_256 = [&](const unsigned (&own)[4], const unsigned (&oth)[4]) -> unsigned {
                unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    lo = min(lo, min(own[g], oth[g]));
                    hi = max(hi, max(own[g], oth[g]));
                }
                lo = __reduce_min_sync(0xffffffffu, lo);
                hi = __reduce_max_sync(0xffffffffu, hi);
                const int c0 = 31 - __clz((lo ^ hi) | 0x8000u);
                unsigned pre = lo & ~((2u << c0) - 1u);
#pragma unroll 1
                for (int b = c0; b >= 15; --b) {
                    const unsigned cand = pre | (1u << b);
                    unsigned cnt = 0;
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        cnt += __popc(__ballot_sync(0xffffffffu, own[g] >= cand)) +
                               __popc(__ballot_sync(0xffffffffu, oth[g] >= cand));
                    pre = (cnt >= (unsigned)k_eff) ? cand : pre;
                }
                return pre;
            };
            const unsigned l2 = max(kth_of_256(rk, prk), kth_of_256(ck, pck));
            sb.sync();  // gq is read; the wide list may overwrite it
            if (l2 > lmin_w) {
                lmin_w = l2;
                count_under(lmin_w);
            }
        }
        if (n_all >= (unsigned)k_eff && n_all <= (unsigned)WCAP) {
            unsigned *wkey = sm.wkey, *widx = sm.widx;
            {
                unsigned o = off;
                while (mask) {
                    const int v = __ffsll((long long)mask) - 1;
                    mask &= mask - 1ull;
                    widx[o] = t * S + v;
                    wkey[o] = mag_key(X[t * XS + v]);
                    ++o;
                }
            }
            sb.sync();
            auto wide_select = [&](auto wk_tag) {
                constexpr int WK = decltype(wk_tag)::value;
                unsigned keys[WK];
                unsigned hi = 0u;
#pragma unroll
                for (int j = 0; j < WK; ++j) {
                    const unsigned i = (unsigned)j * 32u + lane;
                    keys[j] = (i < n_all) ? wkey[i] : 0u;
                    hi = max(hi, keys[j]);
                }
                hi = __reduce_max_sync(0xffffffffu, hi);
                const int wb0 = 31 - __clz((lmin_w ^ hi) | 1u);
                unsigned thr = lmin_w & ~((2u << wb0) - 1u);
                unsigned n_ge = n_all;  // every entry is >= the bound >= thr; the search stops at exactly k_eff
#pragma unroll 1
                for (int b = wb0; b >= 0 && n_ge != (unsigned)k_eff; --b) {
                    const unsigned cand = thr | (1u << b);
                    unsigned cnt = 0;
#pragma unroll
                    for (int j = 0; j < WK; ++j) cnt += __popc(__ballot_sync(0xffffffffu, keys[j] >= cand));
                    if (cnt >= (unsigned)k_eff) {
                        thr = cand;
                        n_ge = cnt;
                    }
                }
                unsigned n_gt = 0;
#pragma unroll
                for (int j = 0; j < WK; ++j) n_gt += __popc(__ballot_sync(0xffffffffu, keys[j] > thr));
                const unsigned need_eq = (unsigned)k_eff - n_gt;
                unsigned gt_before = 0, eq_before = 0;
                const unsigned lt = (1u << lane) - 1u;
#pragma unroll
                for (int j = 0; j < WK; ++j) {
                    const unsigned key = keys[j];
                    const unsigned gtb = __ballot_sync(0xffffffffu, key > thr);
                    const unsigned eqb = __ballot_sync(0xffffffffu, key == thr);
                    if ((j & 1) == warp) {
                        const unsigned e = eq_before + __popc(eqb & lt);
                        if ((key > thr) || (key == thr && e < need_eq)) {
                            const unsigned pos = gt_before + __popc(gtb & lt) + min(e, need_eq);
                            DemoRecord r;
                            r.idx = (int)widx[j * 32 + lane];
                            const int v = r.idx & (S - 1);
                            const int uo = (r.idx >> LOG2S) * XS;
                            r.val = X[uo + v];
                            rec[pos] = r;
                            if (qdom)  // transform-domain momentum: what stays of a transmitted coefficient
                                X[uo + v] = fmaf(-alpha, r.val, r.val);
                            else
                                recs4[pos] = make_int4(uo, v * S, __float_as_int(alpha * r.val), 0);
                        }
                    }
                    gt_before += __popc(gtb);
                    eq_before += __popc(eqb);
                }
            };
            if (n_all <= 128u)
                wide_select(std::integral_constant<int, 4>{});
            else
                wide_select(std::integral_constant<int, WCAP / 32>{});
            done = true;
        }
    }
    if (!done) select_search(sm, k_eff, rec, alpha, t, bar_id, qdom ? SELECT_QDOM : SELECT_LISTED);
}

// ------------------------------------------------------------------------------------------------
// Last step of the in-line selection: the k_eff largest of the n_all candidates (all >= the bound `lmin_w`, at most
// 32 * NK of them; list 0 holds the first n_w0 in ascending index order, list 1 the rest).  Every warp takes all
// candidates into registers, NK keys per lane in list order, and searches bit by bit, from the first bit where the
// bound and the largest key differ, for a threshold with exactly k_eff keys at or above it; the search stops as
// soon as one is found.  If it runs out of bits, equal keys straddle the k_eff-th place: keys above the threshold
// are kept, keys equal to it in index order until k_eff are reached.  A kept candidate's place among the records
// is the number of kept candidates before it; warp w writes the records of the key groups w, w + 2, ...
// ------------------------------------------------------------------------------------------------
template <int NK, bool QDOM>
__device__ __forceinline__ void ballot_select(const SlotMem &sm, unsigned n_w0, unsigned n_all, unsigned lmin_w, int k_eff,
                                              DemoRecord *rec, float alpha, int lane, int warp)
{
    static_assert(NK == 2 || NK == 4, "two or four keys per lane");
    auto list_pos = [&](unsigned i) { return i < n_w0 ? i : i - n_w0 + (unsigned)CAPWP; };
    unsigned keys[NK];
    unsigned hi = 0u;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
        const unsigned i = (unsigned)j * 32u + lane;
        keys[j] = (i < n_all) ? sm.cand_key[list_pos(i)] : 0u;
        hi = max(hi, keys[j]);
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    const int wb0 = 31 - __clz((lmin_w ^ hi) | 1u);
    unsigned thr = lmin_w & ~((2u << wb0) - 1u);
    unsigned n_ge = n_all;  // every candidate is >= the bound >= thr
#pragma unroll 1
    for (int b = wb0; b >= 0 && n_ge != (unsigned)k_eff; --b) {
        const unsigned cand = thr | (1u << b);
        unsigned cnt = 0;
#pragma unroll
        for (int j = 0; j < NK; ++j) cnt += __popc(__ballot_sync(0xffffffffu, keys[j] >= cand));
        if (cnt >= (unsigned)k_eff) {
            thr = cand;
            n_ge = cnt;
        }
    }
    unsigned gtb[NK], eqb[NK];
    unsigned n_gt = 0;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
        gtb[j] = __ballot_sync(0xffffffffu, keys[j] > thr);
        eqb[j] = __ballot_sync(0xffffffffu, keys[j] == thr);
        n_gt += __popc(gtb[j]);
    }
    const unsigned need_eq = (unsigned)k_eff - n_gt;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll 1
    for (int jj = 0; jj < NK / 2; ++jj) {  // (rolled: one copy of the record write)
        const bool second = (jj != 0);     // key groups 2, 3 (NK = 4 only)
        const unsigned key = second ? (warp ? keys[NK - 1] : keys[NK - 2]) : (warp ? keys[1] : keys[0]);
        const unsigned gb = second ? (warp ? gtb[NK - 1] : gtb[NK - 2]) : (warp ? gtb[1] : gtb[0]);
        const unsigned eb = second ? (warp ? eqb[NK - 1] : eqb[NK - 2]) : (warp ? eqb[1] : eqb[0]);
        // kept / equal candidates in the key groups before this one
        unsigned gt_before = warp ? __popc(second ? gtb[NK - 2] : gtb[0]) : 0u;
        unsigned eq_before = warp ? __popc(second ? eqb[NK - 2] : eqb[0]) : 0u;
        if (second) {
            gt_before += __popc(gtb[0]) + __popc(gtb[1]);
            eq_before += __popc(eqb[0]) + __popc(eqb[1]);
        }
        const unsigned e = eq_before + __popc(eb & lt);
        if ((key > thr) || (key == thr && e < need_eq)) {
            const unsigned pos = gt_before + __popc(gb & lt) + min(e, need_eq);
            const unsigned li = list_pos((unsigned)(2 * jj + warp) * 32u + lane);
            DemoRecord r;
            r.idx = sm.cand_idx[li];
            r.val = sm.cand_val[li];
            rec[pos] = r;
            if (QDOM)  // what stays of a transmitted coefficient: q - alpha q
                sm.X[(r.idx >> LOG2S) * XS + (r.idx & (S - 1))] = fmaf(-alpha, r.val, r.val);
            else
                sm.recs4[pos] = make_int4((r.idx >> LOG2S) * XS, (r.idx & (S - 1)) * S, __float_as_int(alpha * r.val), 0);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Exact top-k of one chunk (Section 2.1 "Top-k Sparsification"): thread t holds the coefficients q[v] = Q[t][v] of
// row t.  Writes the k_eff records in ascending index order to `rec`; ends before the barrier that makes them
// visible.  QDOM = false (momentum kept in the spatial domain): also leaves the pre-decoded row-stage list and the
// tile X cleared for the row stage.  (WIDE = false: no room for the wide list, such chunks go to select_search.)  QDOM = true
// (momentum kept in the transform domain): leaves in X the coefficient tile with every transmitted coefficient q replaced by q - alpha q.
// ------------------------------------------------------------------------------------------------
template <bool QDOM, bool WIDE = true>
__device__ __forceinline__ void select_chunk(const SlotMem &sm, float (&q)[S], int k_eff, DemoRecord *rec, float alpha,
                                             int t, const SlotBarrier<S> &sb, int bar_id, int pad_row)
{
    float *X = sm.X;
    float *tmax = sm.tmax;
    int *cand_idx = sm.cand_idx;
    float *cand_val = sm.cand_val;
    unsigned *cand_key = sm.cand_key;
    int4 *recs4 = sm.recs4;
    unsigned *misc = sm.misc;
    const int lane = t & 31, warp = t >> 5;
    // the row-stage tile starts from zero; every thread clears its own row once it is done with it
    auto zero_row = [&]() {
        if (QDOM) return;  // (the transform-domain kernel keeps the coefficient tile: it is its output)
        float4 *row = reinterpret_cast<float4 *>(X + t * XS);
#pragma unroll
        for (int v4 = 0; v4 < S / 4; ++v4) row[v4] = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // The stash of row t.  With the momentum in the spatial domain it is written in the transform core's own order
    // (position p holds coefficient core_index(p)): the registers of a 128-bit store are then neighbours in the
    // core's output, as the pairs of the inverse cascade are, and no register moves are needed to satisfy both.
    constexpr bool CORE_STASH = !QDOM;
    auto stash_row = [&](auto core_order) {
        float4 *row = reinterpret_cast<float4 *>(X + t * XS);
        fdct::static_for<0, S / 4>([&](auto i) {
            constexpr int v4 = decltype(i)::value;
            constexpr bool CO = decltype(core_order)::value;
            constexpr int i0 = CO ? fdct::core_index<S>(4 * v4) : 4 * v4, i1 = CO ? fdct::core_index<S>(4 * v4 + 1) : 4 * v4 + 1;
            constexpr int i2 = CO ? fdct::core_index<S>(4 * v4 + 2) : 4 * v4 + 2, i3 = CO ? fdct::core_index<S>(4 * v4 + 3) : 4 * v4 + 3;
            row[v4] = make_float4(q[i0], q[i1], q[i2], q[i3]);
        });
    };
    // position of coefficient v in a stash kept in core order: v = (2j + 1) << s sits at (32 >> s) + j, v = 0 at 0
    auto stash_pos = [](int v) {
        if (!CORE_STASH) return v;
        const int sft = __ffs(v | S) - 1;
        return ((S / 2) >> sft) + (v >> (sft + 1));
    };
    // ---- exact top-k (Section 2.1 "Top-k Sparsification") -------------------------------
    if (!QDOM) {
        recs4[t] = make_int4(pad_row, 0, 0, 0);  // list padding (ordered before the record writes by the barriers below)
        if (t == 0) recs4[64] = make_int4(pad_row, 0, 0, 0);
    }
    bool slow = false;
    bool zero_chunk = false;
    unsigned n_cw = 0, off = 0, mlo = 0u, mhi = 0u, lmin_w = 0u;
    {
        // per-thread maximum magnitude (independent chains of 16, 3-input max)
        float tm = 0.f;
#pragma unroll
        for (int ch = 0; ch < S / 16; ++ch) {
            const int b0 = 16 * ch;
            float cm = max3abs(q[b0], q[b0 + 1], q[b0 + 2]);
#pragma unroll
            for (int j = 3; j + 1 < 16; j += 2) cm = max3f(cm, fabsf(q[b0 + j]), fabsf(q[b0 + j + 1]));
            tm = max3f(tm, cm, fabsf(q[b0 + 15]));
        }
        // L = the k_eff-th largest of the 64 row maxima (low 15 mantissa bits cleared): a lower bound of
        // the k_eff-th largest coefficient.  Every warp holds all 64 keys, two ballots per step count them.
        const unsigned tkey = __float_as_uint(tm);
        unsigned *tk = reinterpret_cast<unsigned *>(tmax);
        tk[t] = tkey;
        sb.sync();
        const unsigned okey = tk[t ^ 32];
        const unsigned lo_all = __reduce_min_sync(0xffffffffu, min(tkey, okey));
        const unsigned hi_all = __reduce_max_sync(0xffffffffu, max(tkey, okey));
        zero_chunk = (hi_all == 0u);
        const int b0 = 31 - __clz((lo_all ^ hi_all) | 0x8000u);  // >= 15
        unsigned prefix = lo_all & ~((2u << b0) - 1u);
#pragma unroll 1
        for (int b = zero_chunk ? 14 : b0; b >= 15; --b) {
            const unsigned cand = prefix | (1u << b);
            const unsigned cnt = __popc(__ballot_sync(0xffffffffu, tkey >= cand)) +
                                 __popc(__ballot_sync(0xffffffffu, okey >= cand));
            prefix = (cnt >= (unsigned)k_eff) ? cand : prefix;
        }
        lmin_w = prefix;
        if (!zero_chunk) {
            // candidates: |q| >= L  <=>  |q| > Lm (the float just below L); the sign bit of Lm - |q|
            // is funnel-shifted into a bit mask (independent chains of 16)
            const float L = __uint_as_float(lmin_w);
            const float Lm = (L > 0.f) ? __uint_as_float(lmin_w - 1u) : -1.f;
            unsigned mc[S / 16];
#pragma unroll
            for (int ch = 0; ch < S / 16; ++ch) {
                unsigned mm = 0u;
#pragma unroll
                for (int j = 15; j >= 0; --j)
                    mm = __funnelshift_l(__float_as_uint(Lm - fabsf(q[16 * ch + j])), mm, 1);
                mc[ch] = mm;
            }
            mlo = mc[0] | (mc[1] << 16);
            mhi = mc[2] | (mc[3] << 16);
            const unsigned cnt = __popc(mlo) + __popc(mhi);
            const unsigned inc = warp_inclusive_scan(cnt, lane);
            off = inc - cnt;
            n_cw = __shfl_sync(0xffffffffu, inc, 31);
            if (lane == 0) misc[warp] = n_cw;
        }
    }
    if (zero_chunk) {
        // all coefficients zero: the tie rule gives the records 0 .. k_eff-1 with value 0
        if (t < k_eff) {
            DemoRecord r;
            r.idx = t;
            r.val = 0.f;
            rec[t] = r;
        }
        if (!QDOM && t < k_eff) recs4[t] = make_int4(0, 0, 0, 0);
        zero_row();
        if (QDOM) stash_row(std::false_type{});  // (all zero; the tile is the kernel's output)
    } else {
        // stash the coefficients of row t (own row: no hazard with other threads)
        stash_row(std::integral_constant<bool, CORE_STASH>{});
        {
            const unsigned lbase = warp * CAPWP;
            if (n_cw <= CAPW) {
                // each warp compacts its candidates into its own list (rows of warp 0 precede rows of
                // warp 1, so the concatenation is in ascending index order)
                unsigned o = lbase + off;
                unsigned long long mask = ((unsigned long long)mhi << 32) | mlo;
                while (mask) {
                    const int v = __ffsll((long long)mask) - 1;
                    mask &= mask - 1ull;
                    const float val = X[t * XS + stash_pos(v)];
                    cand_idx[o] = t * S + v;
                    cand_val[o] = val;
                    cand_key[o] = mag_key(val);
                    ++o;
                }
            }
            sb.sync();
            const unsigned n_w0 = misc[0], n_w1 = misc[1];
            // more than a list holds, or fewer candidates than k_eff (NaN coefficients fail the float
            // comparisons above): the out-of-line selection takes over
            slow = (n_w0 > (unsigned)CAPW) || (n_w1 > (unsigned)CAPW) || (n_w0 + n_w1 < (unsigned)k_eff);
            if (!slow) {
                zero_row();  // row t of the stash was read by this thread only
                // the two lists, read one behind the other, are in ascending index order
                if (n_w0 + n_w1 <= 64u)
                    ballot_select<2, QDOM>(sm, n_w0, n_w0 + n_w1, lmin_w, k_eff, rec, alpha, lane, warp);
                else
                    ballot_select<4, QDOM>(sm, n_w0, n_w0 + n_w1, lmin_w, k_eff, rec, alpha, lane, warp);
            }
        }
        if (slow) {
            if (CORE_STASH) stash_row(std::false_type{});  // the out-of-line selection reads the tile in index order
            if constexpr (WIDE)
                select_slow(sm, k_eff, rec, alpha, t, bar_id, lmin_w, QDOM);
            else
                select_search(sm, k_eff, rec, alpha, t, bar_id, QDOM ? SELECT_QDOM : SELECT_LISTED);
            sb.sync();  // every thread is done with the coefficient tile
            zero_row();
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Exact top-k for k > MAX_K_LISTED; same contract as select_chunk, except that with the momentum in the spatial domain
// it leaves row t of X ready for the dense row stage: alpha * q at the kept places, zero elsewhere, position p of the
// row holding coefficient core_index(p).  Ends before the barrier that makes records and tile visible.
// The bound is the k-th largest of the 256 quarter-row maxima (16 coefficients each): for a dense tile about 55
// candidates at k = 49, 175 at k = 128, 245 at k = 160.  Both warps take all candidates into registers and find the
// kept set by the same ballot search as the list variant.
// ------------------------------------------------------------------------------------------------
constexpr int MAX_K_QUARTERS = 192;  // above it the bound admits too many candidates (k = 192: 340 of 512 places)

template <bool QDOM>
__device__ __forceinline__ void select_chunk_big(const SlotMem &sm, float (&q)[S], int k_eff, DemoRecord *rec, float alpha,
                                                 int t, const SlotBarrier<S> &sb, int bar_id)
{
    float *X = sm.X;
    unsigned *misc = sm.misc;
    const int lane = t & 31, warp = t >> 5;
    float *my_row = X + t * XS;
    auto stash_row = [&]() {
        float4 *row = reinterpret_cast<float4 *>(my_row);
#pragma unroll
        for (int v4 = 0; v4 < S / 4; ++v4) row[v4] = make_float4(q[4 * v4], q[4 * v4 + 1], q[4 * v4 + 2], q[4 * v4 + 3]);
    };
    auto zero_row = [&]() {
        float4 *row = reinterpret_cast<float4 *>(my_row);
#pragma unroll
        for (int v4 = 0; v4 < S / 4; ++v4) row[v4] = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // position of coefficient v in core order: v = (2j + 1) << s sits at (32 >> s) + j, v = 0 at 0
    auto core_pos = [](int v) {
        const int sft = __ffs(v | S) - 1;
        return ((S / 2) >> sft) + (v >> (sft + 1));
    };
    bool slow = k_eff > MAX_K_QUARTERS;
    bool zero_chunk = false;
    if (!slow) {
        unsigned own[4], oth[4];
        unsigned *gq = sm.wkey;  // [4][64]
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int b0 = 16 * g;
            float cm = max3abs(q[b0], q[b0 + 1], q[b0 + 2]);
#pragma unroll
            for (int j = 3; j + 1 < 16; j += 2) cm = max3f(cm, fabsf(q[b0 + j]), fabsf(q[b0 + j + 1]));
            own[g] = __float_as_uint(fmaxf(cm, fabsf(q[b0 + 15])));
            gq[g * 64 + t] = own[g];
        }
        sb.sync();  // (row t of the tile is this thread's: every thread has read its row of the transposed tile too)
#pragma unroll
        for (int g = 0; g < 4; ++g) oth[g] = gq[g * 64 + (t ^ 32)];
        unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            lo = min(lo, min(own[g], oth[g]));
            hi = max(hi, max(own[g], oth[g]));
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        zero_chunk = (hi == 0u);
        const int c0 = 31 - __clz((lo ^ hi) | 0x8000u);
        unsigned bound = lo & ~((2u << c0) - 1u);
#pragma unroll 1
        for (int b = zero_chunk ? 14 : c0; b >= 15; --b) {
            const unsigned cand = bound | (1u << b);
            unsigned cnt = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g)
                cnt += __popc(__ballot_sync(0xffffffffu, own[g] >= cand)) + __popc(__ballot_sync(0xffffffffu, oth[g] >= cand));
            bound = (cnt >= (unsigned)k_eff) ? cand : bound;
        }
        if (zero_chunk) {
            // all coefficients zero: the tie rule gives the records 0 .. k_eff-1 with value 0
            for (int r = t; r < k_eff; r += S) {
                DemoRecord z;
                z.idx = r;
                z.val = 0.f;
                rec[r] = z;
            }
            zero_row();
            return;
        }
        // candidates: |q| >= bound, i.e. |q| > the float just below it (see select_chunk)
        const float Lm = bound ? __uint_as_float(bound - 1u) : -1.f;
        unsigned mc[S / 16];
#pragma unroll
        for (int ch = 0; ch < S / 16; ++ch) {
            unsigned mm = 0u;
#pragma unroll
            for (int j = 15; j >= 0; --j) mm = __funnelshift_l(__float_as_uint(Lm - fabsf(q[16 * ch + j])), mm, 1);
            mc[ch] = mm;
        }
        unsigned long long mask = ((unsigned long long)(mc[2] | (mc[3] << 16)) << 32) | (mc[0] | (mc[1] << 16));
        const unsigned cnt = (unsigned)__popcll(mask);
        const unsigned inc = warp_inclusive_scan(cnt, lane);
        if (lane == 31) misc[warp] = inc;
        stash_row();
        sb.sync();  // counts visible; the maxima in the list area are read
        const unsigned n_w0 = misc[0], n_all = n_w0 + misc[1];
        slow = n_all > (unsigned)WCAP || n_all < (unsigned)k_eff;  // (fewer than k: NaN coefficients)
        if (!slow) {
            unsigned *wval = sm.wkey, *widx = sm.widx;
            unsigned o = inc - cnt + (warp ? n_w0 : 0u);
            while (mask) {
                const int v = __ffsll((long long)mask) - 1;
                mask &= mask - 1ull;
                widx[o] = t * S + v;
                wval[o] = __float_as_uint(my_row[v]);
                ++o;
            }
            if (!QDOM) zero_row();
            sb.sync();  // the list is complete, the tile cleared
            auto pick = [&](auto wk_tag) {
                constexpr int WK = decltype(wk_tag)::value;
                unsigned keys[WK];
                unsigned top = 0u;
#pragma unroll
                for (int j = 0; j < WK; ++j) {
                    const unsigned i = (unsigned)j * 32u + lane;
                    keys[j] = (i < n_all) ? (wval[i] & 0x7fffffffu) : 0u;
                    top = max(top, keys[j]);
                }
                top = __reduce_max_sync(0xffffffffu, top);
                const int wb0 = 31 - __clz((bound ^ top) | 1u);
                unsigned thr = bound & ~((2u << wb0) - 1u);
                unsigned n_ge = n_all;  // every entry is >= the bound >= thr; the search stops at exactly k_eff
#pragma unroll 1
                for (int b = wb0; b >= 0 && n_ge != (unsigned)k_eff; --b) {
                    const unsigned cand = thr | (1u << b);
                    unsigned n = 0;
#pragma unroll
                    for (int j = 0; j < WK; ++j) n += __popc(__ballot_sync(0xffffffffu, keys[j] >= cand));
                    if (n >= (unsigned)k_eff) {
                        thr = cand;
                        n_ge = n;
                    }
                }
                unsigned n_gt = 0;
#pragma unroll
                for (int j = 0; j < WK; ++j) n_gt += __popc(__ballot_sync(0xffffffffu, keys[j] > thr));
                const unsigned need_eq = (unsigned)k_eff - n_gt;
                const unsigned lt = (1u << lane) - 1u;
                unsigned gt_before = 0, eq_before = 0;
#pragma unroll
                for (int j = 0; j < WK; ++j) {
                    const unsigned gtb = __ballot_sync(0xffffffffu, keys[j] > thr);
                    const unsigned eqb = __ballot_sync(0xffffffffu, keys[j] == thr);
                    if ((j & 1) == warp) {
                        const unsigned e = eq_before + __popc(eqb & lt);
                        if ((keys[j] > thr) || (keys[j] == thr && e < need_eq)) {
                            const unsigned pos = gt_before + __popc(gtb & lt) + min(e, need_eq);
                            DemoRecord r;
                            r.idx = (int)widx[j * 32 + lane];
                            r.val = __uint_as_float(wval[j * 32 + lane]);
                            rec[pos] = r;
                            float *row = X + (r.idx >> LOG2S) * XS;
                            const int v = r.idx & (S - 1);
                            if (QDOM)
                                row[v] = fmaf(-alpha, r.val, r.val);
                            else
                                row[core_pos(v)] = alpha * r.val;
                        }
                    }
                    gt_before += __popc(gtb);
                    eq_before += __popc(eqb);
                }
            };
            if (n_all <= 256u)
                pick(std::integral_constant<int, 8>{});
            else
                pick(std::integral_constant<int, WCAP / 32>{});
        }
    } else {
        sb.sync();  // every thread has read its row of the transposed tile
        stash_row();
    }
    if (slow) {
        select_search(sm, k_eff, rec, alpha, t, bar_id, QDOM ? SELECT_QDOM : SELECT_DENSE);
        if (!QDOM) {  // index order -> core order (this thread's row)
            float4 *row = reinterpret_cast<float4 *>(my_row);
#pragma unroll
            for (int v4 = 0; v4 < S / 4; ++v4) {
                const float4 f = row[v4];
                q[4 * v4] = f.x;
                q[4 * v4 + 1] = f.y;
                q[4 * v4 + 2] = f.z;
                q[4 * v4 + 3] = f.w;
            }
            fdct::static_for<0, S / 4>([&](auto i) {
                constexpr int v4 = decltype(i)::value;
                row[v4] = make_float4(q[fdct::core_index<S>(4 * v4)], q[fdct::core_index<S>(4 * v4 + 1)],
                                      q[fdct::core_index<S>(4 * v4 + 2)], q[fdct::core_index<S>(4 * v4 + 3)]);
            });
        }
    }
}

}  // namespace sel64
