// Compress kernel for 2-D tensors with chunk size 32: Algorithm 1 worker side / CompressChunks, fused per chunk --
// momentum update, 2-D DCT-II, exact top-k, momentum subtraction.  One warp owns one 32 x 32 chunk; lane t works on
// column t, then row t.
//
// A chunk is small enough that no step needs more than a warp-level barrier, so the chunks of an SM (twenty with bf16
// gradients, sixteen with fp32) run in phases of their own and their loads, transforms, selections and stores overlap.
// Instruction issue bounds it: about 1660 instructions per chunk, issued in 62 % of the cycles, next to which the 10 KB
// that a chunk moves cost less.  The next chunk's tiles come in by 16-byte asynchronous copies (they need no tensor map,
// whose acquisition costs about a microsecond per tensor) as soon as this chunk's have been read; B is parked in tensor
// memory between the load and the residual (in registers only sixteen warps fit: 8192 x 8192 154 us instead of 144); the new
// momentum leaves from registers, 128 consecutive bytes per store.
// One call, k = 8, against eight chunks per CTA in lockstep and the tiles fetched twice: 4096 x 4096 57.8 -> 44.1 us,
// 8192 x 8192 198 -> 144 us (fp32 gradients 200 -> 159 us), 1024 x 1024 10.5 -> 6.9 us.
#include <cuda_bf16.h>

#include "demo_internal.h"
#include "fast_common.cuh"
#include "fast_dct.cuh"
#include "launch.cuh"

namespace {

using namespace fastk;

constexpr int S = 32;
constexpr int XS = S + 4;   // row stride of the transpose tile: conflict-free column access, 128-bit row access
constexpr int LOG2S = 5;
constexpr int WARPS = 4;    // per CTA
constexpr int LIST = 64;    // capacity of the candidate list
// Up to this k the row stage of the inverse runs from the list of records; above it the kept set is searched among all
// coefficients and the row stage is dense (4096 x 4096: k = 32 from the list 52.8 us, any k from 33 to 128 dense 77 us;
// the former radix selection took 167 us at k = 64, 227 us at k = 128).
constexpr int MAX_K_LISTED = 32;
constexpr int MAX_K_ROWS = 12;  // up to this k the 32 row maxima bound the candidates, above it the 64 half-row maxima
constexpr int CTAS = 5;         // per SM, by registers

template <typename GT>
struct Area {  // shared memory of one warp
    float m[S * S];            // landing area of the next chunk's tiles
    GT g[S * S];
    float X[S * XS];           // transpose / coefficient / row-stage tile; its padding columns hold the candidate list
    int4 recs4[S + 1];         // kept records, pre-decoded for the row stage; padded
    // the tensor of the chunk looked up last (read from the tables for every chunk: 4096 x 4096 46.6 instead of 45.7 us)
    float *m_base;
    const GT *g_base;
    DemoRecord *rec_base;
    unsigned begin, c1, n1;
};

// Where a chunk lies.
template <typename GT>
struct Place {
    float *m;  // first element of the tile
    const GT *g;
    DemoRecord *rec;
    int n1;
};

// The k largest of all coefficients, by a bit-by-bit search over the keys in registers: at least k keys are >= `bound`.
// Returns the lane's kept columns as a mask; equal keys at the k-th place are kept in index order.
__device__ __forceinline__ unsigned search_all(const float (&q)[S], unsigned bound, int k, int lane)
{
    unsigned top = 0u;
#pragma unroll
    for (int v = 0; v < S; ++v) top = max(top, mag_key(q[v]));
    top = __reduce_max_sync(0xffffffffu, top);
    auto count_ge = [&](unsigned thr) {
        unsigned n = 0u;
#pragma unroll
        for (int v = 0; v < S; ++v) n += mag_key(q[v]) >= thr;
        return __reduce_add_sync(0xffffffffu, n);
    };
    const int b0 = 31 - __clz((bound ^ top) | 1u);
    unsigned thr = bound & ~((2u << b0) - 1u), n_ge = ~0u;
#pragma unroll 1
    for (int b = b0; b >= 0 && n_ge != (unsigned)k; --b) {
        const unsigned cand = thr | (1u << b);
        const unsigned n = count_ge(cand);
        if (n >= (unsigned)k) {
            thr = cand;
            n_ge = n;
        }
    }
    unsigned gt = 0u, eq = 0u;
#pragma unroll
    for (int v = 0; v < S; ++v) {
        gt |= (unsigned)(mag_key(q[v]) > thr) << v;
        eq |= (unsigned)(mag_key(q[v]) == thr) << v;
    }
    if (n_ge != (unsigned)k) {  // more equal keys than places
        const int need = k - (int)__reduce_add_sync(0xffffffffu, __popc(gt));
        const int n = __popc(eq), before = (int)warp_inclusive_scan(n, lane) - n;
        for (int drop = n - max(0, min(n, need - before)); drop > 0; --drop) eq &= ~(0x80000000u >> __clz(eq));
    }
    return gt | eq;
}

template <typename GT, bool BIGK>
__global__ void __launch_bounds__(WARPS * 32, CTAS) compress32_kernel(DemoCompressArgs a)
{
    const StreamOrder order(a.wait_first);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int t = threadIdx.x & 31;
    Area<GT> &w = reinterpret_cast<Area<GT> *>(smem_raw)[threadIdx.x >> 5];
    float *X = w.X;
    // candidate i (value, index) in the padding columns of the tile
    auto candidate = [&](unsigned i) -> float2 & { return *reinterpret_cast<float2 *>(X + (i & 31u) * XS + S + (i >> 5) * 2u); };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_raw + WARPS * sizeof(Area<GT>));
    const int k = a.k;
    const unsigned n_chunks = (unsigned)a.n_chunks, n_warps = gridDim.x * WARPS;  // (fewer than 2^31)

    int e = 0;
    unsigned next_begin = 0;  // first chunk of the next tensor
    auto locate = [&](unsigned c) {
        if (c >= next_begin) {
            e = next_begin ? demo_seek_entry(a.entries, a.n_entries, e + 1, c) : demo_find_entry(a.entries, a.n_entries, c);
            next_begin = e + 1 < a.n_entries ? (unsigned)a.entries[e + 1].chunk_begin : ~0u;
            const DemoTensorEntry te = a.entries[e];
            if (t == 0) {
                w.m_base = a.m_ptrs[te.tensor];
                w.g_base = static_cast<const GT *>(a.g_ptrs[te.tensor]);
                w.rec_base = a.payload + te.rec_begin;
                w.begin = (unsigned)te.chunk_begin;
                w.c1 = (unsigned)te.c1;
                w.n1 = (unsigned)te.n1;
            }
            __syncwarp();
        }
        const unsigned lc = c - w.begin, k0 = lc / w.c1;
        const size_t off = ((size_t)k0 * w.n1 + (lc - k0 * w.c1)) * S;
        Place<GT> p;
        p.m = w.m_base + off;
        p.g = w.g_base + off;
        p.rec = w.rec_base + (size_t)lc * k;
        p.n1 = (int)w.n1;
        return p;
    };
    auto fetch = [&](const Place<GT> &p) {
        auto copy = [&](auto *dst, const auto *src) {
            constexpr int PER = 16 / sizeof(*src), PIECES = S / PER;  // elements of a piece, pieces of a row
            const int r0 = t / PIECES, x = t % PIECES * PER;
#pragma unroll
            for (int r = 0; r < S; r += 32 / PIECES)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + (r0 + r) * S + x)),
                             "l"(src + (size_t)(r0 + r) * p.n1 + x)
                             : "memory");
        };
        copy(w.m, (const float *)p.m);
        copy(w.g, p.g);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    unsigned c = blockIdx.x * WARPS + (threadIdx.x >> 5);
    Place<GT> p;
    if (c < n_chunks) {
        p = locate(c);
        prefetch_l2(p.m + (size_t)t * p.n1);
        prefetch_l2(p.g + (size_t)t * p.n1);
    }
    order.begin();
    if (!BIGK && c < n_chunks) fetch(p);
    __syncwarp();
    const uint32_t tmem = tmem_alloc_cta(tmem_slot, S);
    const uint32_t taddr = tmem + ((threadIdx.x & ~31u) << 16);  // this warp's lanes: column t of B, parked for the residual
    if (BIGK && c < n_chunks) {  // (with the place kept across the allocation the code comes out 5 to 20 % slower)
        p = locate(c);
        fetch(p);
    }
    // (lane 0) the next chunk, known one chunk ahead: the first two rounds are fixed, the rest is drawn
    unsigned drawn = a.tickets ? c - n_warps : NO_TICKET;
    while (c < n_chunks) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        float b[S];  // column t of B = beta * m + g
#pragma unroll
        for (int i = 0; i < S; ++i) b[i] = fmaf(a.beta, w.m[i * S + t], to_f32(w.g[i * S + t]));
        tmem_st32(taddr, b);
        __syncwarp();  // the landing area is free
        const unsigned nc = 2u * n_warps + __shfl_sync(0xffffffffu, drawn, 0);
        Place<GT> next{};
        if (nc < n_chunks) {
            next = locate(nc);
            fetch(next);
            if (t == 0) drawn = ticket_draw(a.tickets);  // (looked at when the next chunk begins)
        }

        // ---- Q = DCT-II of B: column t, transpose (rows in pair order, fast_dct.cuh), row t ---------------------
        float q[S];  // Q[t][.]
        {
            float u[S], y[S];
            fdct::dct2_pre_paired<S>(b, u);
            fdct::dct_core_ortho_paired<S>(u, y);
            float *Xc = X + fdct::pair_order(t);
            fdct::static_for<0, S>([&](auto i) { Xc[fdct::core_index<S>(decltype(i)::value) * XS] = y[decltype(i)::value]; });
            __syncwarp();
            float x[S];
#pragma unroll
            for (int v4 = 0; v4 < S / 4; ++v4) {
                const float4 f = reinterpret_cast<const float4 *>(X + t * XS)[v4];
                x[4 * v4 + 0] = f.x;
                x[4 * v4 + 1] = f.y;
                x[4 * v4 + 3] = f.z;
                x[4 * v4 + 2] = f.w;
            }
            fdct::dct2_pre_paired<S>(x, u);
            fdct::dct_core_ortho_paired<S>(u, y);
            fdct::static_for<0, S>([&](auto i) { q[fdct::core_index<S>(decltype(i)::value)] = y[decltype(i)::value]; });
        }

        // ---- exact top-k (Section 2.1 "Top-k Sparsification"); records in ascending index order ------------------
        float tm[4];  // maxima of the quarters of the row
#pragma unroll
        for (int h = 0; h < 4; ++h)
            tm[h] = max3f(max3abs(q[8 * h], q[8 * h + 1], q[8 * h + 2]), max3abs(q[8 * h + 3], q[8 * h + 4], q[8 * h + 5]),
                          fmaxf(fabsf(q[8 * h + 6]), fabsf(q[8 * h + 7])));
        const unsigned tkey = __float_as_uint(fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3])));
        const unsigned hi = __reduce_max_sync(0xffffffffu, tkey);
        float4 *row = reinterpret_cast<float4 *>(X + t * XS);  // (from here on row t of the tile is this lane's)
        auto stash_row = [&]() {
#pragma unroll
            for (int v4 = 0; v4 < S / 4; ++v4) row[v4] = make_float4(q[4 * v4], q[4 * v4 + 1], q[4 * v4 + 2], q[4 * v4 + 3]);
        };
        auto zero_row = [&]() {
#pragma unroll
            for (int v4 = 0; v4 < S / 4; ++v4) row[v4] = make_float4(0.f, 0.f, 0.f, 0.f);
        };
        // Writes the records of the kept columns `kept` of row t; note(pos, v, val) for each.
        auto write_kept = [&](unsigned kept, auto note) {
            unsigned pos = __popc(kept);
            pos = warp_inclusive_scan(pos, t) - pos;
            for (; kept; kept &= kept - 1u, ++pos) {
                const int v = __ffs(kept) - 1;
                DemoRecord r;
                r.idx = t * S + v;
                r.val = X[t * XS + v];
                p.rec[pos] = r;
                note(pos, v, r.val);
            }
        };
        float y[S];
        if constexpr (BIGK) {
            // 128 quarter-row maxima are >= the smallest of them: a bound for k <= 128
            const unsigned lo = __reduce_min_sync(0xffffffffu, __float_as_uint(fminf(fminf(tm[0], tm[1]), fminf(tm[2], tm[3]))));
            stash_row();
            const unsigned kept = search_all(q, k <= 4 * S && lo <= 0x7f800000u ? lo : 0u, k, t);
            write_kept(kept, [](unsigned, int, float) {});
            // dense row stage of the inverse: DCT-III of the kept coefficients, back into the row in pair order
            float u[S];
            fdct::static_for<0, S>([&](auto i) {
                constexpr int v = fdct::core_index<S>(decltype(i)::value);
                u[decltype(i)::value] = (kept >> v & 1u) ? a.alpha * q[v] : 0.f;
            });
            fdct::dct_core_ortho_paired<S>(u, y);
            fdct::F2 rp[S / 2];
            fdct::dct3_post_pairs<S>(y, rp);
#pragma unroll
            for (int v4 = 0; v4 < S / 4; ++v4)
                row[v4] = make_float4(fdct::f2_lo(rp[2 * v4]), fdct::f2_hi(rp[2 * v4]), fdct::f2_lo(rp[2 * v4 + 1]),
                                      fdct::f2_hi(rp[2 * v4 + 1]));
            __syncwarp();
        } else {
            if (hi == 0u) {
                // all coefficients zero: the tie rule gives the records 0 .. k-1 with value 0
                if (t < k) {
                    DemoRecord r;
                    r.idx = t;
                    r.val = 0.f;
                    p.rec[t] = r;
                }
                w.recs4[t] = make_int4(0, 0, 0, 0);
                if (t == 0) w.recs4[S] = make_int4(0, 0, 0, 0);
                zero_row();
            } else {
                // bound: the k-th largest of the 32 row maxima (small k) or of the 64 half-row maxima, low 15 mantissa bits cleared
                const bool halves = k > MAX_K_ROWS;
                const unsigned h0 = __float_as_uint(fmaxf(tm[0], tm[1])), h1 = __float_as_uint(fmaxf(tm[2], tm[3]));
                const unsigned lo = __reduce_min_sync(0xffffffffu, halves ? min(h0, h1) : tkey);
                const int b0 = 31 - __clz((lo ^ hi) | 0x8000u);  // >= 15
                unsigned bound = lo & ~((2u << b0) - 1u);
                if (halves) {
#pragma unroll 1
                    for (int bit = b0; bit >= 15; --bit) {
                        const unsigned cand = bound | (1u << bit);
                        const int n = __popc(__ballot_sync(0xffffffffu, h0 >= cand)) + __popc(__ballot_sync(0xffffffffu, h1 >= cand));
                        bound = n >= k ? cand : bound;
                    }
                } else {
#pragma unroll 1
                    for (int bit = b0; bit >= 15; --bit) {
                        const unsigned cand = bound | (1u << bit);
                        bound = __popc(__ballot_sync(0xffffffffu, tkey >= cand)) >= k ? cand : bound;
                    }
                }
                // candidates: |q| >= bound, i.e. |q| > the float just below it: sign bits of the differences, shifted together
                const float below = bound ? __uint_as_float(bound - 1u) : -1.f;
                unsigned mc[2] = {0u, 0u};
#pragma unroll
                for (int j = 15; j >= 0; --j) {
                    mc[0] = __funnelshift_l(__float_as_uint(below - fabsf(q[j])), mc[0], 1);
                    mc[1] = __funnelshift_l(__float_as_uint(below - fabsf(q[16 + j])), mc[1], 1);
                }
                unsigned mask = mc[0] | (mc[1] << 16);
                const unsigned cnt = __popc(mask), inc = warp_inclusive_scan(cnt, t);
                const unsigned n_all = __shfl_sync(0xffffffffu, inc, 31);
                stash_row();
                auto note = [&](unsigned pos, int idx, float val) {
                    const int4 r = make_int4((idx >> LOG2S) * XS, (idx & (S - 1)) * S, __float_as_int(a.alpha * val), 0);
                    w.recs4[pos] = r;
                    if (pos + 1 == (unsigned)k)  // up to a multiple of eight and one more: zeros in the last record's row
                        for (int pad = k; pad <= ((k + 7) & ~7); ++pad) w.recs4[pad] = make_int4(r.x, r.y, 0, 0);
                };
                if (n_all <= (unsigned)LIST && n_all >= (unsigned)k) {
                    for (unsigned o = inc - cnt; mask; mask &= mask - 1u, ++o) {
                        const int v = __ffs(mask) - 1;
                        const float val = X[t * XS + v];
                        candidate(o) = make_float2(val, __int_as_float(t * S + v));
                    }
                    zero_row();
                    __syncwarp();
                    auto key_of = [&](unsigned i) { return mag_key(candidate(i).x); };
                    warp_ballot_select<2>(key_of, n_all, bound, k, t, [&](unsigned pos, unsigned i) {
                        DemoRecord r;
                        const float2 cd = candidate(i);
                        r.val = cd.x;
                        r.idx = __float_as_int(cd.y);
                        p.rec[pos] = r;
                        note(pos, r.idx, r.val);
                    });
                } else {  // tied or concentrated spectra; fewer candidates than k: NaN coefficients, the bound is void
                    const unsigned kept = search_all(q, n_all >= (unsigned)k ? bound : 0u, k, t);
                    __syncwarp();
                    write_kept(kept, [&](unsigned pos, int v, float val) { note(pos, t * S + v, val); });
                    zero_row();
                }
            }
            __syncwarp();
            // row stage of the inverse: T[u][t] = sum over kept (u, v) of alpha * val * C[v][t], the running sum of a row
            // stored after every entry and started again from zero with the next row (no branch)
            float acc = 0.f;
            float *Xt = X + t;
            int4 nx = w.recs4[0];
#pragma unroll 1
            for (int r0 = 0; r0 < k; r0 += 8) {
                int4 rc[9];
                float cv[8];
                rc[0] = nx;
#pragma unroll
                for (int j = 1; j < 9; ++j) rc[j] = w.recs4[r0 + j];
                nx = rc[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) cv[j] = __ldg(a.C + (unsigned)(rc[j].y + t));
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    acc = fmaf(__int_as_float(rc[j].z), cv[j], acc);
                    Xt[rc[j].x] = acc;
                    acc = (rc[j].x != rc[j + 1].x) ? 0.f : acc;
                }
            }
        }
        // ---- column stage; m <- B - alpha * IDCT(kept) -----------------------------------------------------------
        {
            float u[S];
            const float *Xt = X + (BIGK ? fdct::pair_order(t) : t);
            fdct::static_for<0, S>([&](auto i) { u[decltype(i)::value] = Xt[fdct::core_index<S>(decltype(i)::value) * XS]; });
            fdct::dct_core_ortho_paired<S>(u, y);
            fdct::F2 rp[S / 2];  // pair j: rows (2j, 2j+1), swapped for odd j
            fdct::dct3_post_pairs<S>(y, rp);
            tmem_wait_st();
            float b[S];
            tmem_ld32(taddr, b);
            float *m = p.m + t;
            fdct::static_for<0, S>([&](auto i) {
                constexpr int r = decltype(i)::value, j = r / 2;
                const float res = ((r ^ j) & 1) ? fdct::f2_hi(rp[j]) : fdct::f2_lo(rp[j]);
                m[(size_t)r * p.n1] = b[r] - res;
            });
        }
        p = next;
        c = nc;
    }
    if (t == 0) ticket_finish(a.tickets, WARPS);
    tmem_free_cta(tmem, S);
}

template <typename GT, bool BIGK>
cudaError_t launch32(DemoCompressArgs a, DemoLaunch &dev, cudaStream_t stream)
{
    if (a.n_chunks <= 0) return cudaSuccess;
    const void *kernel = (const void *)compress32_kernel<GT, BIGK>;
    const size_t smem = sizeof(Area<GT>) * WARPS + 16;
    const cudaError_t err = demo_allow_smem(dev, kernel);
    if (err != cudaSuccess) return err;
    // by registers and shared memory (1 KB reserved per CTA; tensor memory has room for sixteen, the occupancy calculator
    // does not know about it)
    const int by_smem = (int)(227u * 1024u / (smem + 1024u)), per_sm = by_smem < CTAS ? by_smem : CTAS;
    const long long n_ctas = (a.n_chunks + WARPS - 1) / WARPS;
    long long grid = (long long)dev.sm_count * per_sm;
    if (grid >= n_ctas) {
        grid = n_ctas;
        a.tickets = nullptr;
    }
    void *params[] = {&a};
    return demo_launch_kernel(kernel, grid, WARPS * 32, smem, stream, params);
}

}  // namespace

cudaError_t demo_launch_compress_fast32(const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    if (a.k > MAX_K_LISTED)
        return a.grad_bf16 ? launch32<__nv_bfloat16, true>(a, dev, stream) : launch32<float, true>(a, dev, stream);
    return a.grad_bf16 ? launch32<__nv_bfloat16, false>(a, dev, stream) : launch32<float, false>(a, dev, stream);
}
