// Compress kernel for 2-D tensors with chunk size 64 (the paper's main configuration): Algorithm 1 worker
// side / CompressChunks, fused per chunk -- momentum update, 2-D DCT-II, exact top-k, momentum
// subtraction.  64 threads (a "slot") own one 64 x 64 chunk; thread t works on column t, then row t.
//
// What shapes this kernel is its instruction footprint.  A register-resident 64-point transform is
// ~10 KB of straight-line code; three copies (two forward passes, one inverse) plus fully unrolled
// tile reads do not fit the SM's instruction cache, and warps that sit at different places of such
// a stream starve on instruction fetch.  Here the hot loop is kept near 30 KB so that every slot can
// run on its own, and the phases of different chunks (tile wait, transform, selection, store burst)
// overlap on the SM's pipes instead of following one another:
//   * the three transform passes of a chunk go through ONE copy of the multiplications (the DCT-IV blocks
//     that DCT-II and DCT-III share, fast_dct.cuh) inside a rolled loop; only the butterfly cascades differ;
//   * B = beta*m + g is parked in tensor memory (one tcgen05.st of the thread's column) and read back for
//     the residual, instead of fetching and recombining the two tiles a second time;
//   * the next chunk's tiles are requested as soon as the transpose tile is dead, so they land behind
//     the inverse transform and the store burst of the current chunk;
//   * k > 48 has an instantiation of its own (select64.cuh); everything rare (tied or degenerate chunks, tiles of low
//     rank, k above the bounds of the lists) lives in out-of-line routines that work from the coefficient tile in
//     shared memory.
// Every wait on an mbarrier is bounded: on expiry the slot records DEMO_DEV_TIMEOUT and stops.
#include <cuda_bf16.h>

#include <type_traits>

#include "demo_internal.h"
#include "fast_common.cuh"
#include "fast_dct.cuh"
#include "launch.cuh"
#include "select64.cuh"

namespace {

using namespace fastk;
using namespace sel64;

constexpr int TMEM_COLS_PER_GROUP = 64;  // one column block per four warps (two slots)
constexpr int ROW_AHEAD = 8;              // entries of the row-stage list fetched ahead

// Tile area of a slot:  [0, 64*68*4)  the padded transpose / coefficient / row-stage tile X; its first 16 KB double as
// the landing area of the m tile and as the source of the TMA store of the new momentum;  behind it the landing
// area of the g tile, which between its two uses holds the lists of the selection: wide candidate list and -- at its end -- the
// row-stage list.
constexpr size_t TILE_X_BYTES = (size_t)S * XS * sizeof(float);
template <typename GT>
constexpr size_t region_bytes()
{
    constexpr size_t g_bytes = (size_t)S * S * sizeof(GT);
    constexpr size_t lists = (size_t)(WCAP + 4) * 8 + 65 * 16;  // wide list + row-stage list
    static_assert(lists <= g_bytes, "the selection's lists live in the g landing area");
    return TILE_X_BYTES + g_bytes;
}
template <typename GT>
constexpr size_t slot_bytes()
{
    constexpr size_t raw = region_bytes<GT>() + S * 4 + (CAP + 8) * 3 * 4 + 16 * 4 + 16 + 128;  // (last: SlotWalk)
    return (raw + 127) / 128 * 128;
}

// Thread 0's walk over the chunks: its place in the tensor table, and of the current and the next chunk (by turns) the tile
// and the first record.  In shared memory rather than in registers, which every thread of the kernel would have to spare.
struct SlotWalk {
    DemoTensorEntry te;
    long long next_begin;  // chunk_begin of the entry after te (or "never")
    long long rec[2];
    int e, acquired;       // entry of te; tensor whose maps were acquired last
    int tensor[2], x[2], y[2];

    __device__ __forceinline__ void load(const DemoTensorEntry *entries, int n)
    {
        te = entries[e];
        next_begin = (e + 1 < n) ? entries[e + 1].chunk_begin : 0x7fffffffffffffffLL;
    }
    // Moves on to chunk c (ids only grow) and notes its tile and record offset in `slot`.
    __device__ __forceinline__ void seek(const DemoTensorEntry *entries, int n, unsigned c, int k, int slot)
    {
        if (c >= next_begin) {
            e = demo_seek_entry(entries, n, e + 1, c);
            load(entries, n);
        }
        const unsigned lc = (unsigned)(c - te.chunk_begin);
        const unsigned k0 = lc / (unsigned)te.c1;
        tensor[slot] = te.tensor;
        x[slot] = (int)(lc - k0 * (unsigned)te.c1) * S;
        y[slot] = (int)k0 * S;
        rec[slot] = te.rec_begin + (long long)lc * k;
    }
};
static_assert(sizeof(SlotWalk) <= 128, "reserved in slot_bytes");

// QDOM = false: the momentum buffers hold the momentum itself (the contract of demo_compress).  QDOM = true (opt-in,
// demo_set_momentum_domain): they hold its chunk-wise DCT, tile by tile and transposed (element (r, c) of a tile
// is coefficient (c, r)): the step is then Q = beta*Qm + DCT(g), top-k, Qm <- Q - alpha*Q_kept -- one forward
// transform of the gradient, no inverse transform, no row stage.
// BIGK (k > MAX_K_LISTED): the selection is select_chunk_big and the row stage of the inverse is dense -- a fourth trip
// through the transform core along row t, k of whose coefficients are not zero -- instead of k rank-1 updates.
template <typename GT, int THREADS, bool QDOM, bool BIGK>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) compress64_kernel(DemoCompressArgs a)
{
    const StreamOrder order(a.wait_first);
    constexpr int NCH = THREADS / S;
    constexpr int NGROUPS = (THREADS + 127) / 128;                   // groups of four warps
    constexpr int TMEM_COLS = NGROUPS * TMEM_COLS_PER_GROUP < 32 ? 32 : NGROUPS * TMEM_COLS_PER_GROUP;
    static_assert((TMEM_COLS & (TMEM_COLS - 1)) == 0, "tensor-memory allocations are powers of two");
    constexpr unsigned TILE_BYTES = S * S * sizeof(float) + S * S * sizeof(GT);

    extern __shared__ __align__(128) unsigned char smem_all[];
    const int slot = threadIdx.x / S;
    SlotMem sm;
    sm.raw = smem_all + (size_t)slot * slot_bytes<GT>();
    float *Ms = reinterpret_cast<float *>(sm.raw);             // [S*S] m tile
    GT *Gs = reinterpret_cast<GT *>(sm.raw + TILE_X_BYTES);    // [S*S] g tile
    sm.X = Ms;
    sm.wkey = reinterpret_cast<unsigned *>(sm.raw + TILE_X_BYTES);
    sm.widx = sm.wkey + WCAP + 4;
    sm.tmax = reinterpret_cast<float *>(sm.raw + region_bytes<GT>());
    sm.cand_idx = reinterpret_cast<int *>(sm.tmax + S);
    sm.cand_val = reinterpret_cast<float *>(sm.cand_idx + CAP + 8);
    sm.cand_key = reinterpret_cast<unsigned *>(sm.cand_val + CAP + 8);
    sm.recs4 = reinterpret_cast<int4 *>(sm.raw + region_bytes<GT>()) - 65;
    sm.misc = reinterpret_cast<unsigned *>(sm.cand_key + CAP + 8);
    unsigned long long *bar_mem = reinterpret_cast<unsigned long long *>(sm.misc + 16);
    SlotWalk &walk = *reinterpret_cast<SlotWalk *>(bar_mem + 2);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_all + (size_t)NCH * slot_bytes<GT>());
    float *X = sm.X;
    int4 *recs4 = sm.recs4;

    // "row" of the padding entries of the row-stage list: the scratch line tmax[0..S) seen from X
    constexpr int PAD_ROW = (int)(region_bytes<GT>() / sizeof(float));
    const int t = threadIdx.x % S;
    const int hw_warp = threadIdx.x >> 5;
    const SlotBarrier<S> sb{slot + 1};
    const uint32_t bar = smem_u32(bar_mem);

    const int k_eff = a.k;
    const unsigned n_chunks = (unsigned)a.n_chunks;  // (fewer than 2^31)
    unsigned c = blockIdx.x;

    // (thread 0) the tensor maps of the chunk in walk slot `which`
    auto map_of = [&](const void *maps, int which) {
        return static_cast<const char *>(maps) + (size_t)walk.tensor[which] * TMAP_BYTES;
    };
    // (thread 0) maps that this thread has not used yet are acquired before their first use
    auto acquire_maps = [&](int which) {
        if (walk.tensor[which] != walk.acquired) {
            walk.acquired = walk.tensor[which];
            tmap_acquire(map_of(a.tmap_m, which));
            tmap_acquire(map_of(a.tmap_g, which));
        }
    };
    // (thread 0) request the tiles of a chunk
    auto issue_loads = [&](int which) {
        mbar_expect_tx(bar, TILE_BYTES);
        tma_load_2d(smem_u32(Ms), map_of(a.tmap_m, which), walk.x[which], walk.y[which], bar);
        tma_load_2d(smem_u32(Gs), map_of(a.tmap_g, which), walk.x[which], walk.y[which], bar);
    };

    if (t == 0) {
        mbar_init(bar, 1);
        fence_proxy_async();
    }
    auto first_chunk = [&]() {
        walk.e = demo_find_entry(a.entries, a.n_entries, c);
        walk.acquired = -1;
        walk.load(a.entries, a.n_entries);
        walk.seek(a.entries, a.n_entries, c, k_eff, 0);
        acquire_maps(0);
    };
    if (t == 0 && c < n_chunks && !a.late_lookup) first_chunk();
    order.begin();
    __syncwarp();
    if (hw_warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"((uint32_t)TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    fence_proxy_async();
    const uint32_t tmem_base = *tmem_slot;
    // this thread's lane of tensor memory (a warp reaches the 32 lanes of its quadrant) and its slot's columns
    const uint32_t taddr = tmem_base + ((uint32_t)((hw_warp & 3) * 32) << 16) + (uint32_t)((hw_warp >> 2) * TMEM_COLS_PER_GROUP);

    unsigned phase = 0;
    // (thread 0) the new momentum tile goes out, then -- once the store has read it -- the next chunk's tiles come in
    auto store_and_load_next = [&](int which, bool more) {
        tma_store_2d(map_of(a.tmap_m, which), walk.x[which], walk.y[which], smem_u32(Ms));
        tma_store_commit();
        tma_store_wait_read();
        if (more) issue_loads(which ^ 1);
    };

    static_assert(NCH == 1, "one slot per CTA draws the chunks");
    // (Behind the allocation: requested in front of it, or prefetched in front of begin(), 1184 chunks take 23 instead of 19 us.)
    if (t == 0 && c < n_chunks) {
        if (a.late_lookup) first_chunk();
        issue_loads(0);
        // the slot's next chunk is always known one chunk ahead: the first two rounds are fixed, the rest is drawn
        sm.misc[8] = a.tickets ? gridDim.x + c : NO_TICKET;
    }
    sb.sync();

    int which = 0;  // walk slot of the current chunk
    for (unsigned nc; c < n_chunks; c = nc, which ^= 1) {
        // The next chunk is looked up while this chunk's tiles are on their way: the reads of the tensor table and, where the
        // tensor changes, the acquisition of its maps (a fence of about a microsecond; in a set of 168 matrices of 1024
        // columns it is due at nearly every chunk) cost nothing here.  Behind them thread 0 draws the chunk after it, which
        // the others get to see behind the first transform.  (One call, fixed rounds with the look-up and the fences in front
        // of the loads -> this: 300M-class decoder set 1134 -> 990 us, one matrix of 50304 x 20480 2313 -> 2134 us.)
        nc = sm.misc[8];
        unsigned ticket = 0;
        if (t == 0 && nc < n_chunks) {
            walk.seek(a.entries, a.n_entries, nc, k_eff, which ^ 1);
            acquire_maps(which ^ 1);
            ticket = ticket_draw(a.tickets);  // (not looked at before it is written down, behind the first transform)
        }
        // every thread waits for the tiles by itself; whether the wait expired is settled for the whole slot
        // at the first barrier of pass 0 (no barrier lies in between)
        const bool arrived = mbar_wait_bounded(bar, phase);
        phase ^= 1u;
        bool dead = false;
        // (No L2 prefetch of the next chunk's tiles: on a single launch it gains 0.5 %, but in a step that runs at the
        // board's power limit the extra L2 requests cost 1.4 %.)

        // Three passes through one copy of the transform core: 0 = DCT-II down column t of B = beta*m + g,
        // 1 = DCT-II along row t (followed by the selection and the sparse row stage of the inverse),
        // 2 = DCT-III down column t of the row-stage tile (followed by the residual).  BIGK: 2 = DCT-III along row t of
        // the kept coefficients, 3 = DCT-III down column t.
        constexpr int PASSES = QDOM ? 2 : (BIGK ? 4 : 3);
#pragma unroll 1
        for (int ph = 0; ph < PASSES; ++ph) {
            float w[S], y[S];
            if (ph < 2) {
                float x[S];
                if (ph == 0) {
                    if constexpr (QDOM) {
                        // row t of the stored coefficients (column t of the transposed tile) is parked for pass 1;
                        // the forward transform runs on the gradient alone
                        float mq[S];
#pragma unroll
                        for (int i = 0; i < S; ++i) mq[i] = Ms[i * S + t];
                        tmem_st64(taddr, mq);
#pragma unroll
                        for (int i = 0; i < S; ++i) x[i] = to_f32(Gs[i * S + t]);
                    } else {
#pragma unroll
                        for (int i = 0; i < S; ++i) x[i] = fmaf(a.beta, Ms[i * S + t], to_f32(Gs[i * S + t]));
                        // B = beta*m + g, parked for the residual; column k of the tensor-memory lane takes element
                        // pair_order(k), so that the registers of the store are those of the cascade's pairs
                        float xp[S];
                        fdct::static_for<0, S>([&](auto i) { xp[decltype(i)::value] = x[fdct::pair_order(decltype(i)::value)]; });
                        tmem_st64(taddr, xp);
                    }
                    // every thread has consumed its column of the staged tiles (X aliases them)
                    if (!sb.sync_and(arrived)) {
                        if (t == 0) atomicMax(a.status, DEMO_DEV_TIMEOUT);
                        mbar_wait_bounded(bar, phase ^ 1u);  // give copies in flight one more bounded chance to land
                        dead = true;
                        break;
                    }
                } else {
                    const float4 *row = reinterpret_cast<const float4 *>(X + t * XS);
#pragma unroll
                    for (int v4 = 0; v4 < S / 4; ++v4) {  // (pass 0 stored the rows in pair order)
                        const float4 f = row[v4];
                        x[4 * v4 + 0] = f.x;
                        x[4 * v4 + 1] = f.y;
                        x[4 * v4 + 3] = f.z;
                        x[4 * v4 + 2] = f.w;
                    }
                }
                fdct::dct2_pre_paired<S>(x, w);
            } else if (BIGK && ph == 2) {
                const float4 *row = reinterpret_cast<const float4 *>(X + t * XS);
#pragma unroll
                for (int v4 = 0; v4 < S / 4; ++v4) {  // (the selection left the kept coefficients in core order)
                    const float4 f = row[v4];
                    w[4 * v4 + 0] = f.x;
                    w[4 * v4 + 1] = f.y;
                    w[4 * v4 + 2] = f.z;
                    w[4 * v4 + 3] = f.w;
                }
            } else {
                // column t of the row-stage tile: written by this thread only (no barrier before reading it), or, in pair
                // order within each row, by the dense row stage
                const float *Xt = X + (BIGK ? fdct::pair_order(t) : t);
                fdct::static_for<0, S>([&](auto i) {
                    constexpr int p = decltype(i)::value;
                    w[p] = Xt[fdct::core_index<S>(p) * XS];
                });
            }

            fdct::dct_core_ortho_paired<S>(w, y);

            if (ph == 0) {
                // transpose through shared memory; inside a row the elements sit in pair order, so that the 128-bit
                // row reads of pass 1 deliver the cascade's pairs as they are
                float *Xc = X + fdct::pair_order(t);
                fdct::static_for<0, S>([&](auto i) {
                    constexpr int p = decltype(i)::value;
                    Xc[fdct::core_index<S>(p) * XS] = y[p];
                });
                if (t == 0) sm.misc[8] = nc < n_chunks ? 2u * gridDim.x + ticket : NO_TICKET;  // (all have read the last one: the barrier above)
                sb.sync();
            } else if (BIGK && !QDOM && ph == 2) {
                fdct::F2 rp[S / 2];  // the row of the row-stage tile in pair order
                fdct::dct3_post_pairs<S>(y, rp);
                float4 *row = reinterpret_cast<float4 *>(X + t * XS);
#pragma unroll
                for (int v4 = 0; v4 < S / 4; ++v4)
                    row[v4] = make_float4(fdct::f2_lo(rp[2 * v4]), fdct::f2_hi(rp[2 * v4]), fdct::f2_lo(rp[2 * v4 + 1]),
                                          fdct::f2_hi(rp[2 * v4 + 1]));
                sb.sync();
            } else if (ph == PASSES - 1 && !QDOM) {
                // m <- B - alpha * IDCT(kept): column t of the new momentum goes into a dense tile (the m staging
                // area; the row-stage tile it overlaps is dead for every thread only after the barrier below, so the
                // column is formed in registers first), which one TMA store writes out; the next chunk's tiles are
                // requested as soon as the store has read the tile.
                fdct::F2 rp[S / 2];  // pair p: rows (2p, 2p+1), swapped for odd p
                fdct::dct3_post_pairs<S>(y, rp);
                tmem_wait_st();  // the store of B (pass 0) has long completed
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float b[32];  // columns 32h .. 32h+31 of the lane: B in pair order, i.e. the pairs' own order
                    tmem_ld32(taddr + 32 * h, b);
#pragma unroll
                    for (int q = 0; q < 16; ++q) rp[16 * h + q] = fdct::f2_sub(fdct::f2_make(b[2 * q], b[2 * q + 1]), rp[16 * h + q]);
                }
                sb.sync();  // every thread has read its column of the row-stage tile
                fdct::static_for<0, S / 2>([&](auto i) {
                    constexpr int p = decltype(i)::value;
                    Ms[(2 * p + (p & 1)) * S + t] = fdct::f2_lo(rp[p]);
                    Ms[(2 * p + 1 - (p & 1)) * S + t] = fdct::f2_hi(rp[p]);
                });
                fence_proxy_async();
                sb.sync();
                {
                    // the store of this chunk, then -- once it has read the tile -- the loads of the next chunk
                    if (t == 0) store_and_load_next(which, nc < n_chunks);
                }
            } else {
                // ---- coefficients of row t: q[v] = Q[t][v] ------------------------------------------
                DemoRecord *rec = a.payload + walk.rec[which];
                float q[S];
                fdct::static_for<0, S>([&](auto i) {
                    constexpr int p = decltype(i)::value;
                    q[fdct::core_index<S>(p)] = y[p];
                });
                if constexpr (QDOM) {
                    // Q = beta * Qm + DCT(g); the stored row comes back from tensor memory
                    tmem_wait_st();
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float mq[32];
                        tmem_ld32(taddr + 32 * h, mq);
#pragma unroll
                        for (int j = 0; j < 32; ++j) q[32 * h + j] = fmaf(a.beta, mq[j], q[32 * h + j]);
                    }
                    if constexpr (BIGK)
                        select_chunk_big<true>(sm, q, k_eff, rec, a.alpha, t, sb, slot + 1);
                    else
                        select_chunk<true>(sm, q, k_eff, rec, a.alpha, t, sb, slot + 1, PAD_ROW);
                    sb.sync();  // the tile holds Q - alpha * Q_kept (kept entries were patched by the record writers)
                    float4 rowv[S / 4];
                    {
                        const float4 *row = reinterpret_cast<const float4 *>(X + t * XS);
#pragma unroll
                        for (int v4 = 0; v4 < S / 4; ++v4) rowv[v4] = row[v4];
                    }
                    sb.sync();  // the dense tile below overlaps the coefficient tile
#pragma unroll
                    for (int v4 = 0; v4 < S / 4; ++v4) {
                        Ms[(4 * v4 + 0) * S + t] = rowv[v4].x;
                        Ms[(4 * v4 + 1) * S + t] = rowv[v4].y;
                        Ms[(4 * v4 + 2) * S + t] = rowv[v4].z;
                        Ms[(4 * v4 + 3) * S + t] = rowv[v4].w;
                    }
                    fence_proxy_async();
                    sb.sync();
                    if (t == 0) store_and_load_next(which, nc < n_chunks);
                    continue;
                }
                if constexpr (BIGK) {
                    select_chunk_big<false>(sm, q, k_eff, rec, a.alpha, t, sb, slot + 1);
                    sb.sync();  // records complete, kept coefficients in the tile
                    continue;
                }
                select_chunk<false>(sm, q, k_eff, rec, a.alpha, t, sb, slot + 1, PAD_ROW);
                sb.sync();  // records complete (shared list and global payload), tile zeroed

                // ---- residual: row stage of the inverse from the k_eff records, sparse --------------
                {
                    // T[u][t] = sum over kept (u, v) of alpha * val * C[v][t]; the basis is read through L1
                    float acc = 0.f;
                    // The running sum of a row is stored after every entry (the last store of a row carries the
                    // whole sum) and starts again from zero when the next entry belongs to another row: no branch in
                    // the loop.  The list is padded with zero-valued entries (entry 64 is always one) whose "row" is
                    // a scratch line outside the tile.  Entries and their cosines are fetched ahead of the
                    // dependent accumulation.
                    float *Xt = X + t;
                    int4 nx = recs4[0];
#pragma unroll 1
                    for (int r0 = 0; r0 < k_eff; r0 += ROW_AHEAD) {
                        int4 rc[ROW_AHEAD + 1];
                        float cv[ROW_AHEAD];
                        rc[0] = nx;
#pragma unroll
                        for (int j = 1; j < ROW_AHEAD + 1; ++j) rc[j] = recs4[r0 + j];
                        nx = rc[ROW_AHEAD];
#pragma unroll
                        for (int j = 0; j < ROW_AHEAD; ++j) cv[j] = __ldg(a.C + (unsigned)(rc[j].y + t));
#pragma unroll
                        for (int j = 0; j < ROW_AHEAD; ++j) {
                            acc = fmaf(__int_as_float(rc[j].z), cv[j], acc);
                            Xt[rc[j].x] = acc;
                            acc = (rc[j].x != rc[j + 1].x) ? 0.f : acc;
                        }
                    }
                }
            }
        }
        if (dead) break;
    }
    if (threadIdx.x == 0) ticket_finish(a.tickets);
    // tear-down: every slot of the CTA is done with its tensor-memory columns
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (hw_warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
}

template <typename GT, int THREADS, bool QDOM, bool BIGK>
cudaError_t launch64(const DemoCompressArgs &a, long long largest, DemoLaunch &dev, cudaStream_t stream)
{
    constexpr int NCH = THREADS / S;
    auto kernel = compress64_kernel<GT, THREADS, QDOM, BIGK>;
    const size_t smem = slot_bytes<GT>() * NCH + 16;
    if (a.n_chunks <= 0) return cudaSuccess;
    const cudaError_t err = demo_allow_smem(dev, (const void *)kernel);
    if (err != cudaSuccess) return err;
    // CTAs per SM: registers (launch bounds: 512 threads per SM), shared memory (227 KB, 1 KB reserved per CTA)
    // and tensor memory (512 columns, 64 per four warps).  The occupancy calculator is not asked: it does not
    // know about tensor memory and was seen to answer 1 for this kernel.
    int per_sm = 512 / THREADS;
    const int smem_limit = (int)((227u * 1024u) / (smem + 1024u));
    const int tmem_limit = 512 / (((THREADS + 127) / 128) * TMEM_COLS_PER_GROUP);
    if (per_sm > smem_limit) per_sm = smem_limit;
    if (per_sm > tmem_limit) per_sm = tmem_limit;
    if (per_sm < 1) per_sm = 1;
    const long long groups = (a.n_chunks + NCH - 1) / NCH;
    long long grid = (long long)dev.sm_count * per_sm;
    if (grid > groups) grid = groups;
    DemoCompressArgs b = a;
    if (grid == groups) b.tickets = nullptr;
    // The look-up in front of the wait spares every call its latency, except where a set of several tensors nearly fills the device, up to
    // two and a half times: there all tiles would be requested in the same moment, by many maps, and land late; behind the allocation the
    // look-ups spread the requests.  Steps, early / late / before both: 280 chunks of 9 tensors, seven workers 92.5 / 99.9 / 101.7 us; 800 of
    // 23, two workers 48.1 / 44.3 / 46.0; 976 of 57, six workers 135 / 120 / 120; 1424 of 30, six workers 170.5 / 158.5 / 167.1; 2400 of 65,
    // two workers 91.8 / 85.3 / 88.0; 2640 of 72, one worker 60.3 / 60.2 / 63.1; 3328 of 58, three workers 171 / 178 / 173.
    // The line lies at four chunks per SM, with more than four tensors at three and a quarter, where no tensor holds more than three quarters of
    // the chunks (few maps again).  Steps of two workers, data not in L2: 540 chunks of 60 37.9 / 35.3 / 37.3, of 9 34.7 / 33.6 / 34.9, 500 of 20
    // 34.6 / 33.7 / 35.3, but 450 of 10 31.7 / 32.3 / 33.9, 360 of 40 31.4 / 32.4 / 34.3; compress of three, data in L2: 540 of 60 46.0 / 39.1 /
    // 39.2, 375 of 5 35.1 / 36.9 / 37.0, two, 556 of 15, 500 of them in one, 35.4 / 36.7 / 37.4.  (Not in the transform domain: 440 of 15, three
    // workers 42.4 early, 43.6 late.)
    const bool spread = a.n_entries > 4 && 4 * largest <= 3 * a.n_chunks && !a.momentum_dct;
    const long long line = (spread ? 13LL : 16LL) * dev.sm_count / 4;
    b.late_lookup = a.n_entries > 1 && 2 * groups <= 5 * grid && grid > line;
    void *params[] = {&b};
    return demo_launch_kernel((const void *)kernel, grid, THREADS, smem, stream, params);
}

}  // namespace

// Needs the TMA tensor maps of both tensors.
cudaError_t demo_launch_compress_fast64(const DemoCompressArgs &a, long long largest, DemoLaunch &dev, cudaStream_t stream)
{
    if (a.tmap_m == nullptr || a.tmap_g == nullptr) return cudaErrorNotSupported;
    auto pick = [&](auto gt, auto qdom) {
        using GT = decltype(gt);
        constexpr bool Q = decltype(qdom)::value;
        return a.k > MAX_K_LISTED ? launch64<GT, 64, Q, true>(a, largest, dev, stream) : launch64<GT, 64, Q, false>(a, largest, dev, stream);
    };
    if (a.momentum_dct)
        return a.grad_bf16 ? pick(__nv_bfloat16{}, std::true_type{}) : pick(float{}, std::true_type{});
    return a.grad_bf16 ? pick(__nv_bfloat16{}, std::false_type{}) : pick(float{}, std::false_type{});
}
