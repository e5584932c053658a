// Decode for 2-D tensors, chunk size S in {32, 64} (Decompress&Aggregate + update): S threads own one S x S chunk,
// scatter-add the W payloads in worker order into a shared tile, run two fast DCT-III passes, take the sign and
// update x <- x - lr (sign + wd x).  Also the dispatch of the fast compress and decode kernels by chunk size.
#include <cuda_bf16.h>

#include <type_traits>

#include "demo_internal.h"
#include "fast_common.cuh"
#include "fast_dct.cuh"
#include "launch.cuh"

namespace {

using namespace fastk;

template <int S>
struct Cfg {
    static constexpr int XS = S + 4;  // row stride of the transpose tile: conflict-free scalar
                                      // column access and 128-bit row access
    static constexpr int LOG2S = (S == 64) ? 6 : 5;
    // Row stride of the sender counts (16 bit): a thread goes over its row 16 bytes at a time, and rows 16 bytes apart in their banks keep
    // the threads out of each other's way.  (Rows end to end and one count per access, 32 threads on one bank: 4096 x 4096, W = 1 / 16,
    // count-normalised 92 / 105 us, now 31 / 50; the sum 30 / 36.)
    static constexpr int CS = S + 8;
};

// Bytes of one decode slot: the tile, the walk, the staged records and -- for the count-normalised mean -- one
// 16-bit sender count per coordinate.
template <int S>
__host__ __device__ constexpr size_t decode_slot_bytes(bool counts)
{
    return ((size_t)S * Cfg<S>::XS * 4 + 128 + 2 * STAGE_RECORDS * sizeof(DemoRecord) + (counts ? (size_t)S * Cfg<S>::CS * 2 : 0) + 127) /
           128 * 128;
}

static_assert(sizeof(DecodeWalk) <= 128, "reserved in decode_slot_bytes");

// SIGNS: the parameter-server form -- sign(R) goes out as int8 per element, the parameters are neither read
// nor written (a separate instantiation, so that the update kernel keeps its size).
// The records of a chunk's workers come in batches of STAGE_RECORDS through two staging buffers, the first batch a chunk
// ahead, every further one while the scatter works on the batch before it.
// The x tile comes by 16-byte asynchronous copies, sixteen per thread, not by TMA: a tensor map has to be acquired by every
// CTA that comes to a tensor, a fence that stands in front of the chunk (300M-class set, 168 matrices: 696 us with maps, 725
// with a bulk copy per row, 624 like this; one matrix of that size: 612, 731, 597).
// How the records are added up, by k.  (One instantiation each: the loops of the larger k in the same kernel cost 8 us of the
// 96 of 8192 x 8192, k = 32.)  In all of them a coordinate gets its workers' values in the order of the workers.
//   LISTED: up to 64 records per worker, staged; STAGED: up to 512, staged, in parts of 64, unless they are few enough (s = 32,
//   W k < 256) or only the signs are wanted (s = 64); BARRIERS: straight from the payloads, a barrier per worker.
// 4096 x 4096, STAGED / BARRIERS: s = 64, k = 96 / 129 / 257 W = 8 41 / 42, 49 / 51, 65 / 69 us, W = 32 80 / 92, 112 / 122, 171 / 182;
// s = 32, k = 65 W = 1 36 / 34, W = 2 39 / 39, W = 8 60 / 70, k = 129 W = 1 38 / 37, W = 2 44 / 50; signs, s = 64, k = 96 / 128
// W = 8 36 / 33, k = 200 W = 2 / 8 / 32 29 / 26, 50 / 39, 144 / 138.
// COUNTS: the count-normalised mean.  (As a branch of the same kernels its code cost the sum 2 to 12 %: 4096 x 4096, k = 32, W = 64
// 61.9 -> 55.6 us, s = 32, k = 8, W = 64 101 -> 88, 16 chunks 4.4 -> 4.2.)
enum { LISTED, STAGED, BARRIERS };
template <int S, int THREADS, bool SIGNS, int KMODE, bool COUNTS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) decode_fast_kernel(DemoDecodeArgs a)
{
    const StreamOrder order(a.wait_first);
    using C = Cfg<S>;
    constexpr int XS = C::XS, NCH = THREADS / S;
    constexpr int M = S * S;
    extern __shared__ __align__(128) unsigned char smem_all[];
    const int slot = threadIdx.x / S;
    unsigned char *smem_raw = smem_all + (size_t)slot * decode_slot_bytes<S>(COUNTS);
    const SlotBarrier<S> sb{slot + 1};
    // One tile per slot: the aggregate S, then the row-stage output, and -- once column t has been
    // read back into registers -- the staging area of the x tile, fetched behind the second transform.
    float *St = reinterpret_cast<float *>(smem_raw);  // [S*XS]
    float *Xt = St;                                   // [S*S] (aliases St)
    DecodeWalk &walk = *reinterpret_cast<DecodeWalk *>(St + S * XS);
    DemoRecord *stage_all = reinterpret_cast<DemoRecord *>(reinterpret_cast<unsigned char *>(&walk) + 128);    // [2][STAGE_RECORDS] records of a batch of workers
    unsigned short *Cn = reinterpret_cast<unsigned short *>(stage_all + 2 * STAGE_RECORDS);  // [S*CS] senders per coordinate

    const int t = threadIdx.x % S;

    const int k_eff = a.k;
    const unsigned lr_bits = __float_as_uint(a.lr);
    const float decay = 1.f - a.lr * a.wd;
    const float neg_lr_scale = -a.lr * a.agg_scale;

    // The records of a chunk's first batch of workers (up to STAGE_RECORDS records) are copied into one of two
    // staging buffers by asynchronous copies issued a whole chunk ahead, so that the payload reads of the W
    // workers -- W small pieces from W buffers -- never stand in front of the scatter.  One copy group per chunk.
    // (The records of workers w_first .. of the chunk in walk slot `which`.)
    auto stage_batch = [&](int buf, int which, int w_first) {
        if (KMODE != BARRIERS) {
            const long long off = walk.rec[which];
            const int sh = KMODE == STAGED ? stage_shift(k_eff) : (k_eff > 32) ? 6 : 5;
            DemoRecord *dst = stage_all + buf * STAGE_RECORDS;
#pragma unroll
            for (int i = 0; i < STAGE_RECORDS / S; ++i) {
                const int r = i * S + t, wl = w_first + (r >> sh), j = r & ((1 << sh) - 1);
                if (wl < a.W && j < k_eff)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst + r)),
                                 "l"(a.payloads[wl] + off + j)
                                 : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    // A CTA's slots take NCH neighbouring chunks at a time (a group), the groups on demand.  The group after the current one
    // has to be known during the current one (its records are requested), so a group is drawn two ahead: thread 0 draws at
    // the start of a chunk and writes the result down behind the scatter; the loop-top barrier publishes it.
    __shared__ unsigned drawn[2];
    unsigned group = blockIdx.x, next_group, par = 0;
    long long c = (long long)group * NCH + slot;
    int buf = 0, which = 0;  // staging buffer and walk slot of the current chunk
    if (t == 0 && c < a.n_chunks) {
        walk.e = demo_find_entry(a.entries, a.n_entries, c);
        walk.load(a.entries, a.n_entries);
        walk.seek<S>(a.entries, a.n_entries, c, k_eff, 0);
    }
    sb.sync();
    order.begin();
    if (threadIdx.x == 0) drawn[0] = second_ticket(a.tickets, (unsigned)((a.n_chunks + NCH - 1) / NCH));
    if (c < a.n_chunks) stage_batch(0, 0, 0);
    for (; (long long)group * NCH < a.n_chunks; group = next_group, c = (long long)group * NCH + slot, par ^= 1u, which ^= 1) {
        __syncthreads();  // (publishes the draw; all slots start a chunk together)
        next_group = gridDim.x + drawn[par];  // (NO_TICKET ends the loop: groups are fewer than 2^31)
        if (c >= a.n_chunks) continue;
        const bool more = (long long)next_group * NCH + slot < a.n_chunks;
        unsigned ticket = 0;
        if (threadIdx.x == 0) ticket = ticket_draw(a.tickets);
        if (t == 0 && more) walk.seek<S>(a.entries, a.n_entries, (long long)next_group * NCH + slot, k_eff, which ^ 1);
        if (!SIGNS) {  // row t of the x tile on its way to L2
            const float *xr = a.x_ptrs[walk.tensor[which]] + walk.elem[which] + (size_t)t * walk.n1[which];
            prefetch_l2(xr);
            if (S == 64) prefetch_l2(xr + 32);
        }

        {
            float4 *row = reinterpret_cast<float4 *>(St + t * XS);
#pragma unroll
            for (int v4 = 0; v4 < S / 4; ++v4) row[v4] = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (COUNTS)
                for (int v = 0; v < S; v += 8) *reinterpret_cast<uint4 *>(Cn + t * C::CS + v) = make_uint4(0u, 0u, 0u, 0u);
        }
        // (an empty group where there is no next chunk: the waits count groups)
        auto stage_next_chunk = [&](int into) {
            if (more)
                stage_batch(into, which ^ 1, 0);
            else
                asm volatile("cp.async.commit_group;" ::: "memory");
        };
        DemoRecord *stage = stage_all + buf * STAGE_RECORDS;
        // S = sum over workers in worker order (Decompress&Aggregate).
        if constexpr (KMODE != BARRIERS) {
            // Every warp owns the 32 rows of the tile its threads cleared and will transform (rows 32 w .. 32 w + 31
            // for warp w of the slot).  The records of up to sixteen workers (512 records) are staged in shared
            // memory with one round of global loads; then every warp walks the staged workers in order, reads ALL
            // records of a worker (lane j: record j, and j + 32 where k > 32) and adds those that fall into its rows.
            // A coordinate is only ever touched by one warp, so the order of the additions -- worker after worker,
            // hence bit-reproducible -- needs nothing but warp-level synchronisation.
            const int lane = t & 31, warp = t >> 5;
            const int sh = KMODE == STAGED ? stage_shift(k_eff) : (k_eff > 32) ? 6 : 5;  // a worker's records take 2^sh staging entries
            const int wb = STAGE_RECORDS >> sh;           // workers per batch: 16, 8 or fewer
            for (int w0 = 0; w0 < a.W; w0 += wb) {
                // this batch's copies have landed (requested a chunk or a batch ago), for all threads; the tile is cleared, the
                // next chunk looked up, and both warps are done with the other buffer: it takes the batch after this one --
                // of this chunk's workers or, behind the last, the first batch of the slot's next chunk
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                sb.sync();
                stage = stage_all + buf * STAGE_RECORDS;
                buf ^= 1;
                if (w0 + wb < a.W)
                    stage_batch(buf, which, w0 + wb);
                else
                    stage_next_chunk(buf);
                const int nw = min(wb, a.W - w0);
                // Four workers' records are read together, then added one worker after the other without a branch: a record
                // of the other warp's rows goes to a place of this lane's own in the tile's padding (a bank of its own), so
                // that a worker costs one dependent read-add-write.  Indices outside the chunk are noted and reported once.
                // (4096 x 4096, W = 64: 73.8 us with branches around every record -> 63.8; W = 8: 32.5 -> 32.0.)
                const bool two = k_eff > 32;
                const int spare = (32 * warp + lane) * XS + S + (lane >> 3);
                bool bad = false;
                auto add = [&](const DemoRecord &rc, bool have) {
                    const unsigned idx = (unsigned)rc.idx;
                    bad = bad || (have && idx >= (unsigned)M);
                    const bool mine = have && (idx >> (C::LOG2S + 5)) == (unsigned)warp;  // (false for idx >= M)
                    const int at = mine ? (int)(idx >> C::LOG2S) * XS + (int)(idx & (S - 1)) : spare;
                    St[at] += rc.val;
                    if (COUNTS && mine) Cn[(idx >> C::LOG2S) * C::CS + (idx & (S - 1))] += 1;
                };
                if constexpr (KMODE == STAGED) {  // a worker's records in parts of 64, the last one short
                    const int per = (k_eff + 63) >> 6;  // parts of a worker
                    int at = 0, left = k_eff, wl = 0;   // staging place and remaining records of the next part, its worker
                    auto some = [&](auto count) {
                        constexpr int U = decltype(count)::value;
                        DemoRecord rc[U][2];
                        int n[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            n[u] = left;
                            rc[u][0] = stage[at + lane];
                            rc[u][1] = stage[at + lane + 32];
                            at += 64;
                            left -= 64;
                            if (left <= 0) {
                                ++wl;
                                at = wl << sh;
                                left = k_eff;
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            add(rc[u][0], lane < n[u]);
                            add(rc[u][1], lane + 32 < n[u]);
                            __syncwarp();
                        }
                    };
#pragma unroll 1
                    for (int parts = nw * per; parts > 0;) {
                        if (parts >= 4) {
                            some(std::integral_constant<int, 4>{});
                            parts -= 4;
                        } else {
                            some(std::integral_constant<int, 1>{});
                            --parts;
                        }
                    }
                } else {
#pragma unroll 1
                    for (int wl = 0; wl < nw;) {
                        auto some = [&](auto count) {
                            constexpr int U = decltype(count)::value;
                            DemoRecord rc0[U], rc1[U];
    #pragma unroll
                            for (int u = 0; u < U; ++u) {
                                rc0[u] = stage[((wl + u) << sh) + lane];
                                if (two) rc1[u] = stage[((wl + u) << sh) + lane + 32];
                            }
    #pragma unroll
                            for (int u = 0; u < U; ++u) {
                                add(rc0[u], lane < k_eff);
                                if (two) add(rc1[u], lane + 32 < k_eff);
                                __syncwarp();
                            }
                            wl += U;
                        };
                        if (wl + 4 <= nw)
                            some(std::integral_constant<int, 4>{});
                        else
                            some(std::integral_constant<int, 1>{});
                    }
                }
                if (bad) atomicMax(a.status, DEMO_DEV_PAYLOAD);
            }
        } else {
            sb.sync();  // the tile is cleared
            add_from_payloads<S, false>(
                a.payloads, a.W, walk.rec[which], k_eff, t,
                [&](const DemoRecord &rc) {
                    if ((unsigned)rc.idx < (unsigned)M) {
                        St[(rc.idx >> C::LOG2S) * XS + (rc.idx & (S - 1))] += rc.val;
                        if (COUNTS) Cn[(rc.idx >> C::LOG2S) * C::CS + (rc.idx & (S - 1))] += 1;
                    } else {
                        atomicMax(a.status, DEMO_DEV_PAYLOAD);
                    }
                },
                [&] { sb.sync(); });
        }
        if (threadIdx.x == 0) drawn[par ^ 1u] = ticket + tickets_from((unsigned)((a.n_chunks + NCH - 1) / NCH));
        if constexpr (COUNTS) {  // Sparse Top-k Averaging: sum / number of senders, 0/0 = 0 (row t is this thread's)
#pragma unroll 1
            for (int v = 0; v < S; v += 8) {
                const uint4 n8 = *reinterpret_cast<const uint4 *>(Cn + t * C::CS + v);
                if (((n8.x | n8.y | n8.z | n8.w) & 0xfffefffeu) == 0u) continue;  // at most one sender each
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const unsigned n = ((i >> 1) == 0 ? n8.x : (i >> 1) == 1 ? n8.y : (i >> 1) == 2 ? n8.z : n8.w) >> (16 * (i & 1)) & 0xffffu;
                    if (n > 1u) St[t * XS + v + i] = St[t * XS + v + i] / (float)n;
                }
            }
        }
        // Two inverse passes through one copy of the unrolled transform (rolled loop): pass 0 along
        // row t in place, pass 1 down column t; the x tile is fetched while pass 1 computes.
        float r[S];
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            if (pass == 0) {
                const float4 *row = reinterpret_cast<const float4 *>(St + t * XS);
#pragma unroll
                for (int v4 = 0; v4 < S / 4; ++v4) {
                    const float4 f = row[v4];
                    r[4 * v4 + 0] = f.x;
                    r[4 * v4 + 1] = f.y;
                    r[4 * v4 + 2] = f.z;
                    r[4 * v4 + 3] = f.w;
                }
            } else {
#pragma unroll
                for (int u = 0; u < S; ++u) r[u] = St[u * XS + t];
                sb.sync();  // the tile is dead: stage x into it
                if (!SIGNS) {
                    constexpr int PIECES = S / 4;  // 16-byte pieces per row
                    const int n1 = walk.n1[which];
                    const float *src = a.x_ptrs[walk.tensor[which]] + walk.elem[which] + (size_t)(t / PIECES) * n1 + (t % PIECES) * 4;
                    const uint32_t dst = smem_u32(Xt) + t * 16;
#pragma unroll
                    for (int i = 0; i < PIECES; ++i)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * (S * 16)),
                                     "l"(src + (size_t)(i * (S / PIECES)) * n1)
                                     : "memory");
                    asm volatile("cp.async.commit_group;" ::: "memory");
                }
            }
            {
                // inverse transform: the DCT-IV blocks and the butterfly cascade with two sums per instruction
                float w[S], y[S];
                fdct::static_for<0, S>([&](auto i) { w[decltype(i)::value] = r[fdct::core_index<S>(decltype(i)::value)]; });
                fdct::dct_core_ortho_paired<S>(w, y);
                fdct::dct3_post_paired<S>(y, r);
            }
            if (pass == 0) {
                float4 *row = reinterpret_cast<float4 *>(St + t * XS);
#pragma unroll
                for (int v4 = 0; v4 < S / 4; ++v4)
                    row[v4] = make_float4(r[4 * v4], r[4 * v4 + 1], r[4 * v4 + 2], r[4 * v4 + 3]);
                sb.sync();
            }
        }
        if constexpr (SIGNS) {
            signed char *__restrict__ sg = a.sign_ptrs[walk.tensor[which]] + walk.elem[which] + t;
            const size_t n1 = (size_t)walk.n1[which];
#pragma unroll
            for (int i = 0; i < S; ++i) sg[i * n1] = (signed char)((r[i] > 0.f) - (r[i] < 0.f));
            sb.sync();  // the tile is free again
            continue;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");  // (the next chunk's records, requested before, have landed too)
        sb.sync();
        // sign and update:  x - lr (sign(R) + wd x) = x (1 - lr wd) - lr sign(R); -lr sign(R) is lr with
        // its sign flipped where R > 0, and zero where R == 0
        float *__restrict__ x = a.x_ptrs[walk.tensor[which]] + walk.elem[which] + t;
        const size_t n1 = (size_t)walk.n1[which];
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const float rv = r[i];
            float stepv = __uint_as_float(lr_bits ^ (~__float_as_uint(rv) & 0x80000000u));
            stepv = (rv == 0.f) ? 0.f : stepv;
            if (a.phi) stepv = rv * neg_lr_scale;  // phi = identity: -lr * R (R / W for the mean)
            x[i * n1] = fmaf(Xt[i * S + t], decay, stepv);
        }
        sb.sync();  // the tile is free again
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // no copy of this thread may outlive the CTA's shared memory
    if (threadIdx.x == 0) ticket_finish(a.tickets);
}

// The code fits the instruction cache: every slot in a CTA of its own runs best (8192 x 8192 case: 103 us with
// 64-thread CTAs, 108 us with 128, 114 us with 256).
constexpr int DECODE_THREADS = 64;

// Persistent launch: CTAs of `threads` threads (threads / S slots), as many as fit the device, each
// striding over groups of chunks.
template <typename K, typename A>
cudaError_t launch(K kernel, int threads, int nch, size_t smem, DemoLaunch &dev, cudaStream_t stream, A args)
{
    const long long n_chunks = args.n_chunks;
    if (n_chunks <= 0) return cudaSuccess;
    int per_sm = 0;
    const cudaError_t err = demo_resident_ctas(dev, (const void *)kernel, threads, smem, &per_sm);
    if (err != cudaSuccess) return err;
    const long long groups = (n_chunks + nch - 1) / nch;
    long long grid = (long long)dev.sm_count * per_sm;
    if (grid > groups) grid = groups;
    if (grid == groups) args.tickets = nullptr;
    void *params[] = {&args};
    return demo_launch_kernel((const void *)kernel, grid, threads, smem, stream, params);
}

template <int S>
cudaError_t launch_decode(const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    constexpr int TH = DECODE_THREADS;
    constexpr int NCH = TH / S;
    auto pick = [&](auto signs, auto counts) {
        constexpr bool SIGNS = decltype(signs)::value, COUNTS = decltype(counts)::value;
        const size_t smem = decode_slot_bytes<S>(COUNTS) * NCH;
        if (a.k <= 64) return launch(decode_fast_kernel<S, TH, SIGNS, LISTED, COUNTS>, TH, NCH, smem, dev, stream, a);
        if constexpr (!(SIGNS && S == 64))
            if (a.k <= STAGE_RECORDS && (S == 64 || (long long)a.W * a.k >= 256))
                return launch(decode_fast_kernel<S, TH, SIGNS, STAGED, COUNTS>, TH, NCH, smem, dev, stream, a);
        return launch(decode_fast_kernel<S, TH, SIGNS, BARRIERS, COUNTS>, TH, NCH, smem, dev, stream, a);
    };
    if (a.agg == 2) return a.sign_ptrs != nullptr ? pick(std::true_type{}, std::true_type{}) : pick(std::false_type{}, std::true_type{});
    return a.sign_ptrs != nullptr ? pick(std::true_type{}, std::false_type{}) : pick(std::false_type{}, std::false_type{});
}

// One CTA arms an mbarrier with a transaction count that no copy will ever satisfy and waits for it
// with the same bounded wait the production kernels use.
__global__ void wait_selftest_kernel(int *status, long long limit_cycles)
{
    __shared__ __align__(8) unsigned long long bar_mem;
    const uint32_t bar = smem_u32(&bar_mem);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        fence_proxy_async();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_expect_tx(bar, 16);  // 16 bytes that never arrive
    const bool arrived = mbar_wait_bounded(bar, 0, limit_cycles);
    if (!__syncthreads_and(arrived) && threadIdx.x == 0) atomicMax(status, DEMO_DEV_TIMEOUT);
}

}  // namespace

cudaError_t demo_launch_wait_selftest(int *status, long long limit_cycles, cudaStream_t stream)
{
    wait_selftest_kernel<<<1, 64, 0, stream>>>(status, limit_cycles);
    return cudaGetLastError();
}

bool demo_fast_supported(int s) { return s == 128 || s == 64 || s == 32; }

cudaError_t demo_launch_compress_fast(int s, const DemoCompressArgs &a, long long largest, DemoLaunch &dev, cudaStream_t stream)
{
    if (s == 128) return demo_launch_compress_fast128(a, dev, stream);
    if (s == 64) return demo_launch_compress_fast64(a, largest, dev, stream);
    if (s == 32) return demo_launch_compress_fast32(a, dev, stream);
    return cudaErrorInvalidValue;
}

cudaError_t demo_launch_decode_fast(int s, const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    if (s == 128) return demo_launch_decode_fast128(a, dev, stream);
    if (s == 64) return launch_decode<64>(a, dev, stream);
    if (s == 32) return launch_decode<32>(a, dev, stream);
    return cudaErrorInvalidValue;
}
