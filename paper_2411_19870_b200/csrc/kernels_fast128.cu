// Fast kernels for 2-D tensors with chunk size 128: one 256-thread CTA per 128 x 128 chunk.
//
// A 128-point transform does not fit one thread's registers, so it is split by the first stage of the
// same factorisation the 64-point code uses (fast_dct.cuh):
//     DCT-II_128:  u[n] = x[n] + x[127-n],  v[n] = x[n] - x[127-n]   (n < 64)
//                  X[2p] = DCT-II_64(u)[p],  X[2p+1] = DCT-IV_64(v)[p]
// Thread (h, j) = (threadIdx.x / 128, threadIdx.x % 128) owns line j (a column in the first pass, a row
// in the second) and computes its even (h = 0) or odd (h = 1) outputs; h is warp-uniform, so the two
// transform bodies never diverge inside a warp.  The inverse runs the transposed graph:
//     e = DCT-III_64(X[even]),  o = DCT-IV_64(X[odd]),  x[n] = e[n] + o[n],  x[127-n] = e[n] - o[n]
// where thread h of a line finishes n in [32h, 32h+32): the two exchange half of e and o through shared memory.
//
// compress: TMA-staged m and g tiles -> B = beta*m + g (half a column per thread, parked in tensor memory, from where the
// other thread of the column reads it) -> column pass -> row pass ->
// coefficients in shared memory -> exact top-k (bound from the 256 half-row maxima, candidate list, ballot search; radix
// select for degenerate chunks) -> records; sparse row stage of the inverse from the records, half of them by each half of
// the CTA, fast column stage, residual m <- B - alpha * IDCT(kept) against the parked B, one TMA store of the new momentum
// tile.  The next chunk's g tile comes in, and its m tile to L2, as soon as B is formed.  decode: scatter-add of the W payloads
// in worker order, two inverse passes, sign, update; half of the x tile is staged into the (then dead) coefficient tile.
// Two CTAs of a serial chain of phases per SM are what registers (128 for the 64-point halves) and, for compress, shared
// memory allow: shared-memory accesses and issue each take about half of the time.  8192 x 8192, k = 32, bf16 gradients:
// compress 242 -> 222 us (k = 128 313 -> 272) with the halves of the row stage and the early g tile; decode 162 -> 141 us and
// signs 235 -> 131 us with half the exchange (before, the signs form kept two sets of 64 results and spilled), W = 8
// 155 -> 145 and 131 -> 121 us with staged records and the x tile in halves; compress of 2368 chunks 134.0 -> 133.3 us, 592
// 39.6 -> 39.0 with half a column of B per thread (both halves by both before).
// Tiles need the TMA tensor maps; without them the host uses the generic kernels for s = 128.
#include <cuda_bf16.h>

#include <type_traits>

#include "demo_internal.h"
#include "fast_common.cuh"
#include "fast_dct.cuh"
#include "launch.cuh"

namespace {

using namespace fastk;

constexpr int S = 128, H = 64, XS = S + 4, M = S * S, THREADS = 256;
// The decode tile is only ever accessed element-wise: an odd row stride keeps a warp whose lanes walk 32
// different rows (the row pass) on 32 different banks; S + 4 (compress: 128-bit row accesses) gives 4-way
// conflicts there.
constexpr int XSD = S + 1;
constexpr int RECS128 = 128 + 40;     // row-stage list: up to 128 kept records + padding for the look-ahead
constexpr int ROW_AHEAD128 = 8;       // entries of the row-stage list fetched ahead of the accumulation
constexpr int TMEM_COLS128 = 128;     // tensor-memory columns of a compress CTA (two CTAs per SM)
constexpr int CAP128 = 256;           // candidate capacity of the fast top-k (one per thread)
constexpr int CAP128P = CAP128 + 4;   // padded for 128-bit key loads
using SC = fdct::ScaleOrtho<S>;

__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned *warp_tot /*[8]*/)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned inc = warp_inclusive_scan(v, lane);
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    unsigned base = 0;
    for (int w = 0; w < warp; ++w) base += warp_tot[w];
    __syncthreads();
    return base + inc - v;
}

// Forward half-transform of one line: in[n] = x[n] (+/-) x[127-n] already formed; out[p] is
// coefficient 2p (h = 0) or 2p+1 (h = 1) of the orthonormal 128-point DCT-II.
__device__ __forceinline__ void forward_half(int h, float (&in)[H], float (&out)[H])
{
    if (h == 0) {
        fdct::dct2_packed<H, SC>(in, out);
        out[0] *= fdct::dc_scale<S>();
    } else {
        fdct::dct4_paired<H, SC>(in, out);
    }
}
// Inverse half-transform: in[p] = coefficient 2p (h = 0) or 2p+1 (h = 1), result e (h = 0) or o (h = 1).  Thread h of the
// line finishes the elements n and 127-n of n in [32h, 32h+32): it keeps that part of its result and sends the other.
__device__ __forceinline__ void inverse_half(int h, float (&in)[H], float (&keep)[H / 2], float (&send)[H / 2])
{
    float out[H];
    if (h == 0) {
        in[0] *= fdct::dc_scale<S>();
        fdct::dct3_packed<H, SC>(in, out);
#pragma unroll
        for (int q = 0; q < H / 2; ++q) {
            keep[q] = out[q];
            send[q] = out[H / 2 + q];
        }
    } else {
        fdct::dct4_paired<H, SC>(in, out);
#pragma unroll
        for (int q = 0; q < H / 2; ++q) {
            keep[q] = out[H / 2 + q];
            send[q] = out[q];
        }
    }
}
// Elements n (lo) and 127-n (hi) from the kept and the received part: e + o and e - o.
__device__ __forceinline__ void inverse_join(int h, const float (&keep)[H / 2], float (&lo)[H / 2], float (&hi)[H / 2])
{   // (in: hi = the received part)
    if (h == 0) {
#pragma unroll
        for (int q = 0; q < H / 2; ++q) {
            lo[q] = keep[q] + hi[q];
            hi[q] = keep[q] - hi[q];
        }
    } else {
#pragma unroll
        for (int q = 0; q < H / 2; ++q) {
            lo[q] = hi[q] + keep[q];
            hi[q] = hi[q] - keep[q];
        }
    }
}

// The g tile has a landing area of its own behind the tile that m lands in and the transform works in.
template <typename GT>
constexpr size_t compress128_tile_bytes()
{
    return (size_t)S * XS * sizeof(float) + (size_t)M * sizeof(GT);
}
template <typename GT>
constexpr size_t compress128_smem()
{
    return compress128_tile_bytes<GT>() + (256 + 8 + 4) * 4 + RECS128 * 16 + 3 * CAP128P * 4 + 16 + 16;
}

template <typename GT>
__global__ void __launch_bounds__(THREADS, 2) compress_fast128_kernel(DemoCompressArgs a)
{
    const StreamOrder order(a.wait_first);
    constexpr unsigned TILE_BYTES = M * sizeof(float) + M * sizeof(GT);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *Ms = reinterpret_cast<float *>(smem_raw);  // [128*128] m tile
    float *X = Ms;                                    // [128*132] transpose / coefficients / row stage (aliases the m tile)
    GT *Gs = reinterpret_cast<GT *>(X + S * XS);      // [128*128] g tile
    unsigned *hist = reinterpret_cast<unsigned *>(smem_raw + compress128_tile_bytes<GT>());  // [256]
    unsigned *warp_tot = hist + 256;                                                         // [8]
    unsigned *s_state = warp_tot + 8;                                                        // [4]
    int4 *recs4 = reinterpret_cast<int4 *>(s_state + 4);                                     // [RECS128]
    unsigned *cand_key = reinterpret_cast<unsigned *>(recs4 + RECS128);                      // [CAP128P]
    float *cand_val = reinterpret_cast<float *>(cand_key + CAP128P);                         // [CAP128P]
    int *cand_idx = reinterpret_cast<int *>(cand_val + CAP128P);                             // [CAP128P]
    unsigned long long *bar_mem = reinterpret_cast<unsigned long long *>(cand_idx + CAP128P);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar_mem + 2);

    const int tid = threadIdx.x, h = tid >> 7, j = tid & 127;
    const uint32_t bar = smem_u32(bar_mem);
    EntryCursor cur;
    unsigned phase = 0;
    const char *acquired = nullptr;

    auto acquire_maps = [&](const DemoTensorEntry &te) {
        const char *tm_m = static_cast<const char *>(a.tmap_m) + (size_t)te.tensor * TMAP_BYTES;
        if (tid == 0 && tm_m != acquired) {  // tensor maps this thread has not used yet
            acquired = tm_m;
            tmap_acquire(tm_m);
            tmap_acquire(static_cast<const char *>(a.tmap_g) + (size_t)te.tensor * TMAP_BYTES);
        }
    };
    // (thread 0) requests a chunk's g tile, which may come as soon as the one before it has been read, and with it announces
    // both tiles; the m tile follows when the new momentum of the chunk before has left its place.  `ahead`: both only to L2.
    auto issue_tile = [&](const DemoTensorEntry &te, long long c, bool g, bool ahead) {
        const unsigned lc = (unsigned)(c - te.chunk_begin);
        const unsigned k0 = lc / (unsigned)te.c1, k1 = lc - k0 * (unsigned)te.c1;
        const char *tm_g = static_cast<const char *>(a.tmap_g) + (size_t)te.tensor * TMAP_BYTES;
        const char *tm_m = static_cast<const char *>(a.tmap_m) + (size_t)te.tensor * TMAP_BYTES;
        if (ahead) {
            tma_prefetch_2d(tm_g, k1 * S, k0 * S);
        } else {
            if (g) mbar_expect_tx(bar, TILE_BYTES);
            tma_load_2d(g ? smem_u32(Gs) : smem_u32(Ms), g ? tm_g : tm_m, k1 * S, k0 * S, bar);
        }
        if (g || ahead) tma_prefetch_2d(tm_m, k1 * S, k0 * S);
    };

    long long c = blockIdx.x;
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_proxy_async();
    }
    if (c < a.n_chunks) {
        cur.seek(a.entries, a.n_entries, c);
        acquire_maps(cur.te);
        if (tid == 0) issue_tile(cur.te, c, false, true);
    }
    order.begin();
    if (tid == 0 && c < a.n_chunks) {
        issue_tile(cur.te, c, true, false);
        issue_tile(cur.te, c, false, false);
    }
    __syncwarp();
    // Tensor memory as storage: column j of B = beta*m + g is parked in lane j between the forward pass and the residual, by
    // thread (0, j) its rows 0..63 in columns 0..63, by thread (1, j) its rows 127..64 in columns 64..127; each of the two
    // reads back half of both.
    if (tid == 0) tmem_slot[1] = ticket_draw(a.tickets);
    const uint32_t tmem_base = tmem_alloc_cta(tmem_slot, TMEM_COLS128);
    fence_proxy_async();
    const uint32_t taddr = tmem_base + ((uint32_t)(j & ~31) << 16);

    for (long long nc; c < a.n_chunks; c = nc) {
        const DemoTensorEntry te = cur.te;  // the cursor points at chunk c
        const unsigned lc = (unsigned)(c - te.chunk_begin);
        const unsigned k0 = lc / (unsigned)te.c1, k1 = lc - k0 * (unsigned)te.c1;
        const int k_eff = te.k_eff;
        DemoRecord *rec = a.payload + te.rec_begin + (long long)lc * k_eff;

        // the next chunk (drawn during the previous one) is looked up, and its tensor maps acquired, while the tiles are on
        // their way; the cursor moves on.  (Thread 0 wrote the ticket at the end of the previous chunk and overwrites it at
        // the end of this one; the barrier publishes it, those below see to it that every thread has read it.)
        __syncthreads();
        nc = (long long)gridDim.x + tmem_slot[1];
        if (nc < a.n_chunks) {
            cur.seek(a.entries, a.n_entries, nc);
            acquire_maps(cur.te);
        }
        const bool arrived = mbar_wait_bounded(bar, phase);
        phase ^= 1u;
        if (!__syncthreads_and(arrived)) {
            if (tid == 0) atomicMax(a.status, DEMO_DEV_TIMEOUT);
            mbar_wait_bounded(bar, phase ^ 1u);  // give copies in flight one more bounded chance to land
            break;
        }

        // ---- two forward passes through one rolled copy of the half-transforms ---------------------
        float in[H], out[H];
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            if (pass == 0) {
                // Column j of B = beta*m + g: thread h forms the half of it that it will write back (rows 0 .. 63 or 127 .. 64) and parks
                // it in tensor memory (two stores of 32 columns), where the other thread of the column reads it for its own fold,
                // in[n] = B[n][j] +/- B[127-n][j].  (With both halves formed by both threads: twice the shared-memory reads,
                // conversions and multiply-adds.)
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float park[32];
#pragma unroll
                    for (int q = 0; q < 32; ++q) {
                        const int n = 32 * half + q, at = (h ? S - 1 - n : n) * S + j;
                        park[q] = in[n] = fmaf(a.beta, Ms[at], to_f32(Gs[at]));
                    }
                    tmem_st32(taddr + h * H + 32 * half, park);
                }
                tmem_wait_st();
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                fence_proxy_async();
                __syncthreads();  // the staged tiles are consumed (X aliases the m tile)
                if (tid == 0 && nc < a.n_chunks) issue_tile(cur.te, nc, true, false);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float other[32];
                    tmem_ld32(taddr + (h ^ 1) * H + 32 * half, other);
#pragma unroll
                    for (int q = 0; q < 32; ++q) {
                        const int n = 32 * half + q;
                        in[n] = h ? other[q] - in[n] : in[n] + other[q];
                    }
                }
            } else {
                // row j of the column-transformed tile, folded
                const float4 *row = reinterpret_cast<const float4 *>(X + j * XS);
#pragma unroll
                for (int n4 = 0; n4 < H / 4; ++n4) {
                    const float4 lo = row[n4];
                    const float4 hi = row[S / 4 - 1 - n4];  // elements 127-4n4-3 .. 127-4n4
                    in[4 * n4 + 0] = h ? lo.x - hi.w : lo.x + hi.w;
                    in[4 * n4 + 1] = h ? lo.y - hi.z : lo.y + hi.z;
                    in[4 * n4 + 2] = h ? lo.z - hi.y : lo.z + hi.y;
                    in[4 * n4 + 3] = h ? lo.w - hi.x : lo.w + hi.x;
                }
                __syncthreads();  // every thread has read its row before the coefficients overwrite the tile
            }
            forward_half(h, in, out);
            if (pass == 0) {
#pragma unroll
                for (int p = 0; p < H; ++p) X[(2 * p + h) * XS + j] = out[p];  // Y[u][j]
            } else {
                // Q[j][2p + h]: a row keeps its even coefficients in its first half and its odd ones in the second
                // (position 64h + p), so that each thread stores its 64 outputs with 128-bit stores; element-wise
                // stores along a row, with a warp's lanes on 32 different rows, would run into 4-way bank conflicts
                float4 *dst = reinterpret_cast<float4 *>(X + j * XS + H * h);
#pragma unroll
                for (int p4 = 0; p4 < H / 4; ++p4) dst[p4] = make_float4(out[4 * p4], out[4 * p4 + 1], out[4 * p4 + 2], out[4 * p4 + 3]);
            }
            __syncthreads();
        }

        // ---- exact top-k ---------------------------------------------------------------------------
        // thread tid scans one half of row tid/2 as the row pass stored it: the even coefficients (tid even) or the
        // odd ones (tid odd); element e of its half is coefficient 2e + (tid & 1), flat index 128*(tid/2) + 2e + (tid&1).
        // Fast path (k_eff <= 256): the k_eff-th largest of the 256 per-thread maxima is a lower bound L of
        // the k_eff-th largest coefficient (256 groups: the bound is tight, a few dozen candidates); the
        // candidates are listed in index order and searched by ballots, ties to the lowest index.  Everything
        // compares integer magnitude keys, so NaN and Inf are ordered like any other bit pattern.  More
        // than CAP128 candidates (tied or degenerate chunks) or k_eff > 256: radix select below.
        // the row-stage list is padded with zero-valued entries whose "row" is a scratch line, the then unused histogram
        // (ordered before the record writes by the barriers below)
        constexpr int PAD_ROW = (int)(compress128_tile_bytes<GT>() / sizeof(float));
        if (tid < RECS128) recs4[tid] = make_int4(PAD_ROW, 0, 0, 0);
        bool use_radix = k_eff > 256;
        if (!use_radix) {
            const float4 *mine4 = reinterpret_cast<const float4 *>(X + (tid >> 1) * XS + 64 * (tid & 1));
            const int lane = tid & 31, warp = tid >> 5;
            // the two halves of a row sit 256 bytes apart (same banks): the odd one starts 4 pieces later
            const int rot = 4 * (tid & 1);
            // the 64 values stay in registers for the candidate mask (group i4 holds piece (i4 + rot) mod 16)
            float v[64];
            float tm = 0.f;
#pragma unroll
            for (int i4 = 0; i4 < 16; ++i4) {
                const float4 f = mine4[(i4 + rot) & 15];
                v[4 * i4 + 0] = f.x;
                v[4 * i4 + 1] = f.y;
                v[4 * i4 + 2] = f.z;
                v[4 * i4 + 3] = f.w;
                tm = max3f(tm, fabsf(f.x), fabsf(f.y));
                tm = max3f(tm, fabsf(f.z), fabsf(f.w));
            }
            const unsigned tkey = __float_as_uint(tm);
            hist[tid] = tkey;
            __syncthreads();
            if (warp == 0) {
                unsigned k8[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) k8[i] = hist[lane + 32 * i];
                unsigned lo = k8[0], hi = k8[0];
#pragma unroll
                for (int i = 1; i < 8; ++i) {
                    lo = min(lo, k8[i]);
                    hi = max(hi, k8[i]);
                }
                lo = __reduce_min_sync(0xffffffffu, lo);
                hi = __reduce_max_sync(0xffffffffu, hi);
                const int b0 = 31 - __clz((lo ^ hi) | 0x8000u);  // >= 15
                unsigned prefix = lo & ~((2u << b0) - 1u);
#pragma unroll 1
                for (int b = b0; b >= 15; --b) {
                    const unsigned cand = prefix | (1u << b);
                    unsigned cnt = 0;
#pragma unroll
                    for (int i = 0; i < 8; ++i) cnt += __popc(__ballot_sync(0xffffffffu, k8[i] >= cand));
                    prefix = (cnt >= (unsigned)k_eff) ? cand : prefix;
                }
                if (lane == 0) {
                    s_state[2] = prefix;
                    s_state[3] = hi;  // largest magnitude key of the chunk (read before the scan below reuses the word)
                }
            }
            __syncthreads();
            const unsigned lmin = s_state[2];
            // every coefficient zero (a tile that no gradient has touched yet): no selection needed, the tie
            // rule gives the records 0 .. k_eff-1 with value 0
            const bool zero_chunk = s_state[3] == 0u;
            if (zero_chunk) {
                if (tid < k_eff) {
                    DemoRecord r;
                    r.idx = tid;
                    r.val = 0.f;
                    rec[tid] = r;
                    if (k_eff <= 128) recs4[tid] = make_int4((tid >> 7) * XS, (tid & 127) * S, 0, 0);
                }
            } else {
            // candidates of this thread as a bit mask over its 64 values: |q| >= L  <=>  |q| > Lm (the float just
            // below L); the sign bit of Lm - |q| is funnel-shifted into the mask (independent chains of 16), which is
            // then turned from register order into index order
            unsigned long long mask;
            {
                const float Lm = (lmin > 0u) ? __uint_as_float(lmin - 1u) : -1.f;
                unsigned mc[4];
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {
                    unsigned mm = 0u;
#pragma unroll
                    for (int q = 15; q >= 0; --q) mm = __funnelshift_l(__float_as_uint(Lm - fabsf(v[16 * ch + q])), mm, 1);
                    mc[ch] = mm;
                }
                const unsigned long long mreg =
                    ((unsigned long long)(mc[2] | (mc[3] << 16)) << 32) | (unsigned long long)(mc[0] | (mc[1] << 16));
                mask = (tid & 1) ? ((mreg << 16) | (mreg >> 48)) : mreg;
            }
            const unsigned cnt = (unsigned)__popcll(mask);
            const unsigned inc = warp_inclusive_scan(cnt, lane);
            if (lane == 31) warp_tot[warp] = inc;
            __syncthreads();
            unsigned o = inc - cnt, n_cand = 0;
#pragma unroll
            for (int w = 0; w < THREADS / 32; ++w) {
                const unsigned n = warp_tot[w];
                o += w < warp ? n : 0u;
                n_cand += n;
            }
            use_radix = n_cand > (unsigned)CAP128 || n_cand < (unsigned)k_eff;
            if (!use_radix) {
                // The list is in index order: inside a row the candidates of the even-coefficient thread (lane 2r)
                // and of the odd-coefficient thread (lane 2r+1) interleave, so a candidate's place is the row's base
                // plus the candidates of both threads with a smaller coefficient index.
                const unsigned plo = __shfl_xor_sync(0xffffffffu, (unsigned)mask, 1);
                const unsigned phi = __shfl_xor_sync(0xffffffffu, (unsigned)(mask >> 32), 1);
                const unsigned long long pmask = ((unsigned long long)phi << 32) | plo;
                const int odd = tid & 1;
                const unsigned row_base = odd ? o - (unsigned)__popcll(pmask) : o;
                const float *mine = reinterpret_cast<const float *>(mine4);
                unsigned long long left = mask;
                while (left) {
                    const int e = __ffsll((long long)left) - 1;
                    left &= left - 1ull;
                    const unsigned long long below = (1ull << e) - 1ull;
                    // partner coefficients before 2e + odd: 2e' + (1 - odd) with e' < e (even thread) or e' <= e (odd thread)
                    const unsigned long long pbelow = odd ? ((below << 1) | 1ull) : below;
                    const unsigned at = row_base + (unsigned)__popcll(mask & below) + (unsigned)__popcll(pmask & pbelow);
                    const float val = mine[e];
                    cand_key[at] = mag_key(val);
                    cand_val[at] = val;
                    cand_idx[at] = S * (tid >> 1) + 2 * e + odd;
                }
                __syncthreads();
                // the first warp picks the k_eff largest candidates (list order = index order) and writes the records; the
                // others clear the tile for the row stage
                if (warp != 0) {
                    for (int i = tid - 32; i < S * XS / 4; i += THREADS - 32)
                        reinterpret_cast<float4 *>(X)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
                    auto emit = [&](unsigned pos, unsigned li) {
                        DemoRecord r;
                        r.idx = cand_idx[li];
                        r.val = cand_val[li];
                        rec[pos] = r;
                        if (k_eff <= 128)
                            recs4[pos] = make_int4((r.idx >> 7) * XS, (r.idx & 127) * S, __float_as_int(a.alpha * r.val), 0);
                    };
                    auto key_of = [&](unsigned i) { return cand_key[i]; };
                    if (n_cand <= 64u)
                        warp_ballot_select<2>(key_of, n_cand, lmin, k_eff, lane, emit);
                    else
                        warp_ballot_select<8>(key_of, n_cand, lmin, k_eff, lane, emit);
                }
            }
            }  // !zero_chunk
        }
        // ---- radix select on the magnitude bits, then index-ordered compaction -----------------------
        if (use_radix) {
            unsigned thr, need_eq;
            if (tid == 0) {
                s_state[0] = 0u;
                s_state[1] = (unsigned)k_eff;
            }
            // this path works on rows in natural order: every thread turns its half row back (coefficient 2e + (tid&1)
            // from position 64*(tid&1) + e to position 2e + (tid&1)); then thread tid scans the half row
            // [tid/2][64*(tid&1) .. +64): flat indices 64*tid .. 64*tid+63
            {
                float *rowp = X + (tid >> 1) * XS;
                float tmp[64];
#pragma unroll
                for (int i4 = 0; i4 < 16; ++i4) {
                    const float4 f = reinterpret_cast<const float4 *>(rowp + 64 * (tid & 1))[i4];
                    tmp[4 * i4 + 0] = f.x;
                    tmp[4 * i4 + 1] = f.y;
                    tmp[4 * i4 + 2] = f.z;
                    tmp[4 * i4 + 3] = f.w;
                }
                __syncthreads();
#pragma unroll
                for (int e = 0; e < 64; ++e) rowp[2 * e + (tid & 1)] = tmp[e];
                __syncthreads();
            }
            const float *mine = X + (tid >> 1) * XS + 64 * (tid & 1);
#pragma unroll 1
            for (int pass = 0; pass < 4; ++pass) {
                const int shift = 24 - 8 * pass;
                const unsigned mask = (pass == 0) ? 0u : (0xffffffffu << (shift + 8));
                hist[tid] = 0u;
                __syncthreads();
                const unsigned prefix = s_state[0];
#pragma unroll 4
                for (int e = 0; e < 64; ++e) {
                    const unsigned key = mag_key(mine[e]);
                    if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
                }
                __syncthreads();
                if (tid < 32) {
                    const unsigned rem = s_state[1];
                    unsigned local = 0;
#pragma unroll
                    for (int b = 0; b < 8; ++b) local += hist[255 - 8 * tid - b];
                    const unsigned inc = warp_inclusive_scan(local, tid);
                    const unsigned before = inc - local;
                    if (before < rem && rem <= inc) {
                        unsigned cum = before;
                        int b = 255 - 8 * tid;
                        for (int q = 0; q < 8; ++q, --b) {
                            const unsigned hh = hist[b];
                            if (cum + hh >= rem) break;
                            cum += hh;
                        }
                        s_state[1] = rem - cum;
                        s_state[0] = prefix | ((unsigned)b << shift);
                    }
                }
                __syncthreads();
            }
            thr = s_state[0];
            need_eq = s_state[1];
            unsigned gt = 0, eq = 0;
#pragma unroll 4
            for (int e = 0; e < 64; ++e) {
                const unsigned key = mag_key(mine[e]);
                gt += key > thr;
                eq += key == thr;
            }
            const unsigned before = block_exclusive_scan(gt | (eq << 16), warp_tot);
            unsigned gb = before & 0xffffu, eb = before >> 16;
#pragma unroll 1
            for (int e = 0; e < 64; ++e) {
                const float val = mine[e];
                const unsigned key = mag_key(val);
                bool sel = false;
                unsigned pos = 0;
                if (key > thr) {
                    pos = gb + min(eb, need_eq);
                    ++gb;
                    sel = true;
                } else if (key == thr) {
                    if (eb < need_eq) {
                        pos = gb + eb;
                        sel = true;
                    }
                    ++eb;
                }
                if (sel) {
                    const int idx = 64 * tid + e;
                    DemoRecord r;
                    r.idx = idx;
                    r.val = val;
                    rec[pos] = r;
                    if (k_eff <= 128)
                        recs4[pos] = make_int4((idx >> 7) * XS, (idx & 127) * S, __float_as_int(a.alpha * val), 0);
                }
            }
        }
        __syncthreads();  // records complete; the coefficient tile is dead or, without the radix select, already cleared
        if (use_radix) {
            for (int i = tid; i < S * XS / 4; i += THREADS) reinterpret_cast<float4 *>(X)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();
        }

        // ---- residual: sparse row stage T[u][j] = sum over kept (u, v) of val * C[v][j] ------------
        if (k_eff <= 128) {
            // the two halves of the CTA take half of the list each, cut where a row ends
            int cut = k_eff / 2;
            while (cut > 0 && cut < k_eff && recs4[cut].x == recs4[cut - 1].x) ++cut;
            const int r_begin = h ? cut : 0, r_end = h ? k_eff : cut;
            // The running sum of a row is stored after every entry (the last store of a row carries the whole sum)
            // and starts again from zero when the next entry belongs to another row: no branch in the loop.
            // The cosines of a whole batch of entries are requested before the dependent accumulation starts: the
            // 64 KB basis does not stay in what the two CTAs' shared memory leaves of the L1, so most of these
            // loads go to L2 and a batch should pay that latency once.
            float *Xj = X + j;
            float acc = 0.f;
            auto row_stage = [&](auto batch_tag) {
                constexpr int BATCH = decltype(batch_tag)::value;
#pragma unroll 1
                for (int r0 = r_begin; r0 < r_end; r0 += BATCH) {
                    float cv[BATCH];
#pragma unroll
                    for (int q = 0; q < BATCH; ++q) cv[q] = __ldg(a.C + (unsigned)(recs4[r0 + q].y + j));
                    int4 nx = recs4[r0];
#pragma unroll
                    for (int q = 0; q < BATCH; ++q) {
                        const int4 rc = nx;
                        nx = recs4[r0 + q + 1];
                        acc = fmaf(__int_as_float(rc.z), cv[q], acc);
                        Xj[r0 + q < r_end ? rc.x : PAD_ROW] = acc;
                        acc = (rc.x != nx.x) ? 0.f : acc;
                    }
                }
            };
            if (k_eff <= ROW_AHEAD128)
                row_stage(std::integral_constant<int, ROW_AHEAD128>{});
            else
                row_stage(std::integral_constant<int, 3 * ROW_AHEAD128>{});
        } else if (h == 0) {
            // k > 128: the records come from the payload itself
            const float *Cj = a.C + j;
            float acc = 0.f;
            int cur_u = -1;
            for (int r = 0; r < k_eff; ++r) {
                const DemoRecord rc = rec[r];
                const int uo = (rc.idx >> 7) * XS;
                if (uo != cur_u) {
                    if (cur_u >= 0) X[cur_u + j] = acc;
                    acc = 0.f;
                    cur_u = uo;
                }
                acc = fmaf(a.alpha * rc.val, __ldg(Cj + (rc.idx & 127) * S), acc);
            }
            if (cur_u >= 0) X[cur_u + j] = acc;
        }
        __syncthreads();

        // ---- column stage of the inverse (split), residual --------------
#pragma unroll
        for (int p = 0; p < H; ++p) in[p] = X[(2 * p + h) * XS + j];
        fence_proxy_async();
        __syncthreads();  // T is in registers: the tile area is free
        float keep[H / 2], lo[H / 2], hi[H / 2];
        inverse_half(h, in, keep, lo);
        // exchange halves of e and o through the tile area
        float *Ex = X + j;  // [2][32][128]
#pragma unroll
        for (int q = 0; q < H / 2; ++q) Ex[(h * (H / 2) + q) * S] = lo[q];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < H / 2; ++q) hi[q] = Ex[((h ^ 1) * (H / 2) + q) * S];
        inverse_join(h, keep, lo, hi);
        __syncthreads();  // the exchange area is read: the new momentum tile takes its place
        // m <- B - alpha * IDCT(kept): B comes back from tensor memory; the dense tile goes out in one TMA store
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        {
            float b[32];
            tmem_ld32(taddr + 32 * h, b);
            float *Mlo = Ms + (H / 2) * h * S + j, *Mhi = Ms + (S - 1 - (H / 2) * h) * S + j;
#pragma unroll
            for (int q = 0; q < 32; ++q) Mlo[q * S] = b[q] - lo[q];
            tmem_ld32(taddr + H + 32 * h, b);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");  // (the next chunk's stores: behind barriers)
#pragma unroll
            for (int q = 0; q < 32; ++q) Mhi[-q * S] = b[q] - hi[q];
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
            const unsigned ticket = ticket_draw(a.tickets);  // the chunk after the next: drawn behind the store's wait
            tma_store_2d(static_cast<const char *>(a.tmap_m) + (size_t)te.tensor * TMAP_BYTES, (int)(k1 * S), (int)(k0 * S),
                         smem_u32(Ms));
            tma_store_commit();
            tma_store_wait_read();  // the store has read the tile: the next chunk's m tile may land
            if (nc < a.n_chunks) issue_tile(cur.te, nc, false, false);
            tmem_slot[1] = ticket;
        }
    }
    if (tid == 0) ticket_finish(a.tickets);
    tmem_free_cta(tmem_base, TMEM_COLS128);
}

// Decode: the tile, the walk, two staging buffers of records, and the landing area of the upper half of the x tile (before
// that, of the sender counts of the count-normalised mean).
constexpr size_t DECODE128_SMEM = (size_t)S * XSD * 4 + 128 + 2 * STAGE_RECORDS * sizeof(DemoRecord) + M / 2 * sizeof(float);

// SIGNS: the parameter-server form -- sign(R) goes out as int8, the parameters are not touched.
// STAGED: records are staged a chunk ahead and every warp adds those of its 16 rows, worker after worker; otherwise they
// come straight from the payloads with a barrier per worker, ROUND for lists that one round of the threads covers, ROUNDS for longer
// ones (in one instantiation the loop of the longer lists cost signs 4 %).
// The upper half of the x tile comes in behind the scatter and the transforms, the lower half, already in L2, into the dead
// coefficient tile while the upper one is updated; by 16-byte asynchronous copies, without tensor maps (kernels_fast.cu).
// COUNTS: the count-normalised mean (an instantiation of its own, as at s = 32 / 64, where the code for it cost the sum up to 12 %).
enum { STAGED, ROUND, ROUNDS };
template <bool SIGNS, int KMODE, bool COUNTS>
__global__ void __launch_bounds__(THREADS, 2) decode_fast128_kernel(DemoDecodeArgs a)
{
    const StreamOrder order(a.wait_first);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *St = reinterpret_cast<float *>(smem_raw);  // [128*129] aggregate / intermediate; later rows 64.. of x [64*128]
    DecodeWalk &walk = *reinterpret_cast<DecodeWalk *>(St + S * XSD);
    DemoRecord *stage_all = reinterpret_cast<DemoRecord *>(reinterpret_cast<unsigned char *>(&walk) + 128);  // [2][STAGE_RECORDS]
    float *Xh = reinterpret_cast<float *>(stage_all + 2 * STAGE_RECORDS);  // [64*128] rows ..63 of x
    unsigned short *Cn = reinterpret_cast<unsigned short *>(Xh);           // [M] senders per coordinate (agg == 2)
    __shared__ unsigned drawn[2];

    const int tid = threadIdx.x, h = tid >> 7, j = tid & 127, lane = tid & 31, warp = tid >> 5;
    const int k_eff = a.k;
    const unsigned n_chunks = (unsigned)a.n_chunks;  // (fewer than 2^31)
    const unsigned lr_bits = __float_as_uint(a.lr);
    const float decay = 1.f - a.lr * a.wd;
    const float neg_lr_scale = -a.lr * a.agg_scale;

    // the records of workers w_first .. of the chunk in walk slot `which`; one copy group per call
    auto stage_batch = [&](int buf, int which, int w_first) {
        const long long off = walk.rec[which];
        const int sh = stage_shift(k_eff);
        DemoRecord *dst = stage_all + buf * STAGE_RECORDS;
#pragma unroll
        for (int i = 0; i < STAGE_RECORDS / THREADS; ++i) {
            const int r = i * THREADS + tid, wl = w_first + (r >> sh), q = r & ((1 << sh) - 1);
            if (wl < a.W && q < k_eff)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst + r)), "l"(a.payloads[wl] + off + q)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    unsigned c = blockIdx.x, par = 0;
    int buf = 0, which = 0;  // staging buffer and walk slot of the current chunk
    if (tid == 0 && c < n_chunks) {
        walk.e = demo_find_entry(a.entries, a.n_entries, c);
        walk.load(a.entries, a.n_entries);
        walk.seek<S>(a.entries, a.n_entries, c, k_eff, 0);
    }
    __syncthreads();
    if (!SIGNS && c < n_chunks && tid < 128) {  // half a row per thread of the rows that are fetched first on their way to L2
        const float *xr = a.x_ptrs[walk.tensor[0]] + walk.elem[0] + (size_t)(tid >> 1) * walk.n1[0] + (tid & 1) * 64;
        prefetch_l2(xr);
        prefetch_l2(xr + 32);
    }
    order.begin();
    if (tid == 0) drawn[0] = second_ticket(a.tickets, n_chunks);
    if (KMODE == STAGED && c < n_chunks) stage_batch(0, 0, 0);
    for (unsigned nc; c < n_chunks; c = nc, par ^= 1u, which ^= 1) {
        __syncthreads();  // (publishes the draw; the tile and the landing area are free)
        nc = gridDim.x + drawn[par];
        unsigned ticket = 0;
        if (tid == 0) {
            ticket = ticket_draw(a.tickets);
            if (nc < n_chunks) walk.seek<S>(a.entries, a.n_entries, nc, k_eff, which ^ 1);
        }
        // 64 rows of the x tile, one copy group
        auto fetch_rows = [&](float *dst, int row0) {
            const int n1 = walk.n1[which];
            const float *src = a.x_ptrs[walk.tensor[which]] + walk.elem[which] + (size_t)(row0 + warp) * n1 + lane * 4;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + (warp + 8 * i) * S + lane * 4)),
                             "l"(src + (size_t)(8 * i) * n1)
                             : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        if (!SIGNS) {
            if (!COUNTS) fetch_rows(Xh, 0);
            const float *xr = a.x_ptrs[walk.tensor[which]] + walk.elem[which] + (size_t)(64 + (tid >> 2)) * walk.n1[which] + (tid & 3) * 32;
            prefetch_l2(xr);
        }
        for (int i = tid; i < S * XSD / 4; i += THREADS) reinterpret_cast<float4 *>(St)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (COUNTS)
            for (int i = tid; i < M / 2; i += THREADS) reinterpret_cast<unsigned *>(Cn)[i] = 0u;
        // S = sum over workers in worker order (Decompress&Aggregate)
        if constexpr (KMODE == STAGED) {
            const int sh = stage_shift(k_eff), wb = STAGE_RECORDS >> sh;
            for (int w0 = 0; w0 < a.W; w0 += wb) {
                // the records have landed (requested a chunk or a batch ago; only the rows of x are younger), the tile is cleared,
                // the next chunk looked up, and all warps are done with the other buffer
                if (!SIGNS && !COUNTS && w0 == 0)
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                else
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                __syncthreads();
                const DemoRecord *stage = stage_all + buf * STAGE_RECORDS;
                buf ^= 1;
                if (w0 + wb < a.W)
                    stage_batch(buf, which, w0 + wb);
                else if (nc < n_chunks)
                    stage_batch(buf, which ^ 1, 0);
                else
                    asm volatile("cp.async.commit_group;" ::: "memory");
                // branch-free as in kernels_fast.cu: a record of another warp's rows goes to a padding element
                const int spare = (16 * warp + (lane & 15)) * XSD + S;
                bool bad = false;
                const int n_pieces = min(wb, a.W - w0) << (sh - 5), last = (1 << (sh - 5)) - 1;  // 32 records each
#pragma unroll 1
                for (int q0 = 0; q0 < n_pieces; q0 += 4) {
                    DemoRecord rc[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) rc[u] = stage[((q0 + u) << 5 & (STAGE_RECORDS - 1)) + lane];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const bool have = q0 + u < n_pieces && lane < k_eff - (((q0 + u) & last) << 5);
                        const unsigned idx = (unsigned)rc[u].idx;
                        bad = bad || (have && idx >= (unsigned)M);
                        const bool mine = have && (idx >> 11) == (unsigned)warp;  // (false for idx >= M)
                        const int at = mine ? (int)(idx >> 7) * XSD + (int)(idx & 127) : spare;
                        St[at] += rc[u].val;
                        if (COUNTS && mine) Cn[idx] += 1;
                        __syncwarp();
                    }
                }
                if (bad) atomicMax(a.status, DEMO_DEV_PAYLOAD);
            }
        } else {
            __syncthreads();
            add_from_payloads<THREADS, KMODE == ROUND>(
                a.payloads, a.W, walk.rec[which], k_eff, tid,
                [&](const DemoRecord &rc) {
                    if ((unsigned)rc.idx < (unsigned)M) {
                        St[(rc.idx >> 7) * XSD + (rc.idx & 127)] += rc.val;
                        if (COUNTS) Cn[rc.idx] += 1;
                    } else {
                        atomicMax(a.status, DEMO_DEV_PAYLOAD);
                    }
                },
                [] { __syncthreads(); });
        }
        if (tid == 0) drawn[par ^ 1u] = ticket + tickets_from(n_chunks);
        __syncthreads();
        if constexpr (COUNTS) {  // Sparse Top-k Averaging: sum / number of senders, 0/0 = 0
            for (int i = tid; i < M; i += THREADS) {
                const unsigned short n = Cn[i];
                if (n > 1) St[(i >> 7) * XSD + (i & 127)] /= (float)n;
            }
            __syncthreads();
            if (!SIGNS) fetch_rows(Xh, 0);
        }
        // two inverse passes (rolled): both walk "row j" of the tile with unit stride -- pass 0 leaves its result
        // transposed, so that the columns pass 1 needs are rows again and every access below has a fixed offset
        float lo[H / 2], hi[H / 2];
        float *ln = St + j * XSD;  // line j
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            float in[H], keep[H / 2];
#pragma unroll
            for (int p = 0; p < H; ++p) in[p] = ln[2 * p + h];
            __syncthreads();  // every coefficient of the tile has been read
            inverse_half(h, in, keep, lo);
            // exchange halves of e / o inside the line
            float *mine = ln + (H / 2) * h, *theirs = ln + (H / 2) * (h ^ 1);
#pragma unroll
            for (int q = 0; q < H / 2; ++q) mine[q] = lo[q];
            __syncthreads();
#pragma unroll
            for (int q = 0; q < H / 2; ++q) hi[q] = theirs[q];
            inverse_join(h, keep, lo, hi);  // elements 32h + q and 127 - 32h - q
            __syncthreads();  // both halves of every line have read their partner's values
            if (pass == 0) {
                // element n of row j goes to row n, column j
                float *Slo = St + (H / 2) * h * XSD + j, *Shi = St + (S - 1 - (H / 2) * h) * XSD + j;
#pragma unroll
                for (int q = 0; q < H / 2; ++q) {
                    Slo[q * XSD] = lo[q];
                    Shi[-q * XSD] = hi[q];
                }
                __syncthreads();
            }
        }
        // thread (h, j) holds rows 32h + q and 127 - 32h - q of column j
        const ptrdiff_t n1 = walk.n1[which];
        const size_t at_lo = walk.elem[which] + (size_t)((H / 2) * h) * n1 + j, at_hi = walk.elem[which] + (size_t)(S - 1 - (H / 2) * h) * n1 + j;
        if constexpr (SIGNS) {
            signed char *__restrict__ slo = a.sign_ptrs[walk.tensor[which]] + at_lo, *__restrict__ shi = a.sign_ptrs[walk.tensor[which]] + at_hi;
#pragma unroll
            for (int q = 0; q < H / 2; ++q) {
                slo[q * n1] = (signed char)((lo[q] > 0.f) - (lo[q] < 0.f));
                shi[-q * n1] = (signed char)((hi[q] > 0.f) - (hi[q] < 0.f));
            }
            continue;
        }
        fetch_rows(St, 64);
        auto updated = [&](float rv, float xv) {
            float stepv = __uint_as_float(lr_bits ^ (~__float_as_uint(rv) & 0x80000000u));
            stepv = (rv == 0.f) ? 0.f : stepv;
            if (a.phi) stepv = rv * neg_lr_scale;  // phi = identity
            return fmaf(xv, decay, stepv);
        };
        float *__restrict__ xlo = a.x_ptrs[walk.tensor[which]] + at_lo, *__restrict__ xhi = a.x_ptrs[walk.tensor[which]] + at_hi;
        asm volatile("cp.async.wait_group 1;" ::: "memory");  // all but the lower rows
        __syncthreads();
        const float *Xlo = Xh + (H / 2) * h * S + j;
#pragma unroll
        for (int q = 0; q < H / 2; ++q) xlo[q * n1] = updated(lo[q], Xlo[q * S]);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const float *Xhi = St + (63 - (H / 2) * h) * S + j;
#pragma unroll
        for (int q = 0; q < H / 2; ++q) xhi[-q * n1] = updated(hi[q], Xhi[-q * S]);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // no copy may outlive the CTA's shared memory
    if (tid == 0) ticket_finish(a.tickets);
}

template <typename K, typename A>
cudaError_t launch128(K kernel, size_t smem, DemoLaunch &dev, cudaStream_t stream, A args)
{
    const long long n_chunks = args.n_chunks;
    if (n_chunks <= 0) return cudaSuccess;
    const cudaError_t err = demo_allow_smem(dev, (const void *)kernel);
    if (err != cudaSuccess) return err;
    // CTAs per SM: two by the launch bounds (registers), fewer if shared memory (227 KB, 1 KB reserved per CTA) says
    // so.  The occupancy calculator is not asked: it answers 1 for a kernel that allocates tensor memory.
    int per_sm = (int)((227u * 1024u) / (smem + 1024u));
    if (per_sm > 2) per_sm = 2;
    if (per_sm < 1) per_sm = 1;
    long long grid = (long long)dev.sm_count * per_sm;
    if (grid > n_chunks) grid = n_chunks;
    if (grid == n_chunks) args.tickets = nullptr;
    void *params[] = {&args};
    return demo_launch_kernel((const void *)kernel, grid, THREADS, smem, stream, params);
}

}  // namespace

cudaError_t demo_launch_compress_fast128(const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    if (!a.tmap_m || !a.tmap_g) return cudaErrorNotSupported;
    if (a.grad_bf16)
        return launch128(compress_fast128_kernel<__nv_bfloat16>, compress128_smem<__nv_bfloat16>(), dev, stream, a);
    return launch128(compress_fast128_kernel<float>, compress128_smem<float>(), dev, stream, a);
}

cudaError_t demo_launch_decode_fast128(const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    // Staged while the additions are short (k <= 64), and one worker's up to k = 128 in the update form; a further batch of longer lists
    // comes too late.  8192 x 8192, staged / with barriers: k = 32, W = 1 139 / 149 us, W = 8 145 / 169 us, k = 64, W = 8
    // 156 / 164, k = 128, W = 1 139 / 149, W = 8 182 / 165 us; 4096 x 4096, k = 32, W = 64 62 / 103 us, k = 65 .. 128, W = 1
    // 37.3 / 38.1, W = 4 42 / 39, signs W = 1 33.2 / 32.5, W = 4 37.4 / 32.7.
    const bool staged = a.k <= 64 || (a.k <= 128 && a.W == 1 && !a.sign_ptrs);
    auto pick = [&](auto signs, auto counts) {
        constexpr bool SIGNS = decltype(signs)::value, COUNTS = decltype(counts)::value;
        if (staged) return launch128(decode_fast128_kernel<SIGNS, STAGED, COUNTS>, DECODE128_SMEM, dev, stream, a);
        if (a.k <= THREADS) return launch128(decode_fast128_kernel<SIGNS, ROUND, COUNTS>, DECODE128_SMEM, dev, stream, a);
        return launch128(decode_fast128_kernel<SIGNS, ROUNDS, COUNTS>, DECODE128_SMEM, dev, stream, a);
    };
    if (a.agg == 2) return a.sign_ptrs ? pick(std::true_type{}, std::true_type{}) : pick(std::false_type{}, std::true_type{});
    return a.sign_ptrs ? pick(std::true_type{}, std::false_type{}) : pick(std::false_type{}, std::false_type{});
}
