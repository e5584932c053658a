// Kernels for the small chunks: length-s segments of 1-D tensors (any s and basis; a thread per element) and s x s tiles with
// s in {8, 16} (s lanes per tile, 4 or 2 tiles per warp).  A launch takes both lists: the tensors of a small model are done in
// one launch per call, and the norm vectors of a large one beside its tiles.
//
// What bounds them is latency: a chunk holds 8 to 256 elements, so nothing is gained by more threads per chunk (the dense
// kernels, a 256-thread CTA per chunk with radix select and a barrier between all steps, spent 24 us on 2048 tiles of 8 x 8
// and 13 us on 1024 segments), and a warp needs (almost) no block barrier from the loads to the stores:
//   * segments: every thread forms one coefficient, a warp reading the basis by rows of its transpose (the sums run over n in order,
//     so the results are those of the dense kernels bit for bit); the k-th key by a bit-by-bit ballot search;
//   * tiles: lane j holds column j, then row j, in registers (fast_dct.cuh); the transposes go through a tile of the
//     warp's own shared memory; the k-th key by a bit-by-bit search with counts added up over the tile's lanes.
// Measured: 256 x 512 in 8 x 8 tiles plus a vector of 512, two compress calls and a decode: 60.7 -> 30.4 us (the tiles and
// the segments of a call were two launches on two streams).
#include <cuda_bf16.h>

#include <type_traits>

#include "demo_internal.h"
#include "fast_dct.cuh"
#include "launch.cuh"

namespace {

constexpr int THREADS = 128, WARPS = THREADS / 32;
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ unsigned mag_key(float v) { return __float_as_uint(v) & 0x7fffffffu; }

// (warp) the tensor that owns chunk id c.
__device__ __forceinline__ int find_entry_warp(const DemoTensorEntry *entries, int n, long long c)
{
    return demo_find_warp(0, n, [&](int i) { return entries[i].chunk_begin <= c; });
}

// ---- segments -------------------------------------------------------------------------------------------
// Thread i of a segment holds element i: a warp for s <= 32 (lanes above s idle), two for s = 64, a block for s = 128.  Where a
// segment has several warps, each holds all keys (E per lane) and searches for itself; three barriers order the exchange.
template <int S>
struct Seg {
    static constexpr int E = S < 32 ? 1 : S / 32;             // warps per segment = keys per lane
    static constexpr int PER_BLOCK = THREADS / (32 * E);
    static constexpr int PAD = S + 4;
    static __device__ __forceinline__ void sync()
    {
        if constexpr (E == 1)
            __syncwarp();
        else
            __syncthreads();
    }
};

// Elements of a row of the basis that a thread has under way together on the way forward: a launch of few segments is the latency of the
// table's lines.  (Not more at s = 64: with 64 elements a block's 80 registers per thread no longer fit beside the tiles' kernel where one of
// its CTAs has left.)
template <int S>
constexpr int BATCH = S == 128 ? 64 : S < 32 ? S : 32;
template <int B>
__device__ __forceinline__ void load_column(float (&t)[B], const float *__restrict__ at, int stride)
{
#pragma unroll
    for (int u = 0; u < B; ++u) t[u] = __ldg(at + u * stride);
}
// sum_u C[u][i] line[u], u in order.  AHEAD: 64 elements under way together (s = 128).
template <int S, bool AHEAD>
__device__ __forceinline__ float inverse_segment(const float *line, const float *__restrict__ C, int i)
{
    float r = 0.f;
    if constexpr (AHEAD) {
#pragma unroll 1
        for (int u0 = 0; u0 < S; u0 += 64) {
            float t[64];
            load_column(t, C + u0 * S + i, S);
#pragma unroll
            for (int u = 0; u < 64; ++u) r = fmaf(line[u0 + u], t[u], r);
        }
    } else {
#pragma unroll 16
        for (int u = 0; u < S; ++u) r = fmaf(line[u], __ldg(C + u * S + i), r);
    }
    return r;
}

// A warp's first round looks its chunk up and prefetches it in front of the line that StreamOrder draws (launch.cuh).
struct FirstRound {
    const StreamOrder &order;
    bool left;
    __device__ __forceinline__ void begin()
    {
        if (left) order.begin();
        left = false;
    }
};

template <int S, bool AHEAD>
__device__ __forceinline__ void compress_segment(const DemoCompressArgs &a, long long c_own, float *line, FirstRound &first)
{
    constexpr int E = Seg<S>::E;
    const int lane = threadIdx.x & 31, i = threadIdx.x % (32 * E);  // (i >= s only for s < 32)
    const bool valid = c_own < a.n_chunks, on = i < S && valid;
    const long long c = valid ? c_own : a.n_chunks - 1;
    const DemoTensorEntry te = a.entries[find_entry_warp(a.entries, a.n_entries, c)];
    const long long lc = c - te.chunk_begin;
    const size_t off = (size_t)lc * S + i;
    float *__restrict__ m = a.m_ptrs[te.tensor];
    const void *g = a.g_ptrs[te.tensor];
    const int k = te.k_eff;
    if (first.left && on) {
        prefetch_l2(m + off);
        prefetch_l2(static_cast<const char *>(g) + off * (a.grad_bf16 ? 2 : 4));
    }
    first.begin();

    // row i of the basis, as a column of the transposed table (a warp reads 128 consecutive bytes; from the rows, 32 lines per read, sets with
    // many segments of 128 took up to a third longer: 296 tiles of 128 x 128 and a vector of 37888, compress 43.4 us instead of 32.8), the
    // first batch on its way beside the tensors' elements (32 elements at a time, none ahead: one segment of 128 10.8 us a call, now 5.2; from the
    // rows 8.2; of 64 1 / 5000 segments 4.6 / 14.8, 3.6 / 13.3, 5.2 / 37.8)
    const float *Ct = a.C + S * S + (i < S ? i : 0);
    float t[BATCH<S>];
    if constexpr (AHEAD) load_column(t, Ct, S);

    // momentum update  b = beta*m + g  (Algorithm 1, worker side)
    float b = 0.f, q = 0.f;
    if (on) {
        const float gv = a.grad_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16 *>(g)[off]) : static_cast<const float *>(g)[off];
        b = fmaf(a.beta, m[off], gv);
    }
    if (i < S) line[i] = b;
    Seg<S>::sync();
    // q = C b
    if (i < S) {
        if constexpr (AHEAD) {
            constexpr int B = BATCH<S>;
#pragma unroll
            for (int n0 = 0; n0 < S; n0 += B) {
#pragma unroll
                for (int n = 0; n < B; n += 4) {
                    const float4 x = *reinterpret_cast<const float4 *>(line + n0 + n);
                    q = fmaf(x.x, t[n], q);
                    q = fmaf(x.y, t[n + 1], q);
                    q = fmaf(x.z, t[n + 2], q);
                    q = fmaf(x.w, t[n + 3], q);
                }
                if (n0 + B < S) load_column(t, Ct + (n0 + B) * S, S);
            }
        } else {
#pragma unroll 8
            for (int n = 0; n < S; n += 4) {
                const float4 x = *reinterpret_cast<const float4 *>(line + n);
                q = fmaf(x.x, __ldg(Ct + n * S), q);
                q = fmaf(x.y, __ldg(Ct + (n + 1) * S), q);
                q = fmaf(x.z, __ldg(Ct + (n + 2) * S), q);
                q = fmaf(x.w, __ldg(Ct + (n + 3) * S), q);
            }
        }
    }
    Seg<S>::sync();
    // exact top-k: threshold by ballots from the highest bit any key has; keys equal to it are kept in index order
    unsigned key[E], hi = 0u;
    if constexpr (E == 1) {
        key[0] = i < S ? mag_key(q) : 0u;
    } else {
        line[i] = q;
        Seg<S>::sync();
#pragma unroll
        for (int e = 0; e < E; ++e) key[e] = mag_key(line[lane + 32 * e]);
        Seg<S>::sync();
    }
#pragma unroll
    for (int e = 0; e < E; ++e) hi = max(hi, key[e]);
    unsigned thr = 0u;
    int need_eq = S;  // k = s: everything is kept
    if (k < S) {
        hi = __reduce_max_sync(FULL, hi);
        int n_ge = S;
#pragma unroll 1
        for (int bit = 31 - __clz(hi | 1u); bit >= 0 && n_ge != k; --bit) {
            const unsigned cand = thr | (1u << bit);
            int cnt = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) cnt += __popc(__ballot_sync(FULL, key[e] >= cand));
            if (cnt >= k) {
                thr = cand;
                n_ge = cnt;
            }
        }
        int n_gt = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) n_gt += __popc(__ballot_sync(FULL, key[e] > thr));
        need_eq = k - n_gt;
    }
    // this thread's own key is key[i / 32]: how many are kept, and equal, before it
    const unsigned lt = (1u << lane) - 1u;
    const unsigned own = mag_key(q);
    int gt = 0, eq = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const bool elem = lane + 32 * e < S;
        const unsigned gtb = __ballot_sync(FULL, elem && key[e] > thr), eqb = __ballot_sync(FULL, elem && key[e] == thr);
        const unsigned below = e < i / 32 ? FULL : (e == i / 32 ? lt : 0u);
        gt += __popc(gtb & below);
        eq += __popc(eqb & below);
    }
    const bool keep = i < S && (own > thr || (own == thr && eq < need_eq));
    if (keep && valid) {
        DemoRecord r;
        r.idx = i;
        r.val = q;
        a.payload[te.rec_begin + lc * (long long)k + gt + min(eq, need_eq)] = r;
    }
    if (i < S) line[i] = keep ? a.alpha * q : 0.f;
    Seg<S>::sync();
    // m <- b - alpha C^T (kept)
    if (on) m[off] = b - inverse_segment<S, S == 128 && AHEAD>(line, a.C, i);
    Seg<S>::sync();
}

template <int S, bool AHEAD>
__device__ __forceinline__ void decode_segment(const DemoDecodeArgs &a, long long c_own, float *line, unsigned short *senders, FirstRound &first)
{
    constexpr int E = Seg<S>::E;
    const int i = threadIdx.x % (32 * E);
    const bool counts = a.agg == 2;
    const bool valid = c_own < a.n_chunks, on = i < S && valid;
    const long long c = valid ? c_own : a.n_chunks - 1;
    const DemoTensorEntry te = a.entries[find_entry_warp(a.entries, a.n_entries, c)];
    const long long lc = c - te.chunk_begin;
    const size_t off = (size_t)lc * S + i;
    const int k = te.k_eff;
    const long long rec_off = te.rec_begin + lc * (long long)k + i;
    if (first.left && on && !a.sign_ptrs) prefetch_l2(a.x_ptrs[te.tensor] + off);
    first.begin();
    if (i < S) {
        line[i] = 0.f;
        if (counts) senders[i] = 0;
    }
    Seg<S>::sync();
    // sum over workers in worker order (a segment has at most as many records as threads); eight workers' records are
    // fetched together
    for (int w0 = 0; w0 < a.W; w0 += 8) {
        DemoRecord rc[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) rc[w] = (i < k && w0 + w < a.W) ? a.payloads[w0 + w][rec_off] : DemoRecord{-1, 0.f};
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (i < k && w0 + w < a.W) {
                if ((unsigned)rc[w].idx < (unsigned)S) {
                    line[rc[w].idx] += rc[w].val;
                    if (counts) senders[rc[w].idx] += 1;
                } else if (valid) {
                    atomicMax(a.status, DEMO_DEV_PAYLOAD);
                }
            }
            if (w0 + w < a.W) Seg<S>::sync();
        }
    }
    if (counts) {  // Sparse Top-k Averaging: sum / number of senders, 0/0 = 0
        if (i < S) {
            const unsigned short n = senders[i];
            if (n > 1) line[i] = line[i] / (float)n;
        }
        Seg<S>::sync();
    }
    if (on) {
        const float r = inverse_segment<S, AHEAD>(line, a.C, i);
        if (a.sign_ptrs) {
            a.sign_ptrs[te.tensor][off] = (signed char)((r > 0.f) - (r < 0.f));
        } else {
            float *__restrict__ x = a.x_ptrs[te.tensor];
            const float sg = a.phi ? r * a.agg_scale : (float)((r > 0.f) - (r < 0.f));
            const float xv = x[off];
            x[off] = fmaf(-a.lr, fmaf(a.wd, xv, sg), xv);
        }
    }
    Seg<S>::sync();
}

// ---- tiles of 8 x 8 and 16 x 16 ----------------------------------------------------------------------------
template <int S>
struct Tile {
    static constexpr int PER_WARP = 32 / S;
    static constexpr int XS = S + 1;  // row stride: a lane walks a row or a column without bank conflicts among its tile
    static constexpr int FLOATS = PER_WARP * S * XS + 32;  // tiles of a warp start a bank apart
};
template <int S>
__device__ __forceinline__ int segment_sum(int v)
{
#pragma unroll
    for (int d = 1; d < S; d <<= 1) v += __shfl_xor_sync(FULL, v, d);
    return v;
}
// Exclusive prefix sum over the lanes of a tile.
template <int S>
__device__ __forceinline__ int segment_before(int v, int j)
{
    int inc = v;
#pragma unroll
    for (int d = 1; d < S; d <<= 1) {
        const int n = __shfl_up_sync(FULL, inc, d, S);
        if (j >= d) inc += n;
    }
    return inc - v;
}
template <int S>
struct TileRef {
    DemoTensorEntry te;
    long long lc;
    size_t base;  // of this lane's column
};
template <int S>
__device__ __forceinline__ TileRef<S> tile_ref(const DemoTensorEntry *entries, int n, long long c, int j)
{
    TileRef<S> t;
    t.te = entries[demo_find_entry(entries, n, c)];
    t.lc = c - t.te.chunk_begin;
    const long long k0 = t.lc / t.te.c1;
    t.base = (size_t)k0 * S * (size_t)t.te.n1 + (size_t)(t.lc - k0 * t.te.c1) * S + j;
    return t;
}
// Row j of the kept coefficients in q -> column j of C^T Q C in q.
template <int S>
__device__ __forceinline__ void inverse_tile(float (&q)[S], float *X, int j)
{
    constexpr int XS = Tile<S>::XS;
    fdct::dct3_ortho_dense4<S>(q);
#pragma unroll
    for (int v = 0; v < S; ++v) X[j * XS + v] = q[v];
    __syncwarp();
#pragma unroll
    for (int u = 0; u < S; ++u) q[u] = X[u * XS + j];
    __syncwarp();
    fdct::dct3_ortho_dense4<S>(q);
}

template <int S, typename GT>
__device__ __forceinline__ void compress_tiles(const DemoCompressArgs &a, long long group, float *warp_mem, FirstRound &first)
{
    constexpr int XS = Tile<S>::XS, M = S * S;
    const int lane = threadIdx.x & 31, j = lane % S, sub = lane / S;
    float *X = warp_mem + sub * (S * XS + S);
    const long long c_own = group * Tile<S>::PER_WARP + sub;
    const bool on = c_own < a.n_chunks;
    const TileRef<S> t = tile_ref<S>(a.entries, a.n_entries, on ? c_own : a.n_chunks - 1, j);
    const int n1 = t.te.n1, k = t.te.k_eff;
    float *__restrict__ m = a.m_ptrs[t.te.tensor] + t.base;
    const GT *__restrict__ g = static_cast<const GT *>(a.g_ptrs[t.te.tensor]) + t.base;
    if (first.left) {  // row j
        prefetch_l2(m + (size_t)j * n1 - j);
        prefetch_l2(g + (size_t)j * n1 - j);
    }
    first.begin();

    // momentum update  B = beta*m + g, column j  (Algorithm 1, worker side)
    float B[S], q[S];
    {
        GT gv[S];
#pragma unroll
        for (int i = 0; i < S; ++i) {
            B[i] = m[(size_t)i * n1];
            gv[i] = g[(size_t)i * n1];
        }
#pragma unroll
        for (int i = 0; i < S; ++i) q[i] = B[i] = fmaf(a.beta, B[i], (float)gv[i]);
    }
    fdct::dct2_ortho_dense4<S>(q);
#pragma unroll
    for (int u = 0; u < S; ++u) X[u * XS + j] = q[u];
    __syncwarp();
#pragma unroll
    for (int v = 0; v < S; ++v) q[v] = X[j * XS + v];
    __syncwarp();
    fdct::dct2_ortho_dense4<S>(q);  // row j of Q

    // exact top-k: bit-by-bit search for a threshold with exactly k keys at or above it, all tiles of the warp together
    unsigned thr = 0u;
    int need_eq = M;  // k = M: everything is kept
    if (__any_sync(FULL, k < M)) {
        unsigned hi = 0u;
#pragma unroll
        for (int v = 0; v < S; ++v) hi = max(hi, mag_key(q[v]));
        hi = __reduce_max_sync(FULL, hi);
        int n_ge = M;
#pragma unroll 1
        for (int bit = 31 - __clz(hi | 1u); bit >= 0 && __any_sync(FULL, n_ge != k); --bit) {
            const unsigned cand = thr | (1u << bit);
            int cnt = 0;
#pragma unroll
            for (int v = 0; v < S; ++v) cnt += mag_key(q[v]) >= cand;
            cnt = segment_sum<S>(cnt);
            if (cnt >= k && n_ge != k) {
                thr = cand;
                n_ge = cnt;
            }
        }
        int n_gt = 0;
#pragma unroll
        for (int v = 0; v < S; ++v) n_gt += mag_key(q[v]) > thr;
        need_eq = k - segment_sum<S>(n_gt);
    }
    // records in ascending index order (row after row); equal keys in index order until k are reached
    int gt = 0, eq = 0;
#pragma unroll
    for (int v = 0; v < S; ++v) {
        gt += mag_key(q[v]) > thr;
        eq += mag_key(q[v]) == thr;
    }
    const int before = segment_before<S>(gt | eq << 16, j);
    gt = before & 0xffff;
    eq = before >> 16;
    DemoRecord *rec = a.payload + t.te.rec_begin + t.lc * (long long)k;
#pragma unroll
    for (int v = 0; v < S; ++v) {
        const unsigned key = mag_key(q[v]);
        const bool keep = key > thr || (key == thr && eq < need_eq);
        if (keep && on) {
            DemoRecord r;
            r.idx = j * S + v;
            r.val = q[v];
            rec[gt + min(eq, need_eq)] = r;
        }
        gt += key > thr;
        eq += key == thr;
        q[v] = keep ? a.alpha * q[v] : 0.f;
    }
    // m <- B - alpha * IDCT(kept)
    inverse_tile<S>(q, X, j);
    if (on) {
#pragma unroll
        for (int i = 0; i < S; ++i) m[(size_t)i * n1] = B[i] - q[i];
    }
}

template <int S>
__device__ __forceinline__ void decode_tiles(const DemoDecodeArgs &a, long long group, float *warp_mem, unsigned short *warp_counts, FirstRound &first)
{
    constexpr int XS = Tile<S>::XS, M = S * S;
    const int lane = threadIdx.x & 31, j = lane % S, sub = lane / S;
    float *X = warp_mem + sub * (S * XS + S);
    unsigned short *senders = warp_counts + sub * M;
    const bool counts = a.agg == 2;
    const long long c_own = group * Tile<S>::PER_WARP + sub;
    const bool on = c_own < a.n_chunks;
    const TileRef<S> t = tile_ref<S>(a.entries, a.n_entries, on ? c_own : a.n_chunks - 1, j);
    const int n1 = t.te.n1, k = t.te.k_eff;
    const long long rec_off = t.te.rec_begin + t.lc * (long long)k;
    if (first.left && !a.sign_ptrs) prefetch_l2(a.x_ptrs[t.te.tensor] + t.base + (size_t)j * n1 - j);
    first.begin();
#pragma unroll
    for (int v = 0; v < S; ++v) {
        X[j * XS + v] = 0.f;
        if (counts) senders[j * S + v] = 0;
    }
    __syncwarp();
    // sum over workers in worker order; the records of eight workers are fetched together, or, for k > S, eight rounds of
    // one worker's
    auto add = [&](DemoRecord r) {
        if ((unsigned)r.idx < (unsigned)M) {
            X[(r.idx / S) * XS + r.idx % S] += r.val;
            if (counts) senders[r.idx] += 1;
        } else if (on) {
            atomicMax(a.status, DEMO_DEV_PAYLOAD);
        }
    };
    if (__all_sync(FULL, k <= S)) {
        for (int w0 = 0; w0 < a.W; w0 += 8) {
            DemoRecord rc[8];
#pragma unroll
            for (int w = 0; w < 8; ++w) rc[w] = (j < k && w0 + w < a.W) ? a.payloads[w0 + w][rec_off + j] : DemoRecord{-1, 0.f};
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                if (j < k && w0 + w < a.W) add(rc[w]);
                __syncwarp();
            }
        }
    } else {
        for (int w = 0; w < a.W; ++w) {
            for (int r0 = 0; r0 < M; r0 += 8 * S) {  // (k <= M)
                DemoRecord rc[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int i = r0 + r * S + j;
                    rc[r] = i < k ? a.payloads[w][rec_off + i] : DemoRecord{-1, 0.f};
                }
#pragma unroll
                for (int r = 0; r < 8; ++r)
                    if (r0 + r * S + j < k) add(rc[r]);
            }
            __syncwarp();
        }
    }
    float q[S];
#pragma unroll
    for (int v = 0; v < S; ++v) {
        q[v] = X[j * XS + v];
        if (counts) {  // Sparse Top-k Averaging: sum / number of senders, 0/0 = 0
            const unsigned short n = senders[j * S + v];
            if (n > 1) q[v] = q[v] / (float)n;
        }
    }
    __syncwarp();
    inverse_tile<S>(q, X, j);
    if (!on) return;
    if (a.sign_ptrs) {  // parameter-server form: hand out sign(R), the workers apply it
        signed char *__restrict__ sg = a.sign_ptrs[t.te.tensor] + t.base;
#pragma unroll
        for (int i = 0; i < S; ++i) sg[(size_t)i * n1] = (signed char)((q[i] > 0.f) - (q[i] < 0.f));
        return;
    }
    // x <- x - lr * (phi(R) + wd * x), sign(0) = 0
    float *__restrict__ x = a.x_ptrs[t.te.tensor] + t.base;
    float xv[S];
#pragma unroll
    for (int i = 0; i < S; ++i) xv[i] = x[(size_t)i * n1];
#pragma unroll
    for (int i = 0; i < S; ++i) {
        const float sg = a.phi ? q[i] * a.agg_scale : (float)((q[i] > 0.f) - (q[i] < 0.f));
        x[(size_t)i * n1] = fmaf(-a.lr, fmaf(a.wd, xv[i], sg), xv[i]);
    }
}

// ---- kernels: blocks below `seg_blocks` walk the segments, the others the tiles (TILES only) ------------------
template <int S, bool TILES>
constexpr int warp_floats() { return TILES && Tile<S>::FLOATS > Seg<S>::PAD ? Tile<S>::FLOATS : Seg<S>::PAD; }

template <int S, typename GT, bool TILES, bool AHEAD>
__global__ void __launch_bounds__(THREADS) compress_small_kernel(DemoCompressArgs segs, DemoCompressArgs tiles, int seg_blocks)
{
    const StreamOrder order(segs.wait_first);
    FirstRound first{order, true};
    __shared__ __align__(16) float mem[WARPS][warp_floats<S, TILES>()];
    const int warp = threadIdx.x >> 5;
    if (!TILES || (int)blockIdx.x < seg_blocks) {
        // (all threads of a block make the same rounds: a segment beyond the last is computed and not stored)
        constexpr int PB = Seg<S>::PER_BLOCK;
        const int own = warp / Seg<S>::E;
        for (long long c0 = (long long)blockIdx.x * PB; c0 < segs.n_chunks; c0 += (long long)seg_blocks * PB)
            compress_segment<S, AHEAD>(segs, c0 + own, mem[own], first);
    } else if constexpr (TILES) {
        const long long groups = (tiles.n_chunks + Tile<S>::PER_WARP - 1) / Tile<S>::PER_WARP;
        const long long stride = (long long)(gridDim.x - seg_blocks) * WARPS;
        for (long long p = (long long)(blockIdx.x - seg_blocks) * WARPS + warp; p < groups; p += stride)
            compress_tiles<S, GT>(tiles, p, mem[warp], first);
    }
    first.begin();  // (a warp without a round)
}

template <int S, bool TILES, bool AHEAD>
__global__ void __launch_bounds__(THREADS) decode_small_kernel(DemoDecodeArgs segs, DemoDecodeArgs tiles, int seg_blocks)
{
    const StreamOrder order(segs.wait_first);
    FirstRound first{order, true};
    __shared__ __align__(16) float mem[WARPS][warp_floats<S, TILES>()];
    __shared__ unsigned short counts[WARPS][TILES ? Tile<S>::PER_WARP * S * S : S];
    const int warp = threadIdx.x >> 5;
    if (!TILES || (int)blockIdx.x < seg_blocks) {
        // (all threads of a block make the same rounds: a segment beyond the last is computed and not stored)
        constexpr int PB = Seg<S>::PER_BLOCK;
        const int own = warp / Seg<S>::E;
        for (long long c0 = (long long)blockIdx.x * PB; c0 < segs.n_chunks; c0 += (long long)seg_blocks * PB)
            decode_segment<S, AHEAD>(segs, c0 + own, mem[own], counts[own], first);
    } else if constexpr (TILES) {
        const long long groups = (tiles.n_chunks + Tile<S>::PER_WARP - 1) / Tile<S>::PER_WARP;
        const long long stride = (long long)(gridDim.x - seg_blocks) * WARPS;
        for (long long p = (long long)(blockIdx.x - seg_blocks) * WARPS + warp; p < groups; p += stride)
            decode_tiles<S>(tiles, p, mem[warp], counts[warp], first);
    }
    first.begin();
}

// Up to eight blocks per SM for each list (what 64 registers per thread allow).
int blocks_for(long long units, int per_block, int sm_count)
{
    const long long b = (units + per_block - 1) / per_block, cap = 8LL * sm_count;
    return (int)(b < cap ? b : cap);
}
template <class A>
cudaError_t launch(const void *kernel, int segs_per_block, int tiles_per_warp, const A *segs, const A *tiles, DemoLaunch &dev, cudaStream_t stream)
{
    A none{};
    const A &sa = segs ? *segs : none, &ta = tiles ? *tiles : none;
    int seg_blocks = segs ? blocks_for(sa.n_chunks, segs_per_block, dev.sm_count) : 0;
    const int tile_blocks = tiles ? blocks_for(ta.n_chunks, tiles_per_warp * WARPS, dev.sm_count) : 0;
    if (seg_blocks + tile_blocks == 0) return cudaSuccess;
    void *params[] = {const_cast<A *>(&sa), const_cast<A *>(&ta), &seg_blocks};
    return demo_launch_kernel(kernel, seg_blocks + tile_blocks, THREADS, 0, stream, params);
}

// At most two rounds of blocks.
template <int S>
bool few_rounds(long long n_segs, const DemoLaunch &dev)
{
    return n_segs <= 2LL * blocks_for(n_segs, Seg<S>::PER_BLOCK, dev.sm_count) * Seg<S>::PER_BLOCK;
}

template <int S>
cudaError_t compress_small(const DemoCompressArgs *segs, const DemoCompressArgs *tiles, DemoLaunch &dev, cudaStream_t stream)
{
    if constexpr (S <= 16) {
        if (tiles)
            return launch(tiles->grad_bf16 ? (const void *)compress_small_kernel<S, __nv_bfloat16, true, true>
                                           : (const void *)compress_small_kernel<S, float, true, true>,
                          Seg<S>::PER_BLOCK, Tile<S>::PER_WARP, segs, tiles, dev, stream);
    }
    // s = 128: a batch of 64 elements ahead up to two rounds of blocks; beyond, other segments cover the latency, and with half the registers
    // sixteen blocks of an SM instead of eight do (two calls and a decode, data not in L2, 4000 segments 101 us ahead, 92 not, 1000 28 / 29).
    if constexpr (S == 128)
        if (segs && !few_rounds<S>(segs->n_chunks, dev))
            return launch((const void *)compress_small_kernel<S, float, false, false>, Seg<S>::PER_BLOCK, 1, segs, (const DemoCompressArgs *)nullptr, dev, stream);
    return launch((const void *)compress_small_kernel<S, float, false, true>, Seg<S>::PER_BLOCK, 1, segs, (const DemoCompressArgs *)nullptr, dev, stream);
}
template <int S>
cudaError_t decode_small(const DemoDecodeArgs *segs, const DemoDecodeArgs *tiles, DemoLaunch &dev, cudaStream_t stream)
{
    if constexpr (S <= 16) {
        if (tiles)
            return launch((const void *)decode_small_kernel<S, true, false>, Seg<S>::PER_BLOCK, Tile<S>::PER_WARP, segs, tiles, dev, stream);
    }
    // s = 128, up to two rounds of blocks: the inverse reads 64 elements of the basis ahead, with 46 registers per thread; beyond, other segments
    // cover that latency, and with 32 registers the next kernel's blocks find room beside this one's (a decode call, ahead / not: one segment
    // 4.1 / 5.2 us, 600 5.2 / 5.7, 1200 7.5 / 8.3, 2400 13.4 / 11.8, 5000 24.9 / 21.5).  Nor beside tiles, which cover it too (804 tiles and 32
    // segments 44.9 / 44.2).
    if constexpr (S == 128)
        if (segs && segs->wait_first && few_rounds<S>(segs->n_chunks, dev))
            return launch((const void *)decode_small_kernel<S, false, true>, Seg<S>::PER_BLOCK, 1, segs, (const DemoDecodeArgs *)nullptr, dev, stream);
    return launch((const void *)decode_small_kernel<S, false, false>, Seg<S>::PER_BLOCK, 1, segs, (const DemoDecodeArgs *)nullptr, dev, stream);
}

}  // namespace

bool demo_small_tiles_supported(int s) { return s == 8 || s == 16; }

cudaError_t demo_launch_compress_small(int s, const DemoCompressArgs *segs, const DemoCompressArgs *tiles, DemoLaunch &dev,
                                       cudaStream_t stream)
{
    switch (s) {
        case 8: return compress_small<8>(segs, tiles, dev, stream);
        case 16: return compress_small<16>(segs, tiles, dev, stream);
        case 32: return compress_small<32>(segs, nullptr, dev, stream);
        case 64: return compress_small<64>(segs, nullptr, dev, stream);
        case 128: return compress_small<128>(segs, nullptr, dev, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t demo_launch_decode_small(int s, const DemoDecodeArgs *segs, const DemoDecodeArgs *tiles, DemoLaunch &dev,
                                     cudaStream_t stream)
{
    switch (s) {
        case 8: return decode_small<8>(segs, tiles, dev, stream);
        case 16: return decode_small<16>(segs, tiles, dev, stream);
        case 32: return decode_small<32>(segs, nullptr, dev, stream);
        case 64: return decode_small<64>(segs, nullptr, dev, stream);
        case 128: return decode_small<128>(segs, nullptr, dev, stream);
        default: return cudaErrorInvalidValue;
    }
}
