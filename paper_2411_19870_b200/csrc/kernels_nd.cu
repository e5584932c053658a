// Kernels for tensors of any order (up to DEMO_ND_DIMS axes) cut into rectangular chunks
// s_0 x ... x s_{d-1}: the general statement of the method in the paper's appendix ("Multilinear
// Transforms and Chunk-wise Tensor Blocking").  The chunk transform is the multilinear product
// T(B; C_0, ..., C_{d-1}) with the DCT matrix of dimension s_a on axis a, applied one axis after the
// other; chunk extents are run-time values.  One CTA works on one chunk at a time and keeps it in shared
// memory from the momentum update to the residual write-back, so HBM is touched once per operand.
//
// What bounds these kernels is instruction issue and latency, with barriers between the phases, so the work per element
// and the number of phases are what the design cuts:
//   * an axis is transformed line by line, in place, in registers: extents up to 8 and 16 / 32 one line per thread, 64 / 128
//     two threads per line (fast_dct.cuh, dct2_dense4); two equal small last axes (a convolution's kernel window)
//     together; only the other extents are dense contractions from a table, even and odd outputs apart (half the
//     products), into a second tile;
//   * the tile's strides are padded on the host so that neighbouring lines do not share banks, and a line's elements are a
//     constant stride apart; the padding is always zero, so that sweeps over the tile run over plain memory, 16 bytes at a
//     time;
//   * global offsets come from a table of the chunk's contiguous rows, not from four divisions per element, and the loads
//     of eight elements per thread -- of sixteen, in quads, where the rows are whole 16-byte pieces -- are issued together; the next
//     chunk's rows are on their way to L2 during the selection;
//   * addresses along a line are byte offsets, one instruction each, and on a last axis of whole quads four elements one access;
//   * the first axis of the inverse is transformed only along the lines that hold kept coefficients, where it has more than 128 lines;
//   * top-k: the k-th largest of the threads' maxima (from a histogram relative to the largest) bounds the k-th coefficient;
//     the few dozen to few hundred coefficients above it are listed, one warp finds the k-th among them, and the kept ones
//     are put in index order by counting or, where much of a chunk is kept, by going over the tile; radix select only when the
//     list overflows (chunks with many equal magnitudes, k beyond the bound).
// Measured (one call, bf16 gradients, k = 32; dense contractions on every axis with radix select -> this): four
// 512 x 512 x 3 x 3 weights in 32 x 32 x 3 x 3 chunks (9.4 M parameters) compress 381 -> 115 us, decode 219 -> 63;
// 7511 x 512 in 29 x 64: 243 -> 83 / 122 -> 36; 8192 x 8192 in 32 x 128: 2424 -> 1050 / 1155 -> 379; in 16 x 32 (k = 4):
// 3254 -> 1017 / 1509 -> 409.  Quads, byte offsets, L2 ahead and listed lines: in 16 x 32 again 988 -> 882 us, 1024 x 1024 20.5 -> 17.6;
// a set of both kinds (13 M parameters) compress 188 -> 176, decode 80 -> 77.
#include <cuda_bf16.h>

#include <cmath>
#include <cstddef>
#include <type_traits>

#include "demo_internal.h"
#include "fast_dct.cuh"
#include "launch.cuh"

namespace {

constexpr int CAND = 512;       // candidate list
constexpr int DENSE_SHARE = 24;  // select_topk

__device__ __forceinline__ unsigned mag_key(float v) { return __float_as_uint(v) & 0x7fffffffu; }

// Last entry with chunk_begin <= c.
__device__ __forceinline__ int find_nd_entry(const DemoNdEntry *entries, int n, long long c)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (entries[mid].chunk_begin <= c)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Element offset of the chunk's first element: chunk id -> (k_0..k_3) row-major over the chunk grid,
// offset = sum_a k_a s_a stride_a (blocking operator).  A tensor has fewer than 2^31 chunks.
__device__ __forceinline__ size_t chunk_base(const DemoNdEntry &e, unsigned lc)
{
    size_t base = 0;
#pragma unroll
    for (int a = DEMO_ND_DIMS - 1; a >= 0; --a) {
        const unsigned q = lc / (unsigned)e.c[a];
        const unsigned k = lc - q * (unsigned)e.c[a];
        lc = q;
        base += (size_t)k * (size_t)e.s[a] * (size_t)e.stride[a];
    }
    return base;
}

// Offsets of element i (row-major inside the chunk) in the tensor, relative to the chunk's first element, and in the
// tile.  The divisions by the chunk extents are multiplications by inv[a] = ceil(2^32 / s_a), exact for
// i < 2^14 and s_a <= 2^7.
struct Place {
    size_t g;
    int t;
};
__device__ __forceinline__ Place place_of(const DemoNdEntry &e, int i)
{
    Place o{0, 0};
    unsigned r = (unsigned)i;
#pragma unroll
    for (int a = DEMO_ND_DIMS - 1; a >= 0; --a) {
        if (e.s[a] > 1) {
            const unsigned q = __umulhi(r, e.inv[a]);
            const unsigned j = r - q * (unsigned)e.s[a];
            o.g += (size_t)j * (size_t)e.stride[a];
            o.t += (int)j * e.p[a];
            r = q;
        }
    }
    return o;
}
// Row-major index of the element at tile position t (never a padding place).
__device__ __forceinline__ int index_of(const DemoNdEntry &e, int t)
{
    int i = 0;
#pragma unroll
    for (int a = 0; a < DEMO_ND_DIMS; ++a) {
        if (e.s[a] > 1) {
            const int j = t / e.p[a];
            t -= j * e.p[a];
            i = i * e.s[a] + j;
        }
    }
    return i;
}

// Shared memory of a CTA: this, then uint2 rows[cls.rows], float B[max_M] (compress), the tiles.
struct Shared {
    DemoNdEntry e[2];  // current and next chunk, looked up by one thread a chunk ahead
    size_t base[2];
    unsigned ticket, hi, n, n_kept, bound, thr, need_eq, n_eq, state[2], warp_tot[12];
    int n_list;                    // lines in the list, -1: none was made
    unsigned hist[256], fine[256];  // then, together, a bit per line of the first axis
    alignas(16) uint2 cand[CAND];  // candidates (value bits, tile position) in no particular order
    __device__ __forceinline__ unsigned *bits();  // both histograms as one bit map
    __device__ __forceinline__ unsigned *list() { return reinterpret_cast<unsigned *>(cand); }  // tile positions; the candidates are dead
    uint4 kept[CAND / 2];          // the kept ones, two per entry; decode: with cand, two batches of records
};
extern __shared__ __align__(16) unsigned char smem_raw[];
static_assert(offsetof(Shared, fine) == offsetof(Shared, hist) + 256 * sizeof(unsigned), "one bit map");
__device__ __forceinline__ unsigned *Shared::bits() { return reinterpret_cast<unsigned *>(smem_raw + offsetof(Shared, hist)); }
__device__ __forceinline__ Shared *shared() { return reinterpret_cast<Shared *>(smem_raw); }
struct View {
    uint2 *rows;  // (offset in the tensor, offset in the tile) of every row
    float *B, *tile0, *tile1;
};
__host__ __device__ constexpr size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }

__device__ __forceinline__ View carve(const DemoNdClass &k, bool with_b)
{
    View v;
    unsigned char *raw = smem_raw + align16(sizeof(Shared));
    v.rows = reinterpret_cast<uint2 *>(raw);
    raw += align16((size_t)k.rows * 8);
    v.B = reinterpret_cast<float *>(raw);
    raw += with_b ? (size_t)k.max_M * 4 : 0;
    v.tile0 = reinterpret_cast<float *>(raw);
    v.tile1 = v.tile0 + (k.dense_axes ? k.tile : 0);
    return v;
}
size_t shared_bytes(const DemoNdClass &k, bool with_b)
{
    return align16(sizeof(Shared)) + align16((size_t)k.rows * 8) + (with_b ? (size_t)k.max_M * 4 : 0) +
           (size_t)k.tile * 4 * (k.dense_axes ? 2 : 1);
}

__device__ __forceinline__ void locate(Shared *w, int slot, const DemoNdEntry *entries, int n_entries, long long c)
{
    DemoNdEntry &e = w->e[slot];
    const DemoNdEntry &other = w->e[slot ^ 1];
    if (c < e.chunk_begin || c >= e.chunk_end) {
        if (c >= other.chunk_begin && c < other.chunk_end)
            e = other;
        else
            e = entries[find_nd_entry(entries, n_entries, c)];
    }
    w->base[slot] = chunk_base(e, (unsigned)(c - e.chunk_begin));
}

// (one thread) the chunk of a drawn ticket becomes the next one.
__device__ __forceinline__ void take_ticket(Shared *w, int slot, const DemoNdEntry *entries, const DemoNdClass &cls, unsigned ticket)
{
    const long long c = (long long)gridDim.x + ticket;
    if (c < cls.n_chunks) locate(w, slot, entries, cls.n, c);
    w->ticket = ticket;
}

// (all threads) another layout than the previous chunk's: offsets of its rows; the tiles are cleared, because its padding
// lies elsewhere.  A barrier must follow.
__device__ __forceinline__ void enter_layout(const View &v, const DemoNdEntry &e, const DemoNdClass &k)
{
    const int T = blockDim.x;
    if (e.row_table)
        for (int r = threadIdx.x; r * e.row < e.M; r += T) {
            const Place o = place_of(e, r * e.row);
            v.rows[r] = make_uint2((unsigned)o.g, (unsigned)o.t);
        }
    for (int i = threadIdx.x; i < k.tile; i += T) {
        v.tile0[i] = 0.f;
        v.tile1[i] = 0.f;
    }
}
// A chunk's rows on their way to L2, a row per thread.
template <typename T>
__device__ __forceinline__ void prefetch_chunk(const View &v, const DemoNdEntry &e, const T *base)
{
    if (!e.row_table) return;
    for (int r = threadIdx.x; r * e.row < e.M; r += blockDim.x) {
        const T *p = base + v.rows[r].x, *end = p + e.row;
        for (; p < end; p += 128 / sizeof(T)) prefetch_l2(p);
        prefetch_l2(end - 1);
    }
}
// Runs over the chunk's elements, U per thread and round: every thread calls load(j, offset in the tensor) U times without
// a branch in between (the last element again where there is none left), then use(j, index, offset, tile position) for
// those that exist.
template <int U, class Load, class Use>
__device__ __forceinline__ void for_elements(const View &v, const DemoNdEntry &e, Load load, Use use)
{
    const int M = e.M, T = blockDim.x;
    auto walk = [&](auto table) {
        using Off = typename std::conditional<decltype(table)::value, unsigned, size_t>::type;
        const unsigned row = (unsigned)e.row, inv_row = e.inv_row;
        for (int i0 = threadIdx.x; i0 < M; i0 += U * T) {
            Off g[U];
            int t[U];
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int i = min(i0 + j * T, M - 1);
                if constexpr (decltype(table)::value) {
                    const unsigned r = inv_row ? __umulhi((unsigned)i, inv_row) : (unsigned)i;
                    const unsigned d = (unsigned)i - r * row;
                    const uint2 o = v.rows[r];
                    g[j] = o.x + d;
                    t[j] = (int)(o.y + d);
                } else {
                    const Place o = place_of(e, i);
                    g[j] = o.g;
                    t[j] = o.t;
                }
            }
#pragma unroll
            for (int j = 0; j < U; ++j) load(j, g[j]);
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (i0 + j * T < M) use(j, i0 + j * T, g[j], t[j]);
        }
    };
    if (e.row_table)
        walk(std::true_type{});
    else
        walk(std::false_type{});
}

// The same by quads of four neighbouring elements (e.quads): load(j, offset), then use(j, first index, offset, tile position).
template <int U, class Load, class Use>
__device__ __forceinline__ void for_quads(const View &v, const DemoNdEntry &e, Load load, Use use)
{
    const int n = e.M >> 2, T = blockDim.x;
    const unsigned row = (unsigned)e.row >> 2, inv_row = e.inv_row4;
    for (int i0 = threadIdx.x; i0 < n; i0 += U * T) {
        unsigned g[U];
        int t[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int i = min(i0 + j * T, n - 1);
            const unsigned r = inv_row ? __umulhi((unsigned)i, inv_row) : (unsigned)i;
            const unsigned d = 4u * ((unsigned)i - r * row);
            const uint2 o = v.rows[r];
            g[j] = o.x + d;
            t[j] = (int)(o.y + d);
        }
#pragma unroll
        for (int j = 0; j < U; ++j) load(j, g[j]);
#pragma unroll
        for (int j = 0; j < U; ++j)
            if (i0 + j * T < n) use(j, 4 * (i0 + j * T), g[j], t[j]);
    }
}
// Four elements of the tile: in one access where its rows allow, else in four, whose order turns with the thread, so that a warp's 32
// neighbouring quads do not meet in eight banks.
__device__ __forceinline__ float4 turned(float4 f, int r)  // its element j is element (j + r) mod 4 of f
{
    if (r & 1) f = make_float4(f.y, f.z, f.w, f.x);
    if (r & 2) f = make_float4(f.z, f.w, f.x, f.y);
    return f;
}
__device__ __forceinline__ float4 tile_quad(const float *tile, int t, bool whole)
{
    if (whole) return *reinterpret_cast<const float4 *>(tile + t);
    const int r = threadIdx.x >> 3 & 3;
    const float *q = tile + t;
    return turned(make_float4(q[r], q[(r + 1) & 3], q[(r + 2) & 3], q[(r + 3) & 3]), (4 - r) & 3);
}
__device__ __forceinline__ void set_tile_quad(float *tile, int t, bool whole, const float4 &f)
{
    if (whole) {
        *reinterpret_cast<float4 *>(tile + t) = f;
    } else {
        const int r = threadIdx.x >> 3 & 3;
        const float4 v = turned(f, r);
        float *q = tile + t;
        q[r] = v.x;
        q[(r + 1) & 3] = v.y;
        q[(r + 2) & 3] = v.z;
        q[(r + 3) & 3] = v.w;
    }
}
__device__ __forceinline__ float4 grad_quad(const float *g) { return *reinterpret_cast<const float4 *>(g); }
__device__ __forceinline__ uint2 grad_quad(const __nv_bfloat16 *g) { return *reinterpret_cast<const uint2 *>(g); }
__device__ __forceinline__ float4 grad_floats(const float4 &v) { return v; }
__device__ __forceinline__ float4 grad_floats(const uint2 &v)
{   // (bf16 is the upper half of a float)
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                       __uint_as_float(v.y & 0xffff0000u));
}

// ---- one axis of the multilinear product ------------------------------------------------------------
// Every extent is a function of its own (not inlined: dozens of register-resident bodies in one kernel cost each other
// registers).  They get the byte offset of the tile and the slot of the entry, so that the accesses stay shared-memory
// accesses.
__device__ __forceinline__ float *tile_at(unsigned off) { return reinterpret_cast<float *>(smem_raw + off); }
// A line by the byte offsets of its first element and between elements: one instruction per address (as floats, an index
// and a shift each).
struct Line {
    unsigned at, step;
    __device__ __forceinline__ Line(unsigned tile, int first, int p) : at(tile + 4u * (unsigned)first), step(4u * (unsigned)p) {}
    __device__ __forceinline__ float &operator[](int n) const { return *reinterpret_cast<float *>(smem_raw + at + (unsigned)n * step); }
    __device__ __forceinline__ float4 &quad(int n) const { return *reinterpret_cast<float4 *>(smem_raw + at + 16u * (unsigned)n); }
};
__device__ __forceinline__ unsigned tile_offset(const float *X)
{
    return (unsigned)(reinterpret_cast<const unsigned char *>(X) - smem_raw);
}

// Tile position of the first element of line L along axis a (a .. a_last where axes are transformed together): the other
// axes' indices, the last running fastest.
__device__ __forceinline__ int line_base(const DemoNdEntry &e, int a, int a_last, int L)
{
    int t = 0;
    unsigned r = (unsigned)L;
#pragma unroll
    for (int b = DEMO_ND_DIMS - 1; b >= 0; --b) {
        if ((b < a || b > a_last) && e.s[b] > 1) {
            const unsigned q = __umulhi(r, e.inv[b]);
            t += (int)(r - q * (unsigned)e.s[b]) * e.p[b];
            r = q;
        }
    }
    return t;
}

// C[u][n] = a_u cos(pi (2n+1) u / (2S)), the angle reduced to [0, pi/2] in whole numbers.
template <int S>
constexpr double dct_entry(int u, int n)
{
    int m = ((2 * n + 1) * u) % (4 * S);
    if (m > 2 * S) m = 4 * S - m;
    const double c = m > S ? -fdct::c_cos(fdct::kPi * (2 * S - m) / (2.0 * S)) : fdct::c_cos(fdct::kPi * m / (2.0 * S));
    return c * fdct::c_sqrt((u == 0 ? 1.0 : 2.0) / S);
}

template <int S, bool INV>
__device__ __forceinline__ void line_transform(float (&x)[S])
{
    if constexpr ((S & (S - 1)) == 0) {
        if constexpr (INV)
            fdct::dct3_ortho_dense4<S>(x);
        else
            fdct::dct2_ortho_dense4<S>(x);
    } else {
        // even outputs from x[n] + x[S-1-n], odd ones from x[n] - x[S-1-n]: half the products.  (Errors against 64 bits, 5 / 6 / 7 points a
        // side, folded / plain: 8.5 / 7.8 / 6.8e-8 and 8.5 / 8.0 / 7.1e-8; 3 points 7.5 and 7.3e-8: those stay plain.)
        constexpr int H = S / 2;
        float y[S];
        if constexpr (S == 3) {
            fdct::static_for<0, S>([&](auto uu) {
                constexpr int u = decltype(uu)::value;
                float acc = 0.f;
                fdct::static_for<0, S>([&](auto nn) {
                    constexpr int n = decltype(nn)::value;
                    constexpr float c = (float)(INV ? dct_entry<S>(n, u) : dct_entry<S>(u, n));
                    acc = n == 0 ? c * x[0] : fmaf(c, x[n], acc);
                });
                y[u] = acc;
            });
        } else if constexpr (!INV) {
            float u[H + 1], v[H];
            fdct::static_for<0, H>([&](auto nn) {
                constexpr int n = decltype(nn)::value;
                u[n] = x[n] + x[S - 1 - n];
                v[n] = x[n] - x[S - 1 - n];
            });
            u[H] = x[H];  // (odd S: the middle; even S: not used)
            fdct::static_for<0, S>([&](auto uu) {
                constexpr int k = decltype(uu)::value, terms = (k & 1) ? H : (S + 1) / 2;
                float acc = 0.f;
                fdct::static_for<0, terms>([&](auto nn) {
                    constexpr int n = decltype(nn)::value;
                    constexpr float c = (float)dct_entry<S>(k, n);
                    const float t = (k & 1) ? v[n] : u[n];
                    acc = n == 0 ? c * t : fmaf(c, t, acc);
                });
                y[k] = acc;
            });
        } else {
            fdct::static_for<0, (S + 1) / 2>([&](auto nn) {
                constexpr int n = decltype(nn)::value;
                float ev = 0.f, od = 0.f;
                fdct::static_for<0, S>([&](auto uu) {
                    constexpr int k = decltype(uu)::value;
                    constexpr float c = (float)dct_entry<S>(k, n);
                    if constexpr (k & 1)
                        od = k == 1 ? c * x[1] : fmaf(c, x[k], od);
                    else
                        ev = k == 0 ? c * x[0] : fmaf(c, x[k], ev);
                });
                if constexpr (2 * n + 1 == S) {
                    y[n] = ev;
                } else {
                    y[n] = ev + od;
                    y[S - 1 - n] = ev - od;
                }
            });
        }
#pragma unroll
        for (int n = 0; n < S; ++n) x[n] = y[n];
    }
}

// QUADS: the last axis, its lines in whole quads of the tile.  `list`: only the lines that start at these tile positions.
template <int S, bool INV, bool QUADS>
__device__ __noinline__ void lines_whole(unsigned tile, int slot, int a, int n_list)
{
    Shared *s = shared();
    const DemoNdEntry &e = s->e[slot];
    const int lines = n_list >= 0 ? n_list : e.M / S, p = e.p[a];
    for (int L = threadIdx.x; L < lines; L += blockDim.x) {
        const Line q(tile, n_list >= 0 ? (int)s->list()[L] : line_base(e, a, a, L), p);
        float x[S];
        if constexpr (QUADS) {
#pragma unroll
            for (int n = 0; n < S / 4; ++n) {
                const float4 f = q.quad(n);
                x[4 * n] = f.x;
                x[4 * n + 1] = f.y;
                x[4 * n + 2] = f.z;
                x[4 * n + 3] = f.w;
            }
        } else {
#pragma unroll
            for (int n = 0; n < S; ++n) x[n] = q[n];
        }
        line_transform<S, INV>(x);
        if constexpr (QUADS) {
#pragma unroll
            for (int n = 0; n < S / 4; ++n) q.quad(n) = make_float4(x[4 * n], x[4 * n + 1], x[4 * n + 2], x[4 * n + 3]);
        } else {
#pragma unroll
            for (int n = 0; n < S; ++n) q[n] = x[n];
        }
    }
}

// The last two axes, both of extent S: S * S consecutive elements per thread.
template <int S, bool INV>
__device__ __noinline__ void lines_tail(unsigned tile, int slot)
{
    float *X = tile_at(tile);
    const DemoNdEntry &e = shared()->e[slot];
    const int lines = e.M / (S * S);
    for (int L = threadIdx.x; L < lines; L += blockDim.x) {
        float *q = X + line_base(e, 2, 3, L);
        float x[S][S];
#pragma unroll
        for (int i = 0; i < S; ++i)
#pragma unroll
            for (int j = 0; j < S; ++j) x[i][j] = q[i * S + j];
#pragma unroll
        for (int i = 0; i < S; ++i) line_transform<S, INV>(x[i]);
#pragma unroll
        for (int j = 0; j < S; ++j) {
            float col[S];
#pragma unroll
            for (int i = 0; i < S; ++i) col[i] = x[i][j];
            line_transform<S, INV>(col);
#pragma unroll
            for (int i = 0; i < S; ++i) q[i * S + j] = col[i];
        }
    }
}

// Extent 2H, two threads per line: the even outputs are a DCT-II of H points of x[n] + x[2H-1-n], the odd ones a DCT-IV of
// x[n] - x[2H-1-n].  Even warps take one, odd warps the other; the CTA is a multiple of 64 threads.
template <int H, bool INV>
__device__ __noinline__ void lines_split(unsigned tile, int slot, int a)
{
    const DemoNdEntry &e = shared()->e[slot];
    using SC = fdct::ScaleOrtho<2 * H>;
    constexpr float DC = (float)fdct::c_sqrt(0.5);
    const int lines = e.M / (2 * H), p = e.p[a];
    const int h = (threadIdx.x >> 5) & 1;
    const int l0 = (threadIdx.x >> 6) * 32 + (threadIdx.x & 31), per_round = blockDim.x >> 1;
    for (int r0 = 0; r0 < lines; r0 += per_round) {
        const bool active = r0 + l0 < lines;
        const Line q(tile, active ? line_base(e, a, a, r0 + l0) : 0, p);
        float x[H], y[H];
        if (active) {
            if constexpr (!INV) {
#pragma unroll
                for (int n = 0; n < H; ++n) {
                    const float lo = q[n], hi = q[2 * H - 1 - n];
                    x[n] = h ? lo - hi : lo + hi;
                }
                if (h == 0) {
                    fdct::dct2_dense4<H, SC>(x, y);
                    y[0] *= DC;
                } else {
                    fdct::dct4_dense<H, SC>(x, y);
                }
            } else {
#pragma unroll
                for (int n = 0; n < H; ++n) x[n] = q[2 * n + h];
                if (h == 0) {
                    x[0] *= DC;
                    fdct::dct3_dense4<H, SC>(x, y);
                } else {
                    fdct::dct4_dense<H, SC>(x, y);
                }
            }
        }
        __syncthreads();  // both halves of every line of this round are read
        if (active) {
            if constexpr (!INV) {
#pragma unroll
                for (int n = 0; n < H; ++n) q[2 * n + h] = y[n];
            } else {
                if (h == 0) {
#pragma unroll
                    for (int n = 0; n < H; ++n) q[n] = y[n];
                } else {
#pragma unroll
                    for (int n = 0; n < H; ++n) q[2 * H - 1 - n] = y[n];
                }
            }
        }
        if constexpr (INV) {
            __syncthreads();
            if (active) {
#pragma unroll
                for (int i = 0; i < H / 2; ++i) {
                    const int n = i + h * (H / 2);
                    const float ev = q[n], od = q[2 * H - 1 - n];
                    q[n] = ev + od;
                    q[2 * H - 1 - n] = ev - od;
                }
            }
        }
    }
}

// Any other extent, from a table.  Forward: a thread forms 8 even or 8 odd outputs of LPT lines from
// x[n] +- x[s-1-n]; inverse: 8 outputs n and their mirror images from the even and the odd coefficients.
// Table of extent s, h = ceil(s/2), even / odd outputs padded to pe / po (multiples of 8):
//   forward rows n < h: [C[0][n], C[2][n], ... | C[1][n], C[3][n], ...] (the middle n of an odd s halved),
//   inverse rows u < s: C[u][n] for n < h, padded to pe.
__host__ __device__ constexpr int up8(int v) { return (v + 7) & ~7; }
template <int LPT, bool INV>
__device__ __noinline__ void lines_dense(unsigned dst_tile, unsigned src_tile, const float *__restrict__ table, int slot, int a)
{
    const DemoNdEntry &e = shared()->e[slot];
    const int s = e.s[a], p = e.p[a], lines = e.M / s;
    const unsigned step = 4u * (unsigned)p;
    auto at = [](unsigned byte) -> float & { return *reinterpret_cast<float *>(smem_raw + byte); };
    const int h = (s + 1) >> 1, pe = up8(h), po = up8(s >> 1);
    const int groups = INV ? pe >> 3 : (pe + po) >> 3;
    const float *Tb = INV ? table + h * (pe + po) : table;
    const int Q = (lines + LPT - 1) / LPT;
    const int items = groups * Q;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        const int g = it / Q, l0 = it - g * Q;
        unsigned b[LPT];  // bytes into the tile
#pragma unroll
        for (int v = 0; v < LPT; ++v) b[v] = 4u * (unsigned)line_base(e, a, a, min(l0 + v * Q, lines - 1));
        if constexpr (!INV) {
            const bool odd = 8 * g >= pe;
            const float sign = odd ? -1.f : 1.f;
            float acc[LPT][8];
#pragma unroll
            for (int v = 0; v < LPT; ++v)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[v][j] = 0.f;
            const float *tp = Tb + 8 * g;
            unsigned lo[LPT], hi[LPT];
#pragma unroll
            for (int v = 0; v < LPT; ++v) {
                lo[v] = src_tile + b[v];
                hi[v] = lo[v] + (unsigned)(s - 1) * step;
            }
#pragma unroll 4
            for (int n = 0; n < h; ++n, tp += pe + po) {
                const float4 t0 = __ldg(reinterpret_cast<const float4 *>(tp));
                const float4 t1 = __ldg(reinterpret_cast<const float4 *>(tp + 4));
                const float t[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
                for (int v = 0; v < LPT; ++v) {
                    const float xv = fmaf(sign, at(hi[v]), at(lo[v]));
                    lo[v] += step;
                    hi[v] -= step;
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[v][j] = fmaf(t[j], xv, acc[v][j]);
                }
            }
#pragma unroll
            for (int v = 0; v < LPT; ++v) {
                if (l0 + v * Q < lines) {
                    const int u0 = odd ? 2 * (8 * g - pe) + 1 : 16 * g;
                    const unsigned q = dst_tile + b[v] + (unsigned)u0 * step;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (u0 + 2 * j < s) at(q + 2u * (unsigned)j * step) = acc[v][j];
                }
            }
        } else {
            float ev[LPT][8], od[LPT][8];
#pragma unroll
            for (int v = 0; v < LPT; ++v)
#pragma unroll
                for (int j = 0; j < 8; ++j) ev[v][j] = od[v][j] = 0.f;
            const float *tp = Tb + 8 * g;
            unsigned q[LPT];
#pragma unroll
            for (int v = 0; v < LPT; ++v) q[v] = src_tile + b[v];
            auto term = [&](int u, float (&acc)[LPT][8]) {
                const float4 t0 = __ldg(reinterpret_cast<const float4 *>(tp + u * pe));
                const float4 t1 = __ldg(reinterpret_cast<const float4 *>(tp + u * pe + 4));
                const float t[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
                for (int v = 0; v < LPT; ++v) {
                    const float xv = at(q[v]);
                    q[v] += step;
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[v][j] = fmaf(t[j], xv, acc[v][j]);
                }
            };
#pragma unroll 2
            for (int u = 0; u + 1 < s; u += 2) {
                term(u, ev);
                term(u + 1, od);
            }
            if (s & 1) term(s - 1, ev);
#pragma unroll
            for (int v = 0; v < LPT; ++v) {
                if (l0 + v * Q < lines) {
                    const unsigned lo = dst_tile + b[v] + (unsigned)(8 * g) * step, hi = dst_tile + b[v] + (unsigned)(s - 1 - 8 * g) * step;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int n = 8 * g + j;
                        if (n < h) {
                            at(lo + (unsigned)j * step) = ev[v][j] + od[v][j];
                            if (n != s - 1 - n) at(hi - (unsigned)j * step) = ev[v][j] - od[v][j];
                        }
                    }
                }
            }
        }
    }
}

// Extents that are transformed in registers.
constexpr bool in_place_extent(int s) { return s <= 8 || s == 16 || s == 32 || s == 64 || s == 128; }

// The first axis that is transformed, if the kept coefficients' lines along it are worth listing (those it is transformed in by a thread
// per line); else -1.
__device__ __forceinline__ int first_listed(const DemoNdEntry &e)
{
    int a = 0;
    while (a < DEMO_ND_DIMS && e.s[a] == 1) ++a;
    if (a == DEMO_ND_DIMS || (e.tail && a == 2) || !in_place_extent(e.s[a]) || e.s[a] > 32) return -1;
    if (e.M <= 128 * e.s[a]) return -1;  // a round of lines or less (8192 x 8192 in 16 x 32 2033 us listed, 1952 not; 28 M in 32 x 32 x 3 x 3 496 / 511)
    return a;
}

// All axes in turn.  cur / spare: the tile and the second tile (used by dense axes only); swapped as needed.
// n_list >= 0: only the lines in the list are not zero along the first axis (first_listed).
template <bool INV, bool BIG>
__device__ __forceinline__ void transform_chunk(float *&cur, float *&spare, int slot, const float *tables, int n_list)
{
    const DemoNdEntry &e = shared()->e[slot];
    unsigned tile = tile_offset(cur), other = tile_offset(spare);
#pragma unroll 1
    for (int a = 0; a < DEMO_ND_DIMS; ++a) {
        const int s = e.s[a];
        if (s == 1) continue;
        if (e.tail && a == 2) {
            switch (s) {
                case 2: lines_tail<2, INV>(tile, slot); break;
                case 3: lines_tail<3, INV>(tile, slot); break;
                case 4: lines_tail<4, INV>(tile, slot); break;
                case 5: lines_tail<5, INV>(tile, slot); break;
                case 6: lines_tail<6, INV>(tile, slot); break;
                default: lines_tail<7, INV>(tile, slot); break;
            }
            __syncthreads();
            break;
        }
        const int list = n_list;
        n_list = -1;
        auto whole = [&](auto extent) {
            constexpr int S = decltype(extent)::value;
            if constexpr (S % 4 == 0) {
                if (a == DEMO_ND_DIMS - 1 && e.quads == 2) {
                    lines_whole<S, INV, true>(tile, slot, a, list);
                    return;
                }
            }
            lines_whole<S, INV, false>(tile, slot, a, list);
        };
        switch (s) {
            case 2: whole(std::integral_constant<int, 2>{}); break;
            case 3: whole(std::integral_constant<int, 3>{}); break;
            case 4: whole(std::integral_constant<int, 4>{}); break;
            case 5: whole(std::integral_constant<int, 5>{}); break;
            case 6: whole(std::integral_constant<int, 6>{}); break;
            case 7: whole(std::integral_constant<int, 7>{}); break;
            case 8: whole(std::integral_constant<int, 8>{}); break;
            case 16: whole(std::integral_constant<int, 16>{}); break;
            case 32: whole(std::integral_constant<int, 32>{}); break;
            case 64: lines_split<32, INV>(tile, slot, a); break;
            case 128:
                if constexpr (BIG) lines_split<64, INV>(tile, slot, a);
                break;
            default: {
                // two lines per thread where that still occupies the CTA
                const int lines = e.M / s, pe = up8((s + 1) >> 1), groups = (INV ? pe : pe + up8(s >> 1)) >> 3;
                if (groups * ((lines + 1) >> 1) >= (int)blockDim.x)
                    lines_dense<2, INV>(other, tile, tables + e.basis[a], slot, a);
                else
                    lines_dense<1, INV>(other, tile, tables + e.basis[a], slot, a);
                const unsigned t = tile;
                tile = other;
                other = t;
            }
        }
        __syncthreads();
    }
    cur = tile_at(tile);
    spare = tile_at(other);
}

__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned *warp_tot)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned n = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += n;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    unsigned base = 0;
    for (int w = 0; w < warp; ++w) base += warp_tot[w];
    __syncthreads();
    return base + inc - v;
}

// (one warp) the bin of hist[0..256), taken in ascending order, where the running count reaches `rank`, and the count
// before it; bin 256 if it never does.
__device__ __forceinline__ void find_bin(const unsigned *hist, unsigned rank, unsigned *bin, unsigned *before_bin)
{
    const int lane = threadIdx.x & 31;
    unsigned h[8], local = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        h[j] = hist[8 * lane + j];
        local += h[j];
    }
    unsigned inc = local;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned n = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += n;
    }
    unsigned cum = inc - local, b = 256, bb = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (cum < rank && cum + h[j] >= rank) {
            b = 8 * lane + j;
            bb = cum;
        }
        cum += h[j];
    }
    const unsigned who = __ballot_sync(0xffffffffu, b < 256u);
    const int src = who ? __ffs(who) - 1 : 0;
    *bin = __shfl_sync(0xffffffffu, b, src);
    *before_bin = __shfl_sync(0xffffffffu, bb, src);
}

// Records of the coefficients with keys above thr (>= 1: never the padding) and of the first need_eq equal to it, in index order; X
// left with alpha * kept, zero elsewhere; ends with a barrier.  A warp has neighbouring quads of the tile (tile positions are in
// index order): the warps count theirs, then number them.
__device__ __noinline__ void compact(unsigned tile, int slot, DemoRecord *rec, float alpha, unsigned thr, unsigned need_eq)
{
    Shared *s = shared();
    const DemoNdEntry &e = s->e[slot];
    float4 *X4 = reinterpret_cast<float4 *>(tile_at(tile));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, quads = e.tile >> 2;
    const int rounds = (quads + (int)blockDim.x - 1) / (int)blockDim.x, q0 = warp * rounds * 32 + lane;
    auto count = [&](const float4 &f) {  // above | equal << 16
        const unsigned k[4] = {mag_key(f.x), mag_key(f.y), mag_key(f.z), mag_key(f.w)};
        unsigned n = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) n += (k[j] > thr ? 1u : 0u) + (k[j] == thr ? 0x10000u : 0u);
        return n;
    };
    unsigned n = 0;
    for (int r = 0; r < rounds; ++r)
        if (q0 + 32 * r < quads) n += count(X4[q0 + 32 * r]);
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) s->warp_tot[warp] = n;
    __syncthreads();
    unsigned before = 0;
    for (int w = 0; w < warp; ++w) before += s->warp_tot[w];
    for (int r = 0; r < rounds; ++r) {
        const int q = q0 + 32 * r;
        const bool have = q < quads;
        float4 f = have ? X4[q] : make_float4(0.f, 0.f, 0.f, 0.f);
        const unsigned own = count(f);
        unsigned inc = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += v;
        }
        unsigned gt = (before + inc - own) & 0xffffu, eq = (before + inc - own) >> 16;
        before += __shfl_sync(0xffffffffu, inc, 31);
        float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned key = mag_key(v[j]);
            const bool above = key > thr, equal = key == thr;
            const bool keep = above || (equal && eq < need_eq);
            if (keep) {
                DemoRecord out;
                out.idx = index_of(e, 4 * q + j);
                out.val = v[j];
                rec[gt + min(eq, need_eq)] = out;
            }
            gt += above;
            eq += equal;
            v[j] = keep ? alpha * v[j] : 0.f;
        }
        if (have) X4[q] = make_float4(v[0], v[1], v[2], v[3]);
    }
    __syncthreads();
}

// Exact top-k by radix select on the magnitude bits (the padding's zeros are taken out of the counts), index-ordered compaction; leaves
// alpha * kept in X, zero elsewhere.
__device__ __noinline__ void select_radix(unsigned tile, int slot, DemoRecord *rec, float alpha)
{
    float *X = tile_at(tile);
    Shared *s = shared();
    const DemoNdEntry &e = s->e[slot];
    const int tid = threadIdx.x, T = blockDim.x, M = e.M, k_eff = e.k_eff, quads = e.tile >> 2;
    if (tid == 0) {
        s->state[0] = 0u;               // prefix of the key found so far
        s->state[1] = (unsigned)k_eff;  // rank still to resolve inside the prefix class
    }
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        const unsigned mask = (pass == 0) ? 0u : (0xffffffffu << (shift + 8));
        for (int i = tid; i < 256; i += T) s->hist[i] = 0u;
        __syncthreads();
        const unsigned prefix = s->state[0];
        auto note = [&](float v) {
            const unsigned key = mag_key(v);
            if ((key & mask) == prefix) atomicAdd(&s->hist[255u - ((key >> shift) & 255u)], 1u);
        };
        for (int i = tid; i < quads; i += T) {
            const float4 f = reinterpret_cast<const float4 *>(X)[i];
            note(f.x);
            note(f.y);
            note(f.z);
            note(f.w);
        }
        __syncthreads();
        if (tid < 32) {
            unsigned bin, before;
            const unsigned rem = s->state[1];
            if (tid == 0 && prefix == 0u) s->hist[255] -= (unsigned)(4 * quads - M);
            __syncwarp();
            find_bin(s->hist, rem, &bin, &before);
            __syncwarp();
            if (tid == 0) {
                s->state[1] = rem - before;
                s->state[0] = prefix | ((255u - bin) << shift);
            }
        }
        __syncthreads();
    }
    const unsigned thr = s->state[0], need_eq = s->state[1];
    if (thr) {
        compact(tile, slot, rec, alpha, thr, need_eq);
        return;
    }
    // fewer than k coefficients are not zero: zeros are kept too, but not those of the padding
    const int per = (M + T - 1) / T;
    const int start = tid * per;
    const int stop = min(M, start + per);
    unsigned gt = 0, eq = 0;
    for (int i = start; i < stop; ++i) {
        const unsigned key = mag_key(X[place_of(e, i).t]);
        gt += key > thr;
        eq += key == thr;
    }
    const unsigned before = block_exclusive_scan(gt | (eq << 16), s->warp_tot);
    unsigned gb = before & 0xffffu, eb = before >> 16;
    for (int i = start; i < stop; ++i) {
        const int t = place_of(e, i).t;
        const float v = X[t];
        const unsigned key = mag_key(v);
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
            DemoRecord r;
            r.idx = i;
            r.val = v;
            rec[pos] = r;
        }
        X[t] = sel ? alpha * v : 0.f;  // the residual removes alpha times the kept part
    }
    __syncthreads();
}

// (one warp) the k_eff-th largest of n candidate keys, NK per lane: threshold, how many equal to it are kept and exist.
template <int NK>
__device__ __noinline__ void find_threshold(unsigned n, unsigned bound, int k_eff)
{
    const int lane = threadIdx.x & 31;
    Shared *s = shared();
    unsigned keys[NK];
    unsigned top = 0u;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
        const unsigned i = (unsigned)j * 32u + lane;
        keys[j] = i < n ? (s->cand[i].x & 0x7fffffffu) : 0u;
        top = max(top, keys[j]);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    const int b0 = 31 - __clz((bound ^ top) | 1u);
    unsigned thr = bound & ~((2u << b0) - 1u);
    unsigned n_ge = n;  // every candidate is >= the bound >= thr
#pragma unroll 1
    for (int b = b0; b >= 0 && n_ge != (unsigned)k_eff; --b) {
        const unsigned cand = thr | (1u << b);
        unsigned cnt = 0;
#pragma unroll
        for (int j = 0; j < NK; ++j) cnt += __popc(__ballot_sync(0xffffffffu, keys[j] >= cand));
        if (cnt >= (unsigned)k_eff) {
            thr = cand;
            n_ge = cnt;
        }
    }
    unsigned n_gt = 0;
#pragma unroll
    for (int j = 0; j < NK; ++j) n_gt += __popc(__ballot_sync(0xffffffffu, keys[j] > thr));
    if (lane == 0) {
        s->thr = thr;
        s->need_eq = (unsigned)k_eff - n_gt;
        s->n_eq = n_ge - n_gt;
    }
}

// Exact top-k of the coefficients in X (complete for all threads): records in ascending index order to `rec`, X left
// with alpha * kept and zero elsewhere; ends with a barrier.  hist, fine, hi, n and n_kept were cleared before a barrier.
__device__ __forceinline__ void select_topk(float *X, int slot, DemoRecord *rec, float alpha)
{
    const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
    Shared *s = shared();
    const DemoNdEntry &e = s->e[slot];
    const int k_eff = e.k_eff, quads = e.tile >> 2;
    float4 *X4 = reinterpret_cast<float4 *>(X);
    if (k_eff == e.M) {  // everything is kept
        for (int i = tid; i < e.M; i += T) {
            const int t = place_of(e, i).t;
            DemoRecord r;
            r.idx = i;
            r.val = X[t];
            rec[i] = r;
            X[t] = alpha * r.val;
        }
        __syncthreads();
        return;
    }
    // Long lists of a small chunk are numbered by going over the tile twice, short ones by counting the records below each: k^2 / 2
    // comparisons, which pays up to k^2 = 24 M (one call, counting / numbering: 512 x 512 x 3 x 3 in 16 x 16 x 3 x 3 k = 192 / 256 56 / 66
    // and 64 / 66 us; 1024 x 1024 in 16 x 32 k = 64 / 128 / 256 34 / 48 / 81 and 34 / 38 / 37 us).
    const bool dense = k_eff * k_eff > DENSE_SHARE * e.M;
    // group maxima: a thread's quads as one group, or -- where k is not well below the number of threads -- as four
    const bool four = 2 * k_eff > T;
    unsigned key[4] = {0u, 0u, 0u, 0u};
#pragma unroll 4
    for (int i = tid; i < quads; i += T) {
        const float4 f = X4[i];
        key[0] = max(key[0], mag_key(f.x));
        key[1] = max(key[1], mag_key(f.y));
        key[2] = max(key[2], mag_key(f.z));
        key[3] = max(key[3], mag_key(f.w));
    }
    const unsigned mine = max(max(key[0], key[1]), max(key[2], key[3]));
    {
        const unsigned mx = __reduce_max_sync(0xffffffffu, mine);
        if (lane == 0) atomicMax(&s->hi, mx);
    }
    __syncthreads();
    const unsigned hi = s->hi;
    if (hi == 0u) {
        // all coefficients zero: the tie rule gives the records 0 .. k_eff-1 with value 0
        for (int r = tid; r < k_eff; r += T) {
            DemoRecord z;
            z.idx = r;
            z.val = 0.f;
            rec[r] = z;
        }
        __syncthreads();
        return;
    }
    // their histogram, 16 bins per octave below the largest, then one of 256 steps inside the bin that holds the k-th group:
    // the lower edge of that step bounds the k-th coefficient from below.  (The edge of the first bin alone, up to 6 % below,
    // is not enough: with error feedback the magnitudes crowd just below the threshold.)
    auto each_group = [&](auto f) {
        if (four) {
#pragma unroll
            for (int g = 0; g < 4; ++g) f(key[g]);
        } else {
            f(mine);
        }
    };
    each_group([&](unsigned q) { atomicAdd(&s->hist[min(255u, (hi >> 19) - (q >> 19))], 1u); });
    __syncthreads();
    if (tid < 32) {
        unsigned bin, before;
        find_bin(s->hist, (unsigned)k_eff, &bin, &before);
        if (tid == 0) {
            s->state[0] = bin < 255u ? (hi >> 19) - bin : 0u;
            s->state[1] = (unsigned)k_eff - before;
        }
    }
    __syncthreads();
    const unsigned top12 = s->state[0];
    if (top12) {
        each_group([&](unsigned q) {
            if (q >> 19 == top12) atomicAdd(&s->fine[255u - ((q >> 11) & 255u)], 1u);
        });
        __syncthreads();
        if (tid < 32) {
            unsigned step, before;
            find_bin(s->fine, s->state[1], &step, &before);
            if (tid == 0) s->bound = top12 << 19 | (255u - step) << 11;
        }
    } else if (tid == 0) {
        s->bound = 1u;  // fewer than k groups near the largest
    }
    __syncthreads();
    const unsigned bound = s->bound;  // (>= 1: the padding is never a candidate)
    // (a thread whose maximum is below the bound has none; the quads of a thread take their places in the list together)
    if (mine >= bound) {
#pragma unroll 2
        for (int i = tid; i < quads; i += T) {
            const float4 f = X4[i];
            const bool c[4] = {mag_key(f.x) >= bound, mag_key(f.y) >= bound, mag_key(f.z) >= bound, mag_key(f.w) >= bound};
            if (c[0] || c[1] || c[2] || c[3]) {
                unsigned at = atomicAdd(&s->n, (unsigned)c[0] + (unsigned)c[1] + (unsigned)c[2] + (unsigned)c[3]);
                const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (c[j] && at < (unsigned)CAND) s->cand[at] = make_uint2(__float_as_uint(v[j]), (unsigned)(4 * i + j));
                    at += c[j];
                }
            }
        }
    }
    __syncthreads();
    const int n = (int)s->n;
    if (n > CAND || n < k_eff) {
        select_radix(tile_offset(X), slot, rec, alpha);
        return;
    }
    // one warp finds the threshold, the others clear the tile
    if (tid < 32) {
        if (n <= 64)
            find_threshold<2>((unsigned)n, bound, k_eff);
        else if (n <= 128)
            find_threshold<4>((unsigned)n, bound, k_eff);
        else if (n <= 256)
            find_threshold<8>((unsigned)n, bound, k_eff);
        else
            find_threshold<16>((unsigned)n, bound, k_eff);
    }
    const int listed = first_listed(e);
    if (!dense && (T == 32 || tid >= 32)) {
        const int first = T == 32 ? tid : tid - 32, step = T == 32 ? 32 : T - 32;
        for (int i = first; i < quads; i += step) X4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (listed >= 0)
            for (int i = first; i < 512; i += step) s->bits()[i] = 0u;
        if (tid == T - 1 && listed >= 0) s->n_list = 0;
    }
    uint2 *kept = reinterpret_cast<uint2 *>(s->kept);
    if (tid == 0 && (k_eff & 1)) kept[k_eff] = make_uint2(0u, 0xffffffffu);  // completes the last pair: behind everything
    __syncthreads();
    const unsigned thr = s->thr, need_eq = s->need_eq;
    if (dense) {  // (thr < bound: exactly the candidates are kept)
        compact(tile_offset(X), slot, rec, alpha, thr < bound ? bound - 1u : thr, thr < bound ? 0u : need_eq);
        return;
    }
    const bool ties = need_eq != s->n_eq;
    for (int i = tid; i < n; i += T) {
        const uint2 c = s->cand[i];
        const unsigned mag = c.x & 0x7fffffffu;
        bool keep = mag >= thr;
        if (keep && ties && mag == thr) {  // equal keys straddle the k-th place: the lowest positions (in index order) are kept
            unsigned ahead = 0;
            for (int j = 0; j < n; ++j) ahead += (s->cand[j].x & 0x7fffffffu) == thr && s->cand[j].y < c.y;
            keep = ahead < need_eq;
        }
        if (keep) kept[atomicAdd(&s->n_kept, 1u)] = c;
    }
    __syncthreads();
    // a record's place is the number of kept positions below its own (tile positions are in index order)
    const int pairs = (k_eff + 1) >> 1;
    for (int i = tid; i < k_eff; i += T) {
        const uint2 c = kept[i];
        int pos = 0;
#pragma unroll 4
        for (int j = 0; j < pairs; ++j) {
            const uint4 q = s->kept[j];
            pos += (q.y < c.y ? 1 : 0) + (q.w < c.y ? 1 : 0);
        }
        DemoRecord r;
        r.idx = index_of(e, (int)c.y);
        r.val = __uint_as_float(c.x);
        rec[pos] = r;
        X[c.y] = alpha * r.val;
        if (listed >= 0) {  // the line's first place identifies it: the first axis has the largest stride
            const unsigned line = c.y % (unsigned)e.p[listed];
            if (!(atomicOr(&s->bits()[line >> 5], 1u << (line & 31u)) >> (line & 31u) & 1u)) s->list()[atomicAdd(&s->n_list, 1)] = line;
        }
    }
    __syncthreads();
}

// Decode: records of one of the two batches; place of a record outside its chunk; longest list that one warp adds.
constexpr int STAGE = CAND, WARP_K = 32;
constexpr unsigned SKIP = 0xffffffffu;
static_assert(offsetof(Shared, kept) == offsetof(Shared, cand) + STAGE * sizeof(uint2), "the batches are neighbours");

// Registers: 80 per thread (768 threads per SM); 128 with extents of 128.
constexpr int MAX_THREADS = 384, MAX_THREADS_BIG = 256;

template <typename GT, bool BIG>
__global__ void __launch_bounds__(BIG ? MAX_THREADS_BIG : MAX_THREADS, 2) compress_nd_kernel(DemoNdCompressArgs a)
{
    const StreamOrder order(a.wait_first);
    const View v = carve(a.cls, true);
    Shared *s = shared();
    float *tile0 = v.tile0, *tile1 = v.tile1;
    const int tid = threadIdx.x, T = blockDim.x;
    if (tid < 2) s->e[tid].chunk_begin = 1, s->e[tid].chunk_end = 0;  // no tensor yet
    __syncthreads();
    if (tid == 0 && blockIdx.x < a.cls.n_chunks) locate(s, 0, a.entries, a.cls.n, blockIdx.x);
    __syncthreads();
    int layout = -1, slot = 0;
    if (!BIG && blockIdx.x < a.cls.n_chunks) {  // (in the kernels of the large extents it spills registers of the loop below)
        layout = s->e[0].layout;
        enter_layout(v, s->e[0], a.cls);
        __syncthreads();
        prefetch_chunk(v, s->e[0], a.m_ptrs[s->e[0].tensor] + s->base[0]);
        prefetch_chunk(v, s->e[0], static_cast<const GT *>(a.g_ptrs[s->e[0].tensor]) + s->base[0]);
    }
    order.begin();

    for (long long c = blockIdx.x; c < a.cls.n_chunks; c = (long long)gridDim.x + s->ticket, slot ^= 1) {
        // cleared for this chunk's selection; the barriers up to it order the writes
        for (int i = tid; i < 256; i += T) s->hist[i] = s->fine[i] = 0u;
        if (tid == 0) s->hi = 0u, s->n = 0u, s->n_kept = 0u, s->n_list = -1;
        __syncthreads();
        const DemoNdEntry &e = s->e[slot];
        if (e.layout != layout) {
            layout = e.layout;
            enter_layout(v, e, a.cls);
            __syncthreads();
        }
        unsigned ticket = 0;  // (last thread) the CTA's next chunk, drawn now, looked up below
        if (tid == T - 1) ticket = ticket_draw(a.tickets);
        const size_t base = s->base[slot];
        float *__restrict__ m = a.m_ptrs[e.tensor] + base;
        const GT *__restrict__ g = static_cast<const GT *>(a.g_ptrs[e.tensor]) + base;

        // momentum update  B = beta*m + g  on the chunk (Algorithm 1, worker side)
        const bool whole = e.quads == 2;
        if (e.quads) {
            constexpr int U = BIG ? 2 : 4;
            float4 mv[U];
            decltype(grad_quad(g)) gv[U];
            for_quads<U>(
                v, e,
                [&](int j, unsigned off) {
                    mv[j] = *reinterpret_cast<const float4 *>(m + off);
                    gv[j] = grad_quad(g + off);
                },
                [&](int j, int i, unsigned, int t) {
                    const float4 gf = grad_floats(gv[j]);
                    const float4 b = make_float4(fmaf(a.beta, mv[j].x, gf.x), fmaf(a.beta, mv[j].y, gf.y), fmaf(a.beta, mv[j].z, gf.z),
                                                 fmaf(a.beta, mv[j].w, gf.w));
                    *reinterpret_cast<float4 *>(v.B + i) = b;
                    set_tile_quad(tile0, t, whole, b);
                });
        } else {
            constexpr int U = 8;
            float mv[U];
            GT gv[U];
            for_elements<U>(
                v, e,
                [&](int j, auto off) {
                    mv[j] = m[off];
                    gv[j] = g[off];
                },
                [&](int j, int i, auto, int t) {
                    const float b = fmaf(a.beta, mv[j], (float)gv[j]);
                    v.B[i] = b;
                    tile0[t] = b;
                });
        }
        if (tid == T - 1) take_ticket(s, slot ^ 1, a.entries, a.cls, ticket);
        __syncthreads();
        transform_chunk<false, BIG>(tile0, tile1, slot, a.tables, -1);  // Q = T(B; C_0, ..., C_{d-1})
        // the next chunk on its way to L2; not of small chunks, where going over the rows is a part of the work (4096 x 4096 in 8 x 16, two calls
        // 1397 us, 1337 without; in 16 x 32 523 / 521; but 28 M elements in 32 x 32 x 3 x 3 496 / 506)
        if (e.M >= 1024 && (long long)gridDim.x + s->ticket < a.cls.n_chunks && s->e[slot ^ 1].layout == layout) {
            const DemoNdEntry &ne = s->e[slot ^ 1];
            prefetch_chunk(v, ne, a.m_ptrs[ne.tensor] + s->base[slot ^ 1]);
            prefetch_chunk(v, ne, static_cast<const GT *>(a.g_ptrs[ne.tensor]) + s->base[slot ^ 1]);
        }
        select_topk(tile0, slot, a.payload + e.rec_begin + (c - e.chunk_begin) * (long long)e.k_eff, a.alpha);
        // momentum subtraction  m <- B - alpha * T(kept; C_0^T, ..., C_{d-1}^T)
        transform_chunk<true, BIG>(tile0, tile1, slot, a.tables, s->n_list);
        if (e.quads)
            for_quads<2>(v, e, [](int, unsigned) {}, [&](int, int i, unsigned off, int t) {
                const float4 b = *reinterpret_cast<const float4 *>(v.B + i), r = tile_quad(tile0, t, whole);
                *reinterpret_cast<float4 *>(m + off) = make_float4(b.x - r.x, b.y - r.y, b.z - r.z, b.w - r.w);
            });
        else
            for_elements<4>(v, e, [](int, auto) {}, [&](int, int i, auto off, int t) { m[off] = v.B[i] - tile0[t]; });
        __syncthreads();
    }
    if (tid == T - 1) ticket_finish(a.tickets);
}

template <bool BIG>
__global__ void __launch_bounds__(BIG ? MAX_THREADS_BIG : MAX_THREADS, 2) decode_nd_kernel(DemoNdDecodeArgs a)
{
    const StreamOrder order(a.wait_first);
    const View v = carve(a.cls, false);
    Shared *s = shared();
    float *tile0 = v.tile0, *tile1 = v.tile1;
    unsigned short *Cn = reinterpret_cast<unsigned short *>(v.tile0 + (size_t)a.cls.tile * (a.cls.dense_axes ? 2 : 1));  // senders (agg == 2)
    const int tid = threadIdx.x, T = blockDim.x;
    const bool counts = a.agg == 2;
    if (tid < 2) s->e[tid].chunk_begin = 1, s->e[tid].chunk_end = 0;
    __syncthreads();
    if (tid == 0 && blockIdx.x < a.cls.n_chunks) locate(s, 0, a.entries, a.cls.n, blockIdx.x);
    __syncthreads();
    int layout = -1, slot = 0;
    if (!BIG && blockIdx.x < a.cls.n_chunks) {  // (in the kernels of the large extents it spills registers of the loop below)
        layout = s->e[0].layout;
        enter_layout(v, s->e[0], a.cls);
        __syncthreads();
        if (!a.sign_ptrs) prefetch_chunk(v, s->e[0], a.x_ptrs[s->e[0].tensor] + s->base[0]);
    }
    order.begin();

    for (long long c = blockIdx.x; c < a.cls.n_chunks; c = (long long)gridDim.x + s->ticket, slot ^= 1) {
        __syncthreads();
        const DemoNdEntry &e = s->e[slot];
        if (e.layout != layout) {
            layout = e.layout;
            enter_layout(v, e, a.cls);
            __syncthreads();
        }
        unsigned ticket = 0;  // (last thread) the CTA's next chunk, drawn now, looked up below
        if (tid == T - 1) ticket = ticket_draw(a.tickets);
        const int M = e.M, k_eff = e.k_eff;
        const long long rec_off = e.rec_begin + (c - e.chunk_begin) * (long long)k_eff;

        // S = sum over workers in worker order (indices are unique inside one worker's chunk).  k <= STAGE: batches of several
        // workers' records come through two buffers, the next batch while this one is added; a thread turns the records that it
        // requested into tile positions, then one warp adds short lists and all threads long ones, with a barrier per worker.  Larger k:
        // straight from the payloads.  (One warp for every k, with the positions inside its serial loop: 2048 x 2048 in 32 x 128, W = 64,
        // k = 8 / 128 / 512 78 / 228 / 828 us instead of 44 / 107 / 236; W = 16, k = 256 111 instead of 60.)
        const int wb = STAGE / k_eff;
        auto request = [&](int w0, int buf) {
            const int n = min(wb, a.W - w0) * k_eff;  // (negative behind the last)
            for (int r = tid; r < n; r += T) {
                const int w = r / k_eff;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(s->cand + buf + r)),
                             "l"(a.payloads[w0 + w] + rec_off + (r - w * k_eff))
                             : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        if (wb) request(0, 0);
        for (int i = tid; i < e.tile >> 2; i += T) reinterpret_cast<float4 *>(tile0)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (counts)
            for (int i = tid; i < e.tile; i += T) Cn[i] = 0;
        if (tid == T - 1) take_ticket(s, slot ^ 1, a.entries, a.cls, ticket);
        auto position = [&](unsigned idx) {
            if (idx < (unsigned)M) return (unsigned)place_of(e, (int)idx).t;
            atomicMax(a.status, DEMO_DEV_PAYLOAD);
            return SKIP;
        };
        // several records of one worker, their tile accesses side by side
        auto add = [&](const uint2 (&r)[4]) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = r[u].x != SKIP ? tile0[r[u].x] : 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (r[u].x != SKIP) {
                    tile0[r[u].x] = v[u] + __uint_as_float(r[u].y);
                    if (counts) Cn[r[u].x] += 1;
                }
        };
        const uint2 none = make_uint2(SKIP, 0u);
        if (wb) {
            for (int w0 = 0, buf = 0; w0 < a.W; w0 += wb, buf ^= STAGE) {
                uint2 *stage = s->cand + buf;
                const int n = min(wb, a.W - w0) * k_eff;
                request(w0 + wb, buf ^ STAGE);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
                for (int r = tid; r < n; r += T) stage[r].x = position(stage[r].x);
                __syncthreads();  // (the first time: the tile is cleared too)
                if (k_eff <= WARP_K) {
                    if (tid < 32) {
                        for (int r0 = 0; r0 < n; r0 += 4 * k_eff) {  // four workers' records are read together
                            uint2 r[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int i = r0 + u * k_eff + tid;
                                r[u] = tid < k_eff && i < n ? stage[i] : none;
                            }
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (r[u].x != SKIP) {
                                    tile0[r[u].x] += __uint_as_float(r[u].y);
                                    if (counts) Cn[r[u].x] += 1;
                                }
                                __syncwarp();
                            }
                        }
                    }
                    __syncthreads();
                } else {
                    for (int r0 = 0; r0 < n; r0 += k_eff) {
                        for (int i0 = tid; i0 < k_eff; i0 += 4 * T) {
                            uint2 r[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) r[u] = i0 + u * T < k_eff ? stage[r0 + i0 + u * T] : none;
                            add(r);
                        }
                        __syncthreads();
                    }
                }
            }
        } else {
            __syncthreads();
            for (int w = 0; w < a.W; ++w) {
                const DemoRecord *rec = a.payloads[w] + rec_off;
                for (int i0 = tid; i0 < k_eff; i0 += 4 * T) {
                    uint2 r[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) r[u] = i0 + u * T < k_eff ? *reinterpret_cast<const uint2 *>(rec + i0 + u * T) : none;
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (i0 + u * T < k_eff) r[u].x = position(r[u].x);
                    add(r);
                }
                __syncthreads();
            }
        }
        if (counts) {  // Sparse Top-k Averaging: sum / number of senders, 0/0 = 0
            for (int i = tid; i < M; i += T) {
                const int t = place_of(e, i).t;
                const unsigned short n = Cn[t];
                if (n > 1) tile0[t] = tile0[t] / (float)n;
            }
            __syncthreads();
        }
        transform_chunk<true, BIG>(tile0, tile1, slot, a.tables, -1);
        if (a.sign_ptrs) {  // parameter-server form: hand out sign(R), the workers apply it
            signed char *__restrict__ sg = a.sign_ptrs[e.tensor] + s->base[slot];
            for_elements<4>(v, e, [](int, auto) {}, [&](int, int, auto off, int t) {
                const float rv = tile0[t];
                sg[off] = (signed char)((rv > 0.f) - (rv < 0.f));
            });
            continue;
        }
        // x <- x - lr * (phi(R) + wd * x), sign(0) = 0
        float *__restrict__ x = a.x_ptrs[e.tensor] + s->base[slot];
        auto updated = [&](float xv, float rv) {
            const float sg = a.phi ? rv * a.agg_scale : (float)((rv > 0.f) - (rv < 0.f));
            return fmaf(-a.lr, fmaf(a.wd, xv, sg), xv);
        };
        if (e.quads) {
            constexpr int U = BIG ? 2 : 4;
            float4 xv[U];
            for_quads<U>(
                v, e, [&](int j, unsigned off) { xv[j] = *reinterpret_cast<const float4 *>(x + off); },
                [&](int j, int, unsigned off, int t) {
                    const float4 r = tile_quad(tile0, t, e.quads == 2);
                    *reinterpret_cast<float4 *>(x + off) =
                        make_float4(updated(xv[j].x, r.x), updated(xv[j].y, r.y), updated(xv[j].z, r.z), updated(xv[j].w, r.w));
                });
            continue;
        }
        constexpr int U = 8;
        float xv[U];
        for_elements<U>(
            v, e, [&](int j, auto off) { xv[j] = x[off]; },
            [&](int j, int, auto off, int t) {
                x[off] = updated(xv[j], tile0[t]);
            });
    }
    if (tid == T - 1) ticket_finish(a.tickets);
}

template <typename K, typename A>
cudaError_t launch_nd(K kernel, size_t smem, DemoLaunch &dev, cudaStream_t stream, A args)
{
    const DemoNdClass &cls = args.cls;
    if (cls.n_chunks <= 0) return cudaSuccess;
    int per_sm = 0;
    const cudaError_t err = demo_resident_ctas(dev, (const void *)kernel, cls.threads, smem, &per_sm);
    if (err != cudaSuccess) return err;
    long long grid = (long long)dev.sm_count * per_sm;
    if (grid > cls.n_chunks) grid = cls.n_chunks;
    if (grid == cls.n_chunks) args.tickets = nullptr;
    void *params[] = {&args};
    return demo_launch_kernel((const void *)kernel, grid, cls.threads, smem, stream, params);
}

}  // namespace

int DemoNdTables::get(int s)
{
    if (of[s] >= 0) return of[s];
    of[s] = (int)data.size();
    const double pi = 3.141592653589793238462643383279502884;
    const int h = (s + 1) / 2, pe = up8(h), po = up8(s / 2);
    auto C = [&](int u, int n) {
        if ((u & 1) && 2 * n == s - 1) return 0.0;
        return std::sqrt((u == 0 ? 1.0 : 2.0) / s) * std::cos(pi * (2.0 * n + 1.0) * u / (2.0 * s));
    };
    for (int n = 0; n < h; ++n) {
        for (int j = 0; j < pe; ++j) data.push_back(2 * j < s ? (float)(C(2 * j, n) * (2 * n == s - 1 ? 0.5 : 1.0)) : 0.f);
        for (int j = 0; j < po; ++j) data.push_back(2 * j + 1 < s ? (float)C(2 * j + 1, n) : 0.f);
    }
    for (int u = 0; u < s; ++u)
        for (int n = 0; n < pe; ++n) data.push_back(n < h ? (float)C(u, n) : 0.f);
    return of[s];
}

// Tile strides: the innermost axis is dense, every outer stride may be padded by a few words.  The padding is the one with
// the fewest bank conflicts of a warp's accesses over the axis passes (32 neighbouring lines at a time), the smaller tile
// where that is equal; at most a sixteenth of the chunk (or 64 words) is spent on it, an eighth where it makes the rows whole quads.  The
// search takes 1 to 60 us of the host's time, 190 for 4 x 8 x 8 x 16, so tensors of the same chunk shape, whose rows are pieces of the tensor
// alike, share one.  (The lines' indices are found once: with the divisions in every trial, fourteen shapes took 1070 us instead of 550.)
void demo_nd_plan(DemoNdEntry *e, DemoNdTables *tables)
{
    const int *s = e->s;
    e->tail = s[2] == s[3] && s[3] >= 2 && s[3] <= 7 ? s[3] : 0;
    // how many trailing elements follow one another in the tensor and, with strides p, in the tile
    auto run_of = [&](const int *p) {
        long long run = 1;
        for (int a = DEMO_ND_DIMS - 1; a >= 0; --a) {
            if (s[a] > 1 && (e->stride[a] != run || p[a] != run)) break;
            run *= s[a];
        }
        return (int)run;
    };
    // 1: the rows are whole 16-byte pieces of the tensor, 2: of the tile too
    auto quads_of = [&](const int *p) {
        const int run = run_of(p);
        if (run % 4) return 0;
        bool tile = true;
        long long in = 1;  // elements of the axes behind a
        for (int a = DEMO_ND_DIMS - 1; a >= 0; --a) {
            if (e->c[a] > 1 && s[a] * e->stride[a] % 4) return 0;  // chunks start on a piece
            if (s[a] > 1 && in >= run) {
                if (e->stride[a] % 4) return 0;
                tile = tile && p[a] % 4 == 0;
            }
            in *= s[a];
        }
        return tile ? 2 : 1;
    };
    // The lines of the first, second and third warp of each axis pass, as indices along the axes (which the strides tried below do not change).
    struct Pass {
        bool pieces;  // may be 16 bytes per thread, eight threads at a time
        int weight, lines, index[96][DEMO_ND_DIMS];
    };
    auto passes_of = [&](Pass *passes) {
        int n = 0;
        for (int a = 0; a < DEMO_ND_DIMS; ++a) {
            if (s[a] == 1 || (e->tail && a == 3)) continue;
            const int last = e->tail && a == 2 ? 3 : a;
            Pass &q = passes[n++];
            q.pieces = a == 3 && s[a] % 4 == 0 && in_place_extent(s[a]) && s[a] <= 32;
            q.weight = last > a ? 2 : 1;
            q.lines = e->M / (s[a] * (last > a ? s[last] : 1));
            if (q.lines > 96) q.lines = 96;
            for (int l = 0; l < q.lines; ++l) {
                int r = l;
                for (int b = DEMO_ND_DIMS - 1; b >= 0; --b) {
                    const bool across = b < a || b > last;
                    q.index[l][b] = across ? r % s[b] : 0;
                    if (across) r /= s[b];
                }
            }
        }
        return n;
    };
    auto conflicts = [](const Pass *passes, int n, const int *p, bool whole) {
        long long cost = 0;
        for (const Pass *q = passes; q < passes + n; ++q) {
            const bool pieces = whole && q->pieces;
            const int lanes = pieces ? 8 : 32, banks = pieces ? 8 : 32;
            for (int first = 0; first < q->lines; first += 32) {
                unsigned char bank[32] = {0};
                int worst = 0;
                for (int l = first; l < q->lines && l < first + lanes; ++l) {
                    const int *x = q->index[l], t = x[0] * p[0] + x[1] * p[1] + x[2] * p[2] + x[3] * p[3];
                    const int v = ++bank[(pieces ? t >> 2 : t) & (banks - 1)];
                    worst = worst > v ? worst : v;
                }
                cost += worst * q->weight;
            }
        }
        // (rows that are not whole pieces cost four accesses instead of one where the chunk comes and goes)
        return 2 * cost + (whole ? 0 : 2);
    };
    // What quads_of reads of the tensor, so that a layout does not depend on which tensor of a chunk shape came first: the first axis from which
    // on the chunk is one piece of the tensor and the strides that are whole quads; 0 where chunks start off the pieces, whatever the tile.
    int rows = 1;
    {
        long long in = 1;
        int axis = DEMO_ND_DIMS;
        bool joined = true;
        for (int a = DEMO_ND_DIMS - 1; a >= 0; --a) {
            if (e->c[a] > 1 && s[a] * e->stride[a] % 4) rows = 0;
            joined = joined && (s[a] == 1 || e->stride[a] == in);
            if (joined) axis = a;
            if (rows && s[a] > 1 && e->stride[a] % 4 == 0) rows |= 16 << a;
            in *= s[a];
        }
        if (rows) rows |= axis << 1;
    }
    const DemoNdTables::Layout *known = nullptr;
    for (const DemoNdTables::Layout &l : tables->layouts)
        if (l.s[0] == s[0] && l.s[1] == s[1] && l.s[2] == s[2] && l.s[3] == s[3] && l.rows == rows) known = &l;
    const int room = e->M / 16 > 64 ? e->M / 16 : 64, room_quads = e->M / 8 > room ? e->M / 8 : room;
    long long best = -1;
    int p[DEMO_ND_DIMS];
    p[3] = 1;
    Pass passes[DEMO_ND_DIMS];
    const int n_passes = known ? 0 : passes_of(passes);
    for (int pad2 = 0; !known && pad2 <= (s[2] > 1 && !e->tail ? 8 : 0); ++pad2) {
        p[2] = s[3] + pad2;
        for (int pad1 = 0; pad1 <= (s[1] > 1 && s[2] * s[3] > 1 ? 8 : 0); ++pad1) {
            p[1] = p[2] * s[2] + pad1;
            for (int pad0 = 0; pad0 <= (s[0] > 1 && s[1] * s[2] * s[3] > 1 ? 31 : 0); ++pad0) {
                p[0] = p[1] * s[1] + pad0;
                const int floats = p[0] * s[0];
                if (floats > e->M + room_quads) break;
                const bool whole = rows && quads_of(p) == 2;
                if (floats > e->M + room && !whole) continue;
                const long long cost = conflicts(passes, n_passes, p, whole) * (1LL << 20) + floats;
                if (best < 0 || cost < best) {
                    best = cost;
                    for (int a = 0; a < DEMO_ND_DIMS; ++a) e->p[a] = p[a];
                    e->tile = (floats + 3) & ~3;
                }
            }
        }
    }
    if (known) {
        for (int a = 0; a < DEMO_ND_DIMS; ++a) e->p[a] = known->p[a];
        e->tile = known->tile;
    } else {
        DemoNdTables::Layout l;
        for (int a = 0; a < DEMO_ND_DIMS; ++a) {
            l.s[a] = s[a];
            l.p[a] = e->p[a];
        }
        l.tile = e->tile;
        l.rows = rows;
        tables->layouts.push_back(l);
    }
    long long span = 0;
    for (int a = 0; a < DEMO_ND_DIMS; ++a) span += (s[a] - 1) * e->stride[a];
    const int run = run_of(e->p);
    e->row = run;
    e->inv_row = run > 1 ? (unsigned)(((1ULL << 32) + (unsigned long long)run - 1) / (unsigned long long)run) : 0u;
    e->inv_row4 = run > 4 ? (unsigned)(((1ULL << 32) + (unsigned long long)run / 4 - 1) / (unsigned long long)(run / 4)) : 0u;
    e->row_table = e->M / run <= DEMO_ND_MAX_ROWS && span < (1LL << 32);
    e->quads = e->row_table ? quads_of(e->p) : 0;
    // threads: enough for every pass over the long axes in whole rounds, and for 32 elements each
    int threads = (e->M + 31) / 32;
    for (int a = 0; a < DEMO_ND_DIMS; ++a) {
        if (!in_place_extent(s[a])) e->basis[a] = tables->get(s[a]);
        if (s[a] <= 8) continue;
        int n = e->M / s[a];
        if (s[a] == 64 || s[a] == 128) n = (n + 31) / 32 * 64;
        if (!in_place_extent(s[a])) n = n * (up8((s[a] + 1) / 2) + up8(s[a] / 2)) / 8 / 2;
        const int rounds = (n + MAX_THREADS - 1) / MAX_THREADS;
        n = (n + rounds - 1) / rounds;
        threads = threads > n ? threads : n;
    }
    threads = (threads + 31) / 32 * 32;
    e->threads = threads > MAX_THREADS ? MAX_THREADS : threads;
}

// Chunks of a class are drawn from a 32-bit counter.
constexpr long long MAX_CLASS_CHUNKS = (1LL << 31) - 1;

// A class is a size bucket with or without extents of 128 (registers) and with or without dense axes (shared memory), so
// that a few chunks of one kind do not set the resources of all others.  Classes that would not fill the device (fewer than
// two chunks per SM) are merged, with one another and, where it has all that they need, with the largest of the others:
// a launch of its own costs more than the wider variant.
void demo_nd_classify(std::vector<DemoNdEntry> &entries, int sm_count, std::vector<DemoNdClass> *classes)
{
    struct Group {
        std::vector<DemoNdEntry> list;
        long long chunks = 0, elems = 0;
        DemoNdClass k{};
        void widen(const DemoNdClass &o)
        {
            k.max_M = k.max_M > o.max_M ? k.max_M : o.max_M;
            k.tile = k.tile > o.tile ? k.tile : o.tile;
            k.rows = k.rows > o.rows ? k.rows : o.rows;
            k.dense_axes |= o.dense_axes;
            k.big |= o.big;
        }
        void take(Group &o)
        {
            if (o.list.empty()) return;
            list.insert(list.end(), o.list.begin(), o.list.end());
            if (o.elems > elems) k.threads = o.k.threads;  // the CTA size of the larger
            chunks += o.chunks;
            elems += o.elems;
            widen(o.k);
            o = Group();
        }
    };
    Group g[16], rest;
    for (const DemoNdEntry &e : entries) {
        Group one;
        one.list.push_back(e);
        one.chunks = e.chunk_end;
        one.elems = e.chunk_end * e.M;
        one.k.threads = e.threads;
        one.k.max_M = (e.M + 3) & ~3;
        one.k.tile = e.tile;
        one.k.rows = e.row_table ? e.M / e.row : 0;
        for (int s : e.s) {
            one.k.big |= s == 128;
            one.k.dense_axes |= !in_place_extent(s);
        }
        const int bucket = e.M <= 512 ? 0 : e.M <= 2048 ? 1 : e.M <= 4096 ? 2 : 3;
        g[bucket * 4 + one.k.big * 2 + one.k.dense_axes].take(one);
    }
    Group *largest = nullptr;
    for (Group &d : g) {
        if (d.list.empty()) continue;
        if (d.chunks < 2LL * sm_count)
            rest.take(d);
        else if (!largest || d.elems > largest->elems)
            largest = &d;
    }
    if (largest && largest->k.max_M >= rest.k.max_M && largest->k.tile >= rest.k.tile && largest->k.big >= rest.k.big &&
        largest->k.dense_axes >= rest.k.dense_axes)
        largest->take(rest);
    entries.clear();
    classes->clear();
    auto same_layout = [](const DemoNdEntry &x, const DemoNdEntry &y) {
        for (int a = 0; a < DEMO_ND_DIMS; ++a)
            if (x.s[a] != y.s[a] || x.stride[a] != y.stride[a] || x.p[a] != y.p[a]) return false;
        return true;
    };
    auto emit_part = [&](const Group &d, size_t first, size_t last) {  // tensors first .. last - 1
        DemoNdClass k = d.k;
        k.first = (int)entries.size();
        k.n = (int)(last - first);
        k.n_chunks = 0;
        bool split = false;
        for (size_t i = first; i < last; ++i) {
            DemoNdEntry e = d.list[i];
            const long long n = e.chunk_end;
            e.chunk_begin = k.n_chunks;
            k.n_chunks += n;
            e.chunk_end = k.n_chunks;
            for (int s : e.s) split = split || s == 64 || s == 128;
            e.layout = k.n_chunks > n && same_layout(entries.back(), e) ? entries.back().layout : (int)entries.size();
            entries.push_back(e);
        }
        // chunks that leave the device's threads idle get more of them, down to eight elements each (256 chunks of 32 x 32, k = 32 / 128:
        // compress 21 / 56 -> 14 / 18 us, decode of 16 workers 18 / 37 -> 13 / 16)
        const long long places = (long long)sm_count * 2 * MAX_THREADS / k.n_chunks, useful = (k.max_M / 8 + 31) / 32 * 32;
        const long long more = (places < useful ? places : useful) / 32 * 32;
        if (more > k.threads) k.threads = (int)(more < MAX_THREADS ? more : MAX_THREADS);
        if (split) k.threads = (k.threads + 63) / 64 * 64;  // two warps per 32 lines
        if (k.big && k.threads > MAX_THREADS_BIG) k.threads = MAX_THREADS_BIG;
        classes->push_back(k);
    };
    auto emit = [&](const Group &d) {
        long long chunks = 0;
        size_t first = 0;
        for (size_t i = 0; i < d.list.size(); ++i) {
            if (chunks + d.list[i].chunk_end > MAX_CLASS_CHUNKS) {  // (no tensor is larger than that)
                emit_part(d, first, i);
                first = i;
                chunks = 0;
            }
            chunks += d.list[i].chunk_end;
        }
        if (first < d.list.size()) emit_part(d, first, d.list.size());
    };
    for (Group &d : g) emit(d);
    emit(rest);
}

cudaError_t demo_launch_compress_nd(const DemoNdCompressArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    const size_t smem = shared_bytes(a.cls, true);
    if (a.cls.big)
        return a.grad_bf16 ? launch_nd(compress_nd_kernel<__nv_bfloat16, true>, smem, dev, stream, a)
                           : launch_nd(compress_nd_kernel<float, true>, smem, dev, stream, a);
    return a.grad_bf16 ? launch_nd(compress_nd_kernel<__nv_bfloat16, false>, smem, dev, stream, a)
                       : launch_nd(compress_nd_kernel<float, false>, smem, dev, stream, a);
}

cudaError_t demo_launch_decode_nd(const DemoNdDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    const size_t smem = shared_bytes(a.cls, false) + (a.agg == 2 ? align16((size_t)a.cls.tile * 2) : 0);
    return a.cls.big ? launch_nd(decode_nd_kernel<true>, smem, dev, stream, a)
                     : launch_nd(decode_nd_kernel<false>, smem, dev, stream, a);
}
