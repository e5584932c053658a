// Tensor-core kernels for caller-supplied orthonormal bases, chunk size 64 (Section 4.2, "Choice of
// Linear Projections": identity, random orthonormal projection).  With an arbitrary basis P the chunk
// transform Q = P B P^T is a dense contraction with no fast factorisation, so it runs on the 5th
// generation tensor cores: tcgen05.mma (kind::tf32) with fp32 accumulators in tensor memory.
//
// A group of 128 threads works on a PAIR of chunks stacked to M = 128; a CTA holds four groups (one CTA per SM) that run
// independently.  What bounds the kernels is latency -- a pair is a serial chain of loads, MMAs, read-backs and
// the selection -- so the design is about how many pairs an SM can hold:
//   * the data operand lives in tensor memory, not in shared memory: thread (c, r) stores its vector as row (c, r) of A (64
//     columns, contracted) and reads its row of D (64 columns) back; the 128 columns of a group are all it needs because
//     the two parts of the 3xTF32 split go through the A columns one after the other: lo * hi, then hi * lo + hi * hi (24
//     MMAs of 128 x 64 x 8, small products first);
//   * the basis is the only operand in shared memory, hi + lo, K-major (contracts over the columns of P: forward) and MN-major
//     (over its rows: inverse), 64 KB for the CTA; a chunk adds one padded fp32 tile for the transposes and the lists of
//     the selection, 20 KB;
//   * the first forward stage contracts over i: thread (c, j) holds column j of B, read straight from global memory, one
//     coalesced row piece per load; a transpose through the tile gives the second stage its rows; the inverse's row stage is
//     k rank-1 updates on the CUDA cores (as in kernels_fast64.cu), its column stage one more tensor-core stage whose result
//     is column j of the residual update: loads and stores of the momentum are coalesced and B is formed again from L2.
// 4096 x 8192, bf16 gradients, two workers: compress k = 32 177 us, decode 102 us (185 and 108 before the look-up in front of the
// wait and the descriptors that move on; 378 and 236 us at
// k = 32 with both operands in shared memory, 64 KB per pair, two pairs per SM and four stages).  A third of compress
// is the two passes over the momentum: the next pair's tiles are brought to L2 during the selection and read 32 rows at a
// time (without: 199 us).  Every wait is bounded: on expiry the group records DEMO_DEV_TIMEOUT and stops, the CTA frees its
// tensor memory and returns.
#include <cuda_bf16.h>

#include "demo_internal.h"
#include "fast_common.cuh"
#include "launch.cuh"
#include "select64.cuh"

namespace {

using namespace fastk;
using namespace sel64;

constexpr int M = S * S;
constexpr int PAIR_THREADS = 128;
constexpr int BLK = 8192;                   // one [64 rows][128 bytes] operand block
constexpr int TMEM_COLS_PER_GROUP = 128;    // A: 64, D: 64
constexpr int TMEM_COLS = 512;

// shared memory (offsets from a 1024-byte aligned base): basis operands (hi, lo: 2 blocks each), chunk areas, barriers
constexpr int OFF_BM_HI = 0;                // MN-major operand
constexpr int OFF_BM_LO = 2 * BLK;
constexpr int OFF_BK_HI = 4 * BLK;          // K-major operand (compress)
constexpr int OFF_BK_LO = 6 * BLK;
constexpr int X_BYTES = S * XS * 4;
constexpr int chunk_bytes(bool wide) { return X_BYTES + 65 * 16 + S * 4 + (CAP + 8) * 12 + 64 + (wide ? 2 * (WCAP + 4) * 4 : 0); }
constexpr int bars_bytes = 4 * 8 + 4 * 4 + 16;  // mbarrier and drawn pair per group, tensor-memory slot

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ float tf32_rn(float v)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
    return __uint_as_float(r);
}

// Shared-memory matrix descriptor: start address, leading / stride byte offsets (all >> 4), descriptor
// version 1, layout 2 = 128-byte swizzle, 1 = 128-byte swizzle with 32-byte atoms.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t layout)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)layout << 61;
    return d;
}
// Instruction descriptor: D fp32, A (tensor memory) and B tf32, B K- or MN-major, N = 64, M = 128.
__host__ __device__ constexpr uint32_t instr_desc(int b_mn)
{
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)b_mn << 16) | ((uint32_t)(S >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// D += A * B with A in tensor memory.
__device__ __forceinline__ void umma_tf32(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// Byte offset of the 16-byte piece q (0..7) of row r in block (2c + cb): MN = true is the 32-byte-atom
// swizzle of MN-major TF32 operands, MN = false the plain 128-byte swizzle of K-major ones.
template <bool MN>
__device__ __forceinline__ uint32_t op_off(int c, int cb, int r, int q)
{
    if (MN) return (2 * c + cb) * BLK + r * 128 + ((((q >> 1) ^ (r & 3)) << 5) | ((q & 1) << 4));
    return (2 * c + cb) * BLK + r * 128 + ((q ^ (r & 7)) << 4);
}
// Piece p (four floats) of row r of the basis, split into the hi and lo operand tiles.
template <bool MN>
__device__ __forceinline__ void write_split(unsigned char *hi, unsigned char *lo, int r, int p, const float4 &h, const float4 &l)
{
    const uint32_t at = op_off<MN>(0, p >> 3, r, p & 7);
    *reinterpret_cast<float4 *>(hi + at) = h;
    *reinterpret_cast<float4 *>(lo + at) = l;
}

// One product, issued by one thread: D (+)= A * basis part, K = 64 in eight steps of 8 (8 columns of A; 32 bytes inside a
// 128-byte row of the K-major basis, second half of K one block further, or 8 K-rows of the MN-major one).  The descriptor is formed once
// and moved on: a thread that builds one per step takes longer than the tensor core for the product.  Rolled: unrolled, its temporaries
// spill the 64 values that every thread holds.
template <bool MN>
__device__ __forceinline__ void issue_product(uint32_t d_tmem, uint32_t a_tmem, uint32_t b, uint32_t acc)
{
    constexpr uint32_t idesc = instr_desc(MN);
    uint64_t desc = MN ? smem_desc(b, BLK, 512, 1) : smem_desc(b, 16, 1024, 2);  // (addresses stay below 2^18: no carry out of the field)
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
#pragma unroll 1
        for (int kk = 0; kk < 4; ++kk) {
            umma_tf32(d_tmem, a_tmem, desc, idesc, acc);
            acc = 1u;
            a_tmem += 8;
            desc += (MN ? 1024 : 32) >> 4;
        }
        if (!MN) desc += (BLK - 4 * 32) >> 4;
    }
}

// Common frame of both kernels: aligned shared memory, per-group mbarrier, tensor memory, split basis.
struct TcFrame {
    unsigned char *sm;         // aligned base
    unsigned *drawn;           // this group's next pair
    uint32_t bar;              // this group's mbarrier
    uint32_t tmem, a_addr, d_addr;  // base of the CTA's tensor memory; this thread's lane of A and of D
    uint32_t a_mma, d_mma;     // A and D of the group as MMA operands
    unsigned phase;
    int g, pt;                 // group, thread inside the group
};

template <int GROUPS>
__device__ __forceinline__ void tc_setup(TcFrame &f, unsigned char *raw, const float *basis, bool need_k_major, int chunk_area,
                                         const StreamOrder &order)
{
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t raw_s = smem_u32(raw);
    f.sm = raw + (((raw_s + 1023u) & ~1023u) - raw_s);
    f.g = tid / PAIR_THREADS;
    f.pt = tid % PAIR_THREADS;
    unsigned char *bars = f.sm + (need_k_major ? 8 : 4) * BLK + 2 * GROUPS * chunk_area;
    unsigned long long *bar_mem = reinterpret_cast<unsigned long long *>(bars);
    f.drawn = reinterpret_cast<unsigned *>(bars + 4 * 8) + f.g;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 4 * 8 + 4 * 4);
    f.bar = smem_u32(bar_mem + f.g);
    f.phase = 0;
    if (f.pt == 0) {
        mbar_init(f.bar, 1);
        fence_proxy_async();
    }
    order.begin();  // (the basis is written by earlier work)
    // (all threads: by 64 of them, a row each, decode of 1024 x 1024 takes 18.3 us instead of 17.9)
    for (int i = tid; i < S * S / 4; i += GROUPS * PAIR_THREADS) {
        const int r = i % S, p = i / S;
        const float4 v = __ldg(reinterpret_cast<const float4 *>(basis + r * S) + p);
        const float4 h = make_float4(tf32_rn(v.x), tf32_rn(v.y), tf32_rn(v.z), tf32_rn(v.w));
        const float4 l = make_float4(tf32_rn(v.x - h.x), tf32_rn(v.y - h.y), tf32_rn(v.z - h.z), tf32_rn(v.w - h.w));
        if (need_k_major) write_split<false>(f.sm + OFF_BK_HI, f.sm + OFF_BK_LO, r, p, h, l);
        write_split<true>(f.sm + OFF_BM_HI, f.sm + OFF_BM_LO, r, p, h, l);
    }
    fence_proxy_async();  // generic-proxy writes -> visible to the tensor core's reads
    f.tmem = tmem_alloc_cta(tmem_slot, TMEM_COLS);
    f.a_mma = f.tmem + (uint32_t)(f.g * TMEM_COLS_PER_GROUP);
    f.d_mma = f.a_mma + S;
    f.a_addr = f.a_mma + ((uint32_t)((warp & 3) * 32) << 16);
    f.d_addr = f.a_addr + S;
}

// One stage on the pair: v becomes this thread's row of (the pair's vectors) * basis, 3xTF32.  False if a wait expired.
template <bool MN>
__device__ __forceinline__ bool tc_stage(TcFrame &f, const SlotBarrier<PAIR_THREADS> &pb, float (&v)[S])
{
    const uint32_t b_hi = smem_u32(f.sm + (MN ? OFF_BM_HI : OFF_BK_HI)), b_lo = smem_u32(f.sm + (MN ? OFF_BM_LO : OFF_BK_LO));
    bool ok = true;
    auto product = [&](auto last) {
        tmem_wait_st();
        tc_fence_before();
        pb.sync();
        if (f.pt == 0) {
            tc_fence_after();
            issue_product<MN>(f.d_mma, f.a_mma, decltype(last)::value ? b_lo : b_hi, decltype(last)::value);
            if (decltype(last)::value) issue_product<MN>(f.d_mma, f.a_mma, b_hi, 1);
            umma_commit(f.bar);
        }
        ok = mbar_wait_bounded(f.bar, f.phase) && ok;
        f.phase ^= 1u;
        tc_fence_after();
    };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float w[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const float x = v[32 * h + i];
            v[32 * h + i] = tf32_rn(x);
            w[i] = tf32_rn(x - v[32 * h + i]);
        }
        tmem_st32(f.a_addr + 32 * h, w);
    }
    product(std::false_type{});  // lo * hi
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float w[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) w[i] = v[32 * h + i];
        tmem_st32(f.a_addr + 32 * h, w);
    }
    product(std::true_type{});  // hi * lo + hi * hi
    if (!pb.sync_and(ok)) return false;
    tc_fence_after();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float w[32];
        tmem_ld32(f.d_addr + 32 * h, w);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[32 * h + i] = w[i];
    }
    tc_fence_before();
    return true;
}

// Where a chunk lies; the entry index only grows.  MANY (more tensors than MANY_TENSORS): the walk over the table skips entries; an
// instantiation of its own, because in the kernels at the register limit the longer code costs 1 % of 4096 x 8192 even with one
// tensor.  (One entry after the other, one chunk per tensor: 1000 tensors compress 219 us instead of 31, 20000 8.1 ms instead of 0.49.)
constexpr int MANY_TENSORS = 32;
struct ChunkRef {
    int tensor, n1;
    size_t elem;         // of the tile's first element
    long long first_rec;
};
template <bool MANY>
__device__ __forceinline__ ChunkRef locate(const DemoTensorEntry *entries, int n, unsigned c, int k, int &e)
{
    if constexpr (MANY)
        e = demo_seek_entry(entries, n, e, c);
    else
        while (e + 1 < n && entries[e + 1].chunk_begin <= c) ++e;
    const DemoTensorEntry te = entries[e];
    const unsigned lc = (unsigned)(c - te.chunk_begin), k0 = lc / (unsigned)te.c1;
    ChunkRef r;
    r.tensor = te.tensor;
    r.n1 = te.n1;
    r.elem = ((size_t)k0 * (unsigned)te.n1 + (lc - k0 * (unsigned)te.c1)) * S;
    r.first_rec = te.rec_begin + (long long)lc * k;
    return r;
}

// Column of the tile that thread r owns: B = beta * m + g (Algorithm 1, worker side); every load of a warp is 128 (m) and 64
// or 128 (g) consecutive bytes.
template <int BATCH, typename GT, class Use>
__device__ __forceinline__ void each_b(const float *m, const GT *g, int n1, float beta, Use use)
{
#pragma unroll
    for (int i0 = 0; i0 < S; i0 += BATCH) {
        float mv[BATCH];
        GT gv[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            mv[i] = m[(size_t)(i0 + i) * n1];
            gv[i] = g[(size_t)(i0 + i) * n1];
        }
        fdct::static_for<0, BATCH>([&](auto i) { use(i0 + decltype(i)::value, fmaf(beta, mv[decltype(i)::value], to_f32(gv[decltype(i)::value]))); });
    }
}

__device__ __forceinline__ void read_row(const float *X, int r, float (&v)[S])
{
#pragma unroll
    for (int j4 = 0; j4 < S / 4; ++j4) {
        const float4 w = reinterpret_cast<const float4 *>(X + r * XS)[j4];
        v[4 * j4] = w.x;
        v[4 * j4 + 1] = w.y;
        v[4 * j4 + 2] = w.z;
        v[4 * j4 + 3] = w.w;
    }
}
__device__ __forceinline__ void write_row(float *X, int r, const float (&v)[S])
{
#pragma unroll
    for (int j4 = 0; j4 < S / 4; ++j4)
        reinterpret_cast<float4 *>(X + r * XS)[j4] = make_float4(v[4 * j4], v[4 * j4 + 1], v[4 * j4 + 2], v[4 * j4 + 3]);
}

// BIGK (k > TC_MAX_K_LISTED): selection from quarter-row maxima with the wide list (3 groups fit), both inverse stages dense.
// From the list / dense, 4096 x 4096, one worker: k = 44 118 / 127 us, k = 48 127 / 127 (part of the lists overflow: there is no room for a
// wide list); 1024 x 1024: 30 / 28 and 40 / 28 us.
constexpr int TC_MAX_K_LISTED = 44;
template <typename GT, int GROUPS, bool BIGK, bool MANY>
__global__ void __launch_bounds__(GROUPS *PAIR_THREADS, 1) compress_tc_kernel(DemoCompressArgs a)
{
    const StreamOrder order(a.wait_first);
    extern __shared__ unsigned char smem_raw[];
    constexpr int AREA = chunk_bytes(BIGK);
    const unsigned n_chunks = (unsigned)a.n_chunks, n_pairs = (n_chunks + 1u) / 2u;
    const int k_eff = a.k;
    // row `row` of a chunk's tiles on its way to L2; e0: an entry at or in front of the chunk's
    auto prefetch_row = [&](unsigned chunk, int row, int e0) {
        const ChunkRef nr = locate<MANY>(a.entries, a.n_entries, chunk, k_eff, e0);
        const size_t at = nr.elem + (size_t)row * nr.n1;
        const float *nm = a.m_ptrs[nr.tensor] + at;
        const GT *ng = static_cast<const GT *>(a.g_ptrs[nr.tensor]) + at;
        prefetch_l2(nm);
        prefetch_l2(nm + 32);
        prefetch_l2(ng);
        if (sizeof(GT) == 4) prefetch_l2(ng + 32);
    };
    {
        const unsigned first = 2u * (blockIdx.x * GROUPS + threadIdx.x / PAIR_THREADS) + (threadIdx.x >> 6 & 1);
        if (first < n_chunks) prefetch_row(first, threadIdx.x & 63, 0);
    }
    TcFrame f;
    tc_setup<GROUPS>(f, smem_raw, a.C, true, AREA, order);
    const int c = f.pt >> 6, r = f.pt & 63;
    const SlotBarrier<PAIR_THREADS> pb{1 + f.g};        // the 128 threads of the pair
    const int bar_id = 1 + GROUPS + 2 * f.g + c;
    const SlotBarrier<S> sb{bar_id};                    // the 64 threads of one chunk
    SlotMem sm;
    sm.raw = f.sm + 8 * BLK + (2 * f.g + c) * AREA;
    sm.X = reinterpret_cast<float *>(sm.raw);
    sm.recs4 = reinterpret_cast<int4 *>(sm.raw + X_BYTES);
    sm.tmax = reinterpret_cast<float *>(sm.recs4 + 65);
    sm.cand_idx = reinterpret_cast<int *>(sm.tmax + S);
    sm.cand_val = reinterpret_cast<float *>(sm.cand_idx + CAP + 8);
    sm.cand_key = reinterpret_cast<unsigned *>(sm.cand_val + CAP + 8);
    sm.misc = reinterpret_cast<unsigned *>(sm.cand_key + CAP + 8);
    sm.wkey = sm.misc + 16;  // (BIGK only)
    sm.widx = sm.wkey + WCAP + 4;
    constexpr int PAD_ROW = (X_BYTES + 65 * 16) / 4;  // the scratch line tmax[0..S) seen from X
    float *X = sm.X;
    bool ok = true;
    int e = 0;

    for (unsigned p = blockIdx.x * GROUPS + f.g; p < n_pairs;) {
        if (f.pt == 0) *f.drawn = gridDim.x * GROUPS + ticket_draw(a.tickets);  // (read by all behind the barriers below)
        const unsigned chunk = 2u * p + c;
        const bool valid = chunk < n_chunks;
        float v[S];
        ChunkRef cr{};
        float *m = nullptr;
        const GT *g = nullptr;
        if (valid) {
            cr = locate<MANY>(a.entries, a.n_entries, chunk, k_eff, e);
            m = a.m_ptrs[cr.tensor] + cr.elem + r;
            g = static_cast<const GT *>(a.g_ptrs[cr.tensor]) + cr.elem + r;
            each_b<32>(m, g, cr.n1, a.beta, [&](int i, float b) { v[i] = b; });
        } else {
#pragma unroll
            for (int i = 0; i < S; ++i) v[i] = 0.f;
        }
        // ---- Q = P B P^T: column j of B -> column j of P B -> row u of P B -> row u of Q ----------------------
        ok = tc_stage<false>(f, pb, v);
        if (!ok) break;
#pragma unroll
        for (int u = 0; u < S; ++u) X[u * XS + r] = v[u];
        sb.sync();
        read_row(X, r, v);
        ok = tc_stage<false>(f, pb, v);
        if (!ok) break;
        const unsigned next = *f.drawn;  // (written before the barriers of the stages; overwritten behind those below)
        // row r of the group's next tiles on its way to L2.  (Without a counter next is NO_TICKET = 2^31 behind the grid, which then has a
        // group for every pair: 2 next wraps to twice the grid's groups, past the last chunk.)
        if (2u * next + c < n_chunks) prefetch_row(2u * next + c, r, e);

        // ---- exact top-k, records, and the row stage of the inverse -------------------------------------------
        if constexpr (BIGK) {
            if (valid) {
                select_chunk_big<false>(sm, v, k_eff, a.payload + cr.first_rec, a.alpha, r, sb, bar_id);
                sb.sync();
                float w[S];
                read_row(X, r, w);  // (core order)
                fdct::static_for<0, S>([&](auto q) { v[fdct::core_index<S>(decltype(q)::value)] = w[decltype(q)::value]; });
            }
            ok = tc_stage<true>(f, pb, v);  // row u of S P
            if (!ok) break;
            write_row(X, r, v);
            sb.sync();
#pragma unroll
            for (int u = 0; u < S; ++u) v[u] = X[u * XS + r];
        } else if (valid) {
            select_chunk<false, false>(sm, v, k_eff, a.payload + cr.first_rec, a.alpha, r, sb, bar_id, PAD_ROW);
            sb.sync();  // records complete, tile cleared
            // T[u][r] = sum over kept (u, w) of alpha * val * P[w][r]: running sums stored after every entry (kernels_fast64.cu)
            float acc = 0.f;
            float *Xt = X + r;
            int4 nx = sm.recs4[0];
#pragma unroll 1
            for (int r0 = 0; r0 < k_eff; r0 += 8) {
                int4 rc[9];
                float cv[8];
                rc[0] = nx;
#pragma unroll
                for (int j = 1; j < 9; ++j) rc[j] = sm.recs4[r0 + j];
                nx = rc[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) cv[j] = __ldg(a.C + (unsigned)(rc[j].y + r));
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    acc = fmaf(__int_as_float(rc[j].z), cv[j], acc);
                    Xt[rc[j].x] = acc;
                    acc = (rc[j].x != rc[j + 1].x) ? 0.f : acc;
                }
            }
#pragma unroll
            for (int u = 0; u < S; ++u) v[u] = Xt[u * XS];  // (written by this thread only)
        }
        // ---- column stage; momentum subtraction  m <- B - alpha R  (Section 2.1) --------------------------------
        ok = tc_stage<true>(f, pb, v);
        if (!ok) break;
        if (valid) each_b<BIGK ? 16 : 8>(m, g, cr.n1, a.beta, [&](int i, float b) { m[(size_t)i * cr.n1] = b - v[i]; });
        p = next;
    }
    if (!ok && f.pt == 0) atomicMax(a.status, DEMO_DEV_TIMEOUT);
    if (f.pt == 0) ticket_finish(a.tickets, GROUPS);
    tmem_free_cta(f.tmem, TMEM_COLS);
}

template <int GROUPS, bool MANY>
__global__ void __launch_bounds__(GROUPS *PAIR_THREADS, 1) decode_tc_kernel(DemoDecodeArgs a)
{
    const StreamOrder order(a.wait_first);
    extern __shared__ unsigned char smem_raw[];
    constexpr bool counts = GROUPS == 3;  // the count-normalised mean: its counters leave room for three groups
    const int area = X_BYTES + (counts ? M * 2 : 0);
    const unsigned n_chunks = (unsigned)a.n_chunks, n_pairs = (n_chunks + 1u) / 2u;
    const int k_eff = a.k;
    // row `row` of a chunk's x tile on its way to L2
    auto prefetch_row = [&](const ChunkRef &cr, int row) {
        const float *xr = a.x_ptrs[cr.tensor] + cr.elem + (size_t)row * cr.n1;
        prefetch_l2(xr);
        prefetch_l2(xr + 32);
    };
    {
        const unsigned first = 2u * (blockIdx.x * GROUPS + threadIdx.x / PAIR_THREADS) + (threadIdx.x >> 6 & 1);
        int e0 = 0;
        if (first < n_chunks) prefetch_row(locate<MANY>(a.entries, a.n_entries, first, k_eff, e0), threadIdx.x & 63);
    }
    TcFrame f;
    tc_setup<GROUPS>(f, smem_raw, a.C, false, area, order);
    const int c = f.pt >> 6, r = f.pt & 63, lane = f.pt & 31, warp = (f.pt >> 5) & 1;
    const SlotBarrier<PAIR_THREADS> pb{1 + f.g};
    const SlotBarrier<S> sb{1 + GROUPS + 2 * f.g + c};
    float *X = reinterpret_cast<float *>(f.sm + 4 * BLK + (2 * f.g + c) * area);
    unsigned short *Cn = reinterpret_cast<unsigned short *>(X + S * XS);  // senders per coordinate (agg == 2)
    bool ok = true;
    int e = 0;

    for (unsigned p = blockIdx.x * GROUPS + f.g; p < n_pairs;) {
        if (f.pt == 0) *f.drawn = gridDim.x * GROUPS + ticket_draw(a.tickets);
        const unsigned chunk = 2u * p + c;
        const bool valid = chunk < n_chunks;
        float v[S];
        float *x = nullptr;
        ChunkRef cr{};
#pragma unroll
        for (int j = 0; j < S; ++j) v[j] = 0.f;
        if (valid) {
            cr = locate<MANY>(a.entries, a.n_entries, chunk, k_eff, e);
            x = a.x_ptrs[cr.tensor] + cr.elem + r;
            prefetch_row(cr, r);
            write_row(X, r, v);
            if (counts)
                for (int i = 0; i < S; ++i) Cn[r * S + i] = 0;
            // S = sum over workers in worker order (Decompress&Aggregate).  k <= 64: every warp reads all records and adds those
            // of its 32 rows (warp-level order); more: a barrier per worker fixes the order of the additions.
            const DemoRecord *const *payloads = a.payloads;
            if (k_eff <= 64) {
                __syncwarp();  // the warp's rows are cleared
                const int spare = r * XS + S + (lane >> 3);
                bool bad = false;
                auto add = [&](const DemoRecord &rc, bool have) {
                    const unsigned idx = (unsigned)rc.idx;
                    bad = bad || (have && idx >= (unsigned)M);
                    const bool mine = have && (idx >> 11) == (unsigned)warp;
                    const int at = mine ? (int)(idx >> LOG2S) * XS + (int)(idx & (S - 1)) : spare;
                    X[at] += rc.val;
                    if (counts && mine) Cn[idx] += 1;
                };
                for (int w0 = 0; w0 < a.W; w0 += 4) {
                    DemoRecord r0[4], r1[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const DemoRecord *src = payloads[min(w0 + u, a.W - 1)] + cr.first_rec;
                        r0[u] = src[min(lane, k_eff - 1)];
                        if (k_eff > 32) r1[u] = src[min(lane + 32, k_eff - 1)];
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        add(r0[u], lane < k_eff && w0 + u < a.W);
                        if (k_eff > 32) add(r1[u], lane + 32 < k_eff && w0 + u < a.W);
                        __syncwarp();
                    }
                }
                if (bad) atomicMax(a.status, DEMO_DEV_PAYLOAD);
            } else {
                sb.sync();
                for (int w = 0; w < a.W; ++w) {
                    const DemoRecord *rec = payloads[w] + cr.first_rec;
                    for (int i = r; i < k_eff; i += S) {
                        const DemoRecord rc = rec[i];
                        if ((unsigned)rc.idx < (unsigned)M) {
                            X[(rc.idx >> LOG2S) * XS + (rc.idx & (S - 1))] += rc.val;
                            if (counts) Cn[rc.idx] += 1;
                        } else {
                            atomicMax(a.status, DEMO_DEV_PAYLOAD);
                        }
                    }
                    sb.sync();
                }
            }
            read_row(X, r, v);  // (k <= 64: written by this warp only)
            if (counts) {  // Sparse Top-k Averaging: sum / number of senders, 0/0 = 0
#pragma unroll
                for (int j = 0; j < S; ++j) {
                    const unsigned short n = Cn[r * S + j];
                    if (n > 1) v[j] = v[j] / (float)n;
                }
            }
        }
        // ---- R = P^T S P: row u of S -> row u of S P -> column j of S P -> column j of R; x <- x - lr (phi(R) + wd x)
        ok = tc_stage<true>(f, pb, v);
        if (!ok) break;
        const unsigned next = *f.drawn;  // (written before the barriers of this stage, overwritten behind the next one's)
        write_row(X, r, v);
        sb.sync();
#pragma unroll
        for (int u = 0; u < S; ++u) v[u] = X[u * XS + r];
        ok = tc_stage<true>(f, pb, v);
        if (!ok) break;
        if (valid) {
#pragma unroll
            for (int i0 = 0; i0 < S; i0 += 16) {
                float xv[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) xv[i] = x[(size_t)(i0 + i) * cr.n1];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float rv = v[i0 + i];
                    const float sg = a.phi ? rv * a.agg_scale : (float)((rv > 0.f) - (rv < 0.f));
                    x[(size_t)(i0 + i) * cr.n1] = fmaf(-a.lr, fmaf(a.wd, xv[i], sg), xv[i]);
                }
            }
        }
        p = next;
    }
    if (!ok && f.pt == 0) atomicMax(a.status, DEMO_DEV_TIMEOUT);
    if (f.pt == 0) ticket_finish(a.tickets, GROUPS);
    tmem_free_cta(f.tmem, TMEM_COLS);
}

template <typename K, typename A>
cudaError_t launch_tc(K kernel, int groups, int smem, A a, DemoLaunch &dev, cudaStream_t stream)
{
    if (a.n_chunks <= 0) return cudaSuccess;
    const cudaError_t err = demo_allow_smem(dev, (const void *)kernel);
    if (err != cudaSuccess) return err;
    const long long n_ctas = ((a.n_chunks + 1) / 2 + groups - 1) / groups;
    const long long grid = n_ctas < dev.sm_count ? n_ctas : dev.sm_count;  // one CTA per SM: it takes all of the tensor memory
    if (grid == n_ctas) a.tickets = nullptr;
    void *params[] = {&a};
    return demo_launch_kernel((const void *)kernel, grid, groups * PAIR_THREADS, (size_t)smem, stream, params);
}

}  // namespace

bool demo_tc_supported(int s) { return s == S; }

cudaError_t demo_launch_compress_tc(const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    constexpr int FIXED = 8 * BLK + bars_bytes + 1024;  // (last: alignment slack)
    auto pick = [&](auto gt, auto many) {
        using GT = decltype(gt);
        constexpr bool MANY = decltype(many)::value;
        return a.k > TC_MAX_K_LISTED ? launch_tc(compress_tc_kernel<GT, 3, true, MANY>, 3, FIXED + 6 * chunk_bytes(true), a, dev, stream)
                                  : launch_tc(compress_tc_kernel<GT, 4, false, MANY>, 4, FIXED + 8 * chunk_bytes(false), a, dev, stream);
    };
    if (a.n_entries > MANY_TENSORS)
        return a.grad_bf16 ? pick(__nv_bfloat16{}, std::true_type{}) : pick(float{}, std::true_type{});
    return a.grad_bf16 ? pick(__nv_bfloat16{}, std::false_type{}) : pick(float{}, std::false_type{});
}

cudaError_t demo_launch_decode_tc(const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    constexpr int FIXED = 4 * BLK + bars_bytes + 1024;
    auto pick = [&](auto many) {
        constexpr bool MANY = decltype(many)::value;
        if (a.agg == 2)  // the sender counts leave room for three groups
            return launch_tc(decode_tc_kernel<3, MANY>, 3, FIXED + 6 * (X_BYTES + M * 2), a, dev, stream);
        return launch_tc(decode_tc_kernel<4, MANY>, 4, FIXED + 8 * X_BYTES, a, dev, stream);
    };
    return a.n_entries > MANY_TENSORS ? pick(std::true_type{}) : pick(std::false_type{});
}
