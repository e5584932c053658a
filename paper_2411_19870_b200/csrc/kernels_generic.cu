// Generic kernels of the DeMo optimizer transform: s x s tiles of any chunk size s in {8,16,32,64,128}, any basis,
// any k <= M.  One CTA works on one chunk at a time; the chunk stays in shared
// memory from the momentum update to the residual write-back, so HBM is touched once per operand.
// The chunk DCT here is the dense contraction with the precomputed basis (the paper's own cost
// model, Section 2.1 "Complexity Analysis"); the register-resident fast-DCT kernels live in kernels_fast*.cu and
// kernels_small.cu.  These kernels are the path for caller-supplied bases where there is no tensor-core kernel and the
// cross-check of the fast path (DEMO_PATH_GENERIC).
#include <cuda_bf16.h>

#include "demo_internal.h"
#include "generic_common.cuh"

namespace {

// out[r][c] = sum_t L[r*lsr + t*lst] * R[t*rst + c*rsc]   (r < NR, c < NC, t < NT; out row-major)
template <int NR, int NC, int NT>
__device__ __forceinline__ void mm(float *__restrict__ out, const float *__restrict__ L, int lsr, int lst,
                                   const float *__restrict__ R, int rst, int rsc)
{
    constexpr int TR = (NR >= 4) ? 4 : 1;
    constexpr int TC = 4;
    constexpr int tiles_c = NC / TC;
    constexpr int n_tiles = (NR / TR) * tiles_c;
    for (int tile = threadIdx.x; tile < n_tiles; tile += GEN_THREADS) {
        const int r0 = (tile / tiles_c) * TR, c0 = (tile % tiles_c) * TC;
        float acc[TR][TC];
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) acc[i][j] = 0.f;
#pragma unroll 4
        for (int t = 0; t < NT; ++t) {
            float l[TR], rr[TC];
#pragma unroll
            for (int i = 0; i < TR; ++i) l[i] = L[(r0 + i) * lsr + t * lst];
#pragma unroll
            for (int j = 0; j < TC; ++j) rr[j] = R[t * rst + (c0 + j) * rsc];
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(l[i], rr[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) out[(r0 + i) * NC + c0 + j] = acc[i][j];
    }
}

// Forward chunk transform  Q = C B C^T.  Result in `q_out`, `tmp` is scratch.
template <int S>
__device__ __forceinline__ void forward_dct(const float *Bt, float *tmp, float *q_out, const float *C)
{
    mm<S, S, S>(tmp, Bt, S, 1, C, 1, S);  // tmp[i][v] = sum_j B[i][j] C[v][j]
    __syncthreads();
    mm<S, S, S>(q_out, C, S, 1, tmp, S, 1);  // Q[u][v] = sum_i C[u][i] tmp[i][v]
    __syncthreads();
}

// Inverse chunk transform  R = C^T Q C.  Result in `r_out`, `tmp` is scratch.
template <int S>
__device__ __forceinline__ void inverse_dct(const float *Qt, float *tmp, float *r_out, const float *C)
{
    mm<S, S, S>(tmp, Qt, S, 1, C, S, 1);   // tmp[u][j] = sum_v Q[u][v] C[v][j]
    __syncthreads();
    mm<S, S, S>(r_out, C, 1, S, tmp, S, 1);   // R[i][j] = sum_u C[u][i] tmp[u][j]
    __syncthreads();
}

template <int S>
__global__ void __launch_bounds__(GEN_THREADS) compress_generic_kernel(DemoCompressArgs a)
{
    const StreamOrder order(a.wait_first);
    order.begin();
    constexpr int M = S * S;
    extern __shared__ float smem[];
    float *Bt = smem;
    float *X1 = Bt + M;
    float *X2 = X1 + M;
    unsigned *hist = reinterpret_cast<unsigned *>(X2 + M);  // [256]
    unsigned *warp_tot = hist + 256;                        // [8]
    unsigned *s_state = warp_tot + 8;                       // [2]
    const int tid = threadIdx.x;

    for (long long c = blockIdx.x; c < a.n_chunks; c += gridDim.x) {
        const DemoTensorEntry te = a.entries[demo_find_entry(a.entries, a.n_entries, c)];
        const long long lc = c - te.chunk_begin;
        const long long k0 = lc / te.c1;
        const int k1 = (int)(lc - k0 * te.c1);
        const size_t base = (size_t)k0 * S * (size_t)te.n1 + (size_t)k1 * S;
        float *__restrict__ m = a.m_ptrs[te.tensor];
        const void *g = a.g_ptrs[te.tensor];
        const int k_eff = te.k_eff;

        // momentum update  B = beta*m + g  on the chunk (Algorithm 1, worker side)
        for (int i = tid; i < M; i += GEN_THREADS) {
            const int r = i / S, j = i - r * S;
            const size_t off = base + (size_t)r * te.n1 + j;
            const float gv = a.grad_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(g)[off])
                                         : reinterpret_cast<const float *>(g)[off];
            Bt[i] = fmaf(a.beta, m[off], gv);
        }
        __syncthreads();

        float *Q = X2;  // coefficients
        float *O = X1;  // the other buffer
        forward_dct<S>(Bt, X1, Q, a.C);

        // top-k: threshold by radix select, then index-ordered compaction into the payload
        unsigned thr, need_eq;
        radix_select(Q, M, k_eff, hist, s_state, &thr, &need_eq);
        constexpr int PER = (M + GEN_THREADS - 1) / GEN_THREADS;
        const int start = tid * PER;
        unsigned gt = 0, eq = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int i = start + j;
            if (i < M) {
                const unsigned key = mag_key(Q[i]);
                gt += key > thr;
                eq += key == thr;
            }
        }
        const unsigned before = block_exclusive_scan(gt | (eq << 16), warp_tot);
        unsigned gb = before & 0xffffu, eb = before >> 16;
        DemoRecord *rec = a.payload + te.rec_begin + lc * (long long)k_eff;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int i = start + j;
            if (i < M) {
                const float v = Q[i];
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
                O[i] = sel ? a.alpha * v : 0.f;  // the residual removes alpha times the kept part
            }
        }
        __syncthreads();

        // momentum subtraction  m <- B - IDCT(kept coefficients)
        float *R = O;
        inverse_dct<S>(O, Q, R, a.C);
        for (int i = tid; i < M; i += GEN_THREADS) {
            const int r = i / S, j = i - r * S;
            m[base + (size_t)r * te.n1 + j] = Bt[i] - R[i];
        }
        __syncthreads();
    }
}

template <int S>
__global__ void __launch_bounds__(GEN_THREADS) decode_generic_kernel(DemoDecodeArgs a)
{
    const StreamOrder order(a.wait_first);
    order.begin();
    constexpr int M = S * S;
    extern __shared__ float smem[];
    float *St = smem;
    float *X1 = St + M;
    unsigned short *Cn = reinterpret_cast<unsigned short *>(X1 + M);  // [M] senders per coordinate (agg == 2 only)
    const int tid = threadIdx.x;
    const bool counts = a.agg == 2;

    for (long long c = blockIdx.x; c < a.n_chunks; c += gridDim.x) {
        const DemoTensorEntry te = a.entries[demo_find_entry(a.entries, a.n_entries, c)];
        const long long lc = c - te.chunk_begin;
        const long long k0 = lc / te.c1;
        const int k1 = (int)(lc - k0 * te.c1);
        const size_t base = (size_t)k0 * S * (size_t)te.n1 + (size_t)k1 * S;
        float *__restrict__ x = a.x_ptrs[te.tensor];
        const int k_eff = te.k_eff;
        const long long rec_off = te.rec_begin + lc * (long long)k_eff;

        for (int i = tid; i < M; i += GEN_THREADS) {
            St[i] = 0.f;
            if (counts) Cn[i] = 0;
        }
        __syncthreads();
        // aggregate: S = sum over workers, in worker order (Decompress&Aggregate); indices are
        // unique inside one worker's chunk, so a barrier per worker fixes the summation order
        for (int w = 0; w < a.W; ++w) {
            const DemoRecord *rec = a.payloads[w] + rec_off;
            for (int i = tid; i < k_eff; i += GEN_THREADS) {
                const DemoRecord r = rec[i];
                if ((unsigned)r.idx < (unsigned)M) {
                    St[r.idx] += r.val;
                    if (counts) Cn[r.idx] += 1;
                } else {
                    atomicMax(a.status, DEMO_DEV_PAYLOAD);
                }
            }
            __syncthreads();
        }
        if (counts) {  // Sparse Top-k Averaging: sum / number of senders, 0/0 = 0
            for (int i = tid; i < M; i += GEN_THREADS) {
                const unsigned short n = Cn[i];
                if (n > 1) St[i] = St[i] / (float)n;
            }
            __syncthreads();
        }
        float *R = St;
        inverse_dct<S>(St, X1, R, a.C);
        // x <- x - lr * (sign(R) + wd * x), sign(0) = 0
        for (int i = tid; i < M; i += GEN_THREADS) {
            const int r = i / S, j = i - r * S;
            const size_t off = base + (size_t)r * te.n1 + j;
            const float rv = R[i];
            if (a.sign_ptrs) {  // parameter-server form: hand out sign(R), the workers apply it
                a.sign_ptrs[te.tensor][off] = (signed char)((rv > 0.f) - (rv < 0.f));
                continue;
            }
            const float sg = a.phi ? rv * a.agg_scale : (float)((rv > 0.f) - (rv < 0.f));
            const float xv = x[off];
            x[off] = fmaf(-a.lr, fmaf(a.wd, xv, sg), xv);
        }
        __syncthreads();
    }
}

// x <- x - lr (sign + wd x) with the signs a parameter server handed out (Algorithm 1, last two lines); same arithmetic as
// the decode kernels.  Bound by HBM (9 bytes per parameter).  Four consecutive elements per thread.
// BLOCKS: a block takes pieces of 1024 elements of one tensor, a grid apart, and looks the tensor up once per piece (168 matrices,
// 454 M parameters: 632 us, 6.5 TB/s, against 780 us with a search for every four elements; pieces of 8 or 16 elements per thread,
// with their loads together, 7 % longer).  Otherwise a thread takes pieces of four elements and searches for each: for sets whose
// small tensors would leave blocks mostly idle (20000 vectors of 8 / 64 / 128 elements 5.5 / 8.2 / 11 us against 158 with a block per
// vector).
template <bool BLOCKS>
__global__ void __launch_bounds__(GEN_THREADS) apply_signs_kernel(DemoApplySignsArgs a)
{
    constexpr int PIECE = demo_apply_pieces[BLOCKS ? 0 : 1];
    static_assert(PIECE == (BLOCKS ? 4 * GEN_THREADS : 4), "four elements per thread");
    const int lane = threadIdx.x & 31, at = BLOCKS ? (int)threadIdx.x * 4 : 0;
    const long long first = BLOCKS ? blockIdx.x : (long long)blockIdx.x * GEN_THREADS + threadIdx.x;
    const long long stride = BLOCKS ? gridDim.x : (long long)gridDim.x * GEN_THREADS;
    int e = 0;  // the last entry with piece_begin <= q
    auto update = [&](float xv, signed char s) { return fmaf(-a.lr, fmaf(a.wd, xv, (float)s), xv); };
    for (long long q = first; q < a.n_pieces; q += stride) {
        auto below = [&](int i) { return a.entries[i].piece_begin <= q; };
        if constexpr (BLOCKS) {
            const int next = e + 1 + lane, n = __popc(__ballot_sync(0xffffffffu, next < a.n_entries && below(next)));
            e += n;
            if (n == 32) e = demo_find_warp(e, a.n_entries - e, below);
        } else {
            int hi = a.n_entries - 1;
            while (e < hi) {
                const int mid = (e + hi + 1) >> 1;
                if (below(mid))
                    e = mid;
                else
                    hi = mid - 1;
            }
        }
        const DemoFlatEntry en = a.entries[e];
        const long long i0 = (q - en.piece_begin) * PIECE, left = en.n - i0;
        float *__restrict__ x = a.x_ptrs[en.tensor] + i0;
        const signed char *__restrict__ sg = a.sign_ptrs[en.tensor] + i0;
        if (left >= PIECE) {  // tensors start 16-byte aligned, so the pieces are aligned too
            const float4 xv = *reinterpret_cast<const float4 *>(x + at);
            const char4 sv = *reinterpret_cast<const char4 *>(sg + at);
            *reinterpret_cast<float4 *>(x + at) = make_float4(update(xv.x, sv.x), update(xv.y, sv.y), update(xv.z, sv.z), update(xv.w, sv.w));
        } else {
            for (int i = BLOCKS ? threadIdx.x : 0; i < (int)left; i += BLOCKS ? GEN_THREADS : 1) x[i] = update(x[i], sg[i]);
        }
    }
}

template <int S>
cudaError_t compress_dispatch(const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    const size_t extra = (256 + 8 + 2) * sizeof(unsigned);
    return launch_persistent(compress_generic_kernel<S>, 3 * S * S * sizeof(float) + extra, a.n_chunks, dev, stream, &a);
}

template <int S>
cudaError_t decode_dispatch(const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    return launch_persistent(decode_generic_kernel<S>, 2 * S * S * sizeof(float) + S * S * 2, a.n_chunks, dev, stream, &a);
}

}  // namespace

cudaError_t demo_launch_compress_generic(int s, const DemoCompressArgs &a, DemoLaunch &dev,
                                         cudaStream_t stream)
{
    switch (s) {
        case 8: return compress_dispatch<8>(a, dev, stream);
        case 16: return compress_dispatch<16>(a, dev, stream);
        case 32: return compress_dispatch<32>(a, dev, stream);
        case 64: return compress_dispatch<64>(a, dev, stream);
        case 128: return compress_dispatch<128>(a, dev, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t demo_launch_apply_signs(const DemoApplySignsArgs &a, DemoLaunch &dev, cudaStream_t stream)
{
    if (a.n_pieces <= 0) return cudaSuccess;
    const bool blocks = a.piece == demo_apply_pieces[0];
    const auto kernel = blocks ? apply_signs_kernel<true> : apply_signs_kernel<false>;
    const long long need = blocks ? a.n_pieces : (a.n_pieces + GEN_THREADS - 1) / GEN_THREADS;
    int per_sm = 0;
    const cudaError_t err = demo_resident_ctas(dev, (const void *)kernel, GEN_THREADS, 0, &per_sm);
    if (err != cudaSuccess) return err;
    long long grid = (long long)dev.sm_count * per_sm;
    if (grid > need) grid = need;
    // An ordinary launch: resident beside the last CTAs of decode_signs, these would keep that kernel's split of the SM into
    // shared memory and L1 to their end, and the L1 left (28 KB) does not hold the loads in flight (632 -> about 830 us).
    kernel<<<(unsigned)grid, GEN_THREADS, 0, stream>>>(a);
    return cudaGetLastError();
}

cudaError_t demo_launch_decode_generic(int s, const DemoDecodeArgs &a, DemoLaunch &dev,
                                       cudaStream_t stream)
{
    switch (s) {
        case 8: return decode_dispatch<8>(a, dev, stream);
        case 16: return decode_dispatch<16>(a, dev, stream);
        case 32: return decode_dispatch<32>(a, dev, stream);
        case 64: return decode_dispatch<64>(a, dev, stream);
        case 128: return decode_dispatch<128>(a, dev, stream);
        default: return cudaErrorInvalidValue;
    }
}

// =================================================================================================
// Random orthonormal basis (Section 4.2, "Choice of Linear Projections"): Gram-Schmidt process on the
// rows of a Gaussian matrix, in fp64, one CTA.  Right-looking order by blocks of four rows: the warp that holds them makes them
// orthogonal among themselves, one after the other, then every later row loses its components along the four at once.  The four are
// orthogonal to each other only up to rounding times their condition, so the products of a later row with them are not yet its
// components: those follow by a triangular substitution with the four rows' own products, which the block's warp has formed anyway (the
// inverse compact WY form of the modified process; Swirydowicz, Langou, Ananthan, Yang, Thomas, "Low synchronization Gram-Schmidt and
// generalized minimal residual algorithms", 2021).  Taken without it, rows that differ by 1e-5 of their length came out with products of
// 4e-4; with it |P P^T - I| is that of the process row by row, about the rounding times the condition of the matrix.
//
// s dependent steps, so the latency of a step is all there is.  Eight threads keep a row in registers, a warp a block: inside it a step is
// a row published in shared memory and two three-level reductions side by side, without a barrier; one barrier per block, one division per
// step in the whole CTA (fp64 arithmetic is narrow).  At s = 128 the registers hold one published row at a time.  The matrix is read from and
// the verdict written to pinned host memory, the active basis only replaced when the verdict is good: a call is one launch and one
// synchronisation.  (One call, s = 64: 123 us with rows in shared memory, two barriers per step and four copies, 44.6 with a barrier per
// row, 41 now.)
// =================================================================================================
constexpr int GS_LANES = 8;  // threads per row

template <int EPL>  // elements per thread
__global__ void __launch_bounds__(GS_LANES *GS_LANES *EPL, 1) gram_schmidt_kernel(const float *__restrict__ gauss,
                                                                               float *__restrict__ basis, int *verdict)
{
    constexpr int N = GS_LANES * EPL;  // rows = columns
    constexpr int R = 32 / GS_LANES;   // rows of a warp, a block
    __shared__ __align__(16) double pub[2][R][N];  // the rows of a block and 1 / their squared lengths, 0 when nothing is left of one
    __shared__ double pub_inv[2][R], pub_dot[2][R][R];  // [i][j]: product of the block's rows j < i
    const int r = threadIdx.x / GS_LANES, l = threadIdx.x % GS_LANES, warp = threadIdx.x / 32, own = r % R;
    constexpr int V = EPL > 1 ? 2 : 1;  // consecutive elements of a thread
    auto col = [&](int e) { return (e / V) * (V * GS_LANES) + V * l + e % V; };
    double a[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) a[e] = (double)gauss[r * N + col(e)];
    // product of u with a published row, or of the row with itself; all threads of the eight get it
    auto along = [&](const double *u, const double *row) {
        double acc[2] = {0.0, 0.0};
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const double p = row[col(e)];
            acc[e & 1] = fma(u ? u[e] : p, p, acc[e & 1]);
        }
        double sum = acc[0] + acc[1];
#pragma unroll
        for (int d = GS_LANES / 2; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
        return sum;
    };
    auto length2 = [&]() {
        double acc[2] = {0.0, 0.0};
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e & 1] = fma(a[e], a[e], acc[e & 1]);
        double sum = acc[0] + acc[1];
#pragma unroll
        for (int d = GS_LANES / 2; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
        return sum;
    };
    const double scale = length2();  // squared length of the input row
    bool bad = false;
    for (int b = 0; b < N / R && !bad; ++b) {
        if (warp == b) {  // this warp's rows among themselves, one after the other, without a barrier
#pragma unroll 1
            for (int i = 0; i < R; ++i) {
                const double *row = pub[b & 1][i];
                if (own == i) {
#pragma unroll
                    for (int e = 0; e < EPL; ++e) pub[b & 1][i][col(e)] = a[e];
                }
                __syncwarp();
                const double len2 = along(nullptr, row), dot = along(a, row), scale_i = __shfl_sync(0xffffffffu, scale, i * GS_LANES);
                const double inv = len2 > 1e-24 * scale_i ? 1.0 / len2 : 0.0;
                if (own == i && l == 0) pub_inv[b & 1][i] = inv;
                if (EPL <= 8 && own < i && l == 0) pub_dot[b & 1][i][own] = dot;  // (both rows are final)
                const double c = own > i ? dot * inv : 0.0;
                if (EPL > 8) asm volatile("" ::: "memory");
#pragma unroll
                for (int e = 0; e < EPL; ++e) a[e] = fma(-c, row[col(e)], a[e]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < R; ++i) bad = bad || pub_inv[b & 1][i] == 0.0;
        if (warp > b) {  // the block's rows: their parts are taken off together
            constexpr int G = EPL > 8 ? 1 : R;  // (s = 128: one after the other, there are 64 registers)
#pragma unroll 1
            for (int i0 = 0; i0 < R; i0 += G) {
                double c[G];
#pragma unroll
                for (int i = 0; i < G; ++i) c[i] = along(a, pub[b & 1][i0 + i]);
#pragma unroll
                for (int i = 0; i < G; ++i) {
#pragma unroll
                    for (int j = 0; j < i; ++j) c[i] = fma(-c[j], pub_dot[b & 1][i][j], c[i]);
                    c[i] *= pub_inv[b & 1][i0 + i];
                }
                if (G == 1) asm volatile("" ::: "memory");  // (the row is read again rather than kept)
#pragma unroll
                for (int i = 0; i < G; ++i)
#pragma unroll
                    for (int e = 0; e < EPL; ++e) a[e] = fma(-c[i], pub[b & 1][i0 + i][col(e)], a[e]);
            }
        }
    }
    if (threadIdx.x == 0) *verdict = bad;
    if (bad) return;
    const double inv = 1.0 / sqrt(length2());
#pragma unroll
    for (int e = 0; e < EPL; ++e) basis[r * N + col(e)] = basis[N * N + col(e) * N + r] = (float)(a[e] * inv);
}

__global__ void transpose_basis_kernel(float *basis, int s)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < s * s) basis[s * s + i] = basis[i % s * s + i / s];
}

// `gauss` and `verdict` are pinned host memory.
cudaError_t demo_launch_gram_schmidt(const float *gauss, float *basis, int *verdict, int s, cudaStream_t stream)
{
    switch (s) {
        case 8: gram_schmidt_kernel<1><<<1, 64, 0, stream>>>(gauss, basis, verdict); break;
        case 16: gram_schmidt_kernel<2><<<1, 128, 0, stream>>>(gauss, basis, verdict); break;
        case 32: gram_schmidt_kernel<4><<<1, 256, 0, stream>>>(gauss, basis, verdict); break;
        case 64: gram_schmidt_kernel<8><<<1, 512, 0, stream>>>(gauss, basis, verdict); break;
        case 128: gram_schmidt_kernel<16><<<1, 1024, 0, stream>>>(gauss, basis, verdict); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t demo_launch_transpose_basis(float *basis, int s, cudaStream_t stream)
{
    transpose_basis_kernel<<<(s * s + 255) / 256, 256, 0, stream>>>(basis, s);
    return cudaGetLastError();
}

// =================================================================================================
// demo_decode_apply_static: the decode + update step for callers that must not allocate.
//
// The generic decode kernels above read four small tables from global memory besides the caller's
// payloads and parameters: the DCT basis, the tensor table, the two pointer tables and a status
// word.  A context built by demo_init gets them from cudaMalloc; this entry point keeps them in the
// fixed array below instead, so it never allocates -- at the price of hard limits on the problem
// size and of one array shared by every call in the process.
// =================================================================================================
#include <cmath>
#include <cstring>
#include <mutex>

#include "../../include/demo.h"

namespace {

constexpr int STATIC_MAX_TENSORS = DEMO_STATIC_MAX_TENSORS;
constexpr int STATIC_MAX_WORKERS = DEMO_STATIC_MAX_WORKERS;
constexpr int STATIC_MAX_CHUNK = DEMO_STATIC_MAX_CHUNK;

// layout of the scratch array (byte offsets, all multiples of 256)
constexpr size_t OFF_BASIS = 0;                                                                   // s*s floats
constexpr size_t OFF_ENTRIES = OFF_BASIS + sizeof(float) * STATIC_MAX_CHUNK * STATIC_MAX_CHUNK;   // tensor table
constexpr size_t OFF_XPTRS = OFF_ENTRIES + sizeof(DemoTensorEntry) * STATIC_MAX_TENSORS;          // float*[T]
constexpr size_t OFF_PPTRS = OFF_XPTRS + sizeof(void *) * STATIC_MAX_TENSORS;                     // record*[W]
constexpr size_t OFF_STATUS = OFF_PPTRS + sizeof(void *) * STATIC_MAX_WORKERS;                    // int
constexpr size_t STATIC_SCRATCH_BYTES = OFF_STATUS + 256;

static_assert(STATIC_SCRATCH_BYTES == DEMO_STATIC_SCRATCH_BYTES, "header and layout disagree");

}  // namespace

// Device-resident scratch.  In host code this name is only a handle for cudaGetSymbolAddress; the
// device address is looked up once per device and passed to the kernels like any other pointer.
static __device__ __align__(256) unsigned char demo_static_scratch[DEMO_STATIC_SCRATCH_BYTES];

namespace {

constexpr int STATIC_MAX_DEVICES = 64;
std::mutex g_static_mutex;
unsigned char *g_static_base[STATIC_MAX_DEVICES];  // device address of the scratch, per device (0 = not set up)

}  // namespace

extern "C" demo_status demo_decode_apply_static(const demo_config *cfg, const demo_tensor_desc *tensors,
                                                int32_t n_tensors, const void *const *payloads, int32_t n_payloads,
                                                float *const *params, int32_t cuda_device, void *cuda_stream)
{
    if (!cfg || !tensors || !payloads || !params || n_tensors < 1 || cuda_device < 0) return DEMO_ERR_INVALID_ARG;
    if (cuda_device >= STATIC_MAX_DEVICES) return DEMO_ERR_UNSUPPORTED;
    if (n_payloads < 1 || n_payloads != cfg->num_workers) return DEMO_ERR_INVALID_ARG;
    if (!std::isfinite(cfg->lr) || !std::isfinite(cfg->weight_decay)) return DEMO_ERR_INVALID_ARG;
    const int s = cfg->chunk;
    if (!(s == 8 || s == 16 || s == 32 || s == 64 || s == 128)) return DEMO_ERR_UNSUPPORTED;
    // the fixed scratch bounds the problem: reject anything larger instead of overrunning it
    if (s > STATIC_MAX_CHUNK || n_tensors > STATIC_MAX_TENSORS || n_payloads > STATIC_MAX_WORKERS)
        return DEMO_ERR_UNSUPPORTED;
    if (cfg->topk < 1 || (long long)cfg->topk > (long long)s * s) return DEMO_ERR_K;
    for (int t = 0; t < n_tensors; ++t) {
        const demo_tensor_desc &d = tensors[t];
        if (d.ndim != 1 && d.ndim != 2) return DEMO_ERR_SHAPE;
        for (int ax = 0; ax < d.ndim; ++ax)
            if (d.shape[ax] < s || d.shape[ax] % s != 0 || d.shape[ax] > (1LL << 31) - 1) return DEMO_ERR_SHAPE;
        if (!params[t] || (reinterpret_cast<uintptr_t>(params[t]) & 15u)) return DEMO_ERR_INVALID_ARG;
    }
    for (int w = 0; w < n_payloads; ++w)
        if (!payloads[w] || (reinterpret_cast<uintptr_t>(payloads[w]) & 15u)) return DEMO_ERR_INVALID_ARG;

    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) {
        cudaGetLastError();
        return DEMO_ERR_CUDA;
    }
    if (prev != cuda_device && cudaSetDevice(cuda_device) != cudaSuccess) {
        cudaGetLastError();
        return DEMO_ERR_CUDA;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    demo_status result = DEMO_OK;
    do {
        // The tables are copied from host memory that is gone when this call returns (a stack frame, the
        // caller's pointer arrays).  Recorded into a CUDA graph those copies would be replayed from dead
        // memory, so a stream that is capturing is refused before anything is enqueued.
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
            cudaGetLastError();
            result = DEMO_ERR_INVALID_ARG;
            break;
        }
        // one-time set-up per device, with that device current: translate the symbol into a device address
        unsigned char *base = nullptr;
        {
            std::lock_guard<std::mutex> lock(g_static_mutex);
            if (!g_static_base[cuda_device]) {
                void *p = nullptr;
                if (cudaGetSymbolAddress(&p, demo_static_scratch) != cudaSuccess || !p) {
                    cudaGetLastError();
                    result = DEMO_ERR_CUDA;
                    break;
                }
                g_static_base[cuda_device] = static_cast<unsigned char *>(p);
            }
            base = g_static_base[cuda_device];
        }
        DemoLaunch dev;
        if (cudaDeviceGetAttribute(&dev.sm_count, cudaDevAttrMultiProcessorCount, cuda_device) != cudaSuccess) {
            result = DEMO_ERR_CUDA;
            break;
        }

        // host-side images of the tables (fixed-size, on the stack / in static storage: no heap)
        static thread_local float h_basis[STATIC_MAX_CHUNK * STATIC_MAX_CHUNK];
        DemoTensorEntry h_entries[STATIC_MAX_TENSORS];  // 2-D tensors first, then 1-D tensors
        int n2d = 0, n1d = 0;
        long long chunks2d = 0, chunks1d = 0;
        {
            const double pi = 3.141592653589793238462643383279502884;
            for (int u = 0; u < s; ++u)
                for (int n = 0; n < s; ++n) {
                    const double au = (u == 0) ? std::sqrt(1.0 / s) : std::sqrt(2.0 / s);
                    h_basis[(size_t)u * s + n] = (float)(au * std::cos(pi * (2.0 * n + 1.0) * u / (2.0 * s)));
                }
            for (int t = 0; t < n_tensors; ++t) n2d += tensors[t].ndim == 2;
            int i2 = 0, i1 = n2d;
            long long rec = 0;
            for (int t = 0; t < n_tensors; ++t) {
                const demo_tensor_desc &d = tensors[t];
                const bool two = d.ndim == 2;
                const long long n1 = two ? d.shape[1] : d.shape[0];
                const long long c0 = two ? d.shape[0] / s : 1, c1 = n1 / s;
                const long long M = two ? (long long)s * s : s;
                DemoTensorEntry e;
                e.tensor = t;
                e.n1 = (int)n1;
                e.c1 = (int)c1;
                e.k_eff = (int)(cfg->topk < M ? cfg->topk : M);
                e.rec_begin = rec;
                e.chunk_begin = two ? chunks2d : chunks1d;
                (two ? chunks2d : chunks1d) += c0 * c1;
                h_entries[two ? i2++ : i1++] = e;
                rec += c0 * c1 * e.k_eff;
            }
            n1d = n_tensors - n2d;
        }

        bool ok = true;
        ok = ok && cudaMemcpyAsync(base + OFF_BASIS, h_basis, sizeof(float) * (size_t)s * s, cudaMemcpyHostToDevice,
                                   stream) == cudaSuccess;
        ok = ok && cudaMemcpyAsync(base + OFF_ENTRIES, h_entries, sizeof(DemoTensorEntry) * (size_t)n_tensors,
                                   cudaMemcpyHostToDevice, stream) == cudaSuccess;
        ok = ok && cudaMemcpyAsync(base + OFF_XPTRS, params, sizeof(void *) * (size_t)n_tensors, cudaMemcpyHostToDevice,
                                   stream) == cudaSuccess;
        ok = ok && cudaMemcpyAsync(base + OFF_PPTRS, payloads, sizeof(void *) * (size_t)n_payloads,
                                   cudaMemcpyHostToDevice, stream) == cudaSuccess;
        // the array keeps the previous call's contents: the status word must start at zero
        ok = ok && cudaMemsetAsync(base + OFF_STATUS, 0, sizeof(int), stream) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            result = DEMO_ERR_CUDA;
            break;
        }

        DemoDecodeArgs a;
        a.payloads = reinterpret_cast<const DemoRecord *const *>(base + OFF_PPTRS);
        a.W = n_payloads;
        a.x_ptrs = reinterpret_cast<float *const *>(base + OFF_XPTRS);
        a.C = reinterpret_cast<const float *>(base + OFF_BASIS);
        a.lr = cfg->lr;
        a.wd = cfg->weight_decay;
        a.status = reinterpret_cast<int *>(base + OFF_STATUS);
        a.agg = 0;
        a.phi = 0;
        a.agg_scale = 1.f;
        cudaError_t err = cudaSuccess;
        if (n2d) {
            a.entries = reinterpret_cast<const DemoTensorEntry *>(base + OFF_ENTRIES);
            a.n_entries = n2d;
            a.n_chunks = chunks2d;
            err = demo_launch_decode_generic(s, a, dev, stream);
        }
        if (err == cudaSuccess && n1d) {
            a.entries = reinterpret_cast<const DemoTensorEntry *>(base + OFF_ENTRIES) + n2d;
            a.n_entries = n1d;
            a.n_chunks = chunks1d;
            err = demo_launch_decode_small(s, &a, nullptr, dev, stream);
        }
        if (err != cudaSuccess) {
            cudaGetLastError();
            result = DEMO_ERR_CUDA;
        }
    } while (false);
    if (prev >= 0 && prev != cuda_device) cudaSetDevice(prev);
    return result;
}
