// Internal declarations shared by the host library and the kernel translation units.
// Nothing here is part of the public ABI (see include/demo.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

struct DemoTickets;  // launch.cuh
struct DemoLaunch;   // launch.cuh

// One payload record: flat index inside the chunk + fp32 coefficient (8 bytes, little-endian).
struct DemoRecord {
    int32_t idx;
    float val;
};

// One tensor of a work list.  A work list holds either all 2-D tensors or all 1-D tensors; chunk
// ids run over the list, row-major over each tensor's chunk grid (blocking operator, appendix
// B.1.2 of the paper).
struct DemoTensorEntry {
    long long chunk_begin;  // id of this tensor's first chunk inside the list
    long long rec_begin;    // index of this tensor's first record inside a payload
    int tensor;             // position in the caller's pointer arrays
    int n1;                 // row length in elements (2-D: shape[1]; 1-D: shape[0])
    int c1;                 // chunks per row of the chunk grid
    int k_eff;              // min(k, M)
};

struct DemoCompressArgs {
    const DemoTensorEntry *entries;  // device
    int n_entries;
    long long n_chunks;
    int k;                      // k_eff of the list's tensors (all of one kind and chunk size)
    const void *const *g_ptrs;  // device array indexed by DemoTensorEntry::tensor
    float *const *m_ptrs;       // device array
    DemoRecord *payload;        // device, whole payload of this worker
    const float *C;             // device, s x s orthonormal DCT-II, C[u*s + n], and behind it its transpose
    float beta;
    float alpha;    // momentum-subtraction coefficient: m <- B - alpha * IDCT(kept)
    int grad_bf16;  // 1: gradients are bf16, 0: fp32
    int *status;    // device status word (sticky)
    // TMA tensor maps (128-byte CUtensorMap objects in device memory, indexed like the
    // pointer arrays; box = one s x s tile): s = 64 and 128.
    const void *tmap_m;
    const void *tmap_g;
    int wait_first = 1;  // see StreamOrder (launch.cuh)
    DemoTickets *tickets = nullptr;  // device; the counter of this kernel's chunks
    int late_lookup = 0;  // s = 64: the first chunk is looked up behind the tensor-memory allocation (kernels_fast64.cu)
    // 1: the momentum tensors hold the chunk-wise DCT of the momentum (tiles transposed); only the s = 64 tile
    // kernel with tensor maps implements it
    int momentum_dct = 0;
};

struct DemoDecodeArgs {
    const DemoTensorEntry *entries;
    int n_entries;
    long long n_chunks;
    int k = 0;                          // k_eff of the list's tensors
    const DemoRecord *const *payloads;  // device array [W]
    int W;
    float *const *x_ptrs;  // device array
    const float *C;
    float lr;
    float wd;
    int *status;
    int agg;          // 0 sum, 1 mean over workers, 2 per-coordinate count-normalised mean (0/0 = 0)
    int phi;          // 0 sign, 1 identity
    float agg_scale;  // 1/W for the mean, else 1 (only the identity update sees it)
    // Parameter-server form: when not NULL, write sign(R) in {-1, 0, +1} per element to these int8 tensors
    // (device array indexed like x_ptrs) instead of updating the parameters.
    signed char *const *sign_ptrs = nullptr;
    int wait_first = 1;  // see StreamOrder (launch.cuh)
    DemoTickets *tickets = nullptr;  // device; the counter of this kernel's chunks
};

// Launchers (defined in the kernel translation units).  `s` is the chunk size.  Return the CUDA error of the launch.
// Dense transforms of s x s tiles, any basis (kernels_generic.cu).
cudaError_t demo_launch_compress_generic(int s, const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream);
cudaError_t demo_launch_decode_generic(int s, const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream);
// Segments of 1-D tensors (any s, any basis) and, where `demo_small_tiles_supported` and the basis is the DCT, s x s tiles, in
// one launch (kernels_small.cu).  Either list may be NULL.
bool demo_small_tiles_supported(int s);
cudaError_t demo_launch_compress_small(int s, const DemoCompressArgs *segs, const DemoCompressArgs *tiles, DemoLaunch &dev,
                                       cudaStream_t stream);
cudaError_t demo_launch_decode_small(int s, const DemoDecodeArgs *segs, const DemoDecodeArgs *tiles, DemoLaunch &dev,
                                     cudaStream_t stream);
// Fast-DCT kernels for 2-D tensors; `supported` tells whether chunk size s has one.
bool demo_fast_supported(int s);
// largest: chunks of the list's largest tensor
cudaError_t demo_launch_compress_fast(int s, const DemoCompressArgs &a, long long largest, DemoLaunch &dev, cudaStream_t stream);
cudaError_t demo_launch_decode_fast(int s, const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream);
// s = 32 (kernels_fast32.cu).
cudaError_t demo_launch_compress_fast32(const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream);
// s = 64 with TMA tensor maps (kernels_fast64.cu; cudaErrorNotSupported without them).
cudaError_t demo_launch_compress_fast64(const DemoCompressArgs &a, long long largest, DemoLaunch &dev, cudaStream_t stream);
// s = 128 (kernels_fast128.cu); compress needs the TMA tensor maps (cudaErrorNotSupported without them).
cudaError_t demo_launch_compress_fast128(const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream);
cudaError_t demo_launch_decode_fast128(const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream);

// Tensor-core kernels for 2-D tensors under a caller-supplied basis (kernels_tc.cu): tcgen05 MMAs with
// 3xTF32 splitting, chunk size 64 only.
bool demo_tc_supported(int s);
cudaError_t demo_launch_compress_tc(const DemoCompressArgs &a, DemoLaunch &dev, cudaStream_t stream);
cudaError_t demo_launch_decode_tc(const DemoDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream);

// Self-test of the bounded wait (kernels_fast.cu): one CTA waits, for at most `limit_cycles`, on an
// mbarrier that nothing completes, records DEMO_DEV_TIMEOUT in *status and returns.
cudaError_t demo_launch_wait_selftest(int *status, long long limit_cycles, cudaStream_t stream);

// Gram-Schmidt process on the rows of the s x s matrix `gauss` (device, fp32) in fp64; writes the
// orthonormal rows to `basis` (device, fp32, the transpose behind them) and 1 to *flag when a row has no component left.
cudaError_t demo_launch_gram_schmidt(const float *gauss, float *basis, int *verdict, int s, cudaStream_t stream);
// basis[s*s .. 2 s*s) <- the transpose of basis[0 .. s*s) (kernels_generic.cu; the launcher above writes both)
cudaError_t demo_launch_transpose_basis(float *basis, int s, cudaStream_t stream);

// ---- tensors of any order with rectangular chunks (appendix of the paper: blocking operator and
// multilinear product; kernels_nd.cu) ---------------------------------------------------------------
constexpr int DEMO_ND_DIMS = 4;         // lower orders are padded on the left with axes of extent 1
constexpr int DEMO_ND_MAX_ROWS = 1024;  // contiguous rows of a chunk whose offsets the kernels tabulate

struct DemoNdEntry {
    long long chunk_begin;           // id of this tensor's first chunk inside its class
    long long chunk_end;             // chunk_begin + number of chunks of this tensor
    long long rec_begin;             // index of this tensor's first record inside a payload
    long long stride[DEMO_ND_DIMS];  // element stride of each axis of the (contiguous) tensor
    int tensor;                      // position in the caller's pointer arrays
    int k_eff;                       // min(k, M)
    int M;                           // elements per chunk
    int s[DEMO_ND_DIMS];             // chunk shape
    int c[DEMO_ND_DIMS];             // chunk grid
    unsigned inv[DEMO_ND_DIMS];      // ceil(2^32 / s[a]) for s[a] > 1 (division by multiplication), else 0
    int basis[DEMO_ND_DIMS];         // offset (floats, multiple of 8) of axis a's table, where it is a dense contraction
    // filled in by demo_nd_plan and demo_nd_classify (kernels_nd.cu)
    int p[DEMO_ND_DIMS];             // element strides of the padded tile in shared memory
    int tile;                        // its floats, a multiple of 4
    int tail;                        // > 0: the last two axes are both of this extent and transformed together
    int row;                         // elements that are contiguous both in the tensor and in the tile
    unsigned inv_row;                // ceil(2^32 / row) for row > 1, else 0
    int quads;                       // 1: rows are whole 16-byte pieces of the tensor, 2: and of the tile
    unsigned inv_row4;               // ceil(2^32 / (row / 4)) for row > 4, else 0 (quads only)
    int row_table;                   // 1: the chunk's rows are few and their offsets fit 32 bits
    int threads;                     // CTA size this chunk would choose
    int layout;                      // same number: same strides in the tensor and in the tile
};

// Tensors that share a kernel variant: one launch.
struct DemoNdClass {
    int first, n;        // entries first .. first + n - 1 of the context's list
    long long n_chunks;  // chunk ids run over the class
    int threads;         // CTA size
    int max_M, tile;     // largest chunk / padded tile (floats, multiples of 4)
    int rows;            // longest row table
    int dense_axes;      // some extent is a dense contraction from a table (second tile)
    int big;             // some extent is 128: the variant with 64 registers per half line
};
// Coefficient tables of the dense extents in use, and the tile layouts of the chunk shapes planned so far: `rows` is what the search reads of
// the tensor beside them (demo_nd_plan).
struct DemoNdTables {
    struct Layout {
        int s[DEMO_ND_DIMS], p[DEMO_ND_DIMS], tile, rows;
    };
    std::vector<float> data;
    std::vector<Layout> layouts;
    int of[129];
    DemoNdTables() { for (int &v : of) v = -1; }
    int get(int s);  // offset of the tables of extent s (made on first use)
};
void demo_nd_plan(DemoNdEntry *e, DemoNdTables *tables);
// Sorts `entries` by class, sets their chunk ranges (chunk_end holds the number of chunks before) and lists the classes.
void demo_nd_classify(std::vector<DemoNdEntry> &entries, int sm_count, std::vector<DemoNdClass> *classes);

struct DemoNdCompressArgs {
    const DemoNdEntry *entries;  // device, the class's first
    DemoNdClass cls;
    const void *const *g_ptrs;
    float *const *m_ptrs;
    DemoRecord *payload;
    const float *tables;  // device: DemoNdTables::data
    float beta, alpha;
    int grad_bf16;
    int *status;
    int wait_first = 1;  // see StreamOrder (launch.cuh)
    DemoTickets *tickets = nullptr;  // device; the counter of this kernel's chunks
};

struct DemoNdDecodeArgs {
    const DemoNdEntry *entries;  // device, the class's first
    DemoNdClass cls;
    const DemoRecord *const *payloads;
    int W;
    float *const *x_ptrs;
    const float *tables;
    float lr, wd;
    int *status;
    int agg, phi;
    float agg_scale;
    signed char *const *sign_ptrs = nullptr;  // see DemoDecodeArgs
    int wait_first = 1;
    DemoTickets *tickets = nullptr;
};

// x <- x - lr (sign + wd x) from int8 signs, over every tensor of a context (kernels_generic.cu).
struct DemoFlatEntry {
    long long piece_begin;  // index of this tensor's first piece in the launch
    long long n;            // elements
    int tensor;             // position in the pointer arrays
    int pad;
};
struct DemoApplySignsArgs {
    const DemoFlatEntry *entries;  // device
    int n_entries;
    long long n_pieces;
    int piece;                            // elements per piece: one of demo_apply_pieces
    const signed char *const *sign_ptrs;  // device array
    float *const *x_ptrs;                 // device array
    float lr, wd;
};
constexpr int demo_apply_pieces[2] = {1024, 4};  // a block's, a thread's
cudaError_t demo_launch_apply_signs(const DemoApplySignsArgs &a, DemoLaunch &dev, cudaStream_t stream);

cudaError_t demo_launch_compress_nd(const DemoNdCompressArgs &a, DemoLaunch &dev, cudaStream_t stream);
cudaError_t demo_launch_decode_nd(const DemoNdDecodeArgs &a, DemoLaunch &dev, cudaStream_t stream);

// Locate the tensor that owns chunk id c: the last entry with chunk_begin <= c.
__device__ __forceinline__ int demo_find_entry(const DemoTensorEntry *entries, int n, long long c)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (entries[mid].chunk_begin <= c)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// The last entry at or behind e with chunk_begin <= c (which holds for e): strides that double, then halve, so that the entry after e
// costs one comparison and one d entries away about 2 log2 d.
__device__ __forceinline__ int demo_seek_entry(const DemoTensorEntry *entries, int n, int e, long long c)
{
    int step = 1;
    for (; step < n - e && entries[e + step].chunk_begin <= c; step <<= 1) e += step;
    while (step >>= 1)
        if (step < n - e && entries[e + step].chunk_begin <= c) e += step;
    return e;
}

// (warp) the last i of lo .. lo + n - 1 with below(i), which holds for lo and up to some i.  32 places are compared at once, so up to
// 32 entries take one round of loads, up to 2^20 four.  (In steps of 32 entries instead: decode of 20000 vectors of 64 elements 647 us
// instead of 44, of 100000 15.2 ms instead of 0.22.)
#ifdef __CUDACC__
template <class Below>
__device__ __forceinline__ int demo_find_warp(int lo, int n, Below below)
{
    const int lane = threadIdx.x & 31;
    while (n > 1) {
        const int step = (n + 31) / 32, i = lane * step;
        const int last = __popc(__ballot_sync(0xffffffffu, i < n && below(lo + i))) - 1;
        lo += last * step;
        n = n - last * step < step ? n - last * step : step;
    }
    return lo;
}
#endif

// Status values written by kernels (match demo_status in include/demo.h).
#define DEMO_DEV_TIMEOUT 7
#define DEMO_DEV_PAYLOAD 8
