// Shared declarations of the CUDA side of libstream (not shared with the CPU oracle).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "stream.h"

namespace stream {

// Problem geometry as the kernels see it.
struct Geom {
    int batch, H, G, hpg;       // heads; hpg = H / G
    long long T;
    int d, bq, bk, k_top, causal;
    int n_qb;                   // ceil(T / bq): rows per head
    int N_k;                    // key blocks after padding T to a multiple of lcm(bq, bk)
    int levels;                 // split levels that can change the result (with k = k_top)
    const int32_t *k_row;       // device, [n_qb]: k of each query block (clamped to 1 .. k_top), or NULL = k_top everywhere
    int k_override;             // > 0: every row uses this k (one launch of a several-k build); rows stay k_top wide
    unsigned int *row_tiles;    // device, [batch * H * n_qb] or NULL: tiles scored for each row (single-k builds)
    long long qs_b, qs_h, qs_t; // element strides
    long long ks_b, ks_h, ks_t;
};

// Header at the start of the mask workspace. The first 40 bytes mirror stream_stats.
struct WorkspaceHeader {
    unsigned long long tiles_scored;
    unsigned long long rows;
    unsigned int error;
    unsigned int error_info;
    unsigned long long tile_products;  // 64 x 64 tile products computed (more than tiles_scored where rows share a product)
    unsigned long long tiles_fetched;  // tiles copied into shared memory (the tensor-core block kernel counts them)
    unsigned int work_counter;  // next work item of the persistent kernels
    unsigned int pad[53];
};
static_assert(sizeof(WorkspaceHeader) == 256, "workspace header is 256 bytes");

constexpr int kMaxKTop = 1024;

// Several sparsity constants in one call.
constexpr int kMaxMultiK = 8;
struct MultiK {
    int n;               // 0: a single build (k from the geometry)
    int k[kMaxMultiK];
    int use_cache;       // generic kernel: N_k scores of the row fit in shared memory behind the tiles
};

void set_error(const char *fmt, ...);
stream_status cuda_fail(cudaError_t e, const char *what);

// Launchers (each validates what only it can support and returns UNSUPPORTED otherwise).
// allow_mma: bf16 may go through mma.sync where it fits (false: fp32 FMA whatever the dtype).
stream_status launch_mask_generic(const Geom &g, int dtype, bool allow_mma, const void *q, const void *k, int32_t *mask,
                                  float *score, WorkspaceHeader *ws, cudaStream_t st);
// mask / score: [mk.n][rows][k_top]; a row's tiles are scored once for all k where the cache fits.
stream_status launch_mask_generic_multi(const Geom &g, const MultiK &mk, int dtype, bool allow_mma, const void *q, const void *k,
                                        int32_t *mask, float *score, WorkspaceHeader *ws, cudaStream_t st);
stream_status launch_attn_generic(const Geom &g, int dtype, const void *q, const void *k, const void *v,
                                  const int32_t *mask, float scale, void *out, cudaStream_t st);
// bf16 attention on mma.sync (whatever the tcgen05 kernel does not take, with 16-byte aligned rows).
bool attn_mma_supported(const Geom &g, int dtype, const void *q, const void *k, const void *v, const void *out);
stream_status launch_attn_mma(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale,
                              void *out, cudaStream_t st);
bool mask_tc_supported(const Geom &g, int dtype);  // d = 128, blocks of 64, k_top <= 32
bool mask_tc_auto(const Geom &g, int dtype);       // what the kernel is the better choice for beyond that
stream_status launch_mask_tc(const Geom &g, const void *q, const void *k, int32_t *mask, float *score,
                             WorkspaceHeader *ws, cudaStream_t st);
// The rows of the first n_qb <= whole_query_blocks(g) query blocks, no scores asked for.
stream_status launch_mask_whole(const Geom &g, int n_qb, int32_t *mask, WorkspaceHeader *ws, cudaStream_t st);
// Several k in one launch (mk.n >= 1: mask / score are [mk.n][rows][k_top]); with score_memory
// (mask_tc_score_memory_bytes(g) bytes, device) a (row, block) tile is scored once for all k.
size_t mask_tc_score_memory_bytes(const Geom &g);
stream_status launch_mask_tc_multi(const Geom &g, const MultiK &mk, const void *q, const void *k, int32_t *mask,
                                   float *score, WorkspaceHeader *ws, void *score_memory, cudaStream_t st);
// Per-token masks (block_q = 1) on the tensor cores.
bool mask_tok_supported(const Geom &g, int dtype);
stream_status launch_mask_tok(const Geom &g, const void *q, const void *k, int32_t *mask, float *score,
                              WorkspaceHeader *ws, cudaStream_t st);
bool attn_tc_supported(const Geom &g, int dtype);  // d = 128, blocks of 64
bool attn_tc_auto(const Geom &g, int dtype);       // and d = 64, and blocks of 32
stream_status launch_attn_tc(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask,
                             float scale, void *out, cudaStream_t st);
// bad_flag: device word that gets bit 0 set if a mask entry is >= the number of key blocks.
stream_status launch_vertical(const Geom &g, const int32_t *mask, const float *score, float *vertical, float *kurtosis,
                              unsigned int *bad_flag, cudaStream_t st);
stream_status launch_mask_diff(long long n_rows, int k_a, const int32_t *mask_a, const float *score_a, int k_b,
                               const int32_t *mask_b, int32_t *diff, float *diff_score, cudaStream_t st);
// Attention under masks of short query blocks (block_q < 16) on the tensor cores.
bool attn_tok_supported(const Geom &g, int dtype, const void *q, const void *k, const void *v, const void *out);
stream_status launch_attn_tok(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale,
                              void *out, cudaStream_t st);
// Drain `st` and copy a tensor-core attention kernel's status words (code, block) to out.
stream_status read_attn_status(unsigned int out[2], cudaStream_t st);
stream_status read_attn_tok_status(unsigned int out[2], cudaStream_t st);

// The kernels of mask builds and attention, but for clusters, are launched as programmatic dependents: a kernel may begin while the one before it on the stream
// still runs, as far as this point, behind which that one (and with it all before it) is complete and its
// results are there. So launch latency, barrier setup and TMEM allocation are not waited for. Every thread comes by before it
// touches global memory, and reads it with ordinary loads, cp.async or TMA only: no __ldg and no const __restrict__ inputs.
// Those are for data that nobody writes while the kernel lives, and this one lives while the kernel before still
// writes the mask it reads; such loads may also be moved up across the wait or find a line from before it.
__device__ __forceinline__ void after_previous_kernel() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launch of such a kernel (us in a loop of mask and attention, before and after: 28 / 4 heads, 1500 tokens, 56.1 -> 53.2; 12 / 2
// heads in blocks of 32, 41.0 -> 38.9; 4 heads in fp32, 700 tokens, 40.9 -> 37.8; 32 / 8 heads, 4000 tokens, k = 8, 141 -> 136).
// Clusters (cluster > 1) start as before, after the kernel before: one of them launched early began a microsecond later (18.4 -> 19.5).
template <class... K, class... A>
cudaError_t launch_kernel(void (*kern)(K...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st, unsigned cluster, A &&...args) {
    cudaLaunchAttribute at[1] = {};
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = at;
    c.numAttrs = 1;
    if (cluster > 1) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
    }
    return cudaLaunchKernelEx(&c, kern, std::forward<A>(args)...);
}

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }

// 2^x by the special-function unit (relative error about 2^-22; -inf gives 0).
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Levels until every node is a single block: nodes start with at most ceil(N_k / k) blocks and
// the larger half of n blocks has ceil(n / 2). With N_k > 1 the first level always runs (it is
// where scores are first computed), matching n_it = ceil(log2 N_k) >= 1.
__host__ __device__ inline int levels_for(int N_k, int k) {
    long long sz = ((long long)N_k + k - 1) / k;
    int levels = 0;
    while (sz > 1) { sz = (sz + 1) / 2; ++levels; }
    return N_k > 1 ? (levels > 1 ? levels : 1) : 0;
}

// The sparsity constant of query block qb.
__device__ __forceinline__ int row_k(const Geom &g, int qb) {
    if (g.k_override > 0) return g.k_override;
    if (g.k_row == nullptr) return g.k_top;
    const int k = g.k_row[qb];
    return k < 1 ? 1 : (k > g.k_top ? g.k_top : k);
}

// Split levels of a row that runs with k = kq.
__host__ __device__ inline int row_levels(const Geom &g, int kq) {
    return kq == g.k_top ? g.levels : levels_for(g.N_k, kq);
}

// Last key block a row may look at (C^blk of Algorithm 2 in closed form), -1 if none.
__host__ __device__ inline int last_valid_block(const Geom &g, int qb) {
    long long last_tok = g.causal ? ((long long)qb * g.bq + g.bq - 1) : (g.T - 1);
    if (last_tok > g.T - 1) last_tok = g.T - 1;
    return (int)(last_tok / g.bk);
}

// A row whose allowed blocks are no more than its k keeps them all, whatever their scores: Algorithm 2 then drops nothing on any
// level. How many query blocks, from the first, have such rows: 0 unless k is the same for all.
inline int whole_query_blocks(const Geom &g) {
    if (g.k_row != nullptr) return 0;
    const int k = g.k_override > 0 ? g.k_override : g.k_top;
    if (last_valid_block(g, g.n_qb - 1) < k) return g.n_qb;
    return g.causal ? (int)((long long)k * g.bk / g.bq) : 0;
}

// Writing them, for every head's first n_qb query blocks: allowed blocks, -1 padded, and what scoring them would have counted. A head's
// rows lie one behind the other and are written in pieces of 256 entries, a warp a piece (a warp a row took 18 us for 2560 rows
// of 10 on twelve SMs). 32 bits are enough: no such row looks beyond kMaxKTop blocks.
constexpr unsigned kWholePiece = 256;
__host__ __device__ inline long long whole_pieces(const Geom &g, int n_qb) {
    return (long long)g.batch * g.H * (((long long)n_qb * g.k_top + kWholePiece - 1) / kWholePiece);
}
__device__ __forceinline__ void write_whole_rows(const Geom &g, int n_qb, int warp, int n_warps, int lane, int32_t *mask, WorkspaceHeader *ws) {
    const unsigned k = (unsigned)g.k_top, n = (unsigned)n_qb * k, per_head = (n + kWholePiece - 1) / kWholePiece, pieces = (unsigned)whole_pieces(g, n_qb);
    const unsigned T = (unsigned)g.T, bq = (unsigned)g.bq, bk = (unsigned)g.bk;
    unsigned tiles = 0;
    for (unsigned p = (unsigned)warp; p < pieces; p += (unsigned)n_warps) {
        const unsigned head = p / per_head, x0 = (p - head * per_head) * kWholePiece, x1 = min(x0 + kWholePiece, n);
        int32_t *const to = mask + (long long)head * g.n_qb * g.k_top;
#pragma unroll 1
        for (unsigned x = x0 + (unsigned)lane; x < x1; x += 32) {
            const unsigned qb = x / k, i = x - qb * k, blocks = (g.causal ? min((qb + 1u) * bq, T) - 1u : T - 1u) / bk + 1u;
            to[x] = i < blocks ? (int)i : -1;
            if (i == 0u) {
                const unsigned t = g.levels > 0 ? blocks : 0u;
                tiles += t;
                if (g.row_tiles != nullptr) g.row_tiles[(long long)head * g.n_qb + qb] = t;
            }
        }
    }
    tiles = __reduce_add_sync(0xffffffffu, tiles);
    if (lane == 0 && tiles > 0u) atomicAdd(&ws->tiles_scored, (unsigned long long)tiles);
    if (warp == 0 && lane == 0) atomicAdd(&ws->rows, (unsigned long long)g.batch * g.H * n_qb);
}

}  // namespace stream
