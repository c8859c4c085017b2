// Per-token Stream masks on the tensor cores for sm_100a: block_q = 1 (every query token is a row
// of its own), block_k = 64, bf16, d = 128, k_top <= 32 (Algorithm 2 at its finest query
// granularity, the [heads, T, k] shape of the mask).
//
// A row's candidate tile is now 1 x 64 x 128: eight thousand multiply-adds for 16 KB of keys,
// and every token has candidates of its own from the second level on. Gathering them token by
// token would move 128 times more key bytes than the contraction can use. Instead one CTA takes
// 128 consecutive tokens of one head through the hierarchy together, level by level:
//   - the tokens' candidate blocks of the level are merged into one ascending list (a map of the
//     key blocks, a byte or a bit each, set by the tokens, compacted by one warp);
//   - every block of the list is fetched once by TMA (two per stage) and multiplied with all 128
//     tokens at once: tcgen05.mma, A = the group's Q tile (128 tokens, shared memory), B = the pair
//     of key tiles (N = 128), fp32 accumulators in TMEM (128 columns per stage);
//   - a thread per token reads its lane of the accumulator, takes the masked maximum over each
//     tile's 64 keys (Eq. 4 under C, token level) and keeps it if that block is one of the
//     token's own candidates (which ascend with the list);
//   - then each token ranks its 2k branch scores (higher score, then lower block index), keeps k,
//     and marks its next candidates.
// At the first level all tokens share the candidates; deeper down the merged list approaches
// "every block at the level's stride", so the work is that of a dense Q K^T restricted to the
// strides, at tensor-core rate, and each key tile crosses L2 -> SM once per 128 tokens.
//
// Roles (512 threads): warp 0 TMA producer and list builder, warps 1 and 3 issue the MMAs of the
// even and odd stages (warp 1 owns TMEM), warps 4..7 and 8..11 read the accumulators of the even
// and odd stages (thread = token). Ranking: up to k = 16 a thread of warps 4..7 for its token, above all
// sixteen warps, eight tokens each. The levels are separated by CTA-wide barriers; inside a level the
// roles meet on mbarriers, every wait bounded as in the other tensor-core kernels.
// Bound: the levels' serial parts (32 / 8 heads, T = 4096, k = 16: products 19 000 clocks a group of 128
// tokens, ranking, lists and barriers 21 000 before both were changed; 225 us at first, 148 then, 109 since levels that cannot drop
// anything are passed over and the long groups of all heads come first).
#include <math_constants.h>

#include "tc_common.cuh"

namespace stream {
namespace {

using namespace tc;

constexpr int kThreads = 512;
constexpr int kTok = 128;                    // tokens per group = rows of the A operand
constexpr int kBlk = 64, kD = 128;
constexpr int kStages = 4;                   // key-pair stages in shared memory = accumulator slots in TMEM
constexpr int kHalfTile = kBlk * 128;        // 64 keys x 128 bytes (one 64-channel half)
constexpr int kStageBytes = 4 * kHalfTile;   // [2 channel halves][2 tiles]
constexpr int kQBytes = 2 * kTok * 128;      // [2 channel halves][128 tokens][128 bytes]
constexpr int kPad = kTok + 1;               // row length of the per-token arrays (no bank conflicts either way)
constexpr int kMaxNk = 32768;                // key blocks (bitmap of 4 KB, block ids in 16 bits)
constexpr int kMaxList = kTok * 32;          // a level's merged list cannot be longer

struct Tail {
    unsigned long long full[kStages], empty[kStages], tmem_full[kStages], tmem_empty[kStages], q_full;
    unsigned int tmem_base;
    int abort_flag;
    int item;            // the next group
    int n_list;          // blocks in the current level's list
    int n_nodes[kTok];   // surviving nodes per token
    int n_tiles[kTok];   // tiles the token has needed so far (a warp's ranking keeps them here)
    // Of the group, the same for every token: its levels that rank anything, the nodes before the first of
    // them, the places of their left | right << 16 candidates in its list.
    int n_levels, n_node0;
    unsigned node0[32], place0[32];
    int split_f[32], split_l[32];  // (on the way to the nodes)
};

// Dynamic shared memory behind the 1024-byte aligned base:
//   Q tile | key-pair stages | scores [64][kPad] f32 | nodes [32][kPad] u32 | list u16 | bitmap u32 | Tail
// scores rows 0..31: score of a token's node j (its first allowed block); rows 32..63: score of
// node j's right branch at the current level. At the first level the 64 rows hold the scores of
// the (shared) list positions instead. nodes: first block | (blocks in the node << 16). With up
// to 16 nodes rows 16..31 hold the token's candidates of the level instead: block | (its node << 16).
constexpr int kScoresBytes = 64 * kPad * 4, kNodesBytes = 32 * kPad * 4, kListBytes = kMaxList * 2, kBitmapBytes = kMaxNk / 8;
constexpr int kSmemBytes = kQBytes + kStages * kStageBytes + kScoresBytes + kNodesBytes + kListBytes + kBitmapBytes +
                           (int)sizeof(Tail) + 1024;
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");

constexpr unsigned kDescHi = desc_hi_sw128(1024);            // K-major, 8-row groups 1024 bytes apart
constexpr unsigned kIdesc = idesc_bf16(128, 128, false);     // D fp32, A and B bf16 K-major, M = N = 128

constexpr unsigned kNoBlock = 0xffffu;  // (behind every block)

struct Params {
    Geom g;
    int n_items, n_tb;   // groups; groups per head (ceil(T / 128)), but for
    int walked_heads;    // heads (of the batch * H) whose groups are walked together
    int first_tb;        // those before this one, whose tokens keep all blocks they are allowed
    int32_t *mask;
    float *score;
    WorkspaceHeader *ws;
};

__device__ __forceinline__ bool wait_w(unsigned bar, unsigned parity, Tail *tl, WorkspaceHeader *ws, unsigned code) {
    return mbar_wait_warp(bar, parity, &tl->abort_flag, &ws->error, &ws->error_info, code);
}

__device__ __forceinline__ unsigned pack_node(int f, int len) { return (unsigned)f | ((unsigned)len << 16); }
// First block of a node's right half (of its left half, for a node of one block the one behind it).
__device__ __forceinline__ int right_of(unsigned node) { return (int)(((2u * (node & 0xffffu) + (node >> 16) - 1u) >> 1) + 1u); }
// The score whose score_key this is.
__device__ __forceinline__ float score_of_key(unsigned key) { return __uint_as_float(key ^ ((key & 0x80000000u) ? 0x80000000u : 0xffffffffu)); }

// Sorts n keys of a thread, largest first (Batcher's odd-even merge sort, unrolled: n = 32: 191
// exchanges, 64: 543).
template <int n, int P, int K>
__device__ __forceinline__ void sort_step(unsigned (&key)[n]) {
#pragma unroll
    for (int x = 0; x + K < n; ++x)
        if (x >= K % P && ((x - K % P) & (2 * K - 1)) < K && x / (2 * P) == (x + K) / (2 * P)) {
            const unsigned a = key[x], b = key[x + K];
            key[x] = max(a, b);
            key[x + K] = min(a, b);
        }
    if constexpr (K > 1) sort_step<n, P, K / 2>(key);
    else if constexpr (2 * P < n) sort_step<n, 2 * P, 2 * P>(key);
}

template <int kNodes>  // of a token, at most: 16 or 32
__global__ void __launch_bounds__(kThreads, 1)
mask_tok_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k, Params P) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = aligned_smem(smem_raw);
    const unsigned q_smem = smem_u32(smem), k_smem = q_smem + kQBytes;
    float *scores = (float *)(smem + kQBytes + kStages * kStageBytes);
    unsigned *nodes = (unsigned *)((unsigned char *)scores + kScoresBytes);
    unsigned short *list = (unsigned short *)((unsigned char *)nodes + kNodesBytes);
    unsigned *bitmap = (unsigned *)((unsigned char *)list + kListBytes);
    Tail *tl = (Tail *)((unsigned char *)bitmap + kBitmapBytes);
    const Geom &g = P.g;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned lt = (1u << lane) - 1u;

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(smem_u32(&tl->full[i]), 1); mbar_init(smem_u32(&tl->empty[i]), 1);
            mbar_init(smem_u32(&tl->tmem_full[i]), 1); mbar_init(smem_u32(&tl->tmem_empty[i]), 4);
        }
        mbar_init(smem_u32(&tl->q_full), 1);
        tl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    for (int i = tid; i < kMaxNk / 32; i += kThreads) bitmap[i] = 0u;
    if (warp == 1) tmem_alloc(smem_u32(&tl->tmem_base));  // all 512 columns (one CTA per SM)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = tl->tmem_base;
    after_previous_kernel();

    // the level's wanted blocks: a byte each while they fit (plain stores, the same value from all), else a bit
    unsigned char *const wanted = (unsigned char *)bitmap;
    const bool bytes = g.N_k <= kBitmapBytes;
    auto want = [&](int blk) {
        if (bytes) wanted[blk] = 1;
        else atomicOr(&bitmap[blk >> 5], 1u << (blk & 31));
    };
    constexpr bool kSorted = kNodes == 16;

    // role of this warp inside a level
    const bool is_producer = warp == 0;
    const int mma_which = warp == 1 ? 0 : (warp == 3 ? 1 : -1);            // issues the stages with this parity
    const int epi_grp = (warp >= 4 && warp < 12) ? (warp - 4) >> 2 : -1;   // reads the stages with this parity
    const int epi_tok = (warp & 3) * 32 + lane;                            // its token (TMEM lane)

    const int kq = g.k_top;
    unsigned seq = 0;     // stages so far over the whole kernel (the same in every thread)
    unsigned q_par = 0;
    unsigned long long tiles_needed = 0, products = 0;  // per thread

    for (int id = (int)blockIdx.x;;) {  // (the first group is the CTA's own, the counter deals those behind)
        if (id >= P.n_items || *(volatile int *)&tl->abort_flag) break;
        // late token groups (most allowed blocks) of all the heads walked together first
        const int per = P.walked_heads * P.n_tb, walk = id / per, rem = id - walk * per, heads = min(P.walked_heads, g.batch * g.H - walk * P.walked_heads);
        const int level = rem / heads, bh = walk * P.walked_heads + rem - level * heads, tb = P.first_tb + P.n_tb - 1 - level;
        const int b = bh / g.H, h = bh % g.H, kvh = h / g.hpg;
        const long long tok0 = (long long)tb * kTok;
        const long long tq_max = min(tok0 + kTok - 1, g.T - 1);
        const int q_lim_max = last_valid_block(g, (int)tq_max);

        if (is_producer) {
            if (elect_one()) {
                const unsigned bar = smem_u32(&tl->q_full);
                mbar_arrive_expect_tx(bar, (unsigned)kQBytes);
#pragma unroll
                for (int c = 0; c < 2; ++c) tma_load_4d(q_smem + c * (kQBytes / 2), &tmap_q, bar, c * 64, (int)tok0, h, b);
            }
            __syncwarp();
        }
        // the nodes before the first level that ranks anything, and its list: the same for every token
        if (warp == 0) {
            const FirstNodes<1> first(g, kq, g.levels, q_lim_max, lane, tl->split_f, tl->split_l);
            const unsigned ballots[2] = {__ballot_sync(0xffffffffu, first.left[0]), __ballot_sync(0xffffffffu, first.right[0])};
            const int pos_l = flags_before(ballots, lt), pos_r = pos_l + (first.left[0] ? 1 : 0);
            if (first.left[0]) list[pos_l] = (unsigned short)first.f[0];
            if (first.right[0]) list[pos_r] = (unsigned short)((first.f[0] + first.l[0]) / 2 + 1);
            tl->node0[lane] = first.f[0] <= first.l[0] ? pack_node(first.f[0], first.l[0] - first.f[0] + 1) : 0u;
            tl->place0[lane] = (unsigned)pos_l | ((unsigned)pos_r << 16);
            if (lane == 0) { tl->n_list = flags_all(ballots); tl->n_node0 = first.n; tl->n_levels = g.levels - first.splits; }
        }
        // the token this thread reads accumulators for
        const long long e_tq = tok0 + epi_tok;
        const bool e_ok = epi_grp >= 0 && e_tq < g.T;
        const int e_qlim = e_ok ? last_valid_block(g, (int)e_tq) : -1;
        const int key_end = e_ok ? (int)(g.causal ? e_tq + 1 : g.T) : 0;  // keys the token may look at: those before
        unsigned n_tiles = 0;  // tiles the token has needed so far (its own candidates, not the merged list)
        // the next group's number is fetched beside this one's first products or, where that could leave another CTA without work, its last
        const bool ahead = id + 2 * (int)gridDim.x < P.n_items;

        for (int level = 0;; ++level) {
            __syncthreads();  // the level's list is complete; the ranking of the level before is done
            const bool last = level + 1 == tl->n_levels;
            const int n_list = tl->n_list, n_st = (n_list + 1) >> 1;

            if (warp == 13 && lane == 0 && (ahead ? level == 0 : last))
                tl->item = P.n_items <= (int)gridDim.x ? P.n_items : (int)(gridDim.x + atomicAdd(&P.ws->work_counter, 1u));
            if (is_producer) {
                for (int i = 0; i < n_st; ++i) {
                    const unsigned s = seq + (unsigned)i, buf = s & 3u;
                    if (!wait_w(smem_u32(&tl->empty[buf]), ((s >> 2) & 1u) ^ 1u, tl, P.ws, 601)) break;
                    const bool two = 2 * i + 1 < n_list;
                    const int blk0 = list[2 * i], blk1 = two ? list[2 * i + 1] : 0;
                    if (elect_one()) {
                        const unsigned bar = smem_u32(&tl->full[buf]), dst = k_smem + buf * kStageBytes;
                        mbar_arrive_expect_tx(bar, (unsigned)((two ? 4 : 2) * kHalfTile));
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            tma_load_4d(dst + c * 2 * kHalfTile, &tmap_k, bar, c * 64, blk0 * kBlk, kvh, b);
                            if (two) tma_load_4d(dst + (c * 2 + 1) * kHalfTile, &tmap_k, bar, c * 64, blk1 * kBlk, kvh, b);
                        }
                    }
                    __syncwarp();
                }
                if (lane == 0) products += 2ull * (unsigned long long)n_list;  // 128 tokens x 64 keys each
            } else if (mma_which >= 0) {
                bool ok = true;
                if (level == 0) ok = wait_w(smem_u32(&tl->q_full), q_par, tl, P.ws, 602);
                const unsigned a_lo = desc_lo_sw128(q_smem, 16);
                for (int i = 0; ok && i < n_st; ++i) {
                    const unsigned s = seq + (unsigned)i, buf = s & 3u, par = (s >> 2) & 1u;
                    if ((int)(s & 1u) != mma_which) continue;
                    if (!wait_w(smem_u32(&tl->full[buf]), par, tl, P.ws, 603)) break;
                    if (!wait_w(smem_u32(&tl->tmem_empty[buf]), par ^ 1u, tl, P.ws, 604)) break;
                    tc_fence_after();
                    const unsigned b_lo = desc_lo_sw128(k_smem + buf * kStageBytes, 16), d_tmem = tmem_base + buf * 128;
                    if (elect_one()) {
#pragma unroll
                        for (int c = 0; c < 2; ++c)
#pragma unroll
                            for (int k4 = 0; k4 < 4; ++k4)
                                tc_mma_bf16_split(d_tmem, a_lo + ((c * (kQBytes / 2) + k4 * 32) >> 4), kDescHi,
                                                  b_lo + ((c * 2 * kHalfTile + k4 * 32) >> 4), kDescHi, kIdesc, (c | k4) != 0);
                        tc_commit(smem_u32(&tl->tmem_full[buf]));
                        tc_commit(smem_u32(&tl->empty[buf]));  // the stage is free once these MMAs have read it
                    }
                    __syncwarp();
                }
            } else if (epi_grp >= 0) {
                // This token's next candidate: at the first level every allowed block of the list, later the
                // right branches of its nodes, which ascend with the list: block due & 0xffff, of node
                // due >> 16. (From a ranked token's own list the one behind it is always on its way.)
                const int n_nodes = level > 0 && e_ok ? tl->n_nodes[epi_tok] : 0;
                int cur = -1;
                unsigned due = kNoBlock, next = kNoBlock;
                auto read_next = [&]() {
                    ++cur;
                    if constexpr (kSorted) {
                        next = cur < kNodes && n_nodes > 0 ? nodes[(kNodes + cur) * kPad + epi_tok] : kNoBlock;
                    } else {
                        for (next = kNoBlock; cur < n_nodes; ++cur) {
                            const unsigned nd = nodes[cur * kPad + epi_tok];
                            if ((nd >> 16) > 1u && right_of(nd) <= e_qlim) { next = (unsigned)right_of(nd) | ((unsigned)cur << 16); break; }
                        }
                    }
                };
                auto advance = [&]() {
                    if (kSorted) due = next;
                    if (!kSorted || (due & 0xffffu) != kNoBlock) read_next();
                    if (!kSorted) due = next;
                };
                if (level > 0) {
                    if (kSorted) read_next();
                    advance();
                }
                for (int i = 0; i < n_st; ++i) {
                    const unsigned s = seq + (unsigned)i, buf = s & 3u;
                    // the other group's stage: its blocks are passed over
                    const int blk2[2] = {list[2 * i], 2 * i + 1 < n_list ? list[2 * i + 1] : (int)kNoBlock - 1};
                    if ((int)(s & 1u) != epi_grp) {
                        while ((int)(due & 0xffffu) <= blk2[1]) advance();
                        continue;
                    }
                    if (!wait_w(smem_u32(&tl->tmem_full[buf]), (s >> 2) & 1u, tl, P.ws, 605)) break;
                    tc_fence_after();
#pragma unroll
                    for (int tile = 0; tile < 2; ++tile) {
                        const int blk = blk2[tile];
                        const bool mine = level == 0 ? blk <= e_qlim : blk == (int)(due & 0xffffu);
                        if (!__any_sync(0xffffffffu, mine)) continue;  // (a place behind the list is nobody's)
                        const unsigned taddr = tmem_base + buf * 128 + tile * 64 + ((unsigned)((warp & 3) * 32) << 16);
                        unsigned v[64];
                        tmem_ld_32x32_issue(taddr, v);
                        tmem_ld_32x32_issue(taddr + 32, v + 32);
                        // (while they are on their way:) where this token keeps the tile's score, what comes next
                        const int pos = level == 0 ? 2 * i + tile : 32 + (int)(due >> 16);
                        if (mine && level > 0) advance();
                        // keys of the block this token may look at: a prefix (inside T, not after the token if causal)
                        const int n_hi = key_end - blk * kBlk;
                        tmem_ld_wait();
                        if (__any_sync(0xffffffffu, mine && n_hi < kBlk)) {  // the token's own block, or a block across T
#pragma unroll
                            for (int j = 0; j < 64; ++j) v[j] = j < n_hi ? v[j] : 0xff800000u;
                        }
                        const float best = max_of_64(reinterpret_cast<const float *>(v));
                        if (mine) scores[pos * kPad + epi_tok] = best;
                    }
                    tc_fence_before();
                    mbar_arrive_if(smem_u32(&tl->tmem_empty[buf]), lane == 0);
                }
            }
            seq += (unsigned)n_st;
            if (level == 0) q_par ^= 1u;
            __syncthreads();  // every score of the level is in place
            if (*(volatile int *)&tl->abort_flag) break;  // (set only inside the level: the same answer in every thread)

            // ---- ranking. Up to 16 nodes: a thread per token (the first epilogue group's), which sorts its keys
            // in registers, 32 tokens a warp at once. More do not fit in registers: a warp per token, a
            // lane per node, which spends 240 instructions of a warp on every token, 8000 clocks a level of
            // the 128 against 3000. (32 / 8 heads, 4096 tokens: k = 16 225 us that way, 160 this way; k = 24,
            // spilled, 304 this way, 224 that way.)
            if constexpr (kSorted) {
            if (epi_grp == 0) {
                const int t = epi_tok;
                const int n = !e_ok ? 0 : (level == 0 ? tl->n_node0 : tl->n_nodes[t]);
                // Everything of the token goes to registers first: its nodes, and the keys of their left and
                // right candidates (0: there is none).
                unsigned nd[kNodes], own[2 * kNodes], key[2 * kNodes];
#pragma unroll
                for (int j = 0; j < kNodes; ++j) {
                    unsigned at = (unsigned)j | ((unsigned)(32 + j) << 16);
                    if (level == 0) { nd[j] = j < n ? tl->node0[j] : 0u; at = tl->place0[j]; }
                    else nd[j] = j < n ? nodes[j * kPad + t] : 0u;
                    const bool vl = nd[j] != 0u && (int)(nd[j] & 0xffffu) <= e_qlim, vr = (nd[j] >> 16) > 1u && right_of(nd[j]) <= e_qlim;
                    own[2 * j] = score_key(vl, vl ? scores[(at & 0xffffu) * kPad + t] : 0.f);
                    own[2 * j + 1] = score_key(vr, vr ? scores[(at >> 16) * kPad + t] : 0.f);
                }
                if (level == 0) {
#pragma unroll
                    for (int i = 0; i < 2 * kNodes; ++i) n_tiles += own[i] != 0u ? 1u : 0u;
                }
                // The k-th largest key, always in the same place of the sorted ones: kNodes - k places that
                // no candidate can have are taken by keys above all others.
#pragma unroll
                for (int i = 0; i < 2 * kNodes; ++i) key[i] = i % 2 == 0 && i / 2 >= kq ? 0xffffffffu : own[i];
                sort_step<2 * kNodes, 1, 1>(key);
                const unsigned thr = key[kNodes - 1];
                int above[4] = {0, 0, 0, 0};  // (counting the places taken)
#pragma unroll
                for (int i = 0; i < kNodes - 1; ++i) above[i & 3] += key[i] > thr ? 1 : 0;
                int missing = kNodes - (above[0] + above[1]) - (above[2] + above[3]);
                // what is kept, in order, to its place (nothing is left to be read there)
                unsigned n_new = 0u;
#pragma unroll
                for (int i = 0; i < 2 * kNodes; ++i) {
                    const bool equal = own[i] == thr && thr != 0u && missing > 0;
                    missing -= equal ? 1 : 0;
                    if (equal || own[i] > thr) {
                        const unsigned f = nd[i / 2] & 0xffffu, len = nd[i / 2] >> 16, left = (len + 1u) >> 1;
                        nodes[n_new * kPad + t] = i & 1 ? (f + left) | ((len - left) << 16) : f | (left << 16);
                        scores[n_new * kPad + t] = score_of_key(own[i]);
                        ++n_new;
                    }
                }
                tl->n_nodes[t] = (int)n_new;
                if (!last) {  // the token's candidates of the next level: the right branch of every node that has one
                    unsigned c = 0u;
#pragma unroll
                    for (int j = 0; j < kNodes; ++j) {
                        const unsigned x = j < (int)n_new ? nodes[j * kPad + t] : 0u;
                        const int rb = right_of(x);
                        if ((x >> 16) > 1u && rb <= e_qlim) {
                            nodes[(kNodes + c) * kPad + t] = (unsigned)rb | ((unsigned)j << 16);
                            ++c;
                            want(rb);
                        }
                    }
                    if (c < (unsigned)kNodes) nodes[(kNodes + c) * kPad + t] = kNoBlock;
                    n_tiles += c;
                } else if (e_ok) {
                    tiles_needed += n_tiles;
                    if (g.row_tiles != nullptr) g.row_tiles[((long long)b * g.H + h) * g.n_qb + e_tq] = n_tiles;
                }
            }
            } else {
            for (int i = 0; i < kTok / (kThreads / 32); ++i) {
                const int t = warp * (kTok / (kThreads / 32)) + i;
                const long long tq = tok0 + t;
                if (tq >= g.T) break;  // (uniform) tokens beyond T: no row
                const int q_lim = last_valid_block(g, (int)tq);
                int f, l, m;
                bool vl, vr;
                float sl = -CUDART_INF_F, sr = -CUDART_INF_F;
                if (level == 0) {
                    const unsigned nd = tl->node0[lane], at = tl->place0[lane];
                    f = (int)(nd & 0xffffu); l = f + (int)(nd >> 16) - 1; m = (f + l) / 2;
                    vl = nd != 0u && f <= q_lim; vr = vl && l > f && m + 1 <= q_lim;
                    if (vl) sl = scores[(at & 0xffffu) * kPad + t];
                    if (vr) sr = scores[(at >> 16) * kPad + t];
                    const int n0 = __popc(__ballot_sync(0xffffffffu, vl)) + __popc(__ballot_sync(0xffffffffu, vr));
                    if (lane == 0) { tiles_needed += (unsigned long long)n0; tl->n_tiles[t] = n0; }
                } else {
                    const int n = tl->n_nodes[t];
                    vl = lane < n;
                    const unsigned nd = vl ? nodes[lane * kPad + t] : pack_node(0, 0);
                    f = (int)(nd & 0xffffu); l = f + (int)(nd >> 16) - 1; m = (f + l) / 2;
                    vr = vl && l > f && m + 1 <= q_lim;
                    if (vl) sl = scores[lane * kPad + t];
                    if (vr) sr = scores[(32 + lane) * kPad + t];
                }
                const Keep kp = select_topk(vl, sl, vr, sr, kq, lane);
                const unsigned kl = __ballot_sync(0xffffffffu, kp.l), kr = __ballot_sync(0xffffffffu, kp.r);
                const int pos_l = __popc(kl & lt) + __popc(kr & lt), pos_r = pos_l + (kp.l ? 1 : 0);
                const int n_new = __popc(kl) + __popc(kr);
                __syncwarp();  // every lane has read its node and scores
                if (kp.l) { nodes[pos_l * kPad + t] = pack_node(f, m - f + 1); scores[pos_l * kPad + t] = sl; }
                if (kp.r) { nodes[pos_r * kPad + t] = pack_node(m + 1, l - m); scores[pos_r * kPad + t] = sr; }
                if (lane == 0) tl->n_nodes[t] = n_new;
                __syncwarp();
                const bool live = lane < n_new;
                const unsigned nn = live ? nodes[lane * kPad + t] : pack_node(0, 0);
                const int nf = (int)(nn & 0xffffu), nlen = (int)(nn >> 16);
                if (!last) {
                    // the token's candidates of the next level: the right branch of every node that has one
                    const int rb = (nf + nf + nlen - 1) / 2 + 1;
                    const bool has_r = live && nlen > 1 && rb <= q_lim;
                    if (has_r) want(rb);
                    const unsigned hb = __ballot_sync(0xffffffffu, has_r);
                    if (lane == 0) { tiles_needed += (unsigned long long)__popc(hb); tl->n_tiles[t] += __popc(hb); }
                } else {
                    if (lane == 0 && g.row_tiles != nullptr) g.row_tiles[((long long)b * g.H + h) * g.n_qb + tq] = (unsigned)tl->n_tiles[t];
                }
            }
            }
            if (last) {  // emit I[token, :]: first block of every surviving node, ascending, -1 padded
                __syncthreads();
                for (int i = 0; i < kTok / (kThreads / 32); ++i) {
                    const int t = warp * (kTok / (kThreads / 32)) + i;
                    const long long tq = tok0 + t;
                    if (tq >= g.T) break;  // (uniform) tokens beyond T: no row
                    const bool live = lane < tl->n_nodes[t];
                    const long long o = (((long long)b * g.H + h) * g.n_qb + tq) * g.k_top;
                    if (lane < g.k_top) {
                        P.mask[o + lane] = live ? (int)(nodes[lane * kPad + t] & 0xffffu) : -1;
                        if (P.score != nullptr) P.score[o + lane] = live ? scores[lane * kPad + t] : -CUDART_INF_F;
                    }
                }
            }
            if (last) break;
            __syncthreads();  // the bitmap holds every token's candidates
            if (warp == 0) {  // compact it into the ascending list (and clear it for the level after)
                int base = 0;
                const int n_words = (g.N_k + 31) >> 5;
                for (int w0 = 0; w0 < n_words; w0 += 32) {
                    const int w = w0 + lane;
                    unsigned bits = 0u;
                    if (bytes && w < n_words) {
#pragma unroll
                        for (int x = 0; x < 8; ++x) {
                            const unsigned y = bitmap[8 * w + x];
                            bitmap[8 * w + x] = 0u;
                            bits |= ((y & 1u) | ((y >> 7) & 2u) | ((y >> 14) & 4u) | ((y >> 21) & 8u)) << (4 * x);
                        }
                    } else if (w < n_words) {
                        bits = bitmap[w];
                        bitmap[w] = 0u;
                    }
                    const int cnt = __popc(bits);
                    int incl = cnt;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += y;
                    }
                    int at = base + incl - cnt;
                    while (bits) {
                        const int bit = __ffs(bits) - 1;
                        bits &= bits - 1;
                        list[at++] = (unsigned short)(w * 32 + bit);
                    }
                    base += __shfl_sync(0xffffffffu, incl, 31);
                }
                if (lane == 0) tl->n_list = base;
            }
        }
        if (*(volatile int *)&tl->abort_flag) break;
        if (warp == 0 && lane == 0) atomicAdd(&P.ws->rows, (unsigned long long)(tq_max - tok0 + 1));
        id = tl->item;
        __syncthreads();
    }
    // The tokens' rows that belong to no group: by the CTAs without one, where a quarter of the launch has none, else by all behind their last.
    if (P.first_tb > 0) {
        const int spare = (int)gridDim.x - P.n_items, first = 4 * spare >= (int)gridDim.x ? P.n_items : 0, writer = (int)blockIdx.x - first;
        constexpr int kWarps = kThreads / 32;
        if (writer >= 0) write_whole_rows(g, P.first_tb * kTok, writer * kWarps + warp, ((int)gridDim.x - first) * kWarps, lane, P.mask, P.ws);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tiles_needed += __shfl_xor_sync(0xffffffffu, tiles_needed, o);
    if (lane == 0 && (tiles_needed | products) != 0ull) {
        atomicAdd(&P.ws->tiles_scored, tiles_needed);
        atomicAdd(&P.ws->tile_products, products);
    }
    __syncwarp();

    leave(&tl->abort_flag, tmem_base, warp == 1);
}

}  // namespace

bool mask_tok_supported(const Geom &g, int dtype) {
    return dtype == STREAM_BF16 && g.d == kD && g.bq == 1 && g.bk == kBlk && g.k_top <= 32 && g.levels >= 1 &&
           g.N_k <= kMaxNk && g.k_row == nullptr && g.k_override == 0 && tma_strides_ok(g);
}

stream_status launch_mask_tok(const Geom &g, const void *q, const void *k, int32_t *mask, float *score,
                              WorkspaceHeader *ws, cudaStream_t st) {
    if (((uintptr_t)q & 15) != 0 || ((uintptr_t)k & 15) != 0) {
        set_error("tensor-core mask kernel needs 16-byte aligned q and k");
        return STREAM_ERR_UNSUPPORTED;
    }
    CUtensorMap tq, tk;
    stream_status rc = make_map_bf16_d128(&tq, q, g.T, g.H, g.batch, g.qs_t, g.qs_h, g.qs_b, "q", kTok);
    if (rc != STREAM_OK) return rc;
    rc = make_map_bf16_d128(&tk, k, g.T, g.G, g.batch, g.ks_t, g.ks_h, g.ks_b, "k");
    if (rc != STREAM_OK) return rc;
    Params P;
    P.g = g;
    // tokens that keep every block they are allowed, with no score asked for, need no products: whole groups of them have none
    const int whole = score == nullptr ? whole_query_blocks(g) : 0;
    if (whole == g.n_qb) return launch_mask_whole(g, g.n_qb, mask, ws, st);
    P.first_tb = whole / kTok;
    P.n_tb = (int)((g.T + kTok - 1) / kTok) - P.first_tb;
    const long long n_items = (long long)g.batch * g.H * P.n_tb;
    P.n_items = (int)n_items;
    P.walked_heads = walked_heads(g) * g.hpg;
    P.mask = mask; P.score = score; P.ws = ws;
    const int n_sm = sm_count();
    if (n_sm <= 0) { set_error("cannot read the SM count of the current device"); return STREAM_ERR_CUDA; }
    auto kern = g.k_top <= 16 ? mask_tok_kernel<16> : mask_tok_kernel<32>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(mask_tok)");
    // (a CTA more for every piece of the rows kept whole)
    const long long ctas = n_items + (P.first_tb > 0 ? whole_pieces(g, P.first_tb * kTok) : 0);
    const int grid = (int)(ctas < n_sm ? ctas : n_sm);
    e = launch_kernel(kern, grid, kThreads, kSmemBytes, st, 1, tq, tk, P);
    if (e != cudaSuccess) return cuda_fail(e, "mask_tok launch");
    return STREAM_OK;
}

}  // namespace stream
