// Tensor-core block-sparse attention for sm_100a (Eq. 2 on a Stream mask): bf16, d = 64 or 128, blocks
// of 32 or 64. (What follows is said for d = 128 and blocks of 64; Form has the differences.)
//
// One persistent CTA per SM works through "pairs": two rows (query blocks) of one kv head, as a rule two
// query heads at one query block. For every mask entry e the two rows name one key block each (K_0, K_1,
// usually different); the tiles arrive by TMA (128-byte swizzle), and each row r has its own products,
//     S_r = Q_r K_r^T  (64 x 64),     O_r += P_r V_r  (64 x 128),
// with M = 64: a row's 64 tokens take 16 of every 32 TMEM lanes (token 16 w + i in lane 32 w + 16 r + i),
// so the two rows share the columns of an accumulator and of P. A 64-row product takes the tensor
// cores as long as one of both rows together would (128 x 128 with half of S thrown away, 128 x 128
// under an output-lane mask for O), but less energy, and the chip is at its power limit here:
// 1475 -> 1660 MHz in a long run, 128k tokens (32 / 8 heads, k = 32) 6560 -> 6330 us, four layers of
// 9999 (k = 16) 935 -> 883, 4096 (k = 32) 166 -> 158.
//
// Where both rows name the same block at the same entry its K and V tiles are fetched once and serve both rows' products: at the power
// limit the bytes that an entry brings from L2 are as good as clocks (us, two fetches and one: 32 / 8 heads, 4096 tokens, k = 32,
// where the rows that keep all their blocks have the same lists, 151.0, 145.3; 16384, k = 16, 402.0, 393.4; 131072, k = 32, 6150, 6085;
// four layers of 9999 838.7, 835.3). Only there: a row walks its blocks in its own order, whatever the row beside it holds, so that its
// output is the same bit for bit however a call groups the query heads. (The blocks that both rows name anywhere first: 142.3, 384.4,
// 6047, 823 us, but the order of a row's entries, and with it the rounding of its P, was then a matter of its partner's list.)
// (d = 64, whose tiles are half as long, loses 1 % and is left. One product with M = 128 for both rows of a shared block: Q has to lie in
// TMEM for that, in the place of a second buffer of P, and the two shapes of product into O wait for one another or go
// under lane masks: with shared blocks first 126.5, 380, but 850 us for short lists that took 834.)
//
// Two softmax groups of four warps take a pair's entries in turn (its n-th kept entry belongs to
// group n % 2, so that a pair's arithmetic does not depend on what the CTA did before), so
// that one group's chain of waits, TMEM loads and exponentials runs beside the other's. A thread
// owns one query token (TMEM lane) of its group's entries: it reads the token's 64 logits, applies
// the element-level mask C, and writes P = exp2(scale (s - ref)) as bf16 to TMEM, where the P V
// product takes it as its A operand. The logits are given back as soon as they are in registers.
// A group has two buffers of logits and two of P: its next logits are there when it comes for them
// (with one buffer 421 against 411 us at T = 16384), and P need not wait for the product before. (Three logit buffers with P in
// their place instead hold a buffer through Q K^T, softmax and P V: 140 clocks an entry more.)
//
// `ref` is a per-token reference kept instead of the exact running maximum (bf16 P and fp32 sums
// keep their relative precision whatever the reference, as long as nothing overflows): the
// maximum of the token's first allowed logits, moved (with the token's O lane and sums rescaled)
// only when a logit has outgrown it by about 2^30 in exp2's argument, which the entry's sum of P
// shows. The groups share O, so they share the reference: it lives in shared memory, entry 0's
// group sets it before it computes its P, and entry n's warp looks at it again after entry n - 1's
// warp of the same lanes has published (`turn`), so that a reference that moved meanwhile is seen
// and P computed again. At the end of a pair the groups exchange their sums, normalise and store
// half of the channels each.
//
// What bounds it: an entry's products keep the tensor cores busy for 1050 clocks, its softmax work is
// about 2000 of one group's, and the chip runs at its power limit; an entry takes 1350 to
// 1450 clocks at 1600 to 1660 MHz. (What an issuing warp does between two chains counts all the same: one look at both of
// its barriers instead of two, and one commit fewer, 16384 tokens, k = 16: 408 -> 396 us; 131072, k = 32: 6190 -> 6070.) (With P in shared memory, 64 KB of stores and proxy fences, and one O
// per group: 1560 at 1475 MHz.)
//
// Roles (384 threads): warp 0 brings the K and Q tiles by TMA, warp 2 the V tiles and, ahead of
// everyone else, the pairs' mask rows; warp 1 issues the Q K^T chains and owns TMEM; warp 3 issues
// the P V chains (separate issuing warps, because the thread that issues a chain is held until the
// tensor core has taken it); warps 4..7 and 8..11 are the two softmax groups. Every role
// walks the same sequence of (pair, entry), read from the shared copy of the mask rows; they meet
// only on mbarriers. Every wait is bounded: on a timeout the CTA records a code in a device
// status word, raises a shared abort flag, lets its copies drain and leaves.
#include <math_constants.h>

#include "tc_common.cuh"

namespace stream {

// Status word of the tensor-core attention kernel: 0, or the code of the bounded wait that ran
// out (with the block index beside it). Read by stream_check_device_status.
__device__ unsigned int g_attn_status[2];

namespace {

using namespace tc;

constexpr int kThreads = 384;
constexpr int kHalfTile = 64 * 128;       // 64 rows x 128 bytes
// Blocks of 64: two rows in a unit, one in each half of the lanes. Blocks of 32: four, two stacked in
// each half: their 64 tokens meet the 64 keys of both rows' blocks, a token keeps its own row's half of
// the logits, and the other half of its P stays zero.
// d = 128 in blocks of 64: P goes into the product as bf16. Else: as a sum of two bf16, whose rounding is
// below that of the fp32 sums (what the kernels for the other shapes give, too).
template <int kD_, int kBlk_>
struct Form {
    static constexpr int kD = kD_, kBlk = kBlk_, kHalves = kD / 64;
    static constexpr int kRows = 128 / kBlk, kStack = 64 / kBlk;  // rows of a unit; those stacked in one half of the lanes
    static constexpr bool kSplit = !(kD == 128 && kBlk == 64);
    static constexpr bool kShare = kD == 128 && kBlk == 64;  // a block that both rows name at an entry is fetched once
    static constexpr int kPart = kBlk * 128;           // a row's block of one channel half
    static constexpr int kTile = kHalves * kHalfTile;  // 64 x d: the block of one row or those of two
    static constexpr int kOperand = 2 * kTile;         // two tiles: an entry's K or V, or the Q of a pair
    // Stages of the two rings, out of the operand buffers shared memory has room for beside Q. d = 128: five (a V
    // stage is held from its load until the product of its entry is complete, a whole softmax later:
    // V three, K two), or four when the mask rows are long.
    static constexpr int kMaxKStages = kD == 128 ? 2 : 6, kMaxVStages = kD == 128 ? 3 : 6;
    // Two K stages: one is free when the logits of the entry before last are there, which their own barrier says (its next
    // use is at least two entries later). More: a barrier of the stage's own, and a commit more for the issuing warp.
    static constexpr bool kKByLogits = kMaxKStages == 2;
    // Of `rings` buffers (the host sees to kMinRings at least): the stages of V, of K.
    static constexpr int kMinRings = 4;
    static __host__ __device__ constexpr int v_stages(int rings) { return kMaxVStages < (rings + 1) / 2 ? kMaxVStages : (rings + 1) / 2; }
    static __host__ __device__ constexpr int k_stages(int rings) { return kMaxKStages < rings - v_stages(rings) ? kMaxKStages : rings - v_stages(rings); }
    // TMEM columns: the two logit buffers of group g at 128 g and 64 behind, its P at 256 + 64 g (two
    // buffers, the second 32 behind, or the two parts of one), O at 384.
    static constexpr int kPBufs = kSplit ? 1 : 2;
    static constexpr int kPCol = 256, kOCol = 384;
    static constexpr int kOutBytes = kD;               // of an output token that one group stores (half of the channels)
    static constexpr unsigned kIdescQK = idesc_bf16(64, 64, false);  // B = a K tile, K-major
    static constexpr unsigned kIdescPV = idesc_bf16(64, kD, true);   // B = a V tile, MN-major
};
constexpr int kMaskSlots = 2;               // pairs whose mask rows are resident
constexpr int kMaxKTopTc = 1024;
constexpr float kLazySum = 68719476736.f;   // 2^36 = 64 * 2^30: the 64 P of an entry add up to more only if one of them exceeds 2^30 (its logit has outgrown the reference by 30 in log2 units)

// The pair a CTA works on. h[r], qb[r]: head and query block of row r < R (R = 0: a place of the
// order without a pair).
template <class F>
struct Item {
    int b, kvh, R;
    int h[F::kRows], qb[F::kRows];
};

template <class F>
struct Tail {
    unsigned long long q_full[2], q_free[2];  // q_free: the output staged over the pair's Q has left (8 warps)
    unsigned long long k_full[F::kMaxKStages], k_empty[F::kMaxKStages] /* (kKByLogits: not used) */, v_full[F::kMaxVStages], v_empty[F::kMaxVStages];
    unsigned long long s_full[2][2], s_free[2][2];        // per group and logit buffer: ready / read
    unsigned long long p_full[2][2], p_free[2][2];        // per group and P buffer: published / product added
    unsigned long long o_done, o_free;     // a pair's last product is complete; its O has been read (8 warps)
    // Between the two softmax warps of a lane quarter (one per group): the pair's first references
    // are set; group g has published an entry; both have left their sums.
    unsigned long long ref_set[4], turn[4][2], sums_there[4];
    unsigned long long m_full[kMaskSlots], m_empty[kMaskSlots];
    unsigned long long m_same[kMaskSlots];  // (kShare) bit e: both rows of the pair in that slot name the same block at entry e
    unsigned int tmem_base;
    int abort_flag;
    int m_count[kMaskSlots];  // entries of the pair in each mask slot
    Item<F> m_item[kMaskSlots];  // and the pair itself
    float ref[128], sum[2][128];
};
// Dynamic shared memory: Q (two buffers; a pair's output is staged over its Q) | V stages | K stages |
// Tail | mask rows [kMaskSlots][kRows][row_stride] (-1 where a row has nothing), the operands 1024-byte
// aligned.
constexpr int kFixedOperands = 2;  // Q; behind it the V stages, then the K stages
constexpr int kMaxSmemPerCta = 232448;

constexpr unsigned kRowLanes = 16u << 16;  // row 1's accumulator and P: the upper half of every 32 lanes
constexpr unsigned kHiK = desc_hi_sw128(1024);              // every operand: 8-row (8-key) groups 1024 bytes apart

struct Params {
    Geom g;
    int n_items;           // pairs
    int group_heads;       // kv heads (of the batch * G) whose pairs are walked together
    int row_stride;        // ints per resident mask row (k_top rounded up to a multiple of 4)
    int smem_bytes;        // dynamic shared memory of the launch
    int n_k_stages, n_v_stages;  // set by the kernel from what fits behind its aligned base
    const int32_t *mask;
    __nv_bfloat16 *out;
    float scale_log2;      // logit scale times log2(e)
};

// Bounded wait of a whole converged warp (all lanes get the same answer).
template <class F>
__device__ __forceinline__ bool wait_w(unsigned bar, unsigned parity, Tail<F> *tl, unsigned code) {
    return mbar_wait_warp(bar, parity, &tl->abort_flag, &g_attn_status[0], &g_attn_status[1], code);
}

// The same for two barriers, in one look where both phases are complete: for an issuing warp, which has a chain to
// issue every 700 clocks, each look of its own was 100 of them.
template <class F>
__device__ __forceinline__ bool wait_both_w(unsigned bar_a, unsigned parity_a, unsigned code_a, unsigned bar_b, unsigned parity_b, unsigned code_b, Tail<F> *tl) {
    if (__all_sync(0xffffffffu, mbar_try_wait_both(bar_a, parity_a, bar_b, parity_b))) return true;
    return wait_w(bar_a, parity_a, tl, code_a) && wait_w(bar_b, parity_b, tl, code_b);
}

// Shared copy of the mask rows of the pair in slot `slot`: [kRows][row_stride] ints behind the Tail.
template <class F>
__device__ __forceinline__ int *mask_rows(Tail<F> *tl, const Params &P, int slot) {
    return reinterpret_cast<int *>(tl + 1) + slot * F::kRows * P.row_stride;
}

// The order: `group_heads` kv heads at a time, as many as have K and V in L2 together, and within
// them late query blocks (most kept blocks under a causal mask) first. One kv head after the other,
// every head's short pairs in between, left the CTAs 11 % apart at T = 4096 (32 / 8 heads, k = 32;
// 4 % at T = 16384), this order with the turn of nth_item 1 %. A kv head's rows are counted query block by
// query block, head by head within one, and taken from the last in pairs (fours).
template <class F>
__device__ __forceinline__ Item<F> decode_item(const Params &P, int id) {
    const Geom &g = P.g;
    Item<F> it;
    const int n_rows = g.n_qb * g.hpg, levels = (n_rows + F::kRows - 1) / F::kRows;
    const int per_group = P.group_heads * levels;
    const int grp = id / per_group, rem = id - grp * per_group;
    const int heads = min(P.group_heads, g.batch * g.G - grp * P.group_heads);
    const int level = rem / heads, bh = grp * P.group_heads + (rem - level * heads);
    it.kvh = bh % g.G;
    it.b = bh / g.G;
    const int last = n_rows - 1 - level * F::kRows;
    it.R = min(F::kRows, last + 1);
#pragma unroll
    for (int r = 0; r < F::kRows; ++r) {
        const int row = max(last - r, 0);
        it.qb[r] = row / g.hpg;
        it.h[r] = it.kvh * g.hpg + row % g.hpg;
    }
    return it;
}

// Entry n of a pair: the key block of each row (negative: this row has nothing there). The mask loader
// keeps only the entries where some row has a block, in order, at the front of the resident rows, and
// leaves their number in the Tail.
template <class F>
struct Entry { int blk[F::kRows]; };
template <class F>
__device__ __forceinline__ Entry<F> entry_at(const int *rows, int stride, int n) {
    Entry<F> x;
#pragma unroll
    for (int r = 0; r < F::kRows; ++r) x.blk[r] = rows[r * stride + n];
    return x;
}

// ----------------------------------------------------------------------------------------------
// Roles. All walk the kept entries x_0 .. x_{n-1} of a pair in "rounds": round r handles the
// logits of x_r and the P V product of x_{r-1}.
// ----------------------------------------------------------------------------------------------
// Two warps feed the operand buffers, one the K tiles (with each pair's Q tiles), the other the V tiles
// and the mask rows: the copies one warp issues stream at 47 bytes per clock, and an entry's 64 KB
// would take 1400 clocks that way, more than its two chains. Neither blocks on one thing while another could
// move: every step probes its barrier without waiting. The warps run converged (lane 0's probe
// result is broadcast) and one elected lane issues.
template <class F>
struct LoadStream {
    int round, id;     // pair being walked
    int e;             // current entry (n = pair exhausted), -2 = pair not opened yet
    int n = 0;         // entries of the pair
    unsigned long long same = 0;  // bit x: both rows name the same block at the entry x behind the current one
    Entry<F> cur;
    int b, kvh;
    Ring ring, ms;
};

// Opens the stream's pair (its mask rows must be resident) or closes it; true if it did.
template <class F>
__device__ __forceinline__ bool open_pair(const Params &P, Tail<F> *tl, LoadStream<F> &S) {
    if (!probe_w(smem_u32(&tl->m_full[S.ms.idx]), S.ms.phase)) return false;
    S.b = tl->m_item[S.ms.idx].b;
    S.kvh = tl->m_item[S.ms.idx].kvh;
    S.n = tl->m_count[S.ms.idx];
    if (F::kShare) S.same = tl->m_same[S.ms.idx];
    S.e = 0;
    if (S.n > 0) S.cur = entry_at<F>(mask_rows(tl, P, S.ms.idx), P.row_stride, 0);
    return true;
}
template <class F>
__device__ __forceinline__ void close_pair(const Params &P, Tail<F> *tl, LoadStream<F> &S) {
    __syncwarp();  // (every lane has read what it needs of the slot; so wherever one lane arrives for its warp)
    if (elect_one()) mbar_arrive(smem_u32(&tl->m_empty[S.ms.idx]));
    __syncwarp();
    S.ms.advance(kMaskSlots);
    S.id = nth_item(++S.round);
    S.e = -2;
}
template <class F>
__device__ __forceinline__ void next_entry(const Params &P, Tail<F> *tl, LoadStream<F> &S) {
    S.same >>= 1;
    if (++S.e < S.n) S.cur = entry_at<F>(mask_rows(tl, P, S.ms.idx), P.row_stride, S.e);
}

// After a step that could not move: false if the CTA is aborting or nothing has moved for too long.
template <class F>
__device__ __forceinline__ bool idle_ok(Tail<F> *tl, long long t_last, unsigned code) {
    int stop = 0;
    if ((threadIdx.x & 31) == 0) {  // lane 0 decides for the warp
        if (*(volatile int *)&tl->abort_flag) stop = 1;
        else if (clock64() - t_last > kWaitCycles) {
            *(volatile int *)&tl->abort_flag = 1;
            if (atomicCAS(&g_attn_status[0], 0u, code) == 0u) g_attn_status[1] = blockIdx.x;
            stop = 1;
        }
    }
    if (__shfl_sync(0xffffffffu, stop, 0)) return false;
    __nanosleep(40);  // leave the issue slots to the softmax warps of this scheduler
    return true;
}

template <class F>
__device__ void k_producer_role(const Params &P, const CUtensorMap *tq, const CUtensorMap *tk, Tail<F> *tl, unsigned q_smem,
                                unsigned k_smem) {
    LoadStream<F> S;
    S.round = 0;
    S.id = nth_item(0);
    S.e = -2;
    // (kKByLogits) the last two entries, the older one in the stage that is next: the barrier of their logits (0: none), its phase
    unsigned cnt[2] = {0, 0}, bar_old = 0, bar_new = 0, par_old = 0, par_new = 0;
    auto step = [&]() -> bool {
        if (S.e == -2) return open_pair(P, tl, S);
        if (S.e >= S.n) { close_pair(P, tl, S); return true; }
        // a K stage is free once the logits computed from it are complete
        if constexpr (F::kKByLogits) {
            if (bar_old != 0 && !probe_w(bar_old, par_old)) return false;
            const unsigned gi = (unsigned)(S.e & 1), use = gi ? cnt[1]++ : cnt[0]++;
            bar_old = bar_new; par_old = par_new;
            bar_new = smem_u32(&tl->s_full[gi][use & 1u]); par_new = (use >> 1) & 1u;
        } else {
            if (!probe_w(smem_u32(&tl->k_empty[S.ring.idx]), S.ring.phase ^ 1)) return false;
        }
        if (elect_one()) {
            // [half][row][keys][128 B]; a row without a block at an entry gets block 0, its logits are masked out
            const unsigned bar = smem_u32(&tl->k_full[S.ring.idx]), dst = k_smem + S.ring.idx * F::kOperand;
            const bool both = F::kShare && (S.same & 1u) != 0;  // (in row 0's place)
            mbar_arrive_expect_tx(bar, (unsigned)(both ? F::kTile : F::kOperand));
#pragma unroll
            for (int c = 0; c < F::kHalves; ++c)
#pragma unroll
                for (int r = 0; r < F::kRows; ++r)
                    if (r == 0 || !both) tma_load_4d(dst + c * 2 * kHalfTile + r * F::kPart, tk, bar, c * 64, max(S.cur.blk[r], 0) * F::kBlk, S.kvh, S.b);
        }
        __syncwarp();
        S.ring.advance(P.n_k_stages);
        next_entry(P, tl, S);
        return true;
    };
    // The pairs' Q tiles, as early as a buffer and the pair's mask rows allow, a pair ahead of its K tiles
    // as a rule: asked for behind the pair's first K tiles they came 1200 clocks late. (A pair's mask
    // slot stays until this warp has closed the pair on the K side, which a pair's Q precedes.)
    Ring qs, qm;
    int q_round = 0, q_id = nth_item(0);
    auto q_step = [&]() -> bool {
        if (q_id >= P.n_items || !probe_w(smem_u32(&tl->m_full[qm.idx]), qm.phase)) return false;
        if (tl->m_count[qm.idx] > 0) {
            if (!probe_w(smem_u32(&tl->q_free[qs.idx]), qs.phase ^ 1)) return false;
            if (elect_one()) {
                const Item<F> &it = tl->m_item[qm.idx];
                const unsigned bar = smem_u32(&tl->q_full[qs.idx]);
                mbar_arrive_expect_tx(bar, (unsigned)F::kOperand);
#pragma unroll
                for (int c = 0; c < F::kHalves; ++c)  // [half][row][tokens][128 B] (a missing row has those of another)
#pragma unroll
                    for (int r = 0; r < F::kRows; ++r)
                        tma_load_4d(q_smem + qs.idx * F::kOperand + c * 2 * kHalfTile + r * F::kPart, tq, bar, c * 64, it.qb[r] * F::kBlk, it.h[r], it.b);
            }
            __syncwarp();
            qs.advance(2);
        }
        qm.advance(kMaskSlots);
        q_id = nth_item(++q_round);
        return true;
    };
    long long t_last = clock64();
    while (S.id < P.n_items) {
        // (a pair is closed only when its Q has been asked for: its mask slot is then given back)
        if (((S.e < S.n || S.round < q_round) && step()) || q_step()) t_last = clock64();
        else if (!idle_ok(tl, t_last, 101)) return;
    }
}

// The V tiles, and the pairs' mask rows up to two pairs ahead of everyone else: only the kept entries
// of a pair (an entry is kept if either row has a block there) go to shared memory, in order, with
// their number, so that the other roles index them instead of searching.
template <class F>
__device__ void v_producer_role(const Params &P, const CUtensorMap *tv, Tail<F> *tl, unsigned v_smem, int lane) {
    const Geom &g = P.g;
    LoadStream<F> S;
    S.round = 0;
    S.id = nth_item(0);
    S.e = -2;
    int m_round = 0, m_id = nth_item(0);  // the next pair whose mask rows are due
    bool asked = false;                      // its first 32 entries are on their way to registers
    Item<F> it;
    int first[F::kRows];
    const int32_t *row[F::kRows];
    Ring mw;
    auto fetch = [&](int e, int (&blk)[F::kRows]) {
#pragma unroll
        for (int r = 0; r < F::kRows; ++r) blk[r] = e < g.k_top && r < it.R ? row[r][e] : -1;
    };
    auto mask_step = [&]() -> bool {
        if (m_id >= P.n_items) return false;
        if (!asked) {
            it = decode_item<F>(P, m_id);
#pragma unroll
            for (int r = 0; r < F::kRows; ++r) row[r] = P.mask + (((long long)it.b * g.H + it.h[r]) * g.n_qb + it.qb[r]) * g.k_top;
            fetch(lane, first);
            asked = true;
            return true;
        }
        if (!probe_w(smem_u32(&tl->m_empty[mw.idx]), mw.phase ^ 1)) return false;
        int *dst = mask_rows(tl, P, mw.idx);
        int cnt = 0;
        unsigned same[2] = {0u, 0u};
        for (int base = 0; base < g.k_top; base += 32) {
            int blk[F::kRows];
            bool kept = false;
            if (base > 0) fetch(base + lane, blk);
#pragma unroll
            for (int r = 0; r < F::kRows; ++r) {
                if (base == 0) blk[r] = first[r];
                kept = kept || blk[r] >= 0;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, kept);
            const int pos = cnt + __popc(bal & ((1u << lane) - 1u));
            if (kept) {
#pragma unroll
                for (int r = 0; r < F::kRows; ++r) dst[r * P.row_stride + pos] = blk[r];
            }
            if (F::kShare && base < 64) {
                const bool both = kept && blk[0] == blk[F::kRows - 1];
#pragma unroll
                for (int x = 0; x < 2; ++x) same[x] |= __reduce_or_sync(0xffffffffu, both && pos >> 5 == x ? 1u << (pos & 31) : 0u);
            }
            cnt += __popc(bal);
        }
        __syncwarp();
        if (lane == 0) {
            tl->m_count[mw.idx] = cnt;
            if (F::kShare) tl->m_same[mw.idx] = same[0] | (unsigned long long)same[1] << 32;
            tl->m_item[mw.idx] = it;
            mbar_arrive(smem_u32(&tl->m_full[mw.idx]));
        }
        __syncwarp();
        mw.advance(kMaskSlots);
        m_id = nth_item(++m_round);
        asked = false;
        return true;
    };
    auto step = [&]() -> bool {
        if (S.e == -2) return open_pair(P, tl, S);
        if (S.e >= S.n) { close_pair(P, tl, S); return true; }
        // a V stage is free once the product computed from it is complete
        if (!probe_w(smem_u32(&tl->v_empty[S.ring.idx]), S.ring.phase ^ 1)) return false;
        if (elect_one()) {  // [row][half][keys][128 B]
            const unsigned bar = smem_u32(&tl->v_full[S.ring.idx]), dst = v_smem + S.ring.idx * F::kOperand;
            const bool both = F::kShare && (S.same & 1u) != 0;
            mbar_arrive_expect_tx(bar, (unsigned)(both ? F::kTile : F::kOperand));
#pragma unroll
            for (int r = 0; r < F::kRows; ++r)
                if (r == 0 || !both) tma_load_5d(dst + r * F::kHalves * F::kPart, tv, bar, 0, max(S.cur.blk[r], 0) * F::kBlk, S.kvh, 0, S.b);
        }
        __syncwarp();
        S.ring.advance(P.n_v_stages);
        next_entry(P, tl, S);
        return true;
    };
    long long t_last = clock64();
    while (S.id < P.n_items) {
        if (step() || mask_step()) t_last = clock64();
        else if (!idle_ok(tl, t_last, 102)) return;
    }
}

// The two issuing roles are run by all 32 lanes of their warps, converged: the waits are
// warp-wide, one elected lane issues.

// S_r = Q_r K_r^T of both rows for every kept entry.
template <class F>
__device__ void qk_role(const Params &P, Tail<F> *tl, unsigned q_smem, unsigned k_smem, unsigned tmem_base) {
    Ring ks, ms, qs;
    unsigned cnt[2] = {0, 0};  // entries each group has had over the whole kernel
    const unsigned q_lo0 = desc_lo_sw128(q_smem, 16), k_lo = desc_lo_sw128(k_smem, 16);
    for (int round = 0, id; (id = nth_item(round)) < P.n_items; ++round) {
        if (!wait_w(smem_u32(&tl->m_full[ms.idx]), ms.phase, tl, 207)) return;
        const int n_entries = tl->m_count[ms.idx];  // the issuers need no more than the count and which entries are one tile
        unsigned long long same = F::kShare ? tl->m_same[ms.idx] : 0ull;
        const unsigned q_lo = q_lo0 + qs.idx * (F::kOperand >> 4);
        if (n_entries > 0) {
            if (!wait_w(smem_u32(&tl->q_full[qs.idx]), qs.phase, tl, 201)) return;
            qs.advance(2);
        }
        for (int i = 0; i < n_entries; ++i, same >>= 1) {
            const unsigned gi = (unsigned)(i & 1), use = gi ? cnt[1]++ : cnt[0]++;  // entry i of a pair belongs to group i % 2
            if (!wait_both_w(smem_u32(&tl->k_full[ks.idx]), ks.phase, 202, smem_u32(&tl->s_free[gi][use & 1u]), ((use >> 1) & 1u) ^ 1u, 203, tl)) return;
            tc_fence_after();
            const unsigned d_tmem = tmem_base + gi * 128 + (use & 1u) * 64;
            const unsigned b_lo = k_lo + ks.idx * (F::kOperand >> 4), row_1 = F::kShare && (same & 1u) ? 0u : (unsigned)kHalfTile >> 4;
            if (elect_one()) {
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int c = 0; c < F::kHalves; ++c)
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4)
                            tc_mma_bf16_split(d_tmem + r * kRowLanes, q_lo + (((2 * c + r) * kHalfTile + k4 * 32) >> 4), kHiK,
                                              b_lo + r * row_1 + ((2 * c * kHalfTile + k4 * 32) >> 4), kHiK, F::kIdescQK, (c | k4) != 0);
                tc_commit(smem_u32(&tl->s_full[gi][use & 1u]));
                if (!F::kKByLogits) tc_commit(smem_u32(&tl->k_empty[ks.idx]));
            }
            __syncwarp();
            ks.advance(P.n_k_stages);
        }
        __syncwarp();
        if (elect_one()) mbar_arrive(smem_u32(&tl->m_empty[ms.idx]));
        __syncwarp();
        ms.advance(kMaskSlots);
    }
}

// O_r (+)= P_r V_r of both rows for every kept entry; a pair's first entry starts O afresh.
template <class F>
__device__ void pv_role(const Params &P, Tail<F> *tl, unsigned v_smem, unsigned tmem_base) {
    Ring vs, ms;  // vs: the entry's V stage
    unsigned cnt[2] = {0, 0};  // entries each group has had over the whole kernel
    unsigned free_par = 1;  // (the first wait passes at once)
    // a row's MN-major V block has its two 64-channel halves kPart apart
    const unsigned v_lo = desc_lo_sw128(v_smem, F::kPart), d_tmem = tmem_base + F::kOCol;
    for (int round = 0, id; (id = nth_item(round)) < P.n_items; ++round) {
        if (!wait_w(smem_u32(&tl->m_full[ms.idx]), ms.phase, tl, 208)) return;
        const int n_entries = tl->m_count[ms.idx];
        unsigned long long same = F::kShare ? tl->m_same[ms.idx] : 0ull;
        for (int i = 0; i < n_entries; ++i, same >>= 1) {
            const unsigned gi = (unsigned)(i & 1), use = gi ? cnt[1]++ : cnt[0]++, pb = use % F::kPBufs;
            // (P is there: also, O is rescaled if it had to be)
            if (!wait_both_w(smem_u32(&tl->v_full[vs.idx]), vs.phase, 205, smem_u32(&tl->p_full[gi][pb]), (use / F::kPBufs) & 1u, 204, tl)) return;
            if (i == 0) {
                if (!wait_w(smem_u32(&tl->o_free), free_par, tl, 206)) return;  // the previous pair's O has been read
                free_par ^= 1;
            }
            tc_fence_after();
            const unsigned a_tmem = tmem_base + F::kPCol + gi * 64 + pb * 32, b_lo = v_lo + vs.idx * (F::kOperand >> 4), row_1 = F::kShare && (same & 1u) ? 0u : (unsigned)F::kTile >> 4;
            if (elect_one()) {
#pragma unroll
                for (int r = 0; r < 2; ++r)  // row r of the pair: its P (or the parts of it), its V tile
#pragma unroll
                    for (int part = 0; part < (F::kSplit ? 2 : 1); ++part)
#pragma unroll
                        for (int s4 = 0; s4 < 4; ++s4)  // 16 keys per step: 8 columns of packed bf16
                            tc_mma_bf16_ta(d_tmem + r * kRowLanes, a_tmem + r * kRowLanes + part * 32 + s4 * 8,
                                           b_lo + r * row_1 + ((s4 / (F::kBlk / 16) * F::kHalves * F::kPart + s4 % (F::kBlk / 16) * 2048) >> 4), kHiK, F::kIdescPV, (i | part | s4) != 0);
                tc_commit(smem_u32(&tl->p_free[gi][pb]));
                tc_commit(smem_u32(&tl->v_empty[vs.idx]));
                if (i + 1 == n_entries) tc_commit(smem_u32(&tl->o_done));
            }
            __syncwarp();
            vs.advance(P.n_v_stages);
        }
        __syncwarp();
        if (elect_one()) mbar_arrive(smem_u32(&tl->m_empty[ms.idx]));
        __syncwarp();
        ms.advance(kMaskSlots);
    }
}

// One softmax group: four warps, thread = TMEM lane `row`, token `mq` of the pair's row `half`, for the
// entries n with n % 2 == grp (n numbers the kept entries of each pair, as in every role).
// The waits are warp-wide (same answer in every lane), so the warp stays converged for the
// warp-collective TMEM loads and stores and leaves together if the CTA aborts.
//
// A parity wait needs the phase before it complete in the eyes of the waiting thread: a group sees
// every phase of its own logit and P buffers; what it waits for of the other group's (`turn`) it
// has followed entry by entry within the pair, and everything of earlier pairs is complete after
// o_done.
template <class F>
__device__ void softmax_role(const Params &P, const CUtensorMap *to, Tail<F> *tl, unsigned char *q_ptr, unsigned tmem_base, int t) {
    const Geom &g = P.g;
    const int lane = t & 31, row = t & 127, grp = t >> 7, wq = row >> 5;
    // this thread's row of the pair, its token of the row's query block, its logits' first column (in stacked
    // rows: its row's half)
    const int r_own = (lane >> 4) * F::kStack + (F::kStack == 2 ? wq >> 1 : 0), mq = (F::kStack == 2 ? wq & 1 : wq) * 16 + (lane & 15);
    const int col = F::kStack == 2 ? (wq >> 1) * 32 : 0;
    const unsigned lanes = tmem_base + ((unsigned)(row & ~31) << 16);
    const unsigned turn_own = smem_u32(&tl->turn[wq][grp]), turn_other = smem_u32(&tl->turn[wq][grp ^ 1]);
    unsigned char *const stage = q_ptr + (grp * 4 + wq) * 32 * F::kOutBytes;  // this warp's 32 tokens x half of the channels in a Q buffer
    unsigned n_other = 0;     // entries of the other group before this pair, over the whole kernel
    unsigned n_own = 0;       // entries of this group so far
    const unsigned s_full = smem_u32(&tl->s_full[grp][0]), s_free = smem_u32(&tl->s_free[grp][0]), s_addr = lanes + grp * 128 + col;
    unsigned pair_par = 0;    // phase of the barriers that complete once per pair with entries
    int staged = -1;          // Q buffer whose staged output may still be on its way out
    Ring ms, qs;
    if constexpr (F::kStack == 2) {  // P of the keys that are not this row's stays zero
        unsigned zero[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) zero[i] = 0;
        tmem_st_32x32_issue(lanes + F::kPCol + grp * 64, zero);
        tmem_st_32x32_issue(lanes + F::kPCol + grp * 64 + 32, zero);
        tmem_st_wait();
    }
    auto release_stage = [&]() {
        if (staged < 0) return;
        if (lane == 0) {
            tma_store_wait_read();
            mbar_arrive(smem_u32(&tl->q_free[staged]));
        }
        __syncwarp();
        staged = -1;
    };
    for (int round = 0; nth_item(round) < P.n_items; ++round) {
        if (!wait_w(smem_u32(&tl->m_full[ms.idx]), ms.phase, tl, 305)) return;
        const Item<F> &it = tl->m_item[ms.idx];
        const int h = it.h[r_own], qb = it.qb[r_own], b = it.b;
        const int tq0 = qb * F::kBlk;  // (token numbers fit 32 bits: TMA coordinates)
        const bool row_active = r_own < it.R && tq0 + mq < g.T;
        const int key_end = row_active ? (g.causal ? tq0 + mq + 1 : (int)g.T) : 0;  // keys this token may attend: those before
        const int n_entries = tl->m_count[ms.idx], last_entry = max(n_entries - 1, 0);
        const int *my_row = mask_rows(tl, P, ms.idx) + r_own * P.row_stride;  // this token's row of the pair
        float ref = -CUDART_INF_F, l = 0.f;
        // the entry's key block of this token's row; the keys of it the token may attend, a prefix of n_hi
        auto allowed_keys = [&](int blk) { return blk >= 0 ? max(0, min(key_end - blk * F::kBlk, F::kBlk)) : 0; };
        int n_hi = allowed_keys(grp < n_entries ? my_row[grp] : -1);
        bool masked = __any_sync(0xffffffffu, n_hi != F::kBlk);  // the diagonal block, one across T, a row without one
        for (int n = grp; n < n_entries; n += 2) {  // entry n of a pair belongs to group n % 2
            // the token's 64 logits against its row's key block
            const unsigned sb = n_own & 1u, pb = n_own % F::kPBufs;  // the entry's logit and P buffers
            if (!wait_w(s_full + sb * 8, (n_own >> 1) & 1u, tl, 301)) return;
            tc_fence_after();
            unsigned sr[F::kBlk];
#pragma unroll
            for (int x = 0; x < F::kBlk / 32; ++x) tmem_ld_32x32_issue(s_addr + sb * 64 + 32 * x, sr + 32 * x);
            tmem_ld_wait();
            tc_fence_before();
            mbar_arrive_if(s_free + sb * 8, lane == 0);
            if (masked) {
#pragma unroll
                for (int i = 0; i < F::kBlk; ++i) sr[i] = i < n_hi ? sr[i] : 0xff800000u;
            }
            // the pair's first entry sets the references of the tokens it has keys for
            if (n == 0) {
                ref = max_of<F::kBlk>(reinterpret_cast<const float *>(sr));
                tl->ref[row] = ref;
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&tl->ref_set[wq]));
            } else if (n == 1) {
                if (!wait_w(smem_u32(&tl->ref_set[wq]), pair_par, tl, 307)) return;
                ref = tl->ref[row];
            }
            // P under the present reference, their sum, the packed row. A token without a reference, or
            // with a logit that has outgrown it, shows in the sum, and a reference the other group has
            // moved meanwhile in shared memory: then once more. Whether entry n - 1 of this lane
            // quarter is published, and the P buffer's last product added, is looked up halfway
            // through, so that the latency of it is hidden.
            const unsigned other = n_other + (unsigned)((n - 1) >> 1), turn_par = other & 1u;  // entry n - 1 is the other group's `other`-th
            const int next_blk = my_row[min(n + 2, last_entry)];  // (of no meaning behind the last)
            int next_hi = 0;
            const unsigned p_free = smem_u32(&tl->p_free[grp][pb]), p_par = ((n_own / F::kPBufs) & 1u) ^ 1u;
            const unsigned p_addr = lanes + F::kPCol + grp * 64 + (F::kSplit ? 0 : pb * 32) + col / 2;
            unsigned packed[F::kSplit ? 16 : 32], rest[16];
            float esum;
            for (int attempt = 0;; ++attempt) {
                const float shift = ref == -CUDART_INF_F ? 0.f : -ref * P.scale_log2;
                const unsigned long long scale2 = pack_f32x2(P.scale_log2, P.scale_log2), shift2 = pack_f32x2(shift, shift);
                unsigned long long sum2[4] = {0ull, 0ull, 0ull, 0ull};
                auto weights = [&](int i0) -> bool {
#pragma unroll
                    for (int i = i0; i < i0 + 32; i += 2) {
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(pack_u32x2(sr[i], sr[i + 1]), scale2, shift2), x0, x1);
                        const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                        sum2[(i >> 1) & 3] = add_f32x2(sum2[(i >> 1) & 3], pack_f32x2(p0, p1));
                        const __nv_bfloat162 pk = __floats2bfloat162_rn(p0, p1);
                        packed[F::kSplit ? (i >> 1) & 15 : i >> 1] = *reinterpret_cast<const unsigned *>(&pk);
                        if (F::kSplit) {
                            const float2 top = __bfloat1622float2(pk);
                            const __nv_bfloat162 low = __floats2bfloat162_rn(p0 - top.x, p1 - top.y);
                            rest[(i >> 1) & 15] = *reinterpret_cast<const unsigned *>(&low);
                        }
                    }
                    if (F::kSplit) {  // (half at a time: both parts of a whole row do not fit in registers beside the logits)
                        // the product of the group's last entry, from the same buffer, is complete
                        if (i0 == 0 && !wait_w(p_free, p_par, tl, 309)) return false;
                        tmem_st_32x16_issue(p_addr + (i0 >> 1), packed);
                        tmem_st_32x16_issue(p_addr + 32 + (i0 >> 1), rest);
                    }
                    return true;
                };
                if (!weights(0)) return;
                bool seen = mbar_test_wait(p_free, p_par);
                float now = ref;
                if (n > 0) {
                    seen = mbar_test_wait(turn_other, turn_par) && seen;
                    now = *(volatile float *)&tl->ref[row];
                }
                next_hi = allowed_keys(next_blk);
                if constexpr (F::kBlk == 64) weights(32);
                float e0, e1;
                unpack_f32x2(add_f32x2(add_f32x2(sum2[0], sum2[1]), add_f32x2(sum2[2], sum2[3])), e0, e1);
                esum = e0 + e1;
                bool moved = __float_as_uint(now) != __float_as_uint(ref);
                const bool outgrown = (ref == -CUDART_INF_F && n_hi > 0) || !(esum <= kLazySum);
                // (no attempt beyond the third: a reference moves at most once under each group's hands)
                if (!__any_sync(0xffffffffu, !seen || moved || outgrown)) break;
                if (!wait_w(p_free, p_par, tl, 309)) return;
                if (n > 0) {
                    if (!wait_w(turn_other, turn_par, tl, 308)) return;
                    now = *(volatile float *)&tl->ref[row];
                    moved = __float_as_uint(now) != __float_as_uint(ref);
                }
                if (attempt == 2 || !__any_sync(0xffffffffu, moved || outgrown)) break;
                if (F::kSplit) tmem_st_wait();
                if (moved) {
                    if (ref != -CUDART_INF_F) l *= fast_exp2((ref - now) * P.scale_log2);
                    ref = now;
                }
                const bool move = outgrown && !moved;
                if (__any_sync(0xffffffffu, move)) {
                    float f = 1.f;
                    if (move) {
                        const float mx = max_of<F::kBlk>(reinterpret_cast<const float *>(sr));
                        if (ref != -CUDART_INF_F) f = fast_exp2((ref - mx) * P.scale_log2);
                        ref = mx;
                        tl->ref[row] = ref;
                    }
                    if (n > 0) {  // what has been added up so far is brought to the new reference
                        if (!wait_w(smem_u32(&tl->p_free[grp ^ 1][other % F::kPBufs]), (other / F::kPBufs) & 1u, tl, 302)) return;
                        tc_fence_after();
                        rescale_lane<F::kD>(lanes + F::kOCol, f);
                    }
                    l *= f;
                }
            }
            l += esum;
            if constexpr (!F::kSplit) tmem_st_32x32_issue(p_addr, packed);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();  // lane 0 speaks for all lanes: their references and P come before its arrivals
            mbar_arrive_if(turn_own, lane == 0);
            mbar_arrive_if(smem_u32(&tl->p_full[grp][pb]), lane == 0);
            ++n_own;
            n_hi = next_hi;
            masked = __any_sync(0xffffffffu, n_hi != F::kBlk);
            release_stage();  // the previous pair's output has long been read
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tl->m_empty[ms.idx]));  // (nothing of the slot is read below)
        ms.advance(kMaskSlots);
        if (n_entries > 0) {
            release_stage();
            if (!wait_w(smem_u32(&tl->o_done), pair_par, tl, 303)) return;
            tc_fence_after();
            // both groups' sums, under the pair's last reference
            const float now = tl->ref[row];
            if (ref != -CUDART_INF_F && now != ref) l *= fast_exp2((ref - now) * P.scale_log2);
            tl->sum[grp][row] = l;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tl->sums_there[wq]));
            unsigned ra[F::kD / 2];  // this group stores half of the channels of every token
#pragma unroll
            for (int x = 0; x < F::kD / 64; ++x) tmem_ld_32x32_issue(lanes + F::kOCol + grp * (F::kD / 2) + 32 * x, ra + 32 * x);
            tmem_ld_wait();
            tc_fence_before();
            if (!wait_w(smem_u32(&tl->sums_there[wq]), pair_par, tl, 304)) return;
            const float total = l + tl->sum[grp ^ 1][row];
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tl->o_free));
            const float inv = total > 0.f ? 1.f / total : 0.f;
            // The warp's part goes to the pair's Q buffer, whose last product is complete, and
            // from there to global memory as one TMA store (rows beyond T are left out): a lane's
            // own 128 bytes stored directly would touch 32 lines with every instruction.
            unsigned char *const dst = stage + qs.idx * F::kOperand + lane * F::kOutBytes;
            const int turned = F::kOutBytes == 128 ? lane & 7 : (lane >> 1) & 3;  // the swizzle of the map's 128 or 64 bytes
#pragma unroll
            for (int c = 0; c < F::kOutBytes / 16; ++c) {
                unsigned w[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const __nv_bfloat162 pk = __floats2bfloat162_rn(__uint_as_float(ra[8 * c + 2 * u]) * inv, __uint_as_float(ra[8 * c + 2 * u + 1]) * inv);
                    w[u] = *reinterpret_cast<const unsigned *>(&pk);
                }
                *reinterpret_cast<uint4 *>(dst + ((c ^ turned) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            fence_async_smem();
            __syncwarp();
            const int tok = tq0 + (mq & ~15);
            const int h_1 = __shfl_sync(0xffffffffu, h, 16), tok_1 = __shfl_sync(0xffffffffu, tok, 16);
            const bool there_1 = __shfl_sync(0xffffffffu, (int)row_active, 16) != 0;
            if (lane == 0) {  // lanes 0 and 16 hold the first of the 16 tokens of a row
                const unsigned src = smem_u32(stage + qs.idx * F::kOperand);
                if (row_active) tma_store_4d(to, src, grp * (F::kD / 2), tok, h, b);
                if (there_1) tma_store_4d(to, src + 16 * F::kOutBytes, grp * (F::kD / 2), tok_1, h_1, b);
                tma_store_commit();
            }
            staged = qs.idx;
            qs.advance(2);
            pair_par ^= 1;
            n_other += (unsigned)(grp == 0 ? n_entries >> 1 : (n_entries + 1) >> 1);
        } else if (row_active) {
            uint4 *dst = reinterpret_cast<uint4 *>(P.out + (((long long)b * g.H + h) * g.T + tq0 + mq) * F::kD + grp * (F::kD / 2));
#pragma unroll
            for (int c = 0; c < F::kOutBytes / 16; ++c) dst[c] = make_uint4(0, 0, 0, 0);
        }
    }
    if (lane == 0) tma_store_wait_read();  // shared memory is given back when the CTA leaves
    __syncwarp();
}

template <class F>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
               const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_out, Params P) {  // P by value: n_k_stages is filled in here
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = aligned_smem(smem_raw);
    // what is left behind the aligned base decides the number of V and K stages (the same in every thread)
    const int fixed_bytes = (int)(smem - smem_raw) + (int)sizeof(Tail<F>) + kMaskSlots * F::kRows * P.row_stride * (int)sizeof(int);
    const int n_rings = (P.smem_bytes - fixed_bytes) / F::kOperand - kFixedOperands;  // buffers for the two rings: d = 128: 4 or 5
    static_assert(!F::kKByLogits || (F::k_stages(F::kMinRings) == 2 && F::k_stages(F::kMinRings + 1) == 2), "two K stages, with however many buffers");
    P.n_v_stages = F::v_stages(n_rings);
    P.n_k_stages = F::k_stages(n_rings);
    const unsigned q_smem = smem_u32(smem), v_smem = q_smem + kFixedOperands * F::kOperand, k_smem = v_smem + P.n_v_stages * F::kOperand;
    Tail<F> *tl = (Tail<F> *)(smem + (kFixedOperands + P.n_v_stages + P.n_k_stages) * F::kOperand);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&tl->q_full[i]), 1); mbar_init(smem_u32(&tl->q_free[i]), 8); }
        for (int i = 0; i < F::kMaxKStages; ++i) { mbar_init(smem_u32(&tl->k_full[i]), 1); mbar_init(smem_u32(&tl->k_empty[i]), 1); }
        for (int i = 0; i < F::kMaxVStages; ++i) { mbar_init(smem_u32(&tl->v_full[i]), 1); mbar_init(smem_u32(&tl->v_empty[i]), 1); }
        for (int i = 0; i < 2; ++i) {
            for (int j = 0; j < 2; ++j) { mbar_init(smem_u32(&tl->s_full[i][j]), 1); mbar_init(smem_u32(&tl->s_free[i][j]), 4); mbar_init(smem_u32(&tl->p_full[i][j]), 4); mbar_init(smem_u32(&tl->p_free[i][j]), 1); }
        }
        mbar_init(smem_u32(&tl->o_done), 1);
        mbar_init(smem_u32(&tl->o_free), 8);
        for (int i = 0; i < 4; ++i) {
            mbar_init(smem_u32(&tl->ref_set[i]), 1);
            mbar_init(smem_u32(&tl->turn[i][0]), 1);
            mbar_init(smem_u32(&tl->turn[i][1]), 1);
            mbar_init(smem_u32(&tl->sums_there[i]), 2);
        }
        for (int i = 0; i < kMaskSlots; ++i) { mbar_init(smem_u32(&tl->m_full[i]), 1); mbar_init(smem_u32(&tl->m_empty[i]), 12); }
        tl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tl->tmem_base));  // all columns: one CTA per SM
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = tl->tmem_base;
    after_previous_kernel();

    if (warp == 0) {
        k_producer_role(P, &tmap_q, &tmap_k, tl, q_smem, k_smem);
    } else if (warp == 1) {
        qk_role(P, tl, q_smem, k_smem, tmem_base);
    } else if (warp == 2) {
        v_producer_role(P, &tmap_v, tl, v_smem, lane);
    } else if (warp == 3) {
        pv_role(P, tl, v_smem, tmem_base);
    } else {
        softmax_role(P, &tmap_out, tl, smem, tmem_base, (int)threadIdx.x - 128);
    }
    __syncwarp();

    leave(&tl->abort_flag, tmem_base, warp == 1);
}

}  // namespace

bool attn_tc_supported(const Geom &g, int dtype) { return g.d == 128 && g.bq == 64 && attn_tc_auto(g, dtype); }

// Against the mma.sync kernel, us: d = 64: 16 heads, 8192 tokens, k = 40, not causal: 600 -> 208; 6 heads, 12791
// tokens, k = 5: 57 -> 33. Blocks of 32: 12 heads, 10007 tokens, d = 128, k = 8: 152 -> 72; 32
// heads, 1416 tokens, d = 64, k = 60: 172 -> 96; 16 heads, 834 tokens, d = 128, k = 30: 51 -> 35.
bool attn_tc_auto(const Geom &g, int dtype) {
    return dtype == STREAM_BF16 && (g.d == 64 || g.d == 128) && (g.bq == 32 || g.bq == 64) && g.bk == g.bq &&
           g.k_top <= (g.bq == 64 ? kMaxKTopTc : kMaxKTopTc / 2) && tma_strides_ok(g);
}

namespace {
template <class F>
stream_status launch(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale, void *out,
                     cudaStream_t st) {
    CUtensorMap tq, tk, tv, to;
    stream_status rc = make_map_bf16(&tq, q, g.T, g.H, g.batch, g.qs_t, g.qs_h, g.qs_b, "q", F::kBlk, F::kD);  // 4-D: a block of one channel half
    if (rc != STREAM_OK) return rc;
    rc = make_map_bf16(&tk, k, g.T, g.G, g.batch, g.ks_t, g.ks_h, g.ks_b, "k", F::kBlk, F::kD);
    if (rc != STREAM_OK) return rc;
    rc = make_map5_bf16(&tv, v, g.T, g.G, g.batch, g.ks_t, g.ks_h, g.ks_b, "v", F::kBlk, F::kD);
    if (rc != STREAM_OK) return rc;
    rc = make_map_bf16(&to, out, g.T, g.H, g.batch, F::kD, g.T * F::kD, (long long)g.H * g.T * F::kD, "out", 16, F::kD, F::kD / 2);
    if (rc != STREAM_OK) return rc;
    Params P;
    P.g = g;
    const long long kv_bytes = 2ll * g.T * F::kD * 2;  // K and V of one kv head
    const long long fit = kL2KvBytes / kv_bytes, all = (long long)g.batch * g.G;
    P.group_heads = (int)(fit < 1 ? 1 : (fit > all ? all : fit));
    const long long n_items = all * (((long long)g.n_qb * g.hpg + F::kRows - 1) / F::kRows);
    if (n_items > 0x7fffffffLL - (1 << 20)) { set_error("too many rows for 32-bit indexing"); return STREAM_ERR_UNSUPPORTED; }
    P.n_items = (int)n_items;
    P.mask = mask;
    P.out = (__nv_bfloat16 *)out;
    P.scale_log2 = scale * 1.4426950408889634f;
    const int n_sm = sm_count();
    if (n_sm <= 0) { set_error("cannot read the SM count of the current device"); return STREAM_ERR_CUDA; }
    // room for all ring buffers if the mask rows are short enough, else fewer, but four; 1 KB of slack for the alignment
    // of the base (the kernel counts its stages from what it really gets)
    P.row_stride = (g.k_top + 3) & ~3;
    const int tail_bytes = (int)sizeof(Tail<F>) + kMaskSlots * F::kRows * P.row_stride * (int)sizeof(int);
    int smem_bytes = (kFixedOperands + F::kMaxKStages + F::kMaxVStages) * F::kOperand + tail_bytes + 1024;
    if (smem_bytes > kMaxSmemPerCta) smem_bytes = kMaxSmemPerCta;
    if (smem_bytes < (kFixedOperands + F::kMinRings) * F::kOperand + tail_bytes + 1024) {
        set_error("tensor-core attention kernel: k_top = %d needs more shared memory than one CTA has", g.k_top);
        return STREAM_ERR_UNSUPPORTED;
    }
    P.smem_bytes = smem_bytes;
    P.n_k_stages = P.n_v_stages = 0;
    cudaError_t e = cudaFuncSetAttribute(attn_tc_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmemPerCta);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(attn_tc)");
    const int grid = (int)(n_items < n_sm ? n_items : n_sm);
    e = launch_kernel(attn_tc_kernel<F>, grid, kThreads, smem_bytes, st, 1, tq, tk, tv, to, P);
    if (e != cudaSuccess) return cuda_fail(e, "attn_tc launch");
    return STREAM_OK;
}
}  // namespace

stream_status launch_attn_tc(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask,
                             float scale, void *out, cudaStream_t st) {
    if ((((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out) & 15) != 0) {
        set_error("tensor-core attention kernel needs 16-byte aligned q, k, v and out");
        return STREAM_ERR_UNSUPPORTED;
    }
    if (g.bq == 64) return g.d == 128 ? launch<Form<128, 64>>(g, q, k, v, mask, scale, out, st) : launch<Form<64, 64>>(g, q, k, v, mask, scale, out, st);
    return g.d == 128 ? launch<Form<128, 32>>(g, q, k, v, mask, scale, out, st) : launch<Form<64, 32>>(g, q, k, v, mask, scale, out, st);
}

stream_status read_attn_status(unsigned int out[2], cudaStream_t st) {
    cudaError_t e = cudaMemcpyFromSymbolAsync(out, g_attn_status, 2 * sizeof(unsigned int), 0, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyFromSymbolAsync(attention status)");
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    return STREAM_OK;
}

}  // namespace stream
