// Tensor-core Stream mask kernel for sm_100a: bf16, d = 64 or 128, blocks of 32 or 64, k_top <= 64.
// (Figures: d = 128, blocks of 64, unless they say otherwise.)
//
// One persistent CTA per SM (two smaller ones where two_of_four_rows or two_of_two_rows says so) works through "groups": up to four rows
// of one kv head, its query heads at one query block or, where these are few, at some. Their Q tiles stay in shared memory for the whole
// hierarchy (Algorithm 2).
// Candidate key blocks are fetched by TMA (128-byte swizzle), 128 keys at a time, into a ring of
// stages; one tcgen05.mma chain per (stage, row) computes the keys (128 x d) x Q_row^T (d x block)
// into a TMEM slot of as many columns (on the first level one chain for two rows: a chain of one is
// bound by its operands' way out of shared memory, 48 clocks a step of 16 channels against 64 for
// both); four epilogue warps reduce the slot to the masked tile maxima (Eq. 4 under C). There are two
// such groups of four, each serving one of every issuing warp's two slots: the fixed cost of a
// hand-over (wait, fences, arrive) is larger than the reduction itself, and one group alone would be
// the longest stage of the pipeline. A controller warp per
// row keeps the row's nodes in registers, ranks the 2k branch scores (higher score, then lower block
// index), compacts the survivors with ballots and publishes the next level's fetch list. The
// first level's representatives are the same for every row of a group, so one fetched stage
// serves all its rows (levels that cannot drop anything are passed over before it: FirstNodes); from the second
// level on a left branch inherits its parent's score and only right branches are fetched. With several k per call a group runs the hierarchy once per
// k on the same Q tiles and fetches only blocks whose score it does not have yet.
//
// Nothing of a group's beginning waits for the end of the group before: a dispatcher warp has the next
// group's number before it is needed, publishes its first list while the last one's later levels
// run (the level depends on the query block alone), and replaces a row's Q tile as soon as the row's
// last products are complete, so that the first tiles of the next group arrive behind the last
// products of this one. (One warp doing all of it, and ranking all four rows, kept the issuing
// warps waiting for a group or a list for 17 % (T = 16384, k = 16) to 29 % (several k) of the time.)
//
// What bounds it: the chip's power limit (1500 to 1570 MHz at T = 131072, 1590 at 16384, of 1965) with the tensor cores
// busy 70 to 88 % of the clocks; beside them the way of a stage (a third of it transfer) and the
// serial round of a row's level, list to ranked list, about 3500 clocks, which is what short lists wait for.
//
// Roles (608 threads; builds of two CTAs an SM have 320 or 384, one producer, two issuers and one epilogue group): warps 2 and 14 TMA producers of key tiles (even and odd stage buffers), warps 1,
// 3, 13, 17 MMA issuers (warp 1 owns TMEM), warp 18 dispatcher (groups, first lists, Q tiles), warps 0,
// 12, 16, 15 the controllers of rows 0..3, warps 4..7 and 8..11 the two epilogue groups (TMEM lane
// quarter = warp % 4). All roles walk the same fixed unit order (level 1: stage-major, row-minor;
// later levels: row-major), synchronised by mbarriers only. Every wait is bounded: on
// a timeout the CTA records an error code in the workspace header, raises a shared abort flag,
// drains its own copies and leaves.
#include <math_constants.h>

#include "tc_common.cuh"

namespace stream {
namespace {

using namespace tc;

constexpr int kStageKeys = 128;
constexpr int kFinal = 1 << 16;  // (several k) added to the length of a row's last list

// What a build of the kernel is for: head dimension, block size, two nodes a lane (k_top up to 64) or one
// (up to 32), several k with the score memory, rows of several query blocks in a group, two CTAs an SM (where Q and key tiles
// are small enough).
template <int kD_, int kBlk_, bool kWide_, bool kMulti_, bool kQbRows_ = false, bool kTwo_ = false>
struct Shape {
    static constexpr int kR = kTwo_ && kD_ == 128 && kBlk_ == 64 ? 2 : 4;  // rows (query heads, or query blocks) of a group, at most
    static constexpr int kD = kD_, kBlk = kBlk_;
    static constexpr bool kTwo = kTwo_;
    static constexpr int kThreads = kTwo ? 256 + 32 * kR : 608;
    static constexpr int kEpiGroups = kTwo ? 1 : 2;  // two: group g reduces the chains that land in slot g of their issuing warp; one: all
    static constexpr int kMmaWarps = kTwo ? 2 : 4;   // they take the stages in turn
    static constexpr int kProducers = kTwo ? 1 : 2;  // producer p fills the stage buffers b with b % kProducers == p
    static constexpr int kSlots = 2 * kMmaWarps;     // TMEM accumulator slots, one query block of fp32 columns each: two private ones per issuing warp
    static constexpr int kTmemColumns = kTwo ? kSlots * kBlk_ : 512;
    static constexpr int kListReaders = kProducers + kMmaWarps + 4 * kEpiGroups;  // producer, MMA and epilogue warps; of a first list and the group record also the controllers
    static constexpr bool kMulti = kMulti_, kQbRows = kQbRows_;
    static constexpr int kMaskRows = kQbRows ? kR / kEpiGroups : 1;  // of the rows an epilogue group has of a list, those with masks of their own
    static constexpr int kHalves = kD / 64;                 // 64-channel halves (128 bytes a row)
    static constexpr int kTps = kStageKeys / kBlk;          // tiles of a stage
    static constexpr int kParts = kBlk / 32;                // epilogue warps that share a tile
    static constexpr int kTile = kBlk * 128;                // a tile's part of one half
    static constexpr int kStageHalf = kStageKeys * 128;
    static constexpr int kStageBytes = kHalves * kStageHalf;
    static constexpr int kStages = (kTwo ? 64 : 128) * 1024 / kStageBytes;  // 128 KB of keys on their way to an SM
    static constexpr int kQBytes = kHalves * kR * kTile;    // [channel half][row]
    static constexpr int kNodes = kWide_ ? 2 : 1;           // nodes a lane of a controller holds
    static constexpr int kMaxJobs = 64 * kNodes;            // first list: two candidates per node
    static constexpr int kMaxRowJobs = 32 * kNodes;         // a row's list on a later level: at most one tile per node
    static constexpr int kListRegs = (kMaxJobs / kTps + 31) / 32;  // stages of a list, in lanes
    // A parity wait only means something to a thread that saw the phase before it complete, and an
    // arrival only if it cannot come a phase early. So every stage buffer and every TMEM slot
    // belongs to one issuing warp: stage s of the kernel's whole sequence goes, with all its chains,
    // to warp s % kMmaWarps and lands in buffer s % kStages, and a warp's chains alternate between its
    // own two slots. The other issuing warps touch none of its barriers.
    static_assert(kStages % kMmaWarps == 0, "a stage buffer must always meet the same issuing warp");
};

template <class S>
struct Tail {
    unsigned long long full[S::kHalves][S::kStages];  // by channel half
    unsigned long long empty[S::kStages], tmem_full[S::kSlots], tmem_empty[S::kSlots];
    // Per row: its Q tile is there; the last products of a group with it are complete (one commit of
    // every issuing warp).
    unsigned long long q_full[S::kR], q_free[S::kR];
    // Lists 0..kR-1: the rows' lists of the later levels; list kR: the first level's, with the group
    // record. The scores of the two kinds are kept and reported apart, those of the first level twice
    // (by the parity of the record): the next record's first level may be scored before a row's
    // controller has looked at this one's last, but the one after that is only published when
    // the controllers have read the next record, and are done with this one.
    unsigned long long jobs_ready[S::kR + 1], first_done[2][S::kR], scores_done[S::kR];
    // jobs_ack[i]: every reader of list i has taken what it needs from n_jobs[i], its blocks and, for
    // i = kR, the group record; who publishes the list waits for it before it writes them again.
    // Without it a warp with nothing to do in a short list could still be about to read it when the
    // next one is written, or fall two phases behind jobs_ready[i].
    unsigned long long jobs_ack[S::kR + 1];
    unsigned int tmem_base;
    int abort_flag;
    int grp_id, grp_b, grp_kvh, grp_qb, grp_h0, grp_R;
    int grp_levels;  // levels of this group's rows that have something to rank (they share the query block, hence k)
    int grp_k, grp_pass;
    int grp_nodes, grp_f[32 * S::kNodes], grp_l[32 * S::kNodes];  // the nodes before the first of them: first and last block
    int split_f[32 * S::kNodes], split_l[32 * S::kNodes];         // (the dispatcher's own, on the way there)
    unsigned grp_on[2 * S::kNodes];  // bit i of [2 x], [2 x + 1]: the left, right candidate of node kNodes i + x is on the first list
    int grp_new_q;   // 0: another pass over the same rows (several k), the Q tiles are already there
    int grp_last;    // the last pass over these rows: the Q tiles are given back
    int n_jobs[S::kR + 1];
    int first_blk[S::kMaxJobs], jobs_blk[S::kR][S::kMaxRowJobs];
    float first_part[2][S::kR][S::kMaxJobs][S::kParts], part[S::kR][S::kMaxRowJobs][S::kParts];
    float no_part;   // (written before a list's first tile, not read)
    alignas(16) unsigned keys[S::kR][S::kNodes == 1 ? 64 : 1];  // a row's candidates while it ranks them
    int node_f[S::kR][32 * S::kNodes], node_l[S::kR][32 * S::kNodes];
    float node_s[S::kR][32 * S::kNodes];
};
template <class S>
constexpr int kSmemBytes = S::kQBytes + S::kStages * S::kStageBytes + (int)sizeof(Tail<S>) + 1024;

// Bounded wait of a whole converged warp (all lanes get the same answer) that reports into the
// workspace header; false means the CTA is aborting.
template <class S>
__device__ __forceinline__ bool mbar_wait_w(unsigned bar, unsigned parity, Tail<S> *tl, WorkspaceHeader *ws, unsigned code) {
    return mbar_wait_warp(bar, parity, &tl->abort_flag, &ws->error, &ws->error_info, code);
}

// K-major, 128-byte-swizzled operands with 8-row groups 1024 bytes apart: high descriptor word.
constexpr unsigned kDescHi = desc_hi_sw128(1024);

// D fp32, A and B bf16, both K-major, M = 128, N = the tokens of one row or of two.
template <class S>
constexpr unsigned kIdesc = idesc_bf16(128, S::kBlk, false);
template <class S>
constexpr unsigned kIdescTwo = idesc_bf16(128, 2 * S::kBlk, false);

struct Params {
    Geom g;
    int n_groups, n_chunks;
    int walked_heads;  // kv heads (of the batch * G) whose groups are walked together
    int first_qb;  // the rows of the query blocks before it keep all they are allowed, and belong to no group
    // A group's rows: head_rows query heads, at each of qb_rows query blocks (more than one only where
    // all heads of the kv head are in the group): row r is head r % head_rows at the group's query
    // block minus r / head_rows, which row_head and row_back hold in two bits a row.
    int head_rows, qb_rows;
    unsigned row_head, row_back;
    int32_t *mask;
    float *score;
    WorkspaceHeader *ws;
    // Several sparsity constants in one launch: a group runs the hierarchy once per k, with its Q
    // tiles loaded once, and writes mask slab `pass`. A tile's score does not depend on k, so the
    // controller remembers every (row, block) score of the group in `cache` (one entry per row
    // and key block for each CTA: {group tag, score}) and only lists blocks no earlier pass scored.
    MultiK mk;                      // n = 0: one pass with the geometry's k; else in falling order
    int slab_of[kMaxMultiK];        // mask slab of the pass
    unsigned long long *cache;      // [gridDim.x][kR][N_k], zeroed before the launch; NULL = no sharing
    long long slab;                 // elements between two mask slabs
};

__device__ __forceinline__ unsigned long long cache_pack(unsigned tag, float s) {
    return ((unsigned long long)tag << 32) | (unsigned long long)__float_as_uint(s);
}

// ----------------------------------------------------------------------------------------------
// Roles
// ----------------------------------------------------------------------------------------------
// Run by all 32 lanes of a producer warp, converged (warp-wide waits, one elected lane issues): a
// single diverged lane issues TMA copies several times more slowly. Two producers share the
// stages by buffer parity: one alone is busy more than half of the time with the four copies and
// the barrier arm of a stage, and the issuing warps then wait for data.
template <class S>
__device__ void producer_role(const Params &P, const CUtensorMap *tk, Tail<S> *tl, unsigned k_smem, int which) {
    Ring st;
    unsigned grp_par = 0, jr_par = 0;  // jr_par: bit by bit for the rows
    unsigned long long fetched = 0;  // tiles this warp has asked TMA for
    for (;;) {
        if (!mbar_wait_w(smem_u32(&tl->jobs_ready[S::kR]), grp_par, tl, P.ws, 101)) return;
        grp_par ^= 1;
        if (tl->grp_id < 0) {
            if (elect_one()) atomicAdd(&P.ws->tiles_fetched, fetched);
            return;
        }
        const int b = tl->grp_b, kvh = tl->grp_kvh, R = tl->grp_R, levels = tl->grp_levels;
        unsigned open = S::kMulti && levels > 1 ? (1u << R) - 1u : 0u;  // (several k) rows with a list to come
        for (int level = 0; S::kMulti ? level == 0 || open != 0 : level < levels; ++level) {
            const int lists = level == 0 ? 1 : R;
            for (int x = 0; x < lists; ++x) {
                const int li = level == 0 ? S::kR : x;
                if (S::kMulti && level > 0 && !((open >> x) & 1u)) continue;
                if (level > 0) {
                    if (!mbar_wait_w(smem_u32(&tl->jobs_ready[x]), (jr_par >> x) & 1u, tl, P.ws, 102)) return;
                    jr_par ^= 1u << x;
                }
                int n = tl->n_jobs[li];
                if (S::kMulti && n >= kFinal) { n -= kFinal; open &= ~(1u << x); }
                const int *const list = level == 0 ? tl->first_blk : tl->jobs_blk[x];
                for (int j = 0; j < n; j += S::kTps) {
                    if ((st.idx & (S::kProducers - 1)) != which) { st.advance(S::kStages); continue; }  // the other producer's buffer
                    bool there[S::kTps];
                    int blk[S::kTps];
                    unsigned tiles = 0;
#pragma unroll
                    for (int x = 0; x < S::kTps; ++x) {
                        there[x] = x == 0 || j + x < n;
                        tiles += there[x] ? 1u : 0u;
                        blk[x] = there[x] ? list[j + x] : 0;
                    }
                    fetched += tiles;
                    if (!mbar_wait_w(smem_u32(&tl->empty[st.idx]), st.phase ^ 1, tl, P.ws, 103)) return;
                    if (elect_one()) {
                        // The halves of the channels have a barrier each, so that the products with the
                        // first begin while the second is still coming: with four stages the tensor
                        // cores wait for a stage's way from L2, and this takes a third off it. (12.97 ->
                        // 12.01 ms at T = 131072, k = 32. Giving the halves back one by one as well
                        // costs more in the producers' second wait than it gives: 12.23.)
#pragma unroll
                        for (int c = 0; c < S::kHalves; ++c) {
                            const unsigned bar = smem_u32(&tl->full[c][st.idx]);
                            const unsigned dst = k_smem + st.idx * S::kStageBytes + c * S::kStageHalf;
                            mbar_arrive_expect_tx(bar, tiles * S::kTile);
#pragma unroll
                            for (int x = 0; x < S::kTps; ++x)
                                if (there[x]) tma_load_4d(dst + x * S::kTile, tk, bar, c * 64, blk[x] * S::kBlk, kvh, b);
                        }
                    }
                    __syncwarp();
                    st.advance(S::kStages);
                }
                __syncwarp();  // done reading this list, in every lane
                if (elect_one()) mbar_arrive(smem_u32(&tl->jobs_ack[li]));
                __syncwarp();
            }
        }
    }
}

// kMmaWarps warps take the stages in turn (stage s belongs, with all its chains, to warp
// s % kMmaWarps): the waits, commits and bookkeeping between two chains of one warp take several
// times longer than the tensor core needs for a chain, so one issuing warp would leave it idle
// most of the time. All issuing warps walk the same unit order; each is run by all 32 lanes,
// converged: warp-wide waits, one elected lane issues.
//
// Which of the owner's two TMEM slots a chain lands in is a fixed function of its place in the
// unit order, so that the issuing warp and the epilogue groups agree on it without counting each
// other's chains: on the first level chain r of a stage goes to slot r % 2, later (one chain per
// stage) the chain of stage s goes to slot (s / kMmaWarps) % 2. Both sides keep one phase bit per
// slot they use.
template <class S>
__device__ __forceinline__ int chain_slot(int level, int r, unsigned stage) {
    return level == 0 ? (r & 1) : (int)((stage / S::kMmaWarps) & 1u);
}

template <class S>
__device__ void mma_role(const Params &P, Tail<S> *tl, unsigned q_smem, unsigned k_smem, unsigned tmem_base, int which) {
    unsigned grp_par = 0, jr_par = 0;  // jr_par: bit by bit for the rows
    unsigned q_par = 0;       // bit r: phase of row r's next Q tile
    unsigned stage_seq = 0;   // stages so far, over the whole kernel (the same in every role)
    unsigned slot_par = 0;    // bit i: phase of the next use of this warp's slot i
    const unsigned q_lo = desc_lo_sw128(q_smem, 16);
    const unsigned a_lo0 = desc_lo_sw128(k_smem, 16);
    for (;;) {
        if (!mbar_wait_w(smem_u32(&tl->jobs_ready[S::kR]), grp_par, tl, P.ws, 201)) return;
        grp_par ^= 1;
        if (tl->grp_id < 0) return;
        const int R = tl->grp_R, levels = tl->grp_levels;
        const bool give_back = tl->grp_last != 0;
        unsigned q_due = tl->grp_new_q ? (1u << R) - 1u : 0u;  // rows whose Q tile this warp has yet to see arrive
        unsigned open = S::kMulti && levels > 1 ? (1u << R) - 1u : 0u;  // (several k) rows with a list to come
        for (int level = 0; S::kMulti ? level == 0 || open != 0 : level < levels; ++level) {
            const int lists = level == 0 ? 1 : R;
            for (int x = 0; x < lists; ++x) {
                const int li = level == 0 ? S::kR : x;
                if (S::kMulti && level > 0 && !((open >> x) & 1u)) continue;
                if (level > 0) {
                    if (!mbar_wait_w(smem_u32(&tl->jobs_ready[x]), (jr_par >> x) & 1u, tl, P.ws, 203)) return;
                    jr_par ^= 1u << x;
                }
                int n = tl->n_jobs[li];
                const bool final = S::kMulti ? n >= kFinal || levels == 1 : level + 1 == levels;
                if (S::kMulti && n >= kFinal) { n -= kFinal; open &= ~(1u << x); }
                const unsigned n_st = (unsigned)(n + S::kTps - 1) / S::kTps;  // stages of this list
                __syncwarp();
                if (elect_one()) mbar_arrive(smem_u32(&tl->jobs_ack[li]));  // the count is all this role reads
                __syncwarp();
                const int r0 = level == 0 ? 0 : x, r1 = level == 0 ? R : x + 1;
                const unsigned s_end = stage_seq + n_st;
                // this warp's stages of the list: s = which (mod kMmaWarps)
                for (unsigned s = stage_seq + (((unsigned)which - stage_seq) & (S::kMmaWarps - 1)); s < s_end; s += S::kMmaWarps) {
                    const unsigned sidx = S::kStages == S::kMmaWarps ? (unsigned)which : s % S::kStages, a_lo = a_lo0 + sidx * (S::kStageBytes >> 4);
                    for (int r = r0; r < r1; r += 2) {
                        // first level: rows r and r + 1 in one chain, each in its slot
                        const bool two = level == 0 && r + 1 < r1;
                        const int sl = chain_slot<S>(level, r, s);
                        const int slot = 2 * which + sl;
                        const unsigned rows = two ? 3u << r : 1u << r;
                        for (int i = r; (q_due & rows) != 0; ++i) {
                            if (!((q_due >> i) & 1u)) continue;
                            if (!mbar_wait_w(smem_u32(&tl->q_full[i]), (q_par >> i) & 1u, tl, P.ws, 202)) return;
                            q_par ^= 1u << i;
                            q_due &= ~(1u << i);
                        }
                        if (!mbar_wait_w(smem_u32(&tl->tmem_empty[slot]), ((slot_par >> sl) & 1u) ^ 1u, tl, P.ws, 205)) return;
                        if (two && !mbar_wait_w(smem_u32(&tl->tmem_empty[slot + 1]), ((slot_par >> 1) & 1u) ^ 1u, tl, P.ws, 205)) return;
                        slot_par ^= two ? 3u : 1u << sl;
                        tc_fence_after();
                        const unsigned d_tmem = tmem_base + slot * S::kBlk;
                        const unsigned b_lo = q_lo + r * (S::kTile >> 4);
                        const unsigned idesc = two ? kIdescTwo<S> : kIdesc<S>;
#pragma unroll
                        for (int c = 0; c < S::kHalves; ++c) {
                            if (r == r0) {
                                if (!mbar_wait_w(smem_u32(&tl->full[c][sidx]), (s / S::kStages) & 1u, tl, P.ws, 204)) return;
                                tc_fence_after();
                            }
                            if (elect_one()) {
#pragma unroll
                                for (int k4 = 0; k4 < 4; ++k4)
                                    tc_mma_bf16_split(d_tmem, a_lo + ((c * S::kStageHalf + k4 * 32) >> 4), kDescHi,
                                                      b_lo + ((c * S::kR * S::kTile + k4 * 32) >> 4), kDescHi, idesc, (c | k4) != 0);
                                if (c + 1 == S::kHalves) {
                                    tc_commit(smem_u32(&tl->tmem_full[slot]));
                                    if (two) tc_commit(smem_u32(&tl->tmem_full[slot + 1]));
                                    // the stage is free once its last chain has read it (a commit covers
                                    // all earlier instructions of this thread)
                                    if (r + 2 >= r1) tc_commit(smem_u32(&tl->empty[sidx]));
                                }
                            }
                            __syncwarp();
                        }
                    }
                }
                stage_seq = s_end;
                if (level == 0)  // (a warp without a stage in this list)
                    for (int r = 0; r < R; ++r)
                        if ((q_due >> r) & 1u) {
                            if (!mbar_wait_w(smem_u32(&tl->q_full[r]), (q_par >> r) & 1u, tl, P.ws, 206)) return;
                            q_par ^= 1u << r;
                            q_due &= ~(1u << r);
                        }
                if (give_back && final) {  // the rows' last products with these Q tiles
                    if (elect_one())
                        for (int r = r0; r < r1; ++r) tc_commit(smem_u32(&tl->q_free[r]));
                    __syncwarp();
                }
            }
        }
    }
}

// One epilogue group (four warps, one per TMEM lane quarter). Group `grp` waits for and reduces
// the chains that land in slot `grp` of their issuing warp (chain_slot): a slot's barriers are
// then used by one group only, which sees every phase of them. It steps over the other group's
// chains without looking at them: the bookkeeping of a warp is serial code, and what it spends
// there it cannot spend reducing.
template <class S>
__device__ void epilogue_role(const Params &P, Tail<S> *tl, unsigned tmem_base, int wq, int grp, int lane) {
    const Geom &g = P.g;
    unsigned grp_par = 0, jr_par = 0;  // jr_par: bit by bit for the rows
    unsigned stage_seq = 0;
    unsigned full_par = 0;  // bit 2 w + i: phase of the next use of issuing warp w's slot i
    constexpr int kBlk = S::kBlk;
    const int tile = wq / S::kParts;                       // which tile of the stage this warp's lanes hold
    const int key = (wq % S::kParts) * 32 + lane;          // key index inside the tile
    constexpr int kMmaWarps = S::kMmaWarps, kEpiGroups = S::kEpiGroups;
    const unsigned full_bar = smem_u32(&tl->tmem_full[0]), empty_bar = smem_u32(&tl->tmem_empty[0]);
    const unsigned t_lane = tmem_base + ((unsigned)(wq * 32) << 16);
    const int whole_blocks = (int)(g.T / kBlk);
    for (;;) {
        if (!mbar_wait_w(smem_u32(&tl->jobs_ready[S::kR]), grp_par, tl, P.ws, 301)) return;
        const unsigned set = grp_par;
        grp_par ^= 1;
        if (tl->grp_id < 0) return;
        const int R = tl->grp_R, grp_qb = tl->grp_qb, levels = tl->grp_levels;
        auto qb_of = [&](int r) { return S::kQbRows ? grp_qb - (int)((P.row_back >> (2 * r)) & 3u) : grp_qb; };
        float last = 0.f;  // this lane's maximum of the last tile, and where the tile's goes
        unsigned last_to = smem_u32(&tl->no_part);
        auto put = [&] {
            const float best = warp_max(last);
            asm volatile("{\n.reg .pred p;\nsetp.eq.b32 p, %2, 0;\n@p st.shared.f32 [%0], %1;\n}" ::"r"(last_to), "f"(best), "r"(lane) : "memory");
        };
        // Register x of lane i: this warp's tile of the list's stage 32 x + i (-1: there is none, its
        // maximum is not looked at); bit i of masked[y][x]: that tile is not whole for the y-th of
        // this group's rows that the list serves.
        int my_blk[S::kListRegs];
        unsigned masked[S::kMaskRows][S::kListRegs];
        // One chain of this group: the list's stage i, the kernel's stage s, row r, the y-th, where the maximum goes.
        auto reduce = [&](unsigned s, unsigned i, int r, int y, unsigned slot, unsigned to) -> bool {
            const unsigned at = 2 * (s & (kMmaWarps - 1)) + slot;
            if (!mbar_wait_w(full_bar + at * 8, (full_par >> at) & 1u, tl, P.ws, 303)) return false;
            full_par ^= 1u << at;
            tc_fence_after();
            float best = -CUDART_INF_F;
            const unsigned taddr = t_lane + at * kBlk;
            unsigned m0 = masked[0][0], m1 = masked[0][S::kListRegs - 1];
#pragma unroll
            for (int z = 1; z < S::kMaskRows; ++z)
                if (y == z) { m0 = masked[z][0]; m1 = masked[z][S::kListRegs - 1]; }
            const bool whole = (((S::kListRegs > 1 && i >= 32 ? m1 : m0) >> (i & 31)) & 1u) == 0;
            if (whole) {
                unsigned v[kBlk];
#pragma unroll
                for (int x = 0; x < S::kParts; ++x) tmem_ld_32x32_issue(taddr + 32 * x, v + 32 * x);
                put();  // (the tile before this one, while the loads are on their way)
                tmem_ld_wait();
                // the slot goes back as soon as it is in registers: its issuing warp waits for it
                tc_fence_before();
                mbar_arrive_if(empty_bar + at * 8, lane == 0);
                best = max_of<kBlk>(reinterpret_cast<const float *>(v));
            } else {
                put();
                const int blk = __shfl_sync(0xffffffffu, S::kListRegs > 1 && i >= 32 ? my_blk[S::kListRegs - 1] : my_blk[0], i & 31);
                if (blk >= 0) {  // the diagonal block, or a block across T: rare, so little code rather than little time
                    // allowed queries for this key: inside T, and not before the key if causal
                    const int qb = qb_of(r), m_lim = min(kBlk, (int)g.T - qb * kBlk);
                    const int lo = key >= (int)g.T - blk * kBlk ? kBlk : (g.causal && blk == qb ? key : 0);
#pragma unroll 1
                    for (int i0 = 0; i0 < kBlk; i0 += 8) {
                        unsigned v[8];
                        tmem_ld_32x8_issue(taddr + i0, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int x = 0; x < 8; ++x)
                            if (i0 + x >= lo && i0 + x < m_lim) best = fmaxf(best, __uint_as_float(v[x]));
                    }
                }
                tc_fence_before();
                mbar_arrive_if(empty_bar + at * 8, lane == 0);
            }
            last = best;
            last_to = to;
            return true;
        };
        unsigned open = S::kMulti && levels > 1 ? (1u << R) - 1u : 0u;  // (several k) rows with a list to come
        for (int level = 0; S::kMulti ? level == 0 || open != 0 : level < levels; ++level) {
            const int lists = level == 0 ? 1 : R;
            for (int x = 0; x < lists; ++x) {
                const int li = level == 0 ? S::kR : x;
                if (S::kMulti && level > 0 && !((open >> x) & 1u)) continue;
                if (level > 0) {
                    if (!mbar_wait_w(smem_u32(&tl->jobs_ready[x]), (jr_par >> x) & 1u, tl, P.ws, 302)) return;
                    jr_par ^= 1u << x;
                }
                // All there is to read of the list, at once: a look at it chain by chain, with the
                // comparisons, was a good part of what a warp spends on a chain.
                int n = tl->n_jobs[li];
                if (S::kMulti && n >= kFinal) { n -= kFinal; open &= ~(1u << x); }
                const int *const list = level == 0 ? tl->first_blk : tl->jobs_blk[x];
#pragma unroll
                for (int y = 0; y < S::kListRegs; ++y) {
                    const int at = S::kTps * (32 * y + lane) + tile;
                    my_blk[y] = at < n ? list[at] : -1;
                }
                const int r0 = level == 0 ? (kEpiGroups == 2 ? grp : 0) : x, r1 = level == 0 ? R : x + 1;
#pragma unroll
                for (int z = 0; z < S::kMaskRows; ++z) {
                    if (z > 0 && level > 0) continue;
                    // key blocks without a mask: those before `whole`, but for the diagonal one
                    const int qb = qb_of(r0 + kEpiGroups * z), whole = qb < whole_blocks ? whole_blocks : 0, diag = g.causal ? qb : -1;
#pragma unroll
                    for (int y = 0; y < S::kListRegs; ++y)
                        masked[z][y] = __ballot_sync(0xffffffffu, my_blk[y] < 0 || my_blk[y] >= whole || my_blk[y] == diag);
                }
                __syncwarp();  // (lane 0 speaks for what every lane has read)
                mbar_arrive_if(smem_u32(&tl->jobs_ack[li]), lane == 0);
                const unsigned s_end = stage_seq + (unsigned)(n + S::kTps - 1) / S::kTps;
                // First level: every stage serves all rows, rows grp, grp + 2 are this group's, and each
                // issuing warp needs its slot back from the first before it can issue the second: so
                // the first rows of kMmaWarps stages, then the second ones (stage by stage the group
                // waited for that round trip with other warps' chains ready: 115 -> 99 us at
                // T = 4096, 32 / 8 heads, k = 32). Later one chain per stage, this group's are the
                // stages with (s / kMmaWarps) % 2 == grp.
                const unsigned part = smem_u32(level == 0 ? tl->first_part[set][0] : tl->part[x]) + wq * 4;  // (four warps: the kTps * kParts parts of a stage in order)
                const unsigned row_step = level == 0 ? S::kMaxJobs * S::kParts * 4 : 0;
                for (unsigned base = level == 0 ? stage_seq : stage_seq & ~(unsigned)(kMmaWarps - 1); base < s_end; base += kMmaWarps) {
                    const unsigned later = (base / kMmaWarps) & 1u;  // the slot of a chain behind the first level
                    if (kEpiGroups == 2 && level > 0 && (int)later != grp) continue;
                    const unsigned lo = max(base, stage_seq), hi = min(base + kMmaWarps, s_end);
                    for (int r = r0; r < r1; r += kEpiGroups)
                        for (unsigned s = lo; s < hi; ++s)
                            if (!reduce(s, s - stage_seq, r, S::kQbRows ? (r - r0) / kEpiGroups : 0, level == 0 ? (unsigned)r & 1u : later, part + r * row_step + (s - stage_seq) * 16)) return;
                }
                stage_seq = s_end;
                put();
                last_to = smem_u32(&tl->no_part);
                // this list is done for rows r0..r1: tell their controllers
                __syncwarp();
                if (lane == 0 && (!S::kMulti || level == 0 || n > 0))
                    for (int r = level == 0 ? 0 : x; r < r1; ++r) mbar_arrive(smem_u32(level == 0 ? &tl->first_done[set][r] : &tl->scores_done[r]));
            }
        }
    }
}

// Dispatcher and controllers ------------------------------------------------------------------------
// kMulti: several k per group with the score memory; false compiles the plain single-pass form.

// Is block blk a candidate of the first list of a build with k = kq, whose nodes have been split `splits` times?
__device__ __forceinline__ bool on_first_list(const Geom &g, int kq, int splits, int blk) {
    const int i = (int)(((long long)(blk + 1) * kq - 1) / g.N_k);  // the node that holds blk: the last that begins at or before it
    int f = (int)(((long long)i * g.N_k) / kq), l = (int)(((long long)(i + 1) * g.N_k) / kq) - 1;
    for (int x = 0; x < splits; ++x) {
        const int m = (f + l) / 2;
        if (blk <= m) l = m;
        else f = m + 1;
    }
    return blk == f || blk == (f + l) / 2 + 1;
}

template <class S>
__device__ void dispatcher_role(const Params &P, const CUtensorMap *tq, Tail<S> *tl, unsigned q_smem, int lane) {
    const Geom &g = P.g;
    constexpr bool kMulti = S::kMulti;
    constexpr int kNodes = S::kNodes;
    const unsigned lt = (1u << lane) - 1u;
    int splits_of = 0;  // lane i: of the group's pass i
    unsigned ack_par = 1, q_par = (1u << S::kR) - 1u;  // (the first waits pass at once)
    unsigned long long fetched = 0;  // Q tiles asked of TMA
    // (lane 0) the next group's number, if it has been fetched. The first one's is the CTA's own, the counter deals those behind.
    int next = (int)blockIdx.x;
    auto fetch = [&] { return (int)(gridDim.x + atomicAdd(&P.ws->work_counter, 1u)); };
    for (;;) {
        // the previous list and record have been read by everybody
        if (!mbar_wait_w(smem_u32(&tl->jobs_ack[S::kR]), ack_par, tl, P.ws, 402)) return;
        if (lane == 0 && next < 0) next = fetch();
        const int id = __shfl_sync(0xffffffffu, next, 0);
        const bool done = id >= P.n_groups || *(volatile int *)&tl->abort_flag;
        // the one after it a group ahead, unless that could leave another CTA without work
        next = -1;
        if (lane == 0 && id + 2 * (int)gridDim.x < P.n_groups) next = fetch();
        int b = 0, kvh = 0, qb = 0, h0 = 0, R = 0;
        if (!done) {
            // late (expensive) query blocks of all the heads walked together first
            const int levels = (g.n_qb - P.first_qb + P.qb_rows - 1) / P.qb_rows, per = P.walked_heads * levels * P.n_chunks;
            const int walk = id / per, rem = id - walk * per, heads = min(P.walked_heads, g.batch * g.G - walk * P.walked_heads);
            const int level = rem / (heads * P.n_chunks), at = rem - level * heads * P.n_chunks, head = at / P.n_chunks, chunk = at - head * P.n_chunks;
            const int bkv = walk * P.walked_heads + head;
            b = bkv / g.G; kvh = bkv % g.G;
            qb = g.n_qb - 1 - level * P.qb_rows;
            h0 = kvh * g.hpg + chunk * P.head_rows;
            R = min(P.head_rows, g.hpg - chunk * P.head_rows) * min(P.qb_rows, qb - P.first_qb + 1);
        }
        const int q_lim = last_valid_block(g, qb);
        const int n_pass = (!kMulti || done) ? 1 : P.mk.n;
        for (int pass = 0; pass < n_pass; ++pass) {
            const int kq = done ? g.k_top : (kMulti ? P.mk.k[pass] : row_k(g, qb));
            const int levels = row_levels(g, kq);
            const FirstNodes<kNodes> nodes(g, kq, levels, q_lim, lane, tl->split_f, tl->split_l);
            bool on[2 * kNodes];  // goes on the list
            int cand[2 * kNodes];
            unsigned ballots[2 * kNodes];
#pragma unroll
            for (int x = 0; x < kNodes; ++x) {
                cand[2 * x] = nodes.f[x]; cand[2 * x + 1] = (nodes.f[x] + nodes.l[x]) / 2 + 1;
                on[2 * x] = nodes.left[x] && !done; on[2 * x + 1] = nodes.right[x] && !done;
            }
            // Not what an earlier pass has had on its first list: every row has that score. (What rows have
            // met on later levels is for their controllers to know, which may still be at it.)
            for (int e = 0; kMulti && e < pass; ++e) {
                const int splits = __shfl_sync(0xffffffffu, splits_of, e);
#pragma unroll
                for (int x = 0; x < 2 * kNodes; ++x) on[x] = on[x] && !on_first_list(g, P.mk.k[e], splits, cand[x]);
            }
            if (kMulti && lane == pass) splits_of = nodes.splits;
#pragma unroll
            for (int x = 0; x < 2 * kNodes; ++x) ballots[x] = __ballot_sync(0xffffffffu, on[x]);
            int place = flags_before(ballots, lt);
            if (pass > 0 && !mbar_wait_w(smem_u32(&tl->jobs_ack[S::kR]), ack_par, tl, P.ws, 409)) return;
            ack_par ^= 1;
#pragma unroll
            for (int x = 0; x < 2 * kNodes; ++x)
                if (on[x]) tl->first_blk[place++] = cand[x];
#pragma unroll
            for (int x = 0; x < kNodes; ++x) { tl->grp_f[kNodes * lane + x] = nodes.f[x]; tl->grp_l[kNodes * lane + x] = nodes.l[x]; }
            if (lane == 0) {
                tl->n_jobs[S::kR] = flags_all(ballots);
                tl->grp_id = done ? -1 : id; tl->grp_b = b; tl->grp_kvh = kvh; tl->grp_qb = qb; tl->grp_h0 = h0; tl->grp_R = R;
                tl->grp_levels = levels - nodes.splits;
                tl->grp_k = kq; tl->grp_pass = pass; tl->grp_nodes = nodes.n;
#pragma unroll
                for (int x = 0; x < 2 * kNodes; ++x) tl->grp_on[x] = ballots[x];
                tl->grp_new_q = pass == 0;
                tl->grp_last = pass + 1 == n_pass;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tl->jobs_ready[S::kR]));
            if (done) {
                if (lane == 0) atomicAdd(&P.ws->tiles_fetched, fetched);
                return;
            }
            if (pass > 0) continue;
            for (int r = 0; r < R; ++r) {  // the rows' Q tiles, each once the last group is done with the one before
                if (!mbar_wait_w(smem_u32(&tl->q_free[r]), (q_par >> r) & 1u, tl, P.ws, 405)) return;
                q_par ^= 1u << r;
                if (elect_one()) {
                    const unsigned bar = smem_u32(&tl->q_full[r]);
                    mbar_arrive_expect_tx(bar, (unsigned)(S::kHalves * S::kTile));
#pragma unroll
                    for (int c = 0; c < S::kHalves; ++c) tma_load_4d(q_smem + (c * S::kR + r) * S::kTile, tq, bar, c * 64, (S::kQbRows ? qb - (int)((P.row_back >> (2 * r)) & 3u) : qb) * S::kBlk, h0 + (S::kQbRows ? (int)((P.row_head >> (2 * r)) & 3u) : r), b);
                }
                __syncwarp();
            }
            fetched += (unsigned)R;
        }
    }
}

// Row r of every group. Lane i holds nodes kNodes i .. kNodes i + kNodes - 1 of the row.
template <class S>
__device__ void controller_role(const Params &P, Tail<S> *tl, int r, int lane) {
    const Geom &g = P.g;
    constexpr bool kMulti = S::kMulti;
    constexpr int kNodes = S::kNodes;
    const unsigned lt = (1u << lane) - 1u;
    unsigned grp_par = 0, first_par = 0, sd_par = 0, ack_par = 1;  // first_par: bit by bit for the two sets
    // this CTA's score memory for the row (several k only)
    unsigned long long *const cache = kMulti ? P.cache + ((size_t)blockIdx.x * S::kR + r) * g.N_k : nullptr;
    auto remembered = [&](int blk, unsigned tag, float &score) {
        const unsigned long long e = __ldcg(cache + blk);
        if ((unsigned)(e >> 32) != tag) return false;
        score = __uint_as_float((unsigned)e);
        return true;
    };
    auto tile_max = [](const float (&parts)[S::kParts]) { return S::kParts == 2 ? fmaxf(parts[0], parts[S::kParts - 1]) : parts[0]; };
    unsigned long long tiles_all = 0, rows_all = 0;
    for (;;) {
        if (!mbar_wait_w(smem_u32(&tl->jobs_ready[S::kR]), grp_par, tl, P.ws, 407)) return;
        const unsigned set = grp_par;
        grp_par ^= 1;
        const int id = tl->grp_id, b = tl->grp_b, qb = S::kQbRows ? tl->grp_qb - (int)((P.row_back >> (2 * r)) & 3u) : tl->grp_qb, h = tl->grp_h0 + (S::kQbRows ? (int)((P.row_head >> (2 * r)) & 3u) : r), R = tl->grp_R, levels = tl->grp_levels;
        const int kq = tl->grp_k, pass = tl->grp_pass, first_nodes = tl->grp_nodes;
        unsigned on[2 * kNodes];
        int nf[kNodes], nl[kNodes];       // this lane's nodes
#pragma unroll
        for (int x = 0; x < 2 * kNodes; ++x) on[x] = tl->grp_on[x];
#pragma unroll
        for (int x = 0; x < kNodes; ++x) { nf[x] = tl->grp_f[kNodes * lane + x]; nl[x] = tl->grp_l[kNodes * lane + x]; }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tl->jobs_ack[S::kR]));  // (the list itself is not needed)
        if (id < 0) {
            if (lane == 0) {
                atomicAdd(&P.ws->tiles_scored, tiles_all);
                atomicAdd(&P.ws->rows, rows_all);
            }
            return;
        }
        if (r >= R) continue;
        const int q_lim = last_valid_block(g, qb);
        const unsigned tag = (unsigned)id + 1u;  // marks this group's entries of the score memory (0 = never written)
        // A level's candidates, in ascending order: left and right of every node. cand: what they keep if
        // they survive (first and last block, score); have: it is there.
        float ns[kNodes];                 // its nodes' scores
        bool has[2 * kNodes];
        float sc[2 * kNodes];
        unsigned tiles = 0;               // (row, block) tiles that had no score yet
#pragma unroll
        for (int x = 0; x < kNodes; ++x) {
            const int rb = (nf[x] + nl[x]) / 2 + 1;
            bool miss_l = nf[x] <= nl[x] && nf[x] <= q_lim, miss_r = miss_l && rb <= nl[x] && rb <= q_lim;
            has[2 * x] = miss_l; has[2 * x + 1] = miss_r;
            sc[2 * x] = sc[2 * x + 1] = -CUDART_INF_F;
            if (kMulti) {
                if (miss_l && remembered(nf[x], tag, sc[2 * x])) miss_l = false;
                if (miss_r && remembered(rb, tag, sc[2 * x + 1])) miss_r = false;
            }
            tiles += (unsigned)(__popc(__ballot_sync(0xffffffffu, miss_l)) + __popc(__ballot_sync(0xffffffffu, miss_r)));
        }
        bool need[kNodes];                // the right candidate's score comes from the list
        int my_c[kNodes], n_nodes = 0;
        bool listed = true;               // the level's list holds something (else nobody reports on it)
        for (int level = 0; level < levels; ++level) {
            if (level == 0) {
                if (!mbar_wait_w(smem_u32(&tl->first_done[set][r]), (first_par >> set) & 1u, tl, P.ws, 408)) return;
                first_par ^= 1u << set;
                int place = flags_before(on, lt);
#pragma unroll
                for (int x = 0; x < 2 * kNodes; ++x) {
                    if (!((on[x] >> lane) & 1u)) continue;
                    sc[x] = tile_max(tl->first_part[set][r][place++]);
                    if (kMulti) __stcg(cache + ((x & 1) ? (nf[x >> 1] + nl[x >> 1]) / 2 + 1 : nf[x >> 1]), cache_pack(tag, sc[x]));
                }
            } else {
                if (!kMulti || listed) {
                    if (!mbar_wait_w(smem_u32(&tl->scores_done[r]), sd_par, tl, P.ws, 401)) return;
                    sd_par ^= 1;
                }
#pragma unroll
                for (int x = 0; x < kNodes; ++x) {
                    has[2 * x] = kNodes * lane + x < n_nodes;
                    sc[2 * x] = ns[x];
                    if (need[x]) {
                        sc[2 * x + 1] = tile_max(tl->part[r][my_c[x]]);
                        if (kMulti) __stcg(cache + (nf[x] + nl[x]) / 2 + 1, cache_pack(tag, sc[2 * x + 1]));
                    }
                }
            }
            bool keep[2 * kNodes];
            if constexpr (kNodes == 1) {
                const Keep kp = select_topk_counting(has[0], sc[0], has[1], sc[1], kq, level == 0 ? first_nodes : n_nodes, lane, tl->keys[r]);
                keep[0] = kp.l; keep[1] = kp.r;
            } else {
                select_topk_of<2 * kNodes>(has, sc, kq, lane, keep);
            }
            unsigned kept[2 * kNodes];
#pragma unroll
            for (int x = 0; x < 2 * kNodes; ++x) kept[x] = __ballot_sync(0xffffffffu, keep[x]);
            int place = flags_before(kept, lt);
            __syncwarp();
#pragma unroll
            for (int x = 0; x < 2 * kNodes; ++x) {
                if (!keep[x]) continue;
                const int f = nf[x >> 1], l = nl[x >> 1], m = (f + l) / 2;
                tl->node_f[r][place] = (x & 1) ? m + 1 : f;
                tl->node_l[r][place] = (x & 1) ? l : m;
                tl->node_s[r][place] = sc[x];
                ++place;
            }
            __syncwarp();
            n_nodes = flags_all(kept);
#pragma unroll
            for (int x = 0; x < kNodes; ++x) {
                const bool live = kNodes * lane + x < n_nodes;
                nf[x] = live ? tl->node_f[r][kNodes * lane + x] : 0;
                nl[x] = live ? tl->node_l[r][kNodes * lane + x] : -1;
                ns[x] = live ? tl->node_s[r][kNodes * lane + x] : -CUDART_INF_F;
            }
            if (level + 1 < levels) {
                // next level: only right branches need a tile; left ones keep the node's score
                unsigned due[kNodes];
#pragma unroll
                for (int x = 0; x < kNodes; ++x) {
                    const int rb = (nf[x] + nl[x]) / 2 + 1;
                    has[2 * x + 1] = kNodes * lane + x < n_nodes && nl[x] > nf[x] && rb <= q_lim;
                    sc[2 * x + 1] = -CUDART_INF_F;
                    need[x] = has[2 * x + 1];
                    if (kMulti && need[x] && remembered(rb, tag, sc[2 * x + 1])) need[x] = false;  // an earlier pass (another k) has scored it
                    due[x] = __ballot_sync(0xffffffffu, need[x]);
                }
                // (several k) An empty list is left out, but for the row's last, which says that it is.
                const bool final = kMulti && level + 2 == levels;
                listed = flags_all(due) > 0;
                if (kMulti && !listed && !final) continue;
                if (!mbar_wait_w(smem_u32(&tl->jobs_ack[r]), ack_par, tl, P.ws, 403)) return;
                ack_par ^= 1;
                int at = flags_before(due, lt);
#pragma unroll
                for (int x = 0; x < kNodes; ++x) {
                    my_c[x] = at;
                    if (need[x]) tl->jobs_blk[r][at++] = (nf[x] + nl[x]) / 2 + 1;
                }
                if (lane == 0) tl->n_jobs[r] = flags_all(due) + (final ? kFinal : 0);
                tiles += (unsigned)flags_all(due);
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&tl->jobs_ready[r]));
            } else {
                // emit I[q, :]: first block of every surviving node, ascending, -1 padded
                const long long row = ((long long)b * g.H + h) * g.n_qb + qb;
                const long long o = (kMulti ? P.slab_of[pass] * P.slab : 0ll) + row * g.k_top;
#pragma unroll
                for (int x = 0; x < kNodes; ++x) {
                    const int i = kNodes * lane + x;
                    if (i < g.k_top) {
                        P.mask[o + i] = i < n_nodes ? nf[x] : -1;
                        if (P.score != nullptr) P.score[o + i] = i < n_nodes ? ns[x] : -CUDART_INF_F;
                    }
                }
                if (!kMulti && g.row_tiles != nullptr && lane == 0) g.row_tiles[row] = tiles;
            }
        }
        tiles_all += tiles;
        ++rows_all;
    }
}

template <class S>
__global__ void __launch_bounds__(S::kThreads, S::kTwo ? 2 : 1)
mask_tc_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k, Params P) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = aligned_smem(smem_raw);
    const unsigned q_smem = smem_u32(smem), k_smem = q_smem + S::kQBytes;
    Tail<S> *tl = (Tail<S> *)(smem + S::kQBytes + S::kStages * S::kStageBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < S::kStages; ++i) {
            for (int c = 0; c < S::kHalves; ++c) mbar_init(smem_u32(&tl->full[c][i]), 1);
            mbar_init(smem_u32(&tl->empty[i]), 1);
        }
        for (int i = 0; i < S::kSlots; ++i) { mbar_init(smem_u32(&tl->tmem_full[i]), 1); mbar_init(smem_u32(&tl->tmem_empty[i]), 4); }
        for (int i = 0; i <= S::kR; ++i) { mbar_init(smem_u32(&tl->jobs_ready[i]), 1); mbar_init(smem_u32(&tl->jobs_ack[i]), S::kListReaders + (i == S::kR ? S::kR : 0)); }
        for (int i = 0; i < S::kR; ++i) {
            mbar_init(smem_u32(&tl->q_full[i]), 1); mbar_init(smem_u32(&tl->q_free[i]), S::kMmaWarps);
            mbar_init(smem_u32(&tl->first_done[0][i]), 4 * S::kEpiGroups); mbar_init(smem_u32(&tl->first_done[1][i]), 4 * S::kEpiGroups); mbar_init(smem_u32(&tl->scores_done[i]), 4 * S::kEpiGroups);
        }
        tl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (warp == 1) tmem_alloc<S::kTmemColumns>(smem_u32(&tl->tmem_base));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = tl->tmem_base;
    after_previous_kernel();

    // One call of each role, so that its code is in the instruction cache once, and the roles dealt so
    // that a scheduler (warp % 4) runs little beside its two epilogue warps: three copies of the
    // issuing role and two of the controllers', spread over all schedulers, cost a quarter of the
    // kernel's time in instruction fetches.
    // (Two CTAs an SM: warp 0 producer, 1 and 2 issuers, 3 dispatcher, 4..7 epilogue, 8..11 controllers.)
    constexpr bool kTwo = S::kTwo;
    if (warp >= 4 && warp < (kTwo ? 8 : 12)) {
        epilogue_role(P, tl, tmem_base, warp & 3, (warp - 4) >> 2, lane);
    } else if (warp == 1 || warp == (kTwo ? 2 : 3) || (!kTwo && (warp == 13 || warp == 17))) {
        mma_role(P, tl, q_smem, k_smem, tmem_base, warp == 1 ? 0 : (warp <= 3 ? 1 : (warp == 13 ? 2 : 3)));
    } else if (warp == (kTwo ? 0 : 2) || (!kTwo && warp == 14)) {
        producer_role(P, &tmap_k, tl, k_smem, warp <= 2 ? 0 : 1);
    } else if (warp == (kTwo ? 3 : 18)) {
        dispatcher_role(P, &tmap_q, tl, q_smem, lane);
        // the rows without products, beside the CTA's last group (at the beginning, by warps that the first group needs: 58.4 -> 59.1 us,
        // 28 / 4 heads, 3000 tokens, k = 8)
        if constexpr (!S::kMulti) {
            if (P.first_qb > 0) write_whole_rows(P.g, P.first_qb, (int)blockIdx.x, (int)gridDim.x, lane, P.mask, P.ws);
        }
    } else {
        controller_role(P, tl, kTwo ? warp - 8 : (warp == 0 ? 0 : (warp == 12 ? 1 : (warp == 16 ? 2 : 3))), lane);
    }
    __syncwarp();

    leave<S::kTmemColumns>(&tl->abort_flag, tmem_base, warp == 1);
}

// ----------------------------------------------------------------------------------------------
// Host side
// ----------------------------------------------------------------------------------------------
}  // namespace

bool mask_tc_supported(const Geom &g, int dtype) {
    return g.d == 128 && g.bq == 64 && g.k_top <= 32 && mask_tc_auto(g, dtype);
}

// Against the mma.sync kernel, us: 12 heads, 10007 tokens, d = 128, blocks of 32, k = 8: 221 -> 147; d = 64,
// blocks of 64, k = 40 (above): 409 -> 156; 8 heads, 13232 tokens, k = 59: 880 -> 265; 12 heads, 558 tokens,
// k = 59: 16.4 -> 14.6. (28 heads, 1329 tokens, d = 64, blocks of 32, k = 19: 28.7 -> 32.7, the one
// shape of 26 drawn that lost.)
bool mask_tc_auto(const Geom &g, int dtype) {
    return dtype == STREAM_BF16 && (g.d == 64 || g.d == 128) && (g.bq == 32 || g.bq == 64) && g.bk == g.bq && g.k_top <= 64 &&
           g.levels >= 1 && tma_strides_ok(g);
}

namespace {
// Two CTAs an SM of up to four rows each, where Q and key tiles leave room for them. With lists of a few stages every role of a lone CTA waits
// for the others most of the time; two groups fill each other's gaps (us, one and two: 12 / 2 heads, 10007 tokens in blocks of 32,
// k = 8: 114.9, 94.1; d = 64: 32 / 8 heads, 4000 tokens, k = 16: 76.0, 65.6). Not for d = 128 in blocks of 32 with more than 32 blocks a list
// but in long launches: two stages of 128 keys are too few there for one group to go on while the other waits (us, the better split
// of one and of two, in brackets the rows an SM: 8 / 2 heads, 6835 tokens, k = 64 (8): 66, 84; 28 / 4 heads, 3973, k = 64 (12): 68, 75; 8 / 4 heads,
// 11084, k = 51 (16): 139, 142; 24 / 8 heads, 4918, k = 34 (20): 125, 117; 5369, k = 38, not causal (27): 236, 202; 8 / 2 heads, 17789, k = 45 (30): 396, 398).
bool two_of_four_rows(const Geom &g, int first_qb) {
    return g.d == 64 || (g.bq == 32 && (g.k_top <= 32 || (long long)g.batch * g.H * (g.n_qb - first_qb) >= 18ll * sm_count()));
}
// With d = 128 and blocks of 64 there is room for two CTAs of two rows and two stages each: better with up to eight blocks a list and no more than
// eight groups a CTA (32 / 8 heads, 2500 tokens, k = 8: 45.1 -> 36.9; 28 / 4 heads, 1500, k = 5: 29.8 -> 26.7; 12 / 2 heads, 20000,
// k = 6, not causal: 189 -> 180), worse where the tensor cores are the limit (28 / 4 heads, 6000 tokens, k = 12, not causal: 139 -> 144;
// 32 / 8 heads, 60000, k = 10: 2139 -> 2200; 16384, k = 16: 486 -> 521).
bool two_of_two_rows(const Geom &g) {
    return g.d == 128 && g.bq == 64 && g.k_top <= 8 && g.k_row == nullptr && (long long)g.batch * g.H * g.n_qb <= 2 * 8 * 2ll * sm_count();
}

// CTAs of a launch, the groups they share and the rows of a group. Rows share the key tiles of the first level and its chains of two;
// fewer of them make more and shorter groups. Four rows (of several query blocks, unless k changes from one to the next, where a kv head
// has fewer than four heads) are taken where there are rows for some groups of them a CTA, else two, else one.
struct Split { int grid, head_rows, qb_rows, n_chunks; long long n_groups; };
stream_status split_rows(const Geom &g, int first_qb, int ctas_per_sm, int most_rows, bool several_k, Split *s) {
    const int n_cta = sm_count() * ctas_per_sm;
    if (n_cta <= 0) { set_error("cannot read the SM count of the current device"); return STREAM_ERR_CUDA; }
    s->n_chunks = (g.hpg + most_rows - 1) / most_rows;
    s->head_rows = (g.hpg + s->n_chunks - 1) / s->n_chunks;  // (six heads as 3 + 3, not 4 + 2: 139 -> 135 us at 10007 tokens in blocks of 32, 115 -> 107 at 8221)
    s->qb_rows = g.k_row == nullptr ? most_rows / g.hpg : 1;
    if (s->qb_rows < 1) s->qb_rows = 1;
    for (;;) {
        const int rows = s->head_rows * s->qb_rows;
        s->n_chunks = (g.hpg + s->head_rows - 1) / s->head_rows;
        s->n_groups = (long long)g.batch * g.G * ((g.n_qb - first_qb + s->qb_rows - 1) / s->qb_rows) * s->n_chunks;
        // How many groups a CTA there should be rows for, in halves: from 545 drawn shapes (k = 2 to 64), each timed at every number of rows;
        // over 380 others 2.4 % behind the best of these on average, with the attention behind it 1.3. Rows, not groups: three heads as 2 + 1 make more groups than they have work for (6 / 2
        // heads, 4458 tokens, k = 24: two rows 44.2 us, one 34.8). Some of them, us with four (or three) rows, two and one, in brackets the
        // groups of four a CTA. One CTA an SM: 28 / 4 heads, 3419 tokens, k = 27, not causal (2.9): 83, 74, 101; 8 / 2 heads, 20000, k = 24 (3.9):
        // 210, 195; 8 / 2 heads, 13232, k = 59 (2.0): 186, 157, 188; of several query blocks: 16 heads, 9000, k = 12 (3.5): 118, 124, and with
        // two nodes a lane: 1 head, 80291, k = 37 (2.0): 267, 235. Two CTAs, blocks of 64: 28 / 4 heads, 2500, k = 33, not causal (1.1): 73.6, 56.4, 43.0;
        // 12 / 2 heads, 10922, k = 45 (1.7): 177, 156, 107; 2 heads, 73665, k = 16 (1.9): -, 168, 186; 61140, k = 2, not causal (1.6), with the attention: -, 103, 129. Blocks of 32, where a pair of rows is little
        // more work than a row alone: 12 / 2 heads, 6000, k = 40 (2.0): 75.7, 69.7; 28 / 4 heads, 3000, k = 40, d = 128 (1.5): 61, 55, 70.
        const bool wide = g.k_top > 32;
        int halves;
        bool full = false;
        if (several_k) {
            // A group's passes make it long by themselves, and fewer rows share less. Groups of a build that is not causal, or of several query blocks, are
            // nearly equally long (28 / 4 heads, 2992 tokens, k = 3, 7, 14, not causal (2.5): 115, 146; 24 / 8 heads, 4551, not causal (3.9): 164,
            // 244; 2 heads, 40264 (2.1): two rows 1.3 times four; 8 / 2 heads, 10311, k = 5, 10, 21 (2.2): 201, 149; 5501 (2.3): 114, 97).
            halves = rows > 2 ? (g.causal && s->qb_rows == 1 ? 5 : 3) : 2;
        } else if (ctas_per_sm == 2 && most_rows == 4) {
            halves = rows > 2 ? 6 : (g.bq == 64 ? (wide ? 8 : 6) : (wide ? 3 : 2));
            // Not causal, the groups are equally long: with two nodes a lane also where more than one round of them is five sixths full (16 heads, 8192
            // tokens, k = 40 (1.7): 153, 151, 154, with the attention behind them 350, -, 359; 8 / 2 heads, 16000, k = 60 (1.7): 246, 252; 16 heads, 5345,
            // k = 37 (1.1): 113, 96, 94; but one node a lane: 6 / 2 heads, 17942, k = 5 (1.9): 90, 80).
            const long long rounds = (s->n_groups + n_cta - 1) / n_cta;
            full = wide && rows > 2 && !g.causal && rounds > 1 && 6 * s->n_groups >= 5 * rounds * n_cta;
        } else {
            halves = rows > 2 ? (s->qb_rows > 1 ? (wide ? 6 : 4) : (wide ? 7 : 8)) : 2;
        }
        const long long there = several_k ? s->n_groups : (long long)g.batch * g.H * (g.n_qb - first_qb) / rows;
        if (full || 2 * there >= (long long)halves * n_cta || rows == 1) break;
        if (s->qb_rows > 1) s->qb_rows = (s->qb_rows + 1) / 2;
        else s->head_rows = (s->head_rows + 1) / 2;
    }
    s->grid = (int)(s->n_groups < n_cta ? s->n_groups : n_cta);
    return STREAM_OK;
}
constexpr int kMultiRows = Shape<128, 64, false, true>::kR;

template <class S>
cudaError_t launch(int grid, cudaStream_t st, const CUtensorMap &tq, const CUtensorMap &tk, const Params &P) {
    static_assert((S::kTwo ? 2 : 1) * (kSmemBytes<S> + 1024) <= 228 * 1024, "shared memory of an SM");
    const cudaError_t e = cudaFuncSetAttribute(mask_tc_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes<S>);
    return e == cudaSuccess ? launch_kernel(mask_tc_kernel<S>, grid, S::kThreads, kSmemBytes<S>, st, 1, tq, tk, P) : e;
}

template <int kD, int kBlk, bool kWide, bool kTwo>
cudaError_t launch_rows(const Split &sp, int grid, cudaStream_t st, const CUtensorMap &tq, const CUtensorMap &tk, const Params &P) {
    return sp.qb_rows > 1 ? launch<Shape<kD, kBlk, kWide, false, true, kTwo>>(grid, st, tq, tk, P) : launch<Shape<kD, kBlk, kWide, false, false, kTwo>>(grid, st, tq, tk, P);
}
}  // namespace

size_t mask_tc_score_memory_bytes(const Geom &g) {
    Split sp;
    if (split_rows(g, 0, 1, kMultiRows, true, &sp) != STREAM_OK) return 0;
    return (size_t)sp.grid * kMultiRows * (size_t)g.N_k * sizeof(unsigned long long);
}

stream_status launch_mask_tc(const Geom &g, const void *q, const void *k, int32_t *mask, float *score,
                             WorkspaceHeader *ws, cudaStream_t st) {
    MultiK single = {};
    return launch_mask_tc_multi(g, single, q, k, mask, score, ws, nullptr, st);
}

stream_status launch_mask_tc_multi(const Geom &g, const MultiK &mk, const void *q, const void *k, int32_t *mask,
                                   float *score, WorkspaceHeader *ws, void *score_memory, cudaStream_t st) {
    if (((uintptr_t)q & 15) != 0 || ((uintptr_t)k & 15) != 0) {
        set_error("tensor-core mask kernel needs 16-byte aligned q and k");
        return STREAM_ERR_UNSUPPORTED;
    }
    CUtensorMap tq, tk;
    stream_status rc = make_map_bf16(&tq, q, g.T, g.H, g.batch, g.qs_t, g.qs_h, g.qs_b, "q", g.bq, g.d);
    if (rc != STREAM_OK) return rc;
    rc = make_map_bf16(&tk, k, g.T, g.G, g.batch, g.ks_t, g.ks_h, g.ks_b, "k", g.bk, g.d);
    if (rc != STREAM_OK) return rc;
    Params P;
    P.g = g;
    // The rows of one build that keep every block they are allowed, with no score asked for, need no products.
    P.first_qb = mk.n == 0 && score == nullptr ? whole_query_blocks(g) : 0;
    if (P.first_qb == g.n_qb) return launch_mask_whole(g, g.n_qb, mask, ws, st);
    Split sp;
    const bool two_rows = mk.n == 0 && two_of_two_rows(g);
    const int ctas = (mk.n == 0 && two_of_four_rows(g, P.first_qb)) || two_rows ? 2 : 1;
    rc = split_rows(g, P.first_qb, ctas, two_rows ? 2 : 4, mk.n >= 1, &sp);
    if (rc != STREAM_OK) return rc;
    P.n_groups = (int)sp.n_groups;
    P.walked_heads = walked_heads(g);
    P.n_chunks = sp.n_chunks; P.head_rows = sp.head_rows; P.qb_rows = sp.qb_rows;
    P.row_head = P.row_back = 0;
    for (int r = 0; r < sp.head_rows * sp.qb_rows; ++r) {
        P.row_head |= (unsigned)(r % sp.head_rows) << (2 * r);
        P.row_back |= (unsigned)(r / sp.head_rows) << (2 * r);
    }
    // (more CTAs than groups where they have rows to write)
    const long long writers = P.first_qb > 0 ? whole_pieces(g, P.first_qb) / 4 : 0;
    const int grid = writers > sp.grid ? (int)(writers < ctas * sm_count() ? writers : ctas * sm_count()) : sp.grid;
    P.mask = mask; P.score = score; P.ws = ws;
    // The largest k first: its nodes are the smallest, and where the numbers divide it meets all blocks that
    // the others would, in longer lists than theirs (8, 16, 32 at 32768 tokens: 2360 us, in rising order 2570).
    P.mk.n = mk.n;
    for (int i = 0; i < mk.n; ++i) {
        int at = i;
        for (; at > 0 && P.mk.k[at - 1] < mk.k[i]; --at) { P.mk.k[at] = P.mk.k[at - 1]; P.slab_of[at] = P.slab_of[at - 1]; }
        P.mk.k[at] = mk.k[i];
        P.slab_of[at] = i;
    }
    P.cache = (unsigned long long *)score_memory;
    P.slab = (long long)g.batch * g.H * g.n_qb * g.k_top;
    cudaError_t e = cudaSuccess;
    if (score_memory != nullptr) {  // tag 0 = "no score yet"
        e = cudaMemsetAsync(score_memory, 0, mask_tc_score_memory_bytes(g), st);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(score memory)");
    }
    if (mk.n >= 1 && score_memory == nullptr) { set_error("several k in one launch need the score memory"); return STREAM_ERR_WORKSPACE; }
    if (mk.n >= 1) e = sp.qb_rows > 1 ? launch<Shape<128, 64, false, true, true>>(grid, st, tq, tk, P) : launch<Shape<128, 64, false, true>>(grid, st, tq, tk, P);
    else if (two_rows) e = launch_rows<128, 64, false, true>(sp, grid, st, tq, tk, P);
    else if (g.d == 128 && g.bq == 64) e = g.k_top > 32 ? launch_rows<128, 64, true, false>(sp, grid, st, tq, tk, P) : launch_rows<128, 64, false, false>(sp, grid, st, tq, tk, P);
    else if (g.d == 128 && g.k_top <= 32) e = launch_rows<128, 32, false, true>(sp, grid, st, tq, tk, P);
    else if (g.d == 128) e = ctas == 2 ? launch_rows<128, 32, true, true>(sp, grid, st, tq, tk, P) : launch_rows<128, 32, true, false>(sp, grid, st, tq, tk, P);
    else if (g.bq == 64) e = g.k_top > 32 ? launch_rows<64, 64, true, true>(sp, grid, st, tq, tk, P) : launch_rows<64, 64, false, true>(sp, grid, st, tq, tk, P);
    else e = g.k_top > 32 ? launch_rows<64, 32, true, true>(sp, grid, st, tq, tk, P) : launch_rows<64, 32, false, true>(sp, grid, st, tq, tk, P);
    if (e != cudaSuccess) return cuda_fail(e, "mask_tc launch");
    return STREAM_OK;
}

}  // namespace stream
