// Tensor-core attention under masks of short query blocks (block_q < 16, per-token masks above all) for
// sm_100a: bf16, d = 128, block_k = 64.
//
// With a mask row per token no two tokens share their kept blocks, but 128 neighbouring tokens keep
// most blocks between them. One persistent CTA per SM takes 128 consecutive tokens of one head: their
// blocks are merged into one ascending list (a bit per mask row and block says who keeps it), every
// block is fetched once and multiplied with all 128 tokens,
//     S = Q K^T   (128 x 64, fp32 in TMEM),     O += P V   (128 x 128, fp32 in TMEM),
// and tokens that do not keep it are masked like keys after the token. P = exp2(scale (s - ref)) goes to
// the product as two bf16 numbers, the rounded weight and the rest (relative error 2^-17), A operands
// from TMEM: these shapes have had fp32 weights before, and the second product costs less than
// anything it could be traded for.
//
// Two softmax groups of four warps take a CTA's blocks in turn, thread = token; what they do about the
// reference (`ref`, shared, moved only when a logit has outgrown it by about 2^30) and the order they
// publish in (`turn`) is described in attn_tc.cu. Here a token starts with reference 0 and keeps it if the
// first logits it meets give weights between 2^-40 and 2^36 in sum: a maximum taken first would cost
// every token a look at its own first block.
//
// TMEM columns: logits of group g at 64 g, its two P buffers (32 rounded, 32 rest) at 128 + 128 g and 64
// behind, O at 384. Roles (384 threads): warp 0 brings K, V and Q tiles, warp 1 issues Q K^T, warp 3
// P V, warp 2 merges the masks up to two segments ahead (a segment: 128 tokens, 512 key blocks), warps
// 4..11 the softmax groups. They meet only on mbarriers, every wait bounded as in attn_tc.cu.
//
// Bound: the softmax warps' instructions and the two chains of a block (8 x 48 and 8 x 73 clocks) alike.
// 32 / 8 heads, T = 4096, k = 16, block_q = 1: 973 us on mma.sync (attn_mma.cu), 221 here.
#include <cstddef>
#include <math_constants.h>

#include "tc_common.cuh"

namespace stream {

// Status words, as in attn_tc.cu; read by stream_check_device_status too.
static __device__ unsigned int g_attn_tok_status[2];

namespace {

using namespace tc;

constexpr int kThreads = 384;
constexpr int kTok = 128, kBlk = 64, kD = 128;
constexpr int kHalfTile = kBlk * 128;      // 64 rows x 128 bytes
constexpr int kTile = 2 * kHalfTile;       // a 64 x 128 key or value tile
constexpr int kQTile = 2 * kTok * 128;     // [2 channel halves][128 tokens][128 bytes]
constexpr int kKStages = 4, kVStages = 4;
constexpr int kWindow = 512;               // key blocks of a segment
constexpr int kWords = kWindow / 32;
constexpr int kMaskSlots = 2;
constexpr float kLargeSum = 68719476736.f;          // 2^36: beyond it a weight has exceeded 2^30
constexpr float kSmallSum = 9.094947017729282e-13f;  // 2^-40
constexpr int kPCol = 128, kOCol = 384;

struct Segment {
    int b, h, tok0;      // batch entry, query head, first token
    int block0, n;       // first key block of the window, blocks in the list
    int first, last;     // of the 128 tokens' segments
    int first_row;       // mask row of the first token
};

struct Tail {
    unsigned long long q_full[2], q_free[2];  // q_free: the output staged over the Q tile has left (8 warps)
    unsigned long long k_full[kKStages], k_empty[kKStages], v_full[kVStages], v_empty[kVStages];
    unsigned long long s_full[2], s_free[2], p_full[2][2], p_free[2][2];
    unsigned long long o_done, o_free;
    unsigned long long turn[4][2], sums_there[4];
    unsigned long long m_full[kMaskSlots], m_empty[kMaskSlots];
    unsigned int tmem_base;
    int abort_flag;
    Segment seg[kMaskSlots];
    float ref[kTok], sum[2][kTok];
    unsigned short list[kMaskSlots][kWindow];   // blocks of the segment, counted from block0, ascending
    alignas(16) unsigned bits[kMaskSlots][kTok][kWords];  // per mask row of the 128 tokens (cleared 16 bytes at a time)
};
constexpr int kSmemBytes = 2 * kQTile + (kKStages + kVStages) * kTile + (int)sizeof(Tail) + 1024;
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
static_assert(offsetof(Tail, bits) % 16 == 0 && (2 * kQTile + (kKStages + kVStages) * kTile) % 16 == 0, "16-byte accesses");

constexpr unsigned kIdescQK = idesc_bf16(128, 64, false);   // B = a key tile, K-major
constexpr unsigned kIdescPV = idesc_bf16(128, 128, true);   // B = a value tile, MN-major
constexpr unsigned kHi = desc_hi_sw128(1024);

struct Params {
    Geom g;
    int n_items, n_tb;     // groups of 128 tokens, of one head
    int group_heads;       // kv heads (of the batch * G) whose items are walked together, late tokens (most blocks) first
    const int32_t *mask;
    __nv_bfloat16 *out;
    float scale_log2;
};

__device__ __forceinline__ bool wait_w(unsigned bar, unsigned parity, Tail *tl, unsigned code) {
    return mbar_wait_warp(bar, parity, &tl->abort_flag, &g_attn_tok_status[0], &g_attn_tok_status[1], code);
}

// ----------------------------------------------------------------------------------------------
// Roles
// ----------------------------------------------------------------------------------------------
__device__ void mask_role(const Params &P, Tail *tl, int lane) {
    const Geom &g = P.g;
    const int n_kb = (int)((g.T + kBlk - 1) / kBlk);
    Ring ms;
    for (int round = 0, id; (id = nth_item(round)) < P.n_items; ++round) {
        const int per_group = P.group_heads * g.hpg * P.n_tb, grp = id / per_group, rem = id - grp * per_group;
        const int heads = min(P.group_heads, g.batch * g.G - grp * P.group_heads) * g.hpg;  // query heads of the group
        const int tb = P.n_tb - 1 - rem / heads, bh = grp * P.group_heads * g.hpg + rem % heads;  // (heads of a kv head are neighbours)
        Segment s;
        s.b = bh / g.H; s.h = bh % g.H;
        s.tok0 = tb * kTok;
        s.first_row = s.tok0 / g.bq;
        const int tok_end = (int)min((long long)s.tok0 + kTok, g.T), n_rows = (tok_end - 1) / g.bq - s.first_row + 1;
        const int32_t *m = P.mask + (((long long)s.b * g.H + s.h) * g.n_qb + s.first_row) * g.k_top;
        const int n_entries = n_rows * g.k_top;
        // a causal token has no use for blocks behind it
        const int kb_end = g.causal ? min(n_kb, (tok_end - 1) / kBlk + 1) : n_kb;
        s.first = 1;
        for (s.block0 = 0; s.block0 < kb_end; s.block0 += kWindow) {
            // `nth`: a block that occurs more than once in a row counts as often: one more segment takes the
            // second occurrences, and so on
            for (int nth = 0;; ++nth) {
                if (!wait_w(smem_u32(&tl->m_empty[ms.idx]), ms.phase ^ 1, tl, 401)) return;
                unsigned(*bits)[kWords] = tl->bits[ms.idx];
                for (int i = lane; i < kTok * kWords / 4; i += 32) reinterpret_cast<uint4 *>(&bits[0][0])[i] = make_uint4(0, 0, 0, 0);
                __syncwarp();
                bool again = false;
                for (int i0 = 0; i0 < n_entries; i0 += 128) {
                    int e[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) e[u] = i0 + u * 32 + lane < n_entries ? m[i0 + u * 32 + lane] : -1;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = i0 + u * 32 + lane, rel = e[u] - s.block0;
                        if (e[u] < 0 || rel < 0 || rel >= kWindow || e[u] >= kb_end) continue;
                        const int row = i / g.k_top;
                        if (nth > 0) {
                            int before = 0;
                            for (int j = row * g.k_top; j < i; ++j) before += m[j] == e[u];
                            again |= before > nth;
                            if (before != nth) continue;
                        }
                        const unsigned bit = 1u << (rel & 31);
                        again |= (atomicOr(&bits[row][rel >> 5], bit) & bit) != 0u;
                    }
                }
                again = __any_sync(0xffffffffu, again);
                __syncwarp();
                // lanes w and w + 16: word w over the even and the odd rows
                unsigned any = 0;
                for (int r = lane >> 4; r < kTok; r += 2) any |= bits[r][lane & 15];
                any |= __shfl_xor_sync(0xffffffffu, any, 16);
                int n = 0;
                for (int w = 0; w < kWords; ++w) {
                    const unsigned word = __shfl_sync(0xffffffffu, any, w);
                    if ((word >> lane) & 1u) tl->list[ms.idx][n + __popc(word & ((1u << lane) - 1u))] = (unsigned short)(w * 32 + lane);
                    n += __popc(word);
                }
                s.n = n;
                s.last = !again && s.block0 + kWindow >= kb_end;
                __syncwarp();
                if (lane == 0) {
                    tl->seg[ms.idx] = s;
                    mbar_arrive(smem_u32(&tl->m_full[ms.idx]));
                }
                ms.advance(kMaskSlots);
                s.first = 0;
                if (!again) break;
            }
        }
    }
    if (!wait_w(smem_u32(&tl->m_empty[ms.idx]), ms.phase ^ 1, tl, 402)) return;
    if (lane == 0) {  // the end
        tl->seg[ms.idx].n = -1;
        mbar_arrive(smem_u32(&tl->m_full[ms.idx]));
    }
}

struct LoadStream {
    int e, n;        // entry of the open segment (-2: none is open), its entries
    int b, kvh, block0;
    bool done;
    Ring ring, ms;
};

__device__ void producer_role(const Params &P, const CUtensorMap *tq, const CUtensorMap *tk, const CUtensorMap *tv, Tail *tl,
                              unsigned q_smem, unsigned k_smem, unsigned v_smem) {
    Ring qs;
    LoadStream K, V;
    K.e = V.e = -2;
    K.done = V.done = false;
    bool q_due = false;
    // One step of a stream; true if it did something.
    auto step = [&](LoadStream &S, bool is_k) -> bool {
        if (S.done) return false;
        if (S.e == -2) {
            if (!probe_w(smem_u32(&tl->m_full[S.ms.idx]), S.ms.phase)) return false;
            const Segment &s = tl->seg[S.ms.idx];
            S.n = s.n;
            if (S.n < 0) { S.done = true; return true; }
            S.b = s.b; S.kvh = s.h / P.g.hpg; S.block0 = s.block0;
            S.e = 0;
            if (is_k && s.first) q_due = true;
            return true;
        }
        if (S.e >= S.n && !(is_k && q_due)) {
            __syncwarp();
            if (elect_one()) mbar_arrive(smem_u32(&tl->m_empty[S.ms.idx]));
            __syncwarp();
            S.ms.advance(kMaskSlots);
            S.e = -2;
            return true;
        }
        if (is_k && q_due && (S.e > 0 || S.e >= S.n)) {  // Q goes behind the first K tile, which does not depend on the Q buffer
            if (!probe_w(smem_u32(&tl->q_free[qs.idx]), qs.phase ^ 1)) return false;
            if (elect_one()) {
                const Segment &s = tl->seg[S.ms.idx];
                const unsigned bar = smem_u32(&tl->q_full[qs.idx]);
                mbar_arrive_expect_tx(bar, (unsigned)kQTile);
#pragma unroll
                for (int c = 0; c < 2; ++c) tma_load_4d(q_smem + qs.idx * kQTile + c * (kQTile / 2), tq, bar, c * 64, s.tok0, s.h, s.b);
            }
            __syncwarp();
            q_due = false;
            qs.advance(2);
            return true;
        }
        const unsigned empty = smem_u32(is_k ? &tl->k_empty[S.ring.idx] : &tl->v_empty[S.ring.idx]);
        if (!probe_w(empty, S.ring.phase ^ 1)) return false;
        const int blk = S.block0 + tl->list[S.ms.idx][S.e];
        if (elect_one()) {
            const unsigned bar = smem_u32(is_k ? &tl->k_full[S.ring.idx] : &tl->v_full[S.ring.idx]);
            mbar_arrive_expect_tx(bar, (unsigned)kTile);
            tma_load_5d((is_k ? k_smem : v_smem) + S.ring.idx * kTile, is_k ? tk : tv, bar, 0, blk * kBlk, S.kvh, 0, S.b);
        }
        __syncwarp();
        S.ring.advance(is_k ? kKStages : kVStages);
        ++S.e;
        return true;
    };
    long long t_last = clock64();
    while (!K.done || !V.done) {
        const bool moved_k = step(K, true), moved_v = step(V, false);
        if (moved_k || moved_v) { t_last = clock64(); continue; }
        int stop = 0;
        if ((threadIdx.x & 31) == 0) {
            if (*(volatile int *)&tl->abort_flag) stop = 1;
            else if (clock64() - t_last > kWaitCycles) {
                *(volatile int *)&tl->abort_flag = 1;
                if (atomicCAS(&g_attn_tok_status[0], 0u, 121u) == 0u) g_attn_tok_status[1] = blockIdx.x;
                stop = 1;
            }
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) return;
        __nanosleep(40);
    }
}

__device__ void qk_role(Tail *tl, unsigned q_smem, unsigned k_smem, unsigned tmem_base) {
    Ring ks, ms, qs;
    unsigned cnt[2] = {0, 0};  // entries each group has had over the whole kernel
    int u = 0;                 // entries of these tokens so far
    unsigned q_lo = 0;
    const unsigned q_lo0 = desc_lo_sw128(q_smem, 16), k_lo = desc_lo_sw128(k_smem, 16);
    for (;;) {
        if (!wait_w(smem_u32(&tl->m_full[ms.idx]), ms.phase, tl, 221)) return;
        const int n = tl->seg[ms.idx].n, first = tl->seg[ms.idx].first;
        if (n < 0) return;
        if (first) {
            u = 0;
            q_lo = q_lo0 + qs.idx * (kQTile >> 4);
            if (!wait_w(smem_u32(&tl->q_full[qs.idx]), qs.phase, tl, 222)) return;
            qs.advance(2);
        }
        for (int i = 0; i < n; ++i, ++u) {
            if (!wait_w(smem_u32(&tl->k_full[ks.idx]), ks.phase, tl, 223)) return;
            const unsigned gi = (unsigned)(u & 1), use = gi ? cnt[1]++ : cnt[0]++;
            if (!wait_w(smem_u32(&tl->s_free[gi]), (use & 1u) ^ 1u, tl, 224)) return;
            tc_fence_after();
            const unsigned d_tmem = tmem_base + gi * 64, b_lo = k_lo + ks.idx * (kTile >> 4);
            if (elect_one()) {
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4)
                        tc_mma_bf16_split(d_tmem, q_lo + ((c * (kQTile / 2) + k4 * 32) >> 4), kHi, b_lo + ((c * kHalfTile + k4 * 32) >> 4), kHi,
                                          kIdescQK, (c | k4) != 0);
                tc_commit(smem_u32(&tl->s_full[gi]));
                tc_commit(smem_u32(&tl->k_empty[ks.idx]));
            }
            __syncwarp();
            ks.advance(kKStages);
        }
        __syncwarp();
        if (elect_one()) mbar_arrive(smem_u32(&tl->m_empty[ms.idx]));
        __syncwarp();
        ms.advance(kMaskSlots);
    }
}

__device__ void pv_role(Tail *tl, unsigned v_smem, unsigned tmem_base) {
    Ring vs, ms;
    unsigned cnt[2] = {0, 0};
    int u = 0;
    unsigned free_par = 1;  // (the first wait passes at once)
    const unsigned v_lo = desc_lo_sw128(v_smem, kHalfTile), d_tmem = tmem_base + kOCol;
    for (;;) {
        if (!wait_w(smem_u32(&tl->m_full[ms.idx]), ms.phase, tl, 225)) return;
        const int n = tl->seg[ms.idx].n, first = tl->seg[ms.idx].first, last = tl->seg[ms.idx].last;
        if (n < 0) return;
        if (first) {
            u = 0;
            if (!wait_w(smem_u32(&tl->o_free), free_par, tl, 226)) return;  // the O before has been read
            free_par ^= 1;
        }
        for (int i = 0; i < n; ++i, ++u) {
            if (!wait_w(smem_u32(&tl->v_full[vs.idx]), vs.phase, tl, 227)) return;
            const unsigned gi = (unsigned)(u & 1), use = gi ? cnt[1]++ : cnt[0]++, pb = use & 1u;
            if (!wait_w(smem_u32(&tl->p_full[gi][pb]), (use >> 1) & 1u, tl, 228)) return;
            tc_fence_after();
            const unsigned a_tmem = tmem_base + kPCol + gi * 128 + pb * 64, b_lo = v_lo + vs.idx * (kTile >> 4);
            if (elect_one()) {
#pragma unroll
                for (int part = 0; part < 2; ++part)  // the rounded weights, the rest
#pragma unroll
                    for (int s4 = 0; s4 < 4; ++s4)    // 16 keys per step: 8 columns of packed bf16
                        tc_mma_bf16_ta(d_tmem, a_tmem + part * 32 + s4 * 8, b_lo + ((s4 * 2048) >> 4), kHi, kIdescPV, (u | part | s4) != 0);
                tc_commit(smem_u32(&tl->p_free[gi][pb]));
                tc_commit(smem_u32(&tl->v_empty[vs.idx]));
            }
            __syncwarp();
            vs.advance(kVStages);
        }
        __syncwarp();
        if (elect_one()) {
            if (last) tc_commit(smem_u32(&tl->o_done));
            mbar_arrive(smem_u32(&tl->m_empty[ms.idx]));
        }
        __syncwarp();
        ms.advance(kMaskSlots);
    }
}

__device__ void softmax_role(const Params &P, const CUtensorMap *to, Tail *tl, unsigned char *q_ptr, unsigned tmem_base, int t) {
    const Geom &g = P.g;
    const int lane = t & 31, row = t & 127, grp = t >> 7, wq = row >> 5;
    const unsigned lanes = tmem_base + ((unsigned)(row & ~31) << 16);
    const unsigned turn_own = smem_u32(&tl->turn[wq][grp]), turn_other = smem_u32(&tl->turn[wq][grp ^ 1]);
    const unsigned s_full = smem_u32(&tl->s_full[grp]), s_free = smem_u32(&tl->s_free[grp]), s_addr = lanes + grp * 64;
    unsigned char *const stage = q_ptr + (grp * 4 + wq) * 4096;  // this warp's 32 tokens x 64 channels in a Q buffer
    unsigned n_own = 0, n_other = 0;  // entries of either group so far (n_other: before these tokens)
    unsigned item_par = 0;
    int staged = -1;
    int u0 = 0;                       // entries of these tokens before the segment
    float ref = -CUDART_INF_F, l = 0.f;  // -inf: no reference yet, nothing added; weights are then taken under 0
    Ring ms, qs;
    auto release_stage = [&]() {
        if (staged < 0) return;
        if (lane == 0) {
            tma_store_wait_read();
            mbar_arrive(smem_u32(&tl->q_free[staged]));
        }
        __syncwarp();
        staged = -1;
    };
    for (;;) {
        if (!wait_w(smem_u32(&tl->m_full[ms.idx]), ms.phase, tl, 321)) return;
        const Segment &s = tl->seg[ms.idx];
        const int n = s.n;
        if (n < 0) break;
        const int b = s.b, h = s.h, tok0 = s.tok0, block0 = s.block0, last = s.last;
        const int tq = tok0 + row;
        const int key_end = tq < g.T ? (g.causal ? tq + 1 : (int)g.T) : 0;  // keys this token may attend: those before
        const unsigned *my_bits = tl->bits[ms.idx][tq < g.T ? tq / g.bq - s.first_row : 0];
        const unsigned short *list = tl->list[ms.idx];
        auto allowed_keys = [&](int rel) {
            const int left = min(key_end - (block0 + rel) * kBlk, kBlk);
            return ((my_bits[rel >> 5] >> (rel & 31)) & 1u) ? max(0, left) : 0;
        };
        if (s.first) { u0 = 0; ref = -CUDART_INF_F; l = 0.f; }
        const int i0 = (grp ^ u0) & 1;  // entry u of these tokens belongs to group u % 2
        int n_hi = i0 < n ? allowed_keys(list[i0]) : 0;
        for (int i = i0; i < n; i += 2) {
            const int u = u0 + i;
            const bool masked = __any_sync(0xffffffffu, n_hi != kBlk);
            if (!wait_w(s_full, n_own & 1u, tl, 322)) return;
            tc_fence_after();
            unsigned sr[64];
            tmem_ld_32x32_issue(s_addr, sr);
            tmem_ld_32x32_issue(s_addr + 32, sr + 32);
            tmem_ld_wait();
            tc_fence_before();
            mbar_arrive_if(s_free, lane == 0);
            if (masked) {
#pragma unroll
                for (int k = 0; k < 64; ++k) sr[k] = k < n_hi ? sr[k] : 0xff800000u;
            }
            const unsigned other = n_other + (unsigned)((u - 1) >> 1), turn_par = other & 1u;  // entry u - 1 is the other group's `other`-th
            const unsigned pb = n_own & 1u, p_col = lanes + kPCol + grp * 128 + pb * 64;
            if (!wait_w(smem_u32(&tl->p_free[grp][pb]), ((n_own >> 1) & 1u) ^ 1u, tl, 323)) return;
            int next_hi = 0;
            float esum;
            for (int attempt = 0;; ++attempt) {
                const float shift = ref == -CUDART_INF_F ? 0.f : -ref * P.scale_log2;
                const unsigned long long scale2 = pack_f32x2(P.scale_log2, P.scale_log2), shift2 = pack_f32x2(shift, shift),
                                         minus2 = pack_f32x2(-1.f, -1.f);
                unsigned long long sum2[2] = {0ull, 0ull};
                auto weights = [&](int k0) {
                    unsigned hi[16], lo[16];
#pragma unroll
                    for (int k = 0; k < 32; k += 2) {
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(pack_u32x2(sr[k0 + k], sr[k0 + k + 1]), scale2, shift2), x0, x1);
                        const unsigned long long p = pack_f32x2(fast_exp2(x0), fast_exp2(x1));
                        float p0, p1, d0, d1;
                        unpack_f32x2(p, p0, p1);
                        sum2[(k >> 1) & 1] = add_f32x2(sum2[(k >> 1) & 1], p);
                        const __nv_bfloat162 ph = __floats2bfloat162_rn(p0, p1);
                        const unsigned hw = *reinterpret_cast<const unsigned *>(&ph);
                        unpack_f32x2(fma_f32x2(pack_u32x2(hw << 16, hw & 0xffff0000u), minus2, p), d0, d1);
                        const __nv_bfloat162 pl = __floats2bfloat162_rn(d0, d1);
                        hi[k >> 1] = hw;
                        lo[k >> 1] = *reinterpret_cast<const unsigned *>(&pl);
                    }
                    tmem_st_32x16_issue(p_col + (k0 >> 1), hi);
                    tmem_st_32x16_issue(p_col + 32 + (k0 >> 1), lo);
                };
                weights(0);
                bool seen = true;
                float now = ref;
                if (u > 0) {  // (looked up ahead, so that the latency of it is hidden)
                    seen = mbar_test_wait(turn_other, turn_par);
                    now = *(volatile float *)&tl->ref[row];
                }
                next_hi = allowed_keys(list[min(i + 2, kWindow - 1)] & (kWindow - 1));  // (of no meaning behind the last)
                weights(32);
                float e0, e1;
                unpack_f32x2(add_f32x2(sum2[0], sum2[1]), e0, e1);
                esum = e0 + e1;
                bool moved = __float_as_uint(now) != __float_as_uint(ref);
                bool odd = !(esum <= kLargeSum) || (n_hi > 0 && ref == -CUDART_INF_F);
                if (!__any_sync(0xffffffffu, !seen || moved || odd)) break;
                // Something to settle: only after the entry before this one has been published.
                if (u > 0) {
                    if (!wait_w(turn_other, turn_par, tl, 324)) return;
                    now = *(volatile float *)&tl->ref[row];
                    moved = __float_as_uint(now) != __float_as_uint(ref);
                }
                bool again = false;  // the weights have to be taken under another reference
                if (moved) {
                    // (a token that had none until now has added nothing; under 0 its weights stand)
                    again = now != 0.f || ref != -CUDART_INF_F;
                    if (ref != -CUDART_INF_F) l *= fast_exp2((ref - now) * P.scale_log2);
                    ref = now;
                }
                const bool opens = ref == -CUDART_INF_F && n_hi > 0;
                if (opens && esum >= kSmallSum && esum <= kLargeSum) {
                    ref = 0.f;
                    tl->ref[row] = 0.f;
                }
                const bool move = !again && ((opens && ref == -CUDART_INF_F) || !(esum <= kLargeSum));
                if (attempt == 2 || !__any_sync(0xffffffffu, again || move)) break;
                if (__any_sync(0xffffffffu, move)) {
                    float f = 1.f;
                    if (move) {
                        const float mx = max_of_64(reinterpret_cast<const float *>(sr));
                        if (ref != -CUDART_INF_F) f = fast_exp2((ref - mx) * P.scale_log2);
                        ref = mx;
                        tl->ref[row] = ref;
                    }
                    if (u > 0 && __any_sync(0xffffffffu, f != 1.f)) {  // what has been added up so far is brought to the new reference
                        if (!wait_w(smem_u32(&tl->p_free[grp ^ 1][other & 1u]), (other >> 1) & 1u, tl, 325)) return;
                        tc_fence_after();
                        rescale_lane<kD>(lanes + kOCol, f);
                    }
                    l *= f;
                }
            }
            l += esum;
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            mbar_arrive_if(turn_own, lane == 0);
            mbar_arrive_if(smem_u32(&tl->p_full[grp][pb]), lane == 0);
            ++n_own;
            n_hi = next_hi;
            release_stage();
        }
        u0 += n;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tl->m_empty[ms.idx]));  // (nothing of the slot is read below)
        ms.advance(kMaskSlots);
        if (!last) continue;
        release_stage();
        // tokens that keep nothing: no product has waited for their Q tile, over which the output is staged
        if (u0 == 0 && !wait_w(smem_u32(&tl->q_full[qs.idx]), qs.phase, tl, 328)) return;
        if (!wait_w(smem_u32(&tl->o_done), item_par, tl, 326)) return;
        tc_fence_after();
        // both groups' sums, under the last reference
        const float now = u0 > 0 ? tl->ref[row] : -CUDART_INF_F;
        if (ref != -CUDART_INF_F && now != ref) l *= fast_exp2((ref - now) * P.scale_log2);
        tl->sum[grp][row] = l;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tl->sums_there[wq]));
        unsigned ra[64];  // this group stores channels 64 grp .. 64 grp + 63 of every token
        tmem_ld_32x32_issue(lanes + kOCol + grp * 64, ra);
        tmem_ld_32x32_issue(lanes + kOCol + grp * 64 + 32, ra + 32);
        tmem_ld_wait();
        tc_fence_before();
        if (!wait_w(smem_u32(&tl->sums_there[wq]), item_par, tl, 327)) return;
        const float total = l + tl->sum[grp ^ 1][row];
        if (grp == 0) tl->ref[row] = -CUDART_INF_F;  // for the next tokens, whose first entry is this group's
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tl->o_free));
        const float inv = total > 0.f ? 1.f / total : 0.f;
        unsigned char *const dst = stage + qs.idx * kQTile + lane * 128;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            unsigned w[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                // (without any entry O holds another token's numbers)
                const float a = total > 0.f ? __uint_as_float(ra[8 * c + 2 * v]) * inv : 0.f;
                const float d = total > 0.f ? __uint_as_float(ra[8 * c + 2 * v + 1]) * inv : 0.f;
                const __nv_bfloat162 pk = __floats2bfloat162_rn(a, d);
                w[v] = *reinterpret_cast<const unsigned *>(&pk);
            }
            *reinterpret_cast<uint4 *>(dst + ((c ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0 && tq < g.T) {
            tma_store_4d(to, smem_u32(stage + qs.idx * kQTile), grp * 64, tq, h, b);
            tma_store_commit();
        }
        staged = qs.idx;
        qs.advance(2);
        item_par ^= 1;
        n_other += (unsigned)(grp == 0 ? u0 >> 1 : (u0 + 1) >> 1);
    }
    if (lane == 0) tma_store_wait_read();  // shared memory is given back when the CTA leaves
    __syncwarp();
}

__global__ void __launch_bounds__(kThreads, 1)
attn_tok_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_out, Params P) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = aligned_smem(smem_raw);
    const unsigned q_smem = smem_u32(smem), k_smem = q_smem + 2 * kQTile, v_smem = k_smem + kKStages * kTile;
    Tail *tl = (Tail *)(smem + 2 * kQTile + (kKStages + kVStages) * kTile);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&tl->q_full[i]), 1); mbar_init(smem_u32(&tl->q_free[i]), 8);
            mbar_init(smem_u32(&tl->s_full[i]), 1); mbar_init(smem_u32(&tl->s_free[i]), 4);
            for (int j = 0; j < 2; ++j) { mbar_init(smem_u32(&tl->p_full[i][j]), 4); mbar_init(smem_u32(&tl->p_free[i][j]), 1); }
        }
        for (int i = 0; i < kKStages; ++i) { mbar_init(smem_u32(&tl->k_full[i]), 1); mbar_init(smem_u32(&tl->k_empty[i]), 1); }
        for (int i = 0; i < kVStages; ++i) { mbar_init(smem_u32(&tl->v_full[i]), 1); mbar_init(smem_u32(&tl->v_empty[i]), 1); }
        mbar_init(smem_u32(&tl->o_done), 1);
        mbar_init(smem_u32(&tl->o_free), 8);
        for (int i = 0; i < 4; ++i) {
            mbar_init(smem_u32(&tl->turn[i][0]), 1); mbar_init(smem_u32(&tl->turn[i][1]), 1);
            mbar_init(smem_u32(&tl->sums_there[i]), 2);
        }
        for (int i = 0; i < kMaskSlots; ++i) { mbar_init(smem_u32(&tl->m_full[i]), 1); mbar_init(smem_u32(&tl->m_empty[i]), 12); }
        tl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < kTok) tl->ref[threadIdx.x] = -CUDART_INF_F;
    if (warp == 1) tmem_alloc(smem_u32(&tl->tmem_base));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = tl->tmem_base;
    after_previous_kernel();
    if (warp == 0) {
        producer_role(P, &tmap_q, &tmap_k, &tmap_v, tl, q_smem, k_smem, v_smem);
    } else if (warp == 1) {
        qk_role(tl, q_smem, k_smem, tmem_base);
    } else if (warp == 2) {
        mask_role(P, tl, lane);
    } else if (warp == 3) {
        pv_role(tl, v_smem, tmem_base);
    } else {
        softmax_role(P, &tmap_out, tl, smem, tmem_base, (int)threadIdx.x - 128);
    }
    __syncwarp();
    leave(&tl->abort_flag, tmem_base, warp == 1);
}

}  // namespace

// Blocks of 16 tokens or more are better off with a row's blocks for themselves (attn_mma.cu).
bool attn_tok_supported(const Geom &g, int dtype, const void *q, const void *k, const void *v, const void *out) {
    return dtype == STREAM_BF16 && g.d == kD && g.bq < 16 && g.bk == kBlk && tma_strides_ok(g) && g.T < (1ll << 31) - kTok &&
           (((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out) & 15) == 0;
}

stream_status launch_attn_tok(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale,
                              void *out, cudaStream_t st) {
    CUtensorMap tq, tk, tv, to;
    stream_status rc = make_map_bf16_d128(&tq, q, g.T, g.H, g.batch, g.qs_t, g.qs_h, g.qs_b, "q", kTok);
    if (rc != STREAM_OK) return rc;
    rc = make_map5_bf16(&tk, k, g.T, g.G, g.batch, g.ks_t, g.ks_h, g.ks_b, "k", 64, 128);
    if (rc != STREAM_OK) return rc;
    rc = make_map5_bf16(&tv, v, g.T, g.G, g.batch, g.ks_t, g.ks_h, g.ks_b, "v", 64, 128);
    if (rc != STREAM_OK) return rc;
    rc = make_map_bf16_d128(&to, out, g.T, g.H, g.batch, kD, g.T * kD, (long long)g.H * g.T * kD, "out", 32);
    if (rc != STREAM_OK) return rc;
    Params P;
    P.g = g;
    P.n_tb = (int)((g.T + kTok - 1) / kTok);
    const long long fit = kL2KvBytes / (2ll * g.T * kD * 2), all = (long long)g.batch * g.G;
    P.group_heads = (int)(fit < 1 ? 1 : (fit > all ? all : fit));
    const long long n_items = (long long)g.batch * g.H * P.n_tb;
    if (n_items > 0x7fffffffLL - (1 << 20)) { set_error("too many rows for 32-bit indexing"); return STREAM_ERR_UNSUPPORTED; }
    P.n_items = (int)n_items;
    P.mask = mask;
    P.out = (__nv_bfloat16 *)out;
    P.scale_log2 = scale * 1.4426950408889634f;
    const int n_sm = sm_count();
    if (n_sm <= 0) { set_error("cannot read the SM count of the current device"); return STREAM_ERR_CUDA; }
    cudaError_t e = cudaFuncSetAttribute(attn_tok_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(attn_tok)");
    const int grid = (int)(n_items < n_sm ? n_items : n_sm);
    e = launch_kernel(attn_tok_kernel, grid, kThreads, kSmemBytes, st, 1, tq, tk, tv, to, P);
    if (e != cudaSuccess) return cuda_fail(e, "attn_tok launch");
    return STREAM_OK;
}

stream_status read_attn_tok_status(unsigned int out[2], cudaStream_t st) {
    cudaError_t e = cudaMemcpyFromSymbolAsync(out, g_attn_tok_status, 2 * sizeof(unsigned int), 0, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyFromSymbolAsync(attention status)");
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    return STREAM_OK;
}

}  // namespace stream
