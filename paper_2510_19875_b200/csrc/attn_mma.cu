// Block-sparse attention (Eq. 2 on a Stream mask) on mma.sync for the bf16 shapes that the tcgen05
// kernels do not take: d = 64 / 128 / 256, any block sizes up to 64, per-token masks among them.
//
// A warp owns 16 query tokens: their Q fragments (registers; shared memory for d = 256), their
// output accumulators and softmax statistics. Key and value tiles come to shared memory by
// cp.async, one K and one V buffer per group of warps that walks the same tiles: the next K tile
// is fetched while the present one's softmax and P V run, the next V tile behind P V.
//   - Fragments are read with 16-byte shared loads and no transposition: the contraction of Q K^T
//     may take its channels in any order, so lane t of a quad reads 8 consecutive ones; in P V lane
//     (g, t) reads channels 8 g .. 8 g + 7 of the keys it needs and interleaves two keys' words,
//     which makes physical channel 8 g + j column g of product j. A lane ends up with 16
//     consecutive output channels per 64.
//   - P goes in as two bf16 numbers, the rounded value and the rest (relative error 2^-17): the
//     kernel keeps the precision of the fp32 weights at the price of one more product per P V.
//
// Two ways to walk the mask:
//   rows    (block_q >= 16) a group of ceil(block_q / 16) warps takes one row's kept blocks; several
//           groups share a row's blocks (block n to group n mod S) and add up at the end.
//   merged  (block_q < 16) a CTA takes 64 consecutive tokens, whose rows differ. Their blocks are
//           merged, a window of 128 key blocks at a time, into one ascending list with a bit per
//           row: each tile is fetched once and multiplied for the warps that have a token keeping
//           it; tokens that do not keep it are masked like keys after the token.
//           (d = 128 with blocks of 64 keys: attn_tok.cu.)
// Bound: the latency of dependent steps at 8 to 16 warps per SM (issue slots 41 % busy, mma pipe 23
// to 35 %); hence the register limits below (12 heads, T = 10007, blocks of 32, d = 128, k = 8: 180
// us at two CTAs of four warps per SM, 152 at three, 3220 on the fp32-FMA kernel; 16 heads, T = 8192, d = 64,
// k = 40, not causal: 669, 600 at four, 4640). It serves d = 256, blocks other than 32 and 64, block_q !=
// block_k, and per-token masks beside attn_tok.cu's.
#include "warp_common.cuh"

namespace stream {
namespace {

using namespace wp;

constexpr int kMaxBlock = 64;
constexpr int kWindow = 128;          // merged: key blocks per window
constexpr int kMergedWarps = 4;       // merged: warps (16 tokens each) per group
constexpr int kMaxRows = 16 * kMergedWarps;
constexpr size_t kMaxDynamicSmem = 227 * 1024 - 2048;  // (the merged walk's bits are static)

struct Params {
    Geom g;
    const __nv_bfloat16 *q, *k, *v;
    const int32_t *mask;
    __nv_bfloat16 *out;
    float scale_log2;
    int m_warps, splits;   // warps per group, groups per CTA
    int merged;
    int n_tb;              // merged: token groups per head
};

// A warp's 16 tokens and what they have gathered.
template <int D, int BK>
struct Walk {
    static constexpr int kPitch = D * 2;                 // bytes per key row
    static constexpr int kTileBytes = BK * kPitch;
    static constexpr int kQRegs = D <= 128 ? D / 32 : 0;  // 32-channel groups of Q held in registers

    float o[D / 8][4];
    float m_run[2], l_run[2];      // rows gr and gr + 8 of the warp's 16 tokens
    uint4 qa[kQRegs > 0 ? kQRegs : 1], qc[kQRegs > 0 ? kQRegs : 1];

    __device__ void clear() {
#pragma unroll
        for (int i = 0; i < D / 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) o[i][j] = 0.f;
        m_run[0] = m_run[1] = -CUDART_INF_F;
        l_run[0] = l_run[1] = 0.f;
    }

    // Weights of one tile. lim: keys (a prefix) the lane's two tokens may look at.
    __device__ void tile(const unsigned char *ks, const unsigned char *qs, int lim0, int lim1, float scale_log2, unsigned *p_hi,
                         unsigned *p_lo) {
        const int lane = threadIdx.x & 31, gr = lane >> 2, t = lane & 3;
        float s[BK / 8][4];
#pragma unroll
        for (int n = 0; n < BK / 8; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) s[n][i] = 0.f;
        const unsigned char *kr = ks + gr * kPitch;  // (key n * 8 + gr has the swizzle of gr)
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
            const int at = ((4 * c + t) ^ swz_rows(gr)) << 4;
            uint4 a, a8;
            if (kQRegs > 0) {
                a = qa[c % (kQRegs > 0 ? kQRegs : 1)]; a8 = qc[c % (kQRegs > 0 ? kQRegs : 1)];
            } else {
                a = *(const uint4 *)(qs + gr * kPitch + at); a8 = *(const uint4 *)(qs + (gr + 8) * kPitch + at);
            }
            // (two products of one accumulator never back to back: the second would wait for the first)
            uint4 x[BK / 8];
#pragma unroll
            for (int n = 0; n < BK / 8; ++n) {
                x[n] = *(const uint4 *)(kr + n * 8 * kPitch + at);
                mma_bf16(s[n], a.x, a8.x, a.y, a8.y, x[n].x, x[n].y);
            }
#pragma unroll
            for (int n = 0; n < BK / 8; ++n) mma_bf16(s[n], a.z, a8.z, a.w, a8.w, x[n].z, x[n].w);
        }
        if (__any_sync(0xffffffffu, lim0 < BK || lim1 < BK)) {
#pragma unroll
            for (int n = 0; n < BK / 8; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (n * 8 + 2 * t + (i & 1) >= (i < 2 ? lim0 : lim1)) s[n][i] = -CUDART_INF_F;
        }
        float mx[2] = {m_run[0], m_run[1]};
#pragma unroll
        for (int n = 0; n < BK / 8; ++n) {
            mx[0] = fmaxf(mx[0], fmaxf(s[n][0], s[n][1]));
            mx[1] = fmaxf(mx[1], fmaxf(s[n][2], s[n][3]));
        }
        float base[2], alpha[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 1));
            mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 2));
            const float ref = mx[i] == -CUDART_INF_F ? 0.f : mx[i];
            alpha[i] = fast_exp2((m_run[i] - ref) * scale_log2);  // (nothing gathered yet: 0)
            base[i] = ref * scale_log2;
            m_run[i] = mx[i];
        }
        if (__any_sync(0xffffffffu, alpha[0] != 1.f || alpha[1] != 1.f)) {
#pragma unroll
            for (int i = 0; i < D / 8; ++i) {
                o[i][0] *= alpha[0]; o[i][1] *= alpha[0];
                o[i][2] *= alpha[1]; o[i][3] *= alpha[1];
            }
        }
        float sum[2] = {0.f, 0.f};
#pragma unroll
        for (int n = 0; n < BK / 8; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float p0 = fast_exp2(fmaf(s[n][2 * i], scale_log2, -base[i]));
                const float p1 = fast_exp2(fmaf(s[n][2 * i + 1], scale_log2, -base[i]));
                sum[i] += p0 + p1;
                const __nv_bfloat162 hi = __floats2bfloat162_rn(p0, p1);
                const float2 back = __bfloat1622float2(hi);
                const __nv_bfloat162 lo = __floats2bfloat162_rn(p0 - back.x, p1 - back.y);
                p_hi[2 * n + i] = *reinterpret_cast<const unsigned *>(&hi);
                p_lo[2 * n + i] = *reinterpret_cast<const unsigned *>(&lo);
            }
        // (each lane of a quad keeps its own part of the sum; they meet at the end)
        l_run[0] = l_run[0] * alpha[0] + sum[0];
        l_run[1] = l_run[1] * alpha[1] + sum[1];
    }

    __device__ void add_pv(const unsigned char *vs, const unsigned *p_hi, const unsigned *p_lo) {
        const int lane = threadIdx.x & 31, gr = lane >> 2, t = lane & 3;
#pragma unroll
        for (int j = 0; j < BK / 16; ++j) {
            // keys 2 t, 2 t + 1, 2 t + 8, 2 t + 9 of these 16: swizzle = key mod 8
            const unsigned char *v0 = vs + (j * 16 + 2 * t) * kPitch, *v1 = v0 + kPitch;
#pragma unroll
            for (int cg = 0; cg < D / 64; ++cg) {
                const int a0 = ((8 * cg + gr) ^ (2 * t)) << 4, a1 = ((8 * cg + gr) ^ (2 * t + 1)) << 4;
                const uint4 r0 = *(const uint4 *)(v0 + a0), r1 = *(const uint4 *)(v1 + a1);
                const uint4 r2 = *(const uint4 *)(v0 + 8 * kPitch + a0), r3 = *(const uint4 *)(v1 + 8 * kPitch + a1);
                const unsigned w0[4] = {r0.x, r0.y, r0.z, r0.w}, w1[4] = {r1.x, r1.y, r1.z, r1.w};
                const unsigned w2[4] = {r2.x, r2.y, r2.z, r2.w}, w3[4] = {r3.x, r3.y, r3.z, r3.w};
                unsigned b0[8], b1[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    const unsigned sel = (x & 1) ? 0x7632u : 0x5410u;
                    b0[x] = __byte_perm(w0[x >> 1], w1[x >> 1], sel);
                    b1[x] = __byte_perm(w2[x >> 1], w3[x >> 1], sel);
                    mma_bf16(o[cg * 8 + x], p_hi[4 * j], p_hi[4 * j + 1], p_hi[4 * j + 2], p_hi[4 * j + 3], b0[x], b1[x]);
                }
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    mma_bf16(o[cg * 8 + x], p_lo[4 * j], p_lo[4 * j + 1], p_lo[4 * j + 2], p_lo[4 * j + 3], b0[x], b1[x]);
            }
        }
    }
};

// One [BK][D] tile of block r (token stride ks_t) to shared memory by the `n_thr` threads of a
// group; rows beyond the block or beyond T become zeros.
template <int D, int BK, bool kIsK>
__device__ __forceinline__ void fetch(const Geom &g, unsigned dst, const __nv_bfloat16 *base, int r, int thr, int n_thr) {
    constexpr int per_row = D / 8;
    for (int idx = thr; idx < BK * per_row; idx += n_thr) {
        const int n = idx / per_row, c = idx % per_row;
        const long long tk = (long long)r * g.bk + n;
        const bool in = n < g.bk && tk < g.T;
        const int swz = kIsK ? swz_rows(n) : (n & 7);
        cp_async16(dst + n * D * 2 + ((c ^ swz) << 4), base + (in ? tk : 0) * g.ks_t + c * 8, in ? 16 : 0);
    }
    cp_async_commit();
}

// CTAs of four warps an SM should hold: what the registers allow without spilling in the inner loops.
template <int D, int BK>
constexpr int ctas_per_sm() { return D == 64 ? 4 : (D == 128 && BK <= 32 ? 3 : 2); }

template <int D, int BK, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, WARPS == 4 ? ctas_per_sm<D, BK>() : 1) attn_mma_kernel(Params P) {
    using W = Walk<D, BK>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_n, s_again;
    __shared__ unsigned row_bits[kMaxRows][kWindow / 32];  // merged: the window's blocks each row keeps
    __shared__ unsigned any_bits[kWindow / 32];
    const Geom &g = P.g;
    after_previous_kernel();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, t = lane & 3;
    const int grp = warp / P.m_warps, mw = warp % P.m_warps, g_thr = P.m_warps * 32, g_tid = tid - grp * g_thr;

    int b, h, first_row, n_rows;   // merged: rows first_row .. + n_rows; else the one row
    long long tok0;
    if (P.merged) {
        const int bh = blockIdx.x / P.n_tb, tb = P.n_tb - 1 - (int)(blockIdx.x % P.n_tb);  // late tokens first
        b = bh / g.H; h = bh % g.H;
        tok0 = (long long)tb * kMaxRows;
        first_row = (int)(tok0 / g.bq);
        n_rows = (int)((min(tok0 + kMaxRows, g.T) - 1) / g.bq) - first_row + 1;
    } else {
        const int bh = blockIdx.x / g.n_qb, qb = g.n_qb - 1 - (int)(blockIdx.x % g.n_qb);
        b = bh / g.H; h = bh % g.H;
        tok0 = (long long)qb * g.bq;
        first_row = qb; n_rows = 1;
    }
    const int kvh = h / g.hpg;
    const __nv_bfloat16 *qp = P.q + b * g.qs_b + h * g.qs_h;
    const __nv_bfloat16 *kp = P.k + b * g.ks_b + kvh * g.ks_h, *vp = P.v + b * g.ks_b + kvh * g.ks_h;
    const int32_t *mrow = P.mask + (((long long)b * g.H + h) * g.n_qb + first_row) * g.k_top;

    unsigned char *ks = smem + grp * 2 * W::kTileBytes, *vs = ks + W::kTileBytes;
    int *list = (int *)(smem + P.splits * 2 * W::kTileBytes);
    unsigned char *qs = (unsigned char *)list + (P.merged ? kWindow : ((g.k_top + 3) & ~3)) * 4;  // d = 256 only

    // this warp's 16 tokens
    const int m0 = mw * 16 + gr;                 // token of the lane's first row, counted from tok0
    const long long t0 = tok0 + m0, t1 = t0 + 8;
    const int m_end = P.merged ? kMaxRows : g.bq;  // tokens of this CTA
    const bool ok0 = m0 < m_end && t0 < g.T, ok1 = m0 + 8 < m_end && t1 < g.T;
    W w;
    w.clear();
    if (W::kQRegs > 0) {
#pragma unroll
        for (int c = 0; c < W::kQRegs; ++c) {
            w.qa[c] = ok0 ? *(const uint4 *)(qp + t0 * g.qs_t + 32 * c + 8 * t) : make_uint4(0, 0, 0, 0);
            w.qc[c] = ok1 ? *(const uint4 *)(qp + t1 * g.qs_t + 32 * c + 8 * t) : make_uint4(0, 0, 0, 0);
        }
    } else {
        for (int idx = tid; idx < P.m_warps * 16 * (D / 8); idx += blockDim.x) {
            const int m = idx / (D / 8), c = idx % (D / 8);
            uint4 x = make_uint4(0, 0, 0, 0);
            if (m < m_end && tok0 + m < g.T) x = *(const uint4 *)(qp + (tok0 + m) * g.qs_t + c * 8);
            *(uint4 *)(qs + m * D * 2 + ((c ^ swz_rows(m)) << 4)) = x;
        }
    }
    const unsigned char *qw = qs + mw * 16 * D * 2;

    // Tiles list[grp], list[grp + splits], ... of n. `row0`, `row1`: in the merged walk, the rows of the
    // lane's two tokens, whose bits say whether they keep the window's block; list then holds blocks
    // relative to `block0`.
    auto walk = [&](int n, int block0, int row0, int row1) {
        const unsigned ks_s = smem_addr(ks), vs_s = smem_addr(vs);
        if (grp < n) {
            fetch<D, BK, true>(g, ks_s, kp, block0 + list[grp], g_tid, g_thr);
            fetch<D, BK, false>(g, vs_s, vp, block0 + list[grp], g_tid, g_thr);
        }
        for (int i = grp; i < n; i += P.splits) {
            const int rel = list[i], r = block0 + rel;
            const int r_next = i + P.splits < n ? block0 + list[i + P.splits] : -1;
            const long long k0 = (long long)r * g.bk;
            long long l0 = min((long long)g.bk, g.T - k0), l1 = l0;
            if (g.causal) { l0 = min(l0, t0 - k0 + 1); l1 = min(l1, t1 - k0 + 1); }
            int lim0 = ok0 ? (int)max(0ll, l0) : 0, lim1 = ok1 ? (int)max(0ll, l1) : 0;
            if (P.merged) {
                if (!ok0 || !((row_bits[row0][rel >> 5] >> (rel & 31)) & 1u)) lim0 = 0;
                if (!ok1 || !((row_bits[row1][rel >> 5] >> (rel & 31)) & 1u)) lim1 = 0;
            }
            const bool any = __any_sync(0xffffffffu, lim0 > 0 || lim1 > 0);
            unsigned p_hi[BK / 4], p_lo[BK / 4];
            cp_async_wait<1>();
            group_sync(1 + grp, g_thr);  // the K tile is there
            if (any) w.tile(ks, qw, lim0, lim1, P.scale_log2, p_hi, p_lo);
            group_sync(1 + grp, g_thr);  // everybody is done with it
            if (r_next >= 0) fetch<D, BK, true>(g, ks_s, kp, r_next, g_tid, g_thr);
            else cp_async_commit();
            cp_async_wait<1>();
            group_sync(1 + grp, g_thr);  // the V tile is there
            if (any) w.add_pv(vs, p_hi, p_lo);
            group_sync(1 + grp, g_thr);
            if (r_next >= 0) fetch<D, BK, false>(g, vs_s, vp, r_next, g_tid, g_thr);
        }
        cp_async_wait<0>();
    };

    if (!P.merged) {
        // the row's kept entries, in order
        if (warp == 0) {
            int n = 0;
            for (int j = 0; j < g.k_top; j += 32) {
                const int r = j + lane < g.k_top ? mrow[j + lane] : -1;
                const unsigned bal = __ballot_sync(0xffffffffu, r >= 0);
                if (r >= 0) list[n + __popc(bal & ((1u << lane) - 1u))] = r;
                n += __popc(bal);
            }
            if (lane == 0) s_n = n;
        }
        __syncthreads();
        walk(s_n, 0, 0, 0);
    } else {
        const int row0 = (int)(min(t0, g.T - 1) / g.bq) - first_row, row1 = (int)(min(t1, g.T - 1) / g.bq) - first_row;
        const int n_entries = n_rows * g.k_top, n_kb = (int)((g.T + g.bk - 1) / g.bk);
        for (int block0 = 0; block0 < n_kb; block0 += kWindow) {
            // `nth`: a block that occurs more than once in a row counts as often (occurrence nth of every
            // entry in this round; a second round only if the first met a repetition)
            for (int nth = 0;; ++nth) {
                __syncthreads();  // the previous list and bits are done with
                for (int i = tid; i < kMaxRows * (kWindow / 32); i += blockDim.x) (&row_bits[0][0])[i] = 0u;
                if (tid < kWindow / 32) any_bits[tid] = 0u;
                if (tid == 0) s_again = 0;
                __syncthreads();
                for (int i = tid; i < n_entries; i += blockDim.x) {
                    const int rel = mrow[i] - block0, row = i / g.k_top;
                    if (mrow[i] < 0 || rel < 0 || rel >= kWindow) continue;
                    if (nth > 0) {
                        int before = 0;
                        for (int j = row * g.k_top; j < i; ++j) before += mrow[j] == mrow[i];
                        if (before > nth) s_again = 1;
                        if (before != nth) continue;
                    }
                    const unsigned bit = 1u << (rel & 31);
                    if (atomicOr(&row_bits[row][rel >> 5], bit) & bit) s_again = 1;
                    atomicOr(&any_bits[rel >> 5], bit);
                }
                __syncthreads();
                if (warp == 0) {
                    int n = 0;
#pragma unroll
                    for (int x = 0; x < kWindow / 32; ++x) {
                        const unsigned bits = any_bits[x];
                        if ((bits >> lane) & 1u) list[n + __popc(bits & ((1u << lane) - 1u))] = x * 32 + lane;
                        n += __popc(bits);
                    }
                    if (lane == 0) s_n = n;
                }
                __syncthreads();
                const bool again = s_again != 0;
                walk(s_n, block0, row0, row1);
                if (!again) break;
            }
        }
    }

    // Sum over the groups: the others leave their parts in shared memory, group 0 adds them.
    float *part = (float *)smem;  // [splits - 1][m_warps][D / 2 + 4 floats per lane]
    constexpr int kPart = D / 2 + 4;
    if (P.splits > 1) {
        __syncthreads();
        if (grp > 0) {
            float *x = part + (size_t)((grp - 1) * P.m_warps + mw) * kPart * 32 + lane;
#pragma unroll
            for (int i = 0; i < D / 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) x[(i * 4 + j) * 32] = w.o[i][j];
#pragma unroll
            for (int i = 0; i < 2; ++i) { x[(D / 2 + i) * 32] = w.m_run[i]; x[(D / 2 + 2 + i) * 32] = w.l_run[i]; }
        }
        __syncthreads();
        if (grp > 0) return;
        for (int s = 1; s < P.splits; ++s) {
            const float *x = part + (size_t)((s - 1) * P.m_warps + mw) * kPart * 32 + lane;
            float fo[2], fx[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float mx = x[(D / 2 + i) * 32], lx = x[(D / 2 + 2 + i) * 32];
                const float top = fmaxf(w.m_run[i], mx), ref = top == -CUDART_INF_F ? 0.f : top;
                fo[i] = fast_exp2((w.m_run[i] - ref) * P.scale_log2);
                fx[i] = fast_exp2((mx - ref) * P.scale_log2);
                w.l_run[i] = w.l_run[i] * fo[i] + lx * fx[i];
                w.m_run[i] = top;
            }
#pragma unroll
            for (int i = 0; i < D / 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) w.o[i][j] = w.o[i][j] * fo[j >> 1] + x[(i * 4 + j) * 32] * fx[j >> 1];
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float l = w.l_run[i];
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        const float inv = l > 0.f ? 1.f / l : 0.f;
        if (!(i == 0 ? ok0 : ok1)) continue;
        __nv_bfloat16 *dst = P.out + (((long long)b * g.H + h) * g.T + (i == 0 ? t0 : t1)) * D;
#pragma unroll
        for (int cg = 0; cg < D / 64; ++cg)
#pragma unroll
            for (int half = 0; half < 2; ++half) {  // channels 64 cg + 16 t + 8 half ..
                unsigned x[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const __nv_bfloat162 pk = __floats2bfloat162_rn(w.o[cg * 8 + 2 * j][2 * i + half] * inv, w.o[cg * 8 + 2 * j + 1][2 * i + half] * inv);
                    x[j] = *reinterpret_cast<const unsigned *>(&pk);
                }
                *(uint4 *)(dst + 64 * cg + 16 * t + 8 * half) = make_uint4(x[0], x[1], x[2], x[3]);
            }
    }
}

template <int D, int BK>
stream_status launch(Params P, cudaStream_t st) {
    const Geom &g = P.g;
    using W = Walk<D, BK>;
    P.merged = g.bq < 16;
    P.m_warps = P.merged ? kMergedWarps : (g.bq + 15) / 16;
    P.n_tb = (int)((g.T + kMaxRows - 1) / kMaxRows);
    const long long ctas = (long long)g.batch * g.H * (P.merged ? P.n_tb : g.n_qb);
    // Four warps a CTA (eight when there are too few CTAs to give every SM several): whole groups of
    // m_warps, the splits, as many of them as shared memory has room for (a group of one warp, tiles of 64 keys,
    // d = 256: three).
    const bool wide = ctas < 3ll * sm_count_or_default();
    auto bytes = [&](int splits) {
        size_t walk = (size_t)splits * 2 * W::kTileBytes + (size_t)(P.merged ? kWindow : ((g.k_top + 3) & ~3)) * 4;
        if (W::kQRegs == 0) walk += (size_t)P.m_warps * 16 * D * 2;
        const size_t part = (size_t)(splits - 1) * P.m_warps * (D / 2 + 4) * 32 * 4;
        return walk > part ? walk : part;
    };
    P.splits = (wide ? 8 : 4) / P.m_warps;
    while (P.splits > 1 && bytes(P.splits) > kMaxDynamicSmem) --P.splits;
    const size_t smem = bytes(P.splits);
    auto kern = wide ? attn_mma_kernel<D, BK, 8> : attn_mma_kernel<D, BK, 4>;
    cudaError_t e = allow_smem(kern, kMaxDynamicSmem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(attn_mma)");
    e = launch_kernel(kern, (unsigned)ctas, P.m_warps * P.splits * 32, smem, st, 1, P);
    if (e != cudaSuccess) return cuda_fail(e, "attn_mma launch");
    return STREAM_OK;
}

template <int D>
stream_status dispatch_bk(const Params &P, cudaStream_t st) {
    if (P.g.bk <= 16) return launch<D, 16>(P, st);
    if (P.g.bk <= 32) return launch<D, 32>(P, st);
    return launch<D, 64>(P, st);
}

}  // namespace

bool attn_mma_supported(const Geom &g, int dtype, const void *q, const void *k, const void *v, const void *out) {
    return dtype == STREAM_BF16 && (g.d == 64 || g.d == 128 || g.d == 256) && g.bq <= kMaxBlock && g.bk <= kMaxBlock &&
           rows_16_byte_aligned(q, g.qs_t, g.qs_h, g.qs_b, 2) && rows_16_byte_aligned(k, g.ks_t, g.ks_h, g.ks_b, 2) &&
           ((uintptr_t)v & 15) == 0 && ((uintptr_t)out & 15) == 0;
}

stream_status launch_attn_mma(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale,
                              void *out, cudaStream_t st) {
    Params P = {};
    P.g = g;
    P.q = (const __nv_bfloat16 *)q; P.k = (const __nv_bfloat16 *)k; P.v = (const __nv_bfloat16 *)v;
    P.mask = mask;
    P.out = (__nv_bfloat16 *)out;
    P.scale_log2 = scale * 1.4426950408889634f;
    switch (g.d) {
        case 64: return dispatch_bk<64>(P, st);
        case 128: return dispatch_bk<128>(P, st);
        default: return dispatch_bk<256>(P, st);
    }
}

}  // namespace stream
