// Stream mask kernel for every shape the tcgen05 kernels do not take (Algorithm 2): one CTA per
// (batch, head, query block), its warps taking the candidate tiles of a level in turn.
//
// Two ways to score a tile, behind one controller:
//   MmaScore   bf16, d = 64 / 128 / 256, 16-byte aligned rows: mma.sync m16n8k16, exact products,
//              fp32 accumulation. A warp holds 32 keys x all queries of the row. Key fragments come
//              straight from global memory (L2) in 16-byte loads: the contraction does not care in
//              which order its channels are taken, so lane t of a quad reads 8 consecutive channels
//              and both operands use that order. Query fragments come from shared memory.
//   FmaScore   everything else (fp32; any d, alignment; bf16 when the fp32-FMA kernels are asked
//              for): fp32 FMA, one warp per 32-key x up to 32-query part of a tile, the key rows
//              staged in shared memory 32 channels at a time, one chunk ahead. Channels are added in
//              ascending order, one accumulator per (query, key).
// Bound: the L2 round trip and the barriers of a row's few small levels (issue slots 39 % busy, mma
// pipe 22 % in the MMA form; 59 % in the FMA form), which is why a row gets only four warps and an
// SM several rows: the 7 to 16 tiles of a level leave eight warps unequal work (12 heads,
// T = 10007, blocks of 32, d = 128, bf16, k = 8: 310 us with eight warps a row, 222 with four; 8
// heads, T = 5003, blocks of 32, d = 64, fp32: 246 and 216, and 181 since a unit's divisions are done
// once and not with every chunk). Against 256 threads on one padded 64 x 64 tile at a time, with scalar
// loads and four barriers per tile: the fp32 shape 812 -> 181 us; with the attention, 12 heads, T = 5676, d = 256,
// blocks of 64, k = 33, bf16: 12192 -> 1065; 6 heads, T = 17577, blocks of 16: 37015 -> 793. (The MMA form
// serves d = 256, blocks other than 32 and 64, block_q != block_k and k above 64.)
//
// Follows Algorithm 2 with two exact shortcuts: branches without an allowed block are dropped (they
// score -inf and can never displace a finite score), and a left branch inherits its parent's score
// (same representative).
#include "warp_common.cuh"

namespace stream {
namespace {

using namespace wp;

constexpr int kMaxBlock = 64;
constexpr int kWideWarps = 16;    // warps of a row when there are no more rows than SMs
constexpr int kKeysPerUnit = 32;  // keys of a tile one warp scores at a time

// Which (query m, key n) pairs of query block qb and key block r are allowed, counted from the
// blocks' first tokens: m < n_q, n < n_k and n - m <= diag.
struct Allowed {
    int n_q, n_k, diag;
    __device__ Allowed(const Geom &g, int qb, int r) {
        const long long tq0 = (long long)qb * g.bq, tk0 = (long long)r * g.bk;
        n_q = (int)min((long long)g.bq, g.T - tq0);
        n_k = (int)min((long long)g.bk, g.T - tk0);
        diag = g.causal ? (int)max(-64ll, min(64ll, tq0 - tk0)) : 64;
    }
    __device__ bool all(int q_rows, int k_end) const { return q_rows <= n_q && k_end <= n_k && k_end - 1 <= diag; }
    __device__ bool operator()(int m, int n) const { return m < n_q && n < n_k && n - m <= diag; }
};

// ----------------------------------------------------------------------------------------------
// fp32 FMA
// ----------------------------------------------------------------------------------------------
// Lane (kq = lane / 4, kk = lane % 4) holds queries kq + 8 i (i < RQ) x keys kk + 4 j (j < 8): per
// four channels RQ + 8 16-byte shared loads (conflict-free, broadcast over the lanes) feed 32 RQ FMA.
template <typename T, int D, int RQ, Load kLoad>
struct FmaScore {
    using Elem = T;
    static constexpr bool kRegisters = kLoad == Load::kWide || kLoad == Load::kScalars;
    static constexpr int kSQ = 8 * RQ, kCh = D < 32 ? D : 32, kChunks = D / kCh;
    static constexpr int kRowBytes = kCh * 4, kBufBytes = kKeysPerUnit * kRowBytes, kRing = 2;
    static constexpr int kSwz = kCh / 4 - 1;
    // Warps of a row, CTAs an SM should hold. Rows of up to 16 queries have half the register tile, and a fifth CTA pays (fp32, us: 8
    // heads, 4000 tokens, d = 128, blocks of 16, k = 16: 595 -> 555; 6 heads, 5000 tokens, d = 64, k = 8: 240 -> 223; 4 heads, 5500
    // tokens, d = 32, k = 6: 101 -> 89); 32 queries spill with it (181 -> 217).
    static constexpr int kWarps = 4, kCtas = RQ == 2 ? (kRegisters ? 4 : 5) : (kRegisters && D >= 64 ? 3 : 4);

    static int q_parts(const Geom &g) { return (g.bq + kSQ - 1) / kSQ; }
    static size_t smem_bytes(const Geom &g, int warps) {
        return (size_t)q_parts(g) * kSQ * D * 4 + (size_t)warps * kRing * kBufBytes;
    }

    static __device__ void load_q(const Geom &g, unsigned char *smem, const T *qp, int qb) {
        float *Qs = (float *)smem;
        const int rows = (g.bq + kSQ - 1) / kSQ * kSQ;
        for (int idx = threadIdx.x; idx < rows * D; idx += blockDim.x) {
            const int m = idx / D, c = idx % D;
            const long long tq = (long long)qb * g.bq + m;
            const float x = (m < g.bq && tq < g.T) ? to_float(qp[tq * g.qs_t + c]) : 0.f;
            Qs[m * D + ((((c >> 2) ^ (m & kSwz)) << 2) | (c & 3))] = x;
        }
    }

    // Scores list[0 .. n_list) (slots of `f`) and raises their keys.
    static __device__ void score(const Geom &g, unsigned char *smem, const T *kp, int qb, const int *list, int n_list,
                                 const int *f, unsigned *key) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
        const int nq = (g.bq + kSQ - 1) / kSQ, nk = (g.bk + kKeysPerUnit - 1) / kKeysPerUnit, per = nq * nk;
        const int n_units = n_list * per;
        const int mine = n_units > warp ? (n_units - warp + warps - 1) / warps : 0;
        const int n_chunks = mine * kChunks;
        const float *Qs = (const float *)smem;
        unsigned char *buf = smem + (size_t)nq * kSQ * D * 4 + (size_t)warp * kRing * kBufBytes;
        const unsigned buf_s = smem_addr(buf);
        const int kq = lane >> 2, kk = lane & 3;

        // A unit: slot, its key block, which queries and keys of the tile. (Taken apart once per unit: the
        // divisions are some hundred clocks each.)
        struct Unit { int slot, r, qs, ks; };
        auto unit = [&](int u) {
            const int e = per == 1 ? u : u / per, sub = u - e * per;
            Unit x;
            x.slot = list[e];
            x.r = f[x.slot];
            x.qs = nk == 1 ? sub : sub / nk;
            x.ks = sub - x.qs * nk;
            return x;
        };
        // Chunk q (channels cc) on its way: to its buffer, or (bf16) to registers, from where `put` takes it to the
        // buffer behind the products of the chunk before. (Keys beyond the block are never looked at. Loaded and
        // stored at once, element by element, a chunk waited for its loads.)
        constexpr int kPerKey = kCh / 4, kCopies = kKeysPerUnit * kPerKey / 32;
        uint2 raw[kRegisters ? kCopies : 1];
        auto place = [&](int q, int n, int c4) { return (q & 1) * kBufBytes + n * kRowBytes + ((c4 ^ (n & kSwz)) << 4); };
        auto issue = [&](const Unit &x, int q, int cc) {
            const int n0 = x.ks * kKeysPerUnit, n_end = min(g.bk - n0, kKeysPerUnit);
            const int last = (int)min((long long)g.bk, g.T - (long long)x.r * g.bk) - n0 - 1;  // (the tile's last key inside T stands in for those beyond)
            const T *base = kp + ((long long)x.r * g.bk + n0) * g.ks_t + cc * kCh;
            if constexpr (kLoad == Load::kCopy4) {
                constexpr int n_step = 32 / kCh;  // keys a warp copies at a time
                const int c = lane % kCh;
                const unsigned dst = buf_s + (q & 1) * kBufBytes + (c & 3) * 4;
                const long long step = n_step * g.ks_t;
                int n = lane / kCh;
                const T *src = base + (long long)min(n, last) * g.ks_t + c;
                if (last + 1 >= n_end) {
#pragma unroll 8
                    for (; n < n_end; n += n_step, src += step) cp_async4(dst + n * kRowBytes + (((c >> 2) ^ (n & kSwz)) << 4), src);
                } else {
                    for (; n < n_end; n += n_step) {
                        cp_async4(dst + n * kRowBytes + (((c >> 2) ^ (n & kSwz)) << 4), src);
                        src = base + (long long)min(n + n_step, last) * g.ks_t + c;
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < kCopies; ++i) {
                    const int idx = i * 32 + lane, n = idx / kPerKey, c4 = idx % kPerKey;
                    const T *src = base + (long long)min(n, last) * g.ks_t + c4 * 4;
                    if (n < n_end) {
                        if constexpr (kLoad == Load::kCopy16) cp_async16(buf_s + place(q, n, c4), src, 16);
                        else if constexpr (kLoad == Load::kWide) raw[i] = *(const uint2 *)src;
                        else raw[i] = load4(src);
                    }
                }
            }
            if (!kRegisters) cp_async_commit();
        };
        auto put = [&](int q) {
#pragma unroll
            for (int i = 0; i < kCopies; ++i) {
                const int idx = i * 32 + lane, n = idx / kPerKey, c4 = idx % kPerKey;
                *(float4 *)(buf + place(q, n, c4)) = widen4(raw[i]);
            }
        };

        Unit cur = {}, ahead = {};  // the unit being scored, the one being fetched
        if (n_chunks > 0) {
            ahead = unit(warp);
            issue(ahead, 0, 0);
            if constexpr (kRegisters) put(0);
        }
        float acc[RQ][8];
        for (int q = 0; q < n_chunks; ++q) {
            const int cc = q % kChunks;
            if (cc == 0) cur = ahead;
            if (q + 1 < n_chunks) {
                if (cc == kChunks - 1) ahead = unit(warp + (q + 1) / kChunks * warps);
                __syncwarp();  // every lane is done with the buffer's previous chunk
                issue(ahead, q + 1, (q + 1) % kChunks);
                if (!kRegisters) cp_async_wait<1>();
            } else if (!kRegisters) {
                cp_async_wait<0>();
            }
            __syncwarp();
            if (cc == 0) {
#pragma unroll
                for (int i = 0; i < RQ; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
            }
            const unsigned char *kb = buf + (q & 1) * kBufBytes;
            const float *qrow = Qs + (size_t)cur.qs * kSQ * D;
#pragma unroll 1
            for (int c4 = 0; c4 < kCh / 4; ++c4) {
                float4 a[RQ], b[8];
#pragma unroll
                for (int i = 0; i < RQ; ++i) {
                    const int m = kq + 8 * i;
                    a[i] = *(const float4 *)(qrow + m * D + (((cc * (kCh / 4) + c4) ^ (m & kSwz)) << 2));
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int n = kk + 4 * j;
                    b[j] = *(const float4 *)(kb + n * kRowBytes + ((c4 ^ (n & kSwz)) << 4));
                }
                fma_channel<RQ>(acc, a, b, &float4::x);
                fma_channel<RQ>(acc, a, b, &float4::y);
                fma_channel<RQ>(acc, a, b, &float4::z);
                fma_channel<RQ>(acc, a, b, &float4::w);
            }
            if constexpr (kRegisters) {
                if (q + 1 < n_chunks) put(q + 1);
            }
            if (cc == kChunks - 1) {
                float best = -CUDART_INF_F;
                const Allowed ok(g, qb, cur.r);
                if (ok.all((cur.qs + 1) * kSQ, (cur.ks + 1) * kKeysPerUnit)) {
#pragma unroll
                    for (int i = 0; i < RQ; ++i)
#pragma unroll
                        for (int j = 0; j < 8; ++j) best = fmaxf(best, acc[i][j]);
                } else {
                    const int m0 = cur.qs * kSQ + kq, n0 = cur.ks * kKeysPerUnit + kk;
#pragma unroll
                    for (int i = 0; i < RQ; ++i)
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (ok(m0 + 8 * i, n0 + 4 * j)) best = fmaxf(best, acc[i][j]);
                }
                best = warp_max(best);
                if (lane == 0 && best > -CUDART_INF_F) atomicMax(&key[cur.slot], key_of(best));
            }
        }
    }
};

// ----------------------------------------------------------------------------------------------
// mma.sync
// ----------------------------------------------------------------------------------------------
template <int D, int MT>  // MT: m16 tiles of the query block
struct MmaScore {
    using Elem = __nv_bfloat16;
    static constexpr int kGroups = D / 32;  // 32-channel groups: two k16 steps, one 16-byte load per lane and key
    // 32-channel groups whose key fragments are in registers or on their way (L2 takes some 700 clocks,
    // a group's 8 MT products 64 MT of one scheduler): what fits beside 16 MT accumulators
    static constexpr int kFit = MT == 4 ? 2 : (MT == 2 ? 3 : 4), kAhead = kGroups < kFit ? kGroups : kFit;
    static constexpr int kWarps = 4, kCtas = MT == 4 ? 3 : 4;

    static size_t smem_bytes(const Geom &, int) { return (size_t)MT * 16 * D * 2; }

    static __device__ void load_q(const Geom &g, unsigned char *smem, const __nv_bfloat16 *qp, int qb) {
        for (int idx = threadIdx.x; idx < MT * 16 * (D / 8); idx += blockDim.x) {
            const int m = idx / (D / 8), c = idx % (D / 8);
            const long long tq = (long long)qb * g.bq + m;
            uint4 x = make_uint4(0, 0, 0, 0);
            if (m < g.bq && tq < g.T) x = *(const uint4 *)(qp + tq * g.qs_t + c * 8);
            *(uint4 *)(smem + m * D * 2 + ((c ^ swz_rows(m)) << 4)) = x;
        }
    }

    static __device__ void score(const Geom &g, unsigned char *smem, const __nv_bfloat16 *kp, int qb, const int *list, int n_list,
                                 const int *f, unsigned *key) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
        const int gr = lane >> 2, t = lane & 3;
        const int nk = (g.bk + kKeysPerUnit - 1) / kKeysPerUnit;
        for (int u = warp; u < n_list * nk; u += warps) {
            const int slot = list[u / nk], r = f[slot], ks = u % nk;
            const int n_left = g.bk - ks * kKeysPerUnit;  // keys of the block from here on
            const long long tk0 = min((long long)r * g.bk + ks * kKeysPerUnit + gr, g.T - 1);
            const int beyond = (int)min(g.T - 1 - tk0, 24ll);  // (keys beyond T are read as the last one and never looked at)
            const __nv_bfloat16 *row0 = kp + tk0 * g.ks_t + 8 * t;
            int row[4];
#pragma unroll
            for (int n = 0; n < 4; ++n) row[n] = min(n * 8, beyond) * (int)g.ks_t;
            float acc[MT][4][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[m][n][i] = 0.f;
            uint4 b[kAhead][4];
#pragma unroll
            for (int c = 0; c < kAhead; ++c)
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    if (n * 8 < n_left) b[c][n] = *(const uint4 *)(row0 + row[n] + 32 * c);
#pragma unroll
            for (int c = 0; c < kGroups; ++c) {
                uint4 (&x)[4] = b[c % kAhead];
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const int m0 = m * 16 + gr, ch = 4 * c + t;
                    const uint4 qa = *(const uint4 *)(smem + m0 * D * 2 + ((ch ^ swz_rows(m0)) << 4));
                    const uint4 qc = *(const uint4 *)(smem + (m0 + 8) * D * 2 + ((ch ^ swz_rows(m0 + 8)) << 4));
                    // (two products of one accumulator never back to back: the second would wait for the first)
#pragma unroll
                    for (int n = 0; n < 4; ++n)
                        if (n * 8 < n_left) mma_bf16(acc[m][n], qa.x, qc.x, qa.y, qc.y, x[n].x, x[n].y);
#pragma unroll
                    for (int n = 0; n < 4; ++n)
                        if (n * 8 < n_left) mma_bf16(acc[m][n], qa.z, qc.z, qa.w, qc.w, x[n].z, x[n].w);
                }
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    if (c + kAhead < kGroups && n * 8 < n_left) x[n] = *(const uint4 *)(row0 + row[n] + 32 * (c + kAhead));
            }
            float best = -CUDART_INF_F;
            const Allowed ok(g, qb, r);
            if (ok.all(MT * 16, (ks + 1) * kKeysPerUnit)) {
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int i = 0; i < 4; ++i) best = fmaxf(best, acc[m][n][i]);
            } else {
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (ok(m * 16 + gr + 8 * (i >> 1), ks * kKeysPerUnit + n * 8 + 2 * t + (i & 1))) best = fmaxf(best, acc[m][n][i]);
            }
            best = warp_max(best);
            if (lane == 0 && best > -CUDART_INF_F) atomicMax(&key[slot], key_of(best));
        }
    }
};

// ----------------------------------------------------------------------------------------------
// The row
// ----------------------------------------------------------------------------------------------
// A level's candidates live in slots: node i's left half in slot 2 i, its right half in 2 i + 1
// (last < first: no such candidate), each with the key of its score (0: not known yet). Slots are
// in block order, so the tie rule (lower block index) is the lower slot, and no compaction is
// needed between scoring and ranking.
struct Slots {
    int *at;  // first [n] | last [n] | key [n]
    int n;
    __device__ int *first() const { return at; }
    __device__ int *last() const { return at + n; }
    __device__ unsigned *key() const { return (unsigned *)at + 2 * n; }
};

// kCluster: a row's tiles are dealt to the CTAs of a cluster (a power of two of them). Each keeps all the slots, scores
// those that are its own, hands their keys to the others, and ranks like them.
template <class P, int W, bool kCluster>
__global__ void __launch_bounds__(W * 32, W == kWideWarps ? 1 : P::kCtas)
mask_rows_kernel(Geom g, MultiK mk, int score_bytes, int n_max, const typename P::Elem *q,
                 const typename P::Elem *k, int32_t *__restrict__ mask, float *__restrict__ score, WorkspaceHeader *ws) {
    extern __shared__ __align__(16) unsigned char smem[];
    int *words = (int *)(smem + score_bytes);  // n_max: slots, a multiple of 32
    int par = 0;                               // the present level's slots: the first or the second set
    int *list = words + 6 * n_max;             // slots still without a score
    unsigned *keep = (unsigned *)words + 7 * n_max;  // a bit per slot
    // several k: scores of this row by key block, NaN = not scored yet (a score does not depend on k)
    float *cache = mk.use_cache ? (float *)(keep + n_max / 32) : nullptr;
    __shared__ int s_list, s_valid, s_all;  // s_all (clusters): listed by any of the CTAs
    after_previous_kernel();
    const unsigned n_cta = kCluster ? cluster_size() : 1u, cta = kCluster ? cluster_rank() : 0u;

    const int tid = threadIdx.x, n_thr = blockDim.x;
    // heaviest rows (late query blocks) first
    const long long row_rev = blockIdx.x / n_cta;
    const int qb = g.n_qb - 1 - (int)(row_rev / ((long long)g.batch * g.H));
    const int bh = (int)(row_rev % ((long long)g.batch * g.H));
    const int b = bh / g.H, h = bh % g.H, kvh = h / g.hpg;
    const long long row = ((long long)b * g.H + h) * g.n_qb + qb;
    const long long rows_total = (long long)g.batch * g.H * g.n_qb;
    const typename P::Elem *kp = k + b * g.ks_b + kvh * g.ks_h;
    const int q_lim = last_valid_block(g, qb);

    P::load_q(g, smem, q + b * g.qs_b + h * g.qs_h, qb);
    if (cache != nullptr)
        for (int r = tid; r < g.N_k; r += n_thr) cache[r] = CUDART_NAN_F;
    unsigned tiles = 0;

    // Candidate (fst, lst) into slot c; known = key of its score or 0 (then it goes on the list,
    // unless `cache` knows it).
    auto put = [&](const Slots &s, int c, bool ok, int fst, int lst, unsigned known, bool want) {
        if (ok && known == 0u && want) {
            if (cache != nullptr && !isnan(cache[fst])) known = key_of(cache[fst]);
            else if (!kCluster || (((unsigned)c >> 1) & (n_cta - 1u)) == cta) list[atomicAdd(&s_list, 1)] = c;
            if (kCluster) atomicAdd(&s_all, 1);
        }
        s.first()[c] = fst;
        s.last()[c] = ok ? lst : fst - 1;
        s.key()[c] = ok ? known : 0u;
        if (ok) atomicAdd(&s_valid, 1);
    };
    // Node i = blocks (fst : lst) into its two slots: (fst : m) keeps the node's score, (m + 1 : lst)
    // needs one if it holds an allowed block.
    auto split = [&](const Slots &s, int i, bool ok, int fst, int lst, unsigned known) {
        const int m = (fst + lst) / 2;
        put(s, 2 * i, ok, fst, m, known, true);
        put(s, 2 * i + 1, ok && m + 1 <= lst && m + 1 <= q_lim, m + 1, lst, 0u, true);
    };
    auto pad = [&](const Slots &s, int n) {  // up to a multiple of 32: absent candidates
        const int c = n + tid;
        if (c < ((n + 31) & ~31)) { s.first()[c] = 0; s.last()[c] = -1; s.key()[c] = 0u; }
    };

    const int n_pass = mk.n > 0 ? mk.n : 1;
    for (int pass = 0; pass < n_pass; ++pass) {
        const int kq = mk.n > 0 ? mk.k[pass] : row_k(g, qb);  // this pass's k (= k_top unless told otherwise)
        const int levels = row_levels(g, kq);
        __syncthreads();  // the previous pass is done with the slots
        if (tid == 0) { s_list = 0; s_valid = 0; s_all = 0; }
        __syncthreads();
        // initial nodes tiling [0, N_k); those without an allowed block are absent. With no level to
        // go through (one key block) they are the result, and need a score only if it is asked for.
        int n_slots = levels > 0 ? 2 * kq : kq;
        par = 0;
        const Slots start = {words, n_max};
        for (int i = tid; i < kq; i += n_thr) {
            const int fst = (int)(((long long)i * g.N_k) / kq), lst = (int)(((long long)(i + 1) * g.N_k) / kq) - 1;
            const bool ok = fst <= lst && fst <= q_lim;
            if (levels > 0) split(start, i, ok, fst, lst, 0u);
            else put(start, i, ok, fst, lst, 0u, score != nullptr);
        }
        pad(start, n_slots);
        __syncthreads();

        for (int level = 0;; ++level) {
            const Slots cur = {words + par * 3 * n_max, n_max}, nxt = {words + (par ^ 1) * 3 * n_max, n_max};
            if (kCluster) cluster_arrive();  // the level's slots are written
            const int n_list = s_list, n_valid = s_valid, n_all = kCluster ? s_all : n_list, n_words = (n_slots + 31) >> 5;
            P::score(g, smem, kp, qb, list, n_list, cur.first(), cur.key());
            if (level < levels) tiles += (unsigned)n_all;
            __syncthreads();  // every key of the level is in place
            if (kCluster) {
                cluster_wait();
                for (int i = tid; i < n_list * (int)n_cta; i += n_thr) {
                    const int slot = list[i / (int)n_cta];
                    const unsigned to = (unsigned)i % n_cta;
                    if (to != cta) store_in_cluster(&cur.key()[slot], to, cur.key()[slot]);
                }
                cluster_arrive();
                cluster_wait();
            }
            if (tid == 0) { s_list = 0; s_valid = 0; s_all = 0; }
            if (cache != nullptr)
                for (int i = tid; i < n_list; i += n_thr) cache[cur.first()[list[i]]] = score_of(cur.key()[list[i]]);
            // Top-k by rank: a candidate is beaten by a higher score, or an equal one in a lower slot.
            // (Absent candidates have key 0 and beat nobody.) A warp's 32 slots are consecutive: the
            // words before its own compare with >=, those behind it with >.
            for (int w = tid >> 5; w < n_words; w += n_thr >> 5) {
                const int c = w * 32 + (tid & 31);
                const unsigned mine = cur.key()[c];
                const bool valid = cur.last()[c] >= cur.first()[c];
                bool kept = valid;
                if (n_valid > kq) {
                    int rank = 0;
                    for (int u = 0; u < n_words; ++u) {
                        const uint4 *x = (const uint4 *)(cur.key() + u * 32);
                        if (u == w) {
#pragma unroll
                            for (int v = 0; v < 32; ++v) {
                                const unsigned y = cur.key()[u * 32 + v];
                                rank += (y > mine) || (y == mine && v < (tid & 31));
                            }
                        } else {
                            const unsigned thr = u < w && mine != 0u ? mine - 1u : mine;
#pragma unroll
                            for (int v = 0; v < 8; ++v) {
                                const uint4 y = x[v];
                                rank += (int)(y.x > thr) + (int)(y.y > thr) + (int)(y.z > thr) + (int)(y.w > thr);
                            }
                        }
                    }
                    kept = valid && rank < kq;
                }
                const unsigned bal = __ballot_sync(0xffffffffu, kept);
                if ((tid & 31) == 0) keep[w] = bal;
            }
            __syncthreads();
            // survivors stay in ascending block order: a kept slot becomes the node of its rank in the bits
            const bool last = level + 1 >= levels;
            int n_kept = 0;
            for (int u = 0; u < n_words; ++u) n_kept += __popc(keep[u]);
            const long long o = (pass * rows_total + row) * g.k_top;
            for (int c = tid; c < n_words * 32; c += n_thr) {
                const int w = c >> 5;
                if (!((keep[w] >> (c & 31)) & 1u)) continue;
                int pos = __popc(keep[w] & ((1u << (c & 31)) - 1u));
                for (int u = 0; u < w; ++u) pos += __popc(keep[u]);
                if (last && cta != 0u) continue;
                if (last) {
                    mask[o + pos] = cur.first()[c];
                    if (score != nullptr) score[o + pos] = score_of(cur.key()[c]);
                } else {
                    split(nxt, pos, true, cur.first()[c], cur.last()[c], cur.key()[c]);
                }
            }
            if (last) {
                for (int j = n_kept + tid; j < g.k_top && cta == 0u; j += n_thr) {
                    mask[o + j] = -1;
                    if (score != nullptr) score[o + j] = -CUDART_INF_F;
                }
                break;
            }
            n_slots = 2 * n_kept;
            pad(nxt, n_slots);
            par ^= 1;
            __syncthreads();
        }
    }
    if (tid == 0 && cta == 0u) {
        atomicAdd(&ws->tiles_scored, (unsigned long long)tiles);
        atomicAdd(&ws->rows, 1ull);
        if (g.row_tiles != nullptr) g.row_tiles[row] = tiles;
    }
}

constexpr size_t kMaxDynamicSmem = 227 * 1024 - 1024;  // (the kernel has a few static words too)

// Shared memory of a row with W warps: what scoring takes, the slots, the list, a bit per slot.
template <class P>
size_t row_bytes(const Geom &g, int warps) {
    const int n_max = (2 * g.k_top + 31) & ~31;
    return P::smem_bytes(g, warps) + (size_t)(7 * n_max + n_max / 32) * 4;
}

template <class P, int W, bool kCluster = false>
stream_status launch_w(const Geom &g, MultiK mk, const void *q, const void *k, int32_t *mask, float *score, WorkspaceHeader *ws,
                       cudaStream_t st, int first_qb, int n_cta = 1) {
    const long long rows = (long long)g.batch * g.H * (g.n_qb - first_qb);
    const int n_max = (2 * g.k_top + 31) & ~31;
    const size_t score_bytes = P::smem_bytes(g, W);
    size_t smem = row_bytes<P>(g, W);
    mk.use_cache = mk.n > 1 && smem + sizeof(float) * (size_t)g.N_k <= kMaxDynamicSmem;
    if (mk.use_cache) smem += sizeof(float) * (size_t)g.N_k;
    auto kern = mask_rows_kernel<P, W, kCluster>;
    cudaError_t e = allow_smem(kern, kMaxDynamicSmem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(mask_rows)");
    e = launch_kernel(kern, (unsigned)(rows * n_cta), W * 32, smem, st, (unsigned)n_cta, g, mk, (int)score_bytes, n_max, (const typename P::Elem *)q,
                      (const typename P::Elem *)k, mask, score, ws);
    if (e != cudaSuccess) return cuda_fail(e, "mask_rows launch");
    return STREAM_OK;
}

template <class P>
stream_status launch(const Geom &g, const MultiK &mk, const void *q, const void *k, int32_t *mask, float *score, WorkspaceHeader *ws,
                     cudaStream_t st) {
    // Rows that keep all blocks they are allowed, with no score asked for, are written by a kernel of their own (they are the last of
    // the launch's order). Not where they are few, or where all rows run at once anyway: a launch more is 2 us (16 heads, T = 2000, fp32,
    // blocks of 32, k = 24: 145 -> 135 us), and the
    // row kernel does not bear a way out of its beginning (fp32, T = 5003: 178 -> 189 us by the compiler's other choices).
    int first_qb = mk.n == 0 && score == nullptr ? whole_query_blocks(g) : 0;
    if (first_qb < g.n_qb && (4 * first_qb < g.n_qb || (long long)g.batch * g.H * (g.n_qb - first_qb) < 4 * sm_count_or_default())) first_qb = 0;
    if (first_qb > 0) {
        const stream_status rc = launch_mask_whole(g, first_qb, mask, ws, st);
        if (rc != STREAM_OK || first_qb == g.n_qb) return rc;
    }
    const long long rows = (long long)g.batch * g.H * (g.n_qb - first_qb);
    // Sixteen warps when every row has an SM to itself anyway: a level's tiles then spread over more
    // warps (64 rows, fp32, d = 64, blocks of 32, k = 8: 34.9 us with eight, 32.9 with sixteen, before the
    // divisions went; 28.9 now). With up to two rows an SM, too, if the first level has a tile part for
    // each of them (fp32: 208 rows, blocks of 64, k = 8: four warps 92.8 us, sixteen 59.7; 181 rows, blocks
    // of 16, k = 15, d = 128: 118 and 78; 282 rows with 12 parts each: 26.6 and 30.8). With three rows an SM
    // four warps are the better (343 rows, blocks of 16, k = 8: 42.9 us, sixteen 63.5).
    const int parts = 2 * g.k_top * ((g.bq + 31) / 32) * ((g.bk + kKeysPerUnit - 1) / kKeysPerUnit);
    // Fewer rows than half of the SMs: a row over two, four or eight of them, while each has a tile part for
    // every scheduler (fp32, 28 rows, blocks of 64, k = 11: 65.2 -> 31.3 us; 55 rows, blocks of 32, d = 128, k = 9:
    // 55.3 -> 43.7; the 64 rows above: 28.7 -> 24.6).
    int n_cta = 1;
    while (n_cta < 8 && rows * 2 * n_cta <= sm_count_or_default() && parts >= 8 * n_cta) n_cta *= 2;
    // (d = 256 in fp32, blocks above 32 and k above 624: sixteen warps do not fit, four do)
    const bool fits = row_bytes<P>(g, kWideWarps) <= kMaxDynamicSmem;
    if (fits && n_cta > 1 && mk.n <= 1) return launch_w<P, kWideWarps, true>(g, mk, q, k, mask, score, ws, st, first_qb, n_cta);
    if (fits && rows <= (parts >= kWideWarps ? 2 : 1) * (long long)sm_count_or_default()) return launch_w<P, kWideWarps>(g, mk, q, k, mask, score, ws, st, first_qb);
    return launch_w<P, P::kWarps>(g, mk, q, k, mask, score, ws, st, first_qb);
}

template <typename T, int RQ, Load kLoad>
stream_status fma_d(const Geom &g, const MultiK &mk, const void *q, const void *k, int32_t *mask, float *score,
                    WorkspaceHeader *ws, cudaStream_t st) {
    switch (g.d) {
        case 16: return launch<FmaScore<T, 16, RQ, kLoad>>(g, mk, q, k, mask, score, ws, st);
        case 32: return launch<FmaScore<T, 32, RQ, kLoad>>(g, mk, q, k, mask, score, ws, st);
        case 64: return launch<FmaScore<T, 64, RQ, kLoad>>(g, mk, q, k, mask, score, ws, st);
        case 128: return launch<FmaScore<T, 128, RQ, kLoad>>(g, mk, q, k, mask, score, ws, st);
        case 256: return launch<FmaScore<T, 256, RQ, kLoad>>(g, mk, q, k, mask, score, ws, st);
    }
    set_error("generic mask kernel: head dim %d not in {16, 32, 64, 128, 256}", g.d);
    return STREAM_ERR_UNSUPPORTED;
}

template <typename T, Load kLoad>
stream_status fma_rq(const Geom &g, const MultiK &mk, const void *q, const void *k, int32_t *mask, float *score,
                     WorkspaceHeader *ws, cudaStream_t st) {
    if (g.bq <= 16) return fma_d<T, 2, kLoad>(g, mk, q, k, mask, score, ws, st);  // 16 queries per warp instead of 32
    return fma_d<T, 4, kLoad>(g, mk, q, k, mask, score, ws, st);
}

template <int MT>
stream_status mma_d(const Geom &g, const MultiK &mk, const void *q, const void *k, int32_t *mask, float *score,
                    WorkspaceHeader *ws, cudaStream_t st) {
    switch (g.d) {
        case 64: return launch<MmaScore<64, MT>>(g, mk, q, k, mask, score, ws, st);
        case 128: return launch<MmaScore<128, MT>>(g, mk, q, k, mask, score, ws, st);
        default: return launch<MmaScore<256, MT>>(g, mk, q, k, mask, score, ws, st);
    }
}

// ----------------------------------------------------------------------------------------------
// Builds that drop nothing
// ----------------------------------------------------------------------------------------------
// No row has more allowed blocks than it may keep: every row is its allowed blocks, and no key is read. Bound by the launch (32
// heads, 1000 tokens in blocks of 64, k = 16: 24.0 us with all scores computed, 13.1 a call in a loop, the host's part).
constexpr int kWholeThreads = 256;
__global__ void __launch_bounds__(kWholeThreads) mask_whole_kernel(Geom g, int n_qb, int32_t *mask, WorkspaceHeader *ws) {
    after_previous_kernel();
    write_whole_rows(g, n_qb, (int)(blockIdx.x * kWholeThreads + threadIdx.x) / 32, (int)gridDim.x * (kWholeThreads / 32), (int)threadIdx.x & 31, mask, ws);
}

}  // namespace

stream_status launch_mask_whole(const Geom &g, int n_qb, int32_t *mask, WorkspaceHeader *ws, cudaStream_t st) {
    const long long blocks = (whole_pieces(g, n_qb) + kWholeThreads / 32 - 1) / (kWholeThreads / 32), most = 8 * sm_count_or_default();
    const cudaError_t e = launch_kernel(mask_whole_kernel, (unsigned)(blocks < most ? blocks : most), kWholeThreads, 0, st, 1, g, n_qb, mask, ws);
    return e == cudaSuccess ? STREAM_OK : cuda_fail(e, "mask_whole launch");
}

stream_status launch_mask_generic_multi(const Geom &g, const MultiK &mk, int dtype, bool allow_mma, const void *q, const void *k,
                                        int32_t *mask, float *score, WorkspaceHeader *ws, cudaStream_t st) {
    if (g.bq > kMaxBlock || g.bk > kMaxBlock) {
        set_error("generic mask kernel: block sizes up to %d (got %d, %d)", kMaxBlock, g.bq, g.bk);
        return STREAM_ERR_UNSUPPORTED;
    }
    const int e = dtype == STREAM_F32 ? 4 : 2;
    const bool k_aligned = rows_16_byte_aligned(k, g.ks_t, g.ks_h, g.ks_b, e);
    if (dtype == STREAM_F32) {
        if (k_aligned) return fma_rq<float, Load::kCopy16>(g, mk, q, k, mask, score, ws, st);
        return fma_rq<float, Load::kCopy4>(g, mk, q, k, mask, score, ws, st);
    }
    // d = 16 and 32 would leave most of an mma's channels or lanes unused: they stay on the FMA form
    if (allow_mma && (g.d == 64 || g.d == 128 || g.d == 256) && k_aligned && g.ks_t < (1 << 24) &&
        rows_16_byte_aligned(q, g.qs_t, g.qs_h, g.qs_b, 2)) {
        if (g.bq <= 16) return mma_d<1>(g, mk, q, k, mask, score, ws, st);
        if (g.bq <= 32) return mma_d<2>(g, mk, q, k, mask, score, ws, st);
        return mma_d<4>(g, mk, q, k, mask, score, ws, st);
    }
    if (rows_aligned(k, g.ks_t, g.ks_h, g.ks_b, 2, 8)) return fma_rq<__nv_bfloat16, Load::kWide>(g, mk, q, k, mask, score, ws, st);
    return fma_rq<__nv_bfloat16, Load::kScalars>(g, mk, q, k, mask, score, ws, st);
}

stream_status launch_mask_generic(const Geom &g, int dtype, bool allow_mma, const void *q, const void *k, int32_t *mask,
                                  float *score, WorkspaceHeader *ws, cudaStream_t st) {
    MultiK single = {};
    return launch_mask_generic_multi(g, single, dtype, allow_mma, q, k, mask, score, ws, st);
}

}  // namespace stream
