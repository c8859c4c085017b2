// Block-sparse attention (Eq. 2 on a Stream mask) in fp32 FMA: every dtype, head dimension, block
// size and alignment the ABI accepts (fp32 above all).
//
// One CTA per (batch, head, query block). A warp owns QW query tokens (32, or 16 where the output
// accumulators would not fit) against 32 keys at a time; ceil(block_q / QW) warps make a group that
// walks a sequence of key tiles, and the groups of a CTA take the row's tiles in turn, each with
// softmax statistics and accumulators of its own, added up at the end. One K and one V buffer
// per group, filled by cp.async (bf16, and rows off 16 bytes: through registers): the next K tile arrives behind softmax and P V, the next V tile
// behind the next Q K^T (with three CTAs an SM at d = 64 both are asked for behind P V, and nothing covers them but the
// other CTAs). Inner loops read shared memory 16 bytes at a time, conflict-free:
//   Q K^T   lane (kq, kk): queries kq + 8 i x keys kk + 4 j; QW / 8 + 8 loads per 4 QW FMA
//   P V     lane (ro, co): QW / 4 consecutive queries x channels 4 co + 32 i, P kept key-major
// Bound: latency. 8 to 12 warps an SM wait for their tiles, for each other and for the merge of a row's four parts after two tiles
// each (8 heads, T = 5003, blocks of 32, d = 64, k = 8: 108 us, 24 TFLOP/s; a bare FMA loop reaches 66 of 74.5). The kernel this one replaced padded every tile to 64 x 64 and loaded
// scalars: 8 heads, T = 5003, blocks of 32, d = 64, k = 8: 599 -> 150 us, and 108 since; one head, T = 2048: 82 -> 18 us.
#include "warp_common.cuh"

namespace stream {
namespace {

using namespace wp;

constexpr int kMaxBlock = 64;
constexpr int kKeys = 32;  // keys of a tile
constexpr size_t kMaxDynamicSmem = 220 * 1024;
constexpr size_t kSmemPerSm = 228 * 1024, kSmemPerCtaReserved = 1024 + 128;  // (128: the kernel's static words)

template <typename T>
__device__ __forceinline__ void store4(T *dst, float4 x);
template <>
__device__ __forceinline__ void store4<float>(float *dst, float4 x) {
    dst[0] = x.x; dst[1] = x.y; dst[2] = x.z; dst[3] = x.w;
}
template <>
__device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16 *dst, float4 x) {
    dst[0] = __float2bfloat16_rn(x.x); dst[1] = __float2bfloat16_rn(x.y);
    dst[2] = __float2bfloat16_rn(x.z); dst[3] = __float2bfloat16_rn(x.w);
}

template <int D, int QW>
struct Shape {
    static constexpr int kTileBytes = kKeys * D * 4, kPPitch = QW + 8, kPBytes = kKeys * kPPitch * 4;
    static constexpr int kSwz = (D / 4 - 1) & 7;  // 16-byte columns are permuted within a row by row & kSwz
    static constexpr int kRowPitch = D + 4;                // (eight lanes, eight different 16-byte columns)
    static constexpr int kPart = QW * kRowPitch + 2 * QW;  // floats a warp leaves behind for the final sum
};

// A [32][D] fp32 tile: keys n0 .. n0 + 31 of block r.
template <typename T, int D, Load kLoad, bool kIsK>
__device__ __forceinline__ void fetch(const Geom &g, unsigned char *dst, const T *base, int r, int n0, int thr, int n_thr) {
    constexpr int per_row = D / 4, n_copies = kKeys * per_row;
    if constexpr (kLoad == Load::kWide) {  // eight loads of a thread on their way at a time, not one value after the other
        const long long tk0 = (long long)r * g.bk + n0;
        const int n_in = (int)max(0ll, min((long long)min(g.bk - n0, kKeys), g.T - tk0));  // keys of the tile; the rest become zeros
        constexpr int most = n_copies / 32 < 8 ? n_copies / 32 : 8;
        for (int first = thr; first < n_copies; first += most * n_thr) {
            uint2 x[most];
#pragma unroll
            for (int i = 0; i < most; ++i) {
                const int idx = first + i * n_thr, n = idx / per_row, c = idx % per_row;
                x[i] = n < n_in ? *(const uint2 *)(base + (tk0 + n) * g.ks_t + c * 4) : make_uint2(0, 0);
            }
#pragma unroll
            for (int i = 0; i < most; ++i) {
                const int idx = first + i * n_thr, n = idx / per_row, c = idx % per_row;
                if (idx < n_copies) *(float4 *)(dst + n * D * 4 + ((kIsK ? c ^ (n & Shape<D, 32>::kSwz) : c) << 4)) = widen4(x[i]);
            }
        }
        return;
    }
    for (int idx = thr; idx < n_copies; idx += n_thr) {
        const int n = idx / per_row, c = idx % per_row;
        const long long tk = (long long)r * g.bk + n0 + n;
        const bool in = n0 + n < g.bk && tk < g.T;  // the rest become zeros
        unsigned char *to = dst + n * D * 4 + ((kIsK ? c ^ (n & Shape<D, 32>::kSwz) : c) << 4);
        const T *src = base + (in ? tk : 0) * g.ks_t + c * 4;
        if (kLoad == Load::kCopy16) {
            cp_async16(smem_addr(to), src, in ? 16 : 0);
        } else {
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (in) x = make_float4(to_float(src[0]), to_float(src[1]), to_float(src[2]), to_float(src[3]));
            *(float4 *)to = x;
        }
    }
    if (kLoad == Load::kCopy16) cp_async_commit();
}

// The builds of the kernel. kRow: a row by a CTA. kCluster: its tiles are dealt to the groups of all CTAs of a cluster, which
// read each other's parts at the end. kThree, kFour: as kRow, with three or four CTAs of four warps an SM where the registers of
// kRow let an SM hold two. kThree at d = 64 (one warp a group): P lies over the group's K tile, for the room of the third, and both
// next tiles are fetched behind P V: what a warp then waits for its tiles the other two CTAs' warps cover.
enum class Build { kRow, kCluster, kThree, kFour };

// Threads of a CTA at most, and the CTAs an SM whose registers a thread is held to (0: unbounded). Unbounded, ptxas takes 200 to 250
// at d = 32 and 64. Held to three CTAs d = 32 spills nothing and d = 64 20 to 90 bytes; to four, d = 32 spills 70 to
// 150. At d = 128 and 256 a bound of one CTA lets it take more than it would (8 heads, 5000 tokens, d = 128, blocks of
// 32: 294 -> 274 us; blocks of 16, k = 16: 482 -> 427), but at d = 256 a cluster's kernel then spills (2 heads, 600
// tokens: 57.4 -> 59.4).
template <int D, int QW, Build kBuild>
struct Bounds {
    static constexpr bool kTight = kBuild == Build::kThree || kBuild == Build::kFour;
    static constexpr int kThreads = kTight ? 128 : 256;
    static constexpr int kCtas = kTight ? (kBuild == Build::kThree ? 3 : 4) : (D == 128 || (D == 256 && kBuild == Build::kRow) ? 1 : 0);
};

template <typename T, int D, int QW, Load kLoad, Build kBuild>
__global__ void __launch_bounds__(Bounds<D, QW, kBuild>::kThreads, Bounds<D, QW, kBuild>::kCtas)
attn_generic_kernel(Geom g, int m_warps, int splits, const T *q, const T *k, const T *v, const int32_t *mask, float scale, T *__restrict__ out) {
    constexpr bool kCluster = kBuild == Build::kCluster, kPInK = kBuild == Build::kThree && D == 64;
    using Sh = Shape<D, QW>;
    constexpr bool kAsync = kLoad == Load::kCopy16;
    constexpr int RQ = QW / 8, RO = QW / 4, CO = D < 32 ? 1 : D / 32;
    // (d = 128, us, at 2 and 4: 278.5 against 272.9 for 8 heads, 5000 tokens, blocks of 32; the other dimensions have no registers for it)
    constexpr int kUnrollQK = D == 128 ? 4 : 2, kUnrollPV = D == 128 ? 8 : 4;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_n;
    after_previous_kernel();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = warp / m_warps, mw = warp % m_warps, g_thr = m_warps * 32, g_tid = tid - grp * g_thr;
    const int kq = lane >> 2, kk = lane & 3;   // Q K^T
    const int ro = lane >> 3, co = lane & 7;   // P V
    // late (longer) rows first
    const unsigned n_cta = kCluster ? cluster_size() : 1u, cta = kCluster ? cluster_rank() : 0u, row = blockIdx.x / n_cta;
    const int bh = (int)(row / (unsigned)g.n_qb), qb = g.n_qb - 1 - (int)(row % (unsigned)g.n_qb);
    const int turn = (int)cta * splits + grp, groups = (int)n_cta * splits;  // this group's turn among all of the row's
    const int b = bh / g.H, h = bh % g.H, kvh = h / g.hpg;
    const T *qp = q + b * g.qs_b + h * g.qs_h;
    const T *kp = k + b * g.ks_b + kvh * g.ks_h, *vp = v + b * g.ks_b + kvh * g.ks_h;
    const int32_t *mrow = mask + ((long long)bh * g.n_qb + qb) * g.k_top;

    // Q | per group K, V | per warp P | per warp row factors | kept blocks
    float *Qs = (float *)smem;
    unsigned char *ks = smem + (size_t)m_warps * QW * D * 4 + (size_t)grp * 2 * Sh::kTileBytes, *vs = ks + Sh::kTileBytes;
    unsigned char *pw = smem + (size_t)m_warps * QW * D * 4 + (size_t)splits * 2 * Sh::kTileBytes;
    float *Ps = (float *)(kPInK ? ks + (size_t)mw * Sh::kPBytes : pw + (size_t)warp * Sh::kPBytes);
    if (!kPInK) pw += (size_t)m_warps * splits * Sh::kPBytes;
    float *factor = (float *)pw + warp * QW;
    int *list = (int *)((float *)pw + m_warps * splits * QW);

    for (int idx = tid; idx < m_warps * QW * D; idx += blockDim.x) {
        const int m = idx / D, c = idx % D;
        const long long tq = (long long)qb * g.bq + m;
        const float x = (m < g.bq && tq < g.T) ? to_float(qp[tq * g.qs_t + c]) : 0.f;
        Qs[m * D + ((((c >> 2) ^ (m & Sh::kSwz)) << 2) | (c & 3))] = x;
    }
    if (warp == 0) {  // the row's kept blocks, in order
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

    float o[RO][CO * 4];
#pragma unroll
    for (int i = 0; i < RO; ++i)
#pragma unroll
        for (int j = 0; j < CO * 4; ++j) o[i][j] = 0.f;
    float m_run[RQ], l_run[RQ];
#pragma unroll
    for (int i = 0; i < RQ; ++i) { m_run[i] = -CUDART_INF_F; l_run[i] = 0.f; }
    const float *qw = Qs + (size_t)mw * QW * D;

    const int n_sub = (g.bk + kKeys - 1) / kKeys, n_tiles = s_n * n_sub;
    if (turn < n_tiles) {
        fetch<T, D, kLoad, true>(g, ks, kp, list[turn / n_sub], turn % n_sub * kKeys, g_tid, g_thr);
        fetch<T, D, kLoad, false>(g, vs, vp, list[turn / n_sub], turn % n_sub * kKeys, g_tid, g_thr);
    }
    for (int i0 = turn; i0 < n_tiles; i0 += groups) {
        const int r = list[i0 / n_sub], n0 = i0 % n_sub * kKeys, nxt = i0 + groups;
        const long long k0 = (long long)r * g.bk + n0;
        const int n_keys = (int)max(0ll, min((long long)min(g.bk - n0, kKeys), g.T - k0));
        if (kAsync) cp_async_wait<1>();
        group_sync(1 + grp, g_thr);  // the K tile is there
        float s[RQ][8];
#pragma unroll
        for (int i = 0; i < RQ; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) s[i][j] = 0.f;
#pragma unroll kUnrollQK
        for (int c4 = 0; c4 < D / 4; ++c4) {
            float4 a[RQ], x[8];
#pragma unroll
            for (int i = 0; i < RQ; ++i) a[i] = *(const float4 *)(qw + (kq + 8 * i) * D + ((c4 ^ (kq & Sh::kSwz)) << 2));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int n = kk + 4 * j;
                x[j] = *(const float4 *)(ks + n * D * 4 + ((c4 ^ (n & Sh::kSwz)) << 4));
            }
            fma_channel<RQ>(s, a, x, &float4::x);
            fma_channel<RQ>(s, a, x, &float4::y);
            fma_channel<RQ>(s, a, x, &float4::z);
            fma_channel<RQ>(s, a, x, &float4::w);
        }
        group_sync(1 + grp, g_thr);  // everybody is done with the K tile
        if (!kPInK) {
            if (nxt < n_tiles) fetch<T, D, kLoad, true>(g, ks, kp, list[nxt / n_sub], nxt % n_sub * kKeys, g_tid, g_thr);
            else if (kAsync) cp_async_commit();
        }
        // online softmax; the four lanes of a query share its keys
        bool moved = false;
#pragma unroll
        for (int i = 0; i < RQ; ++i) {
            const int m = mw * QW + kq + 8 * i;
            const long long tq = (long long)qb * g.bq + m;
            int lim = m < g.bq && tq < g.T ? n_keys : 0;
            if (g.causal) lim = (int)max(0ll, min((long long)lim, tq - k0 + 1));
            float mx = m_run[i];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                s[i][j] = kk + 4 * j < lim ? scale * s[i][j] : -CUDART_INF_F;
                mx = fmaxf(mx, s[i][j]);
            }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float ref = mx == -CUDART_INF_F ? 0.f : mx;
            const float alpha = m_run[i] == -CUDART_INF_F ? 0.f : expf(m_run[i] - ref);
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float p = s[i][j] == -CUDART_INF_F ? 0.f : expf(s[i][j] - ref);
                sum += p;
                Ps[(kk + 4 * j) * Sh::kPPitch + kq + 8 * i] = p;
            }
            l_run[i] = l_run[i] * alpha + sum;  // (each lane its own keys' part; they meet at the end)
            m_run[i] = mx;
            if (kk == 0) factor[kq + 8 * i] = alpha;
            moved |= alpha != 1.f;
        }
        moved = __any_sync(0xffffffffu, moved);
        if (kAsync && kPInK) cp_async_wait<0>();
        else if (kAsync) cp_async_wait<1>();
        group_sync(1 + grp, g_thr);  // the V tile and this warp's P are there
        if (moved) {
#pragma unroll
            for (int i = 0; i < RO; ++i) {
                const float f = factor[ro * RO + i];
#pragma unroll
                for (int j = 0; j < CO * 4; ++j) o[i][j] *= f;
            }
        }
        if (D >= 32 || co * 4 < D) {
#pragma unroll kUnrollPV
            for (int n = 0; n < n_keys; ++n) {
                float p[RO];
#pragma unroll
                for (int i = 0; i < RO; i += 4) *(float4 *)(p + i) = *(const float4 *)(Ps + n * Sh::kPPitch + ro * RO + i);
#pragma unroll
                for (int j = 0; j < CO; ++j) {
                    const float4 x = *(const float4 *)(vs + n * D * 4 + (co + 8 * j) * 16);
#pragma unroll
                    for (int i = 0; i < RO; ++i) {
                        o[i][4 * j] = fmaf(p[i], x.x, o[i][4 * j]);
                        o[i][4 * j + 1] = fmaf(p[i], x.y, o[i][4 * j + 1]);
                        o[i][4 * j + 2] = fmaf(p[i], x.z, o[i][4 * j + 2]);
                        o[i][4 * j + 3] = fmaf(p[i], x.w, o[i][4 * j + 3]);
                    }
                }
            }
        }
        group_sync(1 + grp, g_thr);  // done with the V tile and with P
        if (kPInK && nxt < n_tiles) fetch<T, D, kLoad, true>(g, ks, kp, list[nxt / n_sub], nxt % n_sub * kKeys, g_tid, g_thr);
        if (nxt < n_tiles) fetch<T, D, kLoad, false>(g, vs, vp, list[nxt / n_sub], nxt % n_sub * kKeys, g_tid, g_thr);
    }
    if (kAsync) cp_async_wait<0>();

    // Sum over the groups through shared memory (all tiles are done with): every warp leaves its rows'
    // maxima and sums and its accumulators, row by row; the weights of the groups are taken once per
    // row; then all threads add up and store four channels of a row at a time. (One warp per row
    // group doing it alone took a third of a small call: 25.3 -> 18.5 us for 64 rows of 8 blocks.)
    __syncthreads();
    float *part = (float *)smem + (size_t)warp * Sh::kPart;
#pragma unroll
    for (int i = 0; i < RQ; ++i) {
        float l = l_run[i];
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if (kk == 0) { part[kq + 8 * i] = m_run[i]; part[QW + kq + 8 * i] = l; }
    }
    if (D >= 32 || co * 4 < D) {
#pragma unroll
        for (int i = 0; i < RO; ++i)
#pragma unroll
            for (int j = 0; j < CO; ++j)
                *(float4 *)(part + 2 * QW + (ro * RO + i) * Sh::kRowPitch + 4 * co + 32 * j) =
                    make_float4(o[i][4 * j], o[i][4 * j + 1], o[i][4 * j + 2], o[i][4 * j + 3]);
    }
    if constexpr (kCluster) {
        cluster_arrive();
        cluster_wait();
        const size_t step = (size_t)m_warps * Sh::kPart;  // to the same row of the CTA's next group
        float *const weight = (float *)smem + (size_t)splits * step;  // [row][group]
        for (int m = tid; m < m_warps * QW; m += blockDim.x) {
            const float *first = (const float *)smem + (size_t)(m / QW) * Sh::kPart + m % QW;
            float *const w = weight + m * groups;
            float top = -CUDART_INF_F, total = 0.f;
            for (int s = 0; s < groups; ++s) {
                w[s] = load_in_cluster(first + s % splits * step, (unsigned)(s / splits));
                top = fmaxf(top, w[s]);
            }
            const float ref = top == -CUDART_INF_F ? 0.f : top;
            for (int s = 0; s < groups; ++s) {
                w[s] = w[s] == -CUDART_INF_F ? 0.f : expf(w[s] - ref);
                total += w[s] * load_in_cluster(first + s % splits * step + QW, (unsigned)(s / splits));
            }
            const float inv = total > 0.f ? 1.f / total : 0.f;
            for (int s = 0; s < groups; ++s) w[s] *= inv;
        }
        __syncthreads();
        for (int idx = tid + (int)cta * (int)blockDim.x; idx < m_warps * QW * (D / 4); idx += (int)(n_cta * blockDim.x)) {
            const int m = idx / (D / 4), c = idx % (D / 4) * 4;
            const long long tq = (long long)qb * g.bq + m;
            if (m >= g.bq || tq >= g.T) continue;
            const float *first = (const float *)smem + (size_t)(m / QW) * Sh::kPart + 2 * QW + (m % QW) * Sh::kRowPitch + c;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int s = 0; s < groups; ++s) {
                const float f = weight[m * groups + s];
                const float4 y = load4_in_cluster(first + s % splits * step, (unsigned)(s / splits));
                x.x = fmaf(f, y.x, x.x); x.y = fmaf(f, y.y, x.y); x.z = fmaf(f, y.z, x.z); x.w = fmaf(f, y.w, x.w);
            }
            store4(out + ((long long)bh * g.T + tq) * D + c, x);
        }
        cluster_arrive();  // (nobody leaves while its part may still be read)
        cluster_wait();
        return;
    }
    __syncthreads();
    for (int m = tid; m < m_warps * QW; m += blockDim.x) {
        float *first = (float *)smem + (size_t)(m / QW) * Sh::kPart + m % QW;
        const size_t step = (size_t)m_warps * Sh::kPart;  // to the same row of the next group
        float top = -CUDART_INF_F, total = 0.f;
        for (int s = 0; s < splits; ++s) top = fmaxf(top, first[s * step]);
        const float ref = top == -CUDART_INF_F ? 0.f : top;
        for (int s = 0; s < splits; ++s) {
            const float f = first[s * step] == -CUDART_INF_F ? 0.f : expf(first[s * step] - ref);
            total += f * first[s * step + QW];
            first[s * step] = f;
        }
        const float inv = total > 0.f ? 1.f / total : 0.f;
        for (int s = 0; s < splits; ++s) first[s * step] *= inv;
    }
    __syncthreads();
    for (int idx = tid; idx < m_warps * QW * (D / 4); idx += blockDim.x) {
        const int m = idx / (D / 4), c = idx % (D / 4) * 4;
        const long long tq = (long long)qb * g.bq + m;
        if (m >= g.bq || tq >= g.T) continue;
        const float *first = (float *)smem + (size_t)(m / QW) * Sh::kPart;
        const size_t step = (size_t)m_warps * Sh::kPart;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < splits; ++s) {
            const float f = first[s * step + m % QW];
            const float4 y = *(const float4 *)(first + s * step + 2 * QW + (m % QW) * Sh::kRowPitch + c);
            x.x = fmaf(f, y.x, x.x); x.y = fmaf(f, y.y, x.y); x.z = fmaf(f, y.z, x.z); x.w = fmaf(f, y.w, x.w);
        }
        store4(out + ((long long)bh * g.T + tq) * D + c, x);
    }
}

template <typename T, int D, int QW, Load kLoad>
stream_status launch_qw(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale, void *out,
                     cudaStream_t st) {
    using Sh = Shape<D, QW>;
    const int m_warps = (g.bq + QW - 1) / QW;
    const long long rows = (long long)g.batch * g.H * g.n_qb;
    // Four warps a CTA, so that several CTAs share an SM; eight when every row has an SM to itself
    // anyway. Fewer rows than half of the SMs: a row over two, four or eight CTAs, while each has a tile part for
    // every scheduler (28 rows, blocks of 64, k = 11, d = 64: 65.4 -> 34.8 us; 55 rows, blocks of 32, k = 9, d = 128:
    // 38.9 -> 30.7). Not where a row has little to share out, eight tiles of 32 queries and 64 channels or fewer: a CTA alone begins while
    // the kernel before it still runs, as no cluster does (us with the mask build in a graph, cluster and alone: blocks of 32, k = 8: d = 64,
    // 24 rows 32.9, 32.9, 72 rows 41.0, 40.5, d = 32 26.7, 25.5 and 32.8, 30.8, d = 16, 10 rows, 20.5, 18.6; blocks of 16, d = 16, k = 8, 24 rows
    // 21.6, 18.5, but d = 32, 56 rows 27.4, 28.7; blocks of 64, whose rows are two warps' work a tile: k = 2, d = 32, 40 rows 36.9, 34.9, k = 3,
    // d = 64, 24 rows 43.9, 47.2, k = 4 41.1, 50.4, 72 rows 59.5, 65.6, d = 16 36.9, 39.0; more tiles: 64 rows of blocks of 32, d = 64,
    // k = 10, 50.5, 51.3; 72 rows, d = 128, k = 8, 65.5, 69.7).
    // T may have fewer blocks than k_top, and what counts are those that are there: a CTA of a cluster has two tile
    // parts at least, a group half of one (16 rows, T = 29, blocks of 48, k = 9, d = 16: 32 -> 10 us). With up to 64 channels they also decide on
    // the next CTAs, unless each would have just one (us with the mask build, by k_top and by those there: k = 16 and 24, d = 64, three blocks of 64, 12 heads:
    // 43.9, 24.6, six, 3 heads: 59.6, 26.7, four, one head: 23.5 with eight CTAs, 26.7 with four; d = 16, ten blocks of 32: 22.5, 20.5; d = 128
    // gains as often as it loses: four blocks of 32 20.5, 24.6, three 23.4, 20.5); with many
    // rows an idle group takes another CTA's shared memory (2500 rows, k = 1, d = 128, rows off 16 bytes: 397 -> 223).
    const int n_sm = sm_count_or_default(), n_sub = (g.bk + kKeys - 1) / kKeys, tiles = g.k_top * n_sub;
    const int there = (int)std::min((long long)g.k_top, (g.T + g.bk - 1) / g.bk) * n_sub;
    int splits = (rows <= n_sm ? 8 : 4) / m_warps, n_cta = 1;
    const bool small = D <= 64 && there * m_warps <= 8;
    auto worth = [&](int n) { return D > 64 ? tiles * m_warps >= 8 * n : there * m_warps >= 8 * n || (there < tiles && there == 2 * n); };
    while (!small && n_cta < 8 && rows * 2 * n_cta <= n_sm && worth(n_cta) && there >= 3 && there >= 2 * n_cta) n_cta *= 2;
    if (n_cta > 1) splits = std::min({splits, (tiles + n_cta - 1) / n_cta, 2 * ((there + n_cta - 1) / n_cta)});
    else if (rows > n_sm) splits = std::min(splits, rows > 4ll * n_sm ? there : 2 * there);
    auto bytes = [&](int s, bool p_in_k) {
        const size_t walk = (size_t)m_warps * QW * D * 4 + (size_t)s * 2 * Sh::kTileBytes + (size_t)m_warps * s * ((p_in_k ? 0 : Sh::kPBytes) + QW * 4) + (size_t)g.k_top * 4;
        const size_t sum = (size_t)m_warps * s * Sh::kPart * 4 + (n_cta > 1 ? (size_t)m_warps * QW * s * n_cta * 4 : 0);
        return walk > sum ? walk : sum;
    };
    while (splits > 1 && bytes(splits, false) > kMaxDynamicSmem) splits /= 2;
    // More than two CTAs an SM: a round of rows then takes 1.4 times as long, so it is a matter of rounds (us at two, at
    // three; 8 heads, blocks of 32, k = 8). d = 64: 376 rows 49.7, 38.3; 480 to 600 are two rounds either way, 480 52.3, 61.6; 592
    // 53.1, 66.8; 640 74.1, 68.2; 1256 123.6, 108.1. d = 32: 160 rows 17.9, 22.7; 400 34.1, 23.9; 592 34.9, 42.0;
    // 752 50.6, 43.6; 3000 177.6, 149.4; bf16 and rows off 16 bytes alike. Four only for groups of two warps at d = 32 (blocks of
    // 64; two, three, four): 480 rows 113, 104, 100; 720 168, 146, 157; 1000 223, 202, 183. Where the rows have work
    // for two warps only (k = 1 and 2), smaller CTAs fill the SM by themselves (2400 rows, k = 2, d = 64: 81.8, 85.9).
    // A causal head's first rows have fewer than k blocks and come last, so that a round may be some rows over: a sixth of
    // those for a round of two, half for one of three or four (d = 64, causal: 304 rows, k = 4, 29.0, 22.0; 320, k = 16, 61.5, 68.8;
    // 344 69.9, 69.1; 480, k = 16, 93.7, 83.2, k = 4, 31.1, 35.5; not causal: 304 rows, k = 8, 44.4, 37.7). Over 795 calls timed both
    // ways this is 0.4 % off the better of the two, 27 % at worst; a third of them for all rounds 0.7 and 50 %.
    const int warps = m_warps * splits;
    const long long first = g.causal ? (long long)g.batch * g.H * std::min((long long)g.n_qb, (long long)g.k_top * g.bk / g.bq) : 0;
    const long long in_twos = rows - first / 6, in_more = rows - first / 2;
    Build build = n_cta > 1 ? Build::kCluster : Build::kRow;
    if ((D == 64 || (D == 32 && QW == 32)) && n_cta == 1 && (warps == 3 || warps == 4) && in_twos > 2ll * n_sm) {
        auto fit = [&](size_t ctas) { return ctas * (bytes(splits, D == 64) + kSmemPerCtaReserved) <= kSmemPerSm; };
        const bool three = (D == 32 || m_warps * Sh::kPBytes <= Sh::kTileBytes) && fit(3), four = D == 32 && m_warps == 2 && fit(4);
        if (four && ((in_more > 3ll * n_sm && in_more <= 4ll * n_sm) || in_more > 6ll * n_sm)) build = Build::kFour;
        else if (three && (four || in_more <= 3ll * n_sm || in_twos > 4ll * n_sm)) build = Build::kThree;
    }
    const size_t smem = bytes(splits, D == 64 && build == Build::kThree);
    auto kern = build == Build::kCluster ? attn_generic_kernel<T, D, QW, kLoad, Build::kCluster> : attn_generic_kernel<T, D, QW, kLoad, Build::kRow>;
    if constexpr (D == 64 || (D == 32 && QW == 32)) {
        if (build == Build::kThree) kern = attn_generic_kernel<T, D, QW, kLoad, Build::kThree>;
    }
    if constexpr (D == 32 && QW == 32) {
        if (build == Build::kFour) kern = attn_generic_kernel<T, D, QW, kLoad, Build::kFour>;
    }
    cudaError_t e = allow_smem(kern, kMaxDynamicSmem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(attn_generic)");
    e = launch_kernel(kern, (unsigned)(rows * n_cta), (unsigned)(m_warps * splits * 32), smem, st, (unsigned)n_cta, g, m_warps, splits, (const T *)q,
                      (const T *)k, (const T *)v, mask, scale, (T *)out);
    if (e != cudaSuccess) return cuda_fail(e, "attn_generic launch");
    return STREAM_OK;
}

template <typename T, int D, Load kLoad>
stream_status launch(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale, void *out,
                     cudaStream_t st) {
    // 32 tokens a warp are 64 accumulators a lane at d = 64; not where half of them would be padding
    if constexpr (D <= 64) {
        if (g.bq > 16) return launch_qw<T, D, 32, kLoad>(g, q, k, v, mask, scale, out, st);
    }
    return launch_qw<T, D, 16, kLoad>(g, q, k, v, mask, scale, out, st);
}

template <typename T, Load kLoad>
stream_status dispatch_d(const Geom &g, const void *q, const void *k, const void *v, const int32_t *mask, float scale, void *out,
                         cudaStream_t st) {
    switch (g.d) {
        case 16: return launch<T, 16, kLoad>(g, q, k, v, mask, scale, out, st);
        case 32: return launch<T, 32, kLoad>(g, q, k, v, mask, scale, out, st);
        case 64: return launch<T, 64, kLoad>(g, q, k, v, mask, scale, out, st);
        case 128: return launch<T, 128, kLoad>(g, q, k, v, mask, scale, out, st);
        case 256: return launch<T, 256, kLoad>(g, q, k, v, mask, scale, out, st);
    }
    set_error("generic attention kernel: head dim %d not in {16, 32, 64, 128, 256}", g.d);
    return STREAM_ERR_UNSUPPORTED;
}

}  // namespace

stream_status launch_attn_generic(const Geom &g, int dtype, const void *q, const void *k, const void *v,
                                  const int32_t *mask, float scale, void *out, cudaStream_t st) {
    if (g.bq > kMaxBlock || g.bk > kMaxBlock) {
        set_error("generic attention kernel: block sizes up to %d (got %d, %d)", kMaxBlock, g.bq, g.bk);
        return STREAM_ERR_UNSUPPORTED;
    }
    if (dtype != STREAM_F32) {
        if (rows_aligned(k, g.ks_t, g.ks_h, g.ks_b, 2, 8) && ((uintptr_t)v & 7) == 0) return dispatch_d<__nv_bfloat16, Load::kWide>(g, q, k, v, mask, scale, out, st);
        return dispatch_d<__nv_bfloat16, Load::kScalars>(g, q, k, v, mask, scale, out, st);
    }
    const bool aligned = rows_16_byte_aligned(k, g.ks_t, g.ks_h, g.ks_b, 4) && ((uintptr_t)v & 15) == 0;
    if (aligned) return dispatch_d<float, Load::kCopy16>(g, q, k, v, mask, scale, out, st);
    return dispatch_d<float, Load::kScalars>(g, q, k, v, mask, scale, out, st);
}

}  // namespace stream
