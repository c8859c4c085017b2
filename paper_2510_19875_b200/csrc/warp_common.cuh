// Helpers shared by the kernels that run on warp-level instructions (mma.sync, fp32 FMA, cp.async).
#pragma once
#include <math_constants.h>

#include <algorithm>

#include "common.cuh"

namespace stream {
namespace wp {

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// 16 bytes global -> shared without a register; bytes = 0 writes zeros and reads nothing.
__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(unsigned dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// D += A B, m16n8k16, bf16 operands (exact products), fp32 accumulation.
__device__ __forceinline__ void mma_bf16(float *c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float warp_max(float x) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}

// One channel of an RQ x 8 tile: acc += a b^T. (Channel by channel, so that an accumulator's next
// addition is 8 RQ instructions away; four in a row on one accumulator wait for each other.)
template <int RQ>
__device__ __forceinline__ void fma_channel(float (&acc)[RQ][8], const float4 (&a)[RQ], const float4 (&b)[8], float float4::*ch) {
#pragma unroll
    for (int i = 0; i < RQ; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i].*ch, b[j].*ch, acc[i][j]);
}

// Barrier of a group of warps (one warp needs no more than reconvergence). Ids 1.. are the caller's.
__device__ __forceinline__ void group_sync(int id, int threads) {
    if (threads == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The CTAs of a cluster: their number, this one's; a barrier in two halves (what was written before the
// first is seen behind the second, in the other CTAs' shared memory too); a word of another's
// shared memory, at the place of one of this CTA's own.
__device__ __forceinline__ unsigned cluster_size() {
    unsigned n;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n));
    return n;
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ unsigned address_in_cluster(const void *own, unsigned cta) {
    unsigned at;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((unsigned)__cvta_generic_to_shared(own)), "r"(cta));
    return at;
}
__device__ __forceinline__ void store_in_cluster(unsigned *own, unsigned cta, unsigned value) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(address_in_cluster(own, cta)), "r"(value) : "memory");
}
__device__ __forceinline__ float load_in_cluster(const float *own, unsigned cta) {
    float x;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(address_in_cluster(own, cta)) : "memory");
    return x;
}
__device__ __forceinline__ float4 load4_in_cluster(const float *own, unsigned cta) {
    float4 x;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(address_in_cluster(own, cta)) : "memory");
    return x;
}

// Which of the 8 16-byte columns of a 128-byte line a bf16 row keeps chunk c of that line in: c ^
// swz_rows(row). Read as mma operands, 8 lanes (two rows r, r + 1, four consecutive chunks each)
// then meet 8 different columns.
__device__ __forceinline__ int swz_rows(int row) { return ((row & 1) << 2) | ((row >> 1) & 3); }

// fp32 score <-> unsigned key of the same order (-0 first brought to +0; 0 is below every score).
__device__ __forceinline__ unsigned key_of(float s) {
    const unsigned b = __float_as_uint(s + 0.f);
    return b ^ ((b & 0x80000000u) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float score_of(unsigned key) {
    return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
}

// Allows a kernel the dynamic shared memory `most`, whatever this launch takes: the limit belongs to the kernel,
// and one set to the need of a launch would be in the way of another thread's.
template <class Kernel>
cudaError_t allow_smem(Kernel *kern, size_t most) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// How the fp32-FMA kernels bring keys and values to shared memory: 16 or 4 bytes at a time by cp.async (fp32),
// 8 at a time through registers (bf16, widened on the way), element by element (rows off these boundaries).
enum class Load { kCopy16, kCopy4, kWide, kScalars };

// Four bf16 in a row, element by element; as fp32.
__device__ __forceinline__ uint2 load4(const __nv_bfloat16 *src) {
    const unsigned short *x = (const unsigned short *)src;
    const unsigned a = x[0], b = x[1], c = x[2], d = x[3];
    return make_uint2(a | (b << 16), c | (d << 16));
}
__device__ __forceinline__ float4 widen4(uint2 x) {
    return make_float4(__uint_as_float(x.x << 16), __uint_as_float(x.x & 0xffff0000u), __uint_as_float(x.y << 16),
                       __uint_as_float(x.y & 0xffff0000u));
}

inline bool rows_aligned(const void *base, long long s_t, long long s_h, long long s_b, int elem, int bytes) {
    const long long per = bytes / elem;
    return ((uintptr_t)base & (bytes - 1)) == 0 && s_t % per == 0 && s_h % per == 0 && s_b % per == 0;
}
inline bool rows_16_byte_aligned(const void *base, long long s_t, long long s_h, long long s_b, int elem) {
    return rows_aligned(base, s_t, s_h, s_b, elem, 16);
}

// SMs of the current device (148 if it cannot be asked): only used to choose launch shapes.
inline int sm_count_or_default() {
    int dev = 0, n = 148;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n = 148;
    return n;
}

}  // namespace wp
}  // namespace stream
