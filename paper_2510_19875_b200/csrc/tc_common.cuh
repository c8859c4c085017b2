// PTX wrappers and host helpers shared by the tcgen05 / TMA kernels of libstream (sm_100a only).
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace stream {
namespace tc {

constexpr long long kWaitCycles = 1ll << 31;  // ~1 s: far beyond any legitimate wait

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// The first 1024-byte boundary of the dynamic shared memory, as an offset from its start: an address
// that has gone through an integer is a generic one to the compiler, and every access to it a 64-bit
// address and a longer wait.
__device__ __forceinline__ unsigned char *aligned_smem(unsigned char *raw) { return raw + ((0u - smem_u32(raw)) & 1023u); }

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Two barriers' phases at once: the second look is on its way while the first is.
__device__ __forceinline__ bool mbar_try_wait_both(unsigned bar_a, unsigned parity_a, unsigned bar_b, unsigned parity_b) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p, q;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 q, [%3], %4;\nand.pred p, p, q;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar_a), "r"(parity_a), "r"(bar_b), "r"(parity_b)
        : "memory");
    return ok != 0;
}

// The same, but the hardware may keep the thread suspended for up to `ns` nanoseconds while the
// phase is incomplete, instead of returning at once: far fewer shared-memory transactions than
// polling, and the shared-memory port is what these kernels run against.
__device__ __forceinline__ bool mbar_try_wait_suspend(unsigned bar, unsigned parity, unsigned ns) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(ns)
        : "memory");
    return ok != 0;
}

// Non-blocking probe of an mbarrier phase.
__device__ __forceinline__ bool mbar_test_wait(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// The same for a whole converged warp: lane 0's answer.
__device__ __forceinline__ bool probe_w(unsigned bar, unsigned parity) {
    return __shfl_sync(0xffffffffu, (int)mbar_test_wait(bar, parity), 0) != 0;
}

// The part of a bounded wait on an mbarrier phase behind its first look. Returns false if the CTA is aborting, or if this wait ran
// out, in which case it raises the CTA's abort flag and records `code` (first one wins) with the
// block index in the two error words.
static __device__ __noinline__ bool mbar_wait_slow(unsigned bar, unsigned parity, int *abort_flag, unsigned *err_code,
                                                   unsigned *err_info, unsigned code, long long limit) {
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try_wait_suspend(bar, parity, 4000u)) return true;
        if (*(volatile int *)abort_flag) return false;
        if (clock64() - t0 > limit) {
            *(volatile int *)abort_flag = 1;
            if (atomicCAS(err_code, 0u, code) == 0u) *err_info = blockIdx.x;
            return false;
        }
    }
}

// True in exactly one lane of a converged warp (the same lane every time).
__device__ __forceinline__ bool elect_one() {
    unsigned pred;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(pred));
    return pred != 0;
}

// Bounded wait of a whole converged warp: every lane waits, and all lanes get the same
// answer (false as soon as one lane saw the abort flag or ran out of time), so that the warp
// stays converged for the elect_one() that follows.
__device__ __forceinline__ bool mbar_wait_warp(unsigned bar, unsigned parity, int *abort_flag, unsigned *err_code,
                                               unsigned *err_info, unsigned code, long long limit = kWaitCycles) {
    // (one vote on the first look and no divergence on the way: this is what the warps' serial code
    // does most, and a look per lane with a branch of its own costs twice the clocks)
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait_slow(bar, parity, abort_flag, err_code, err_info, code, limit));
}

// Arrival of the lanes that say so (one of a warp, as a rule), without a branch.
__device__ __forceinline__ void mbar_arrive_if(unsigned bar, bool mine) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %1, 0;\n@p mbarrier.arrive.shared::cta.b64 _, [%0];\n}" ::"r"(bar), "r"((unsigned)mine)
                 : "memory");
}

__device__ __forceinline__ void tma_load_4d(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1, int c2,
                                            int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"((unsigned long long)map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

__device__ __forceinline__ void tma_load_5d(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1, int c2,
                                            int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
        ::"r"(dst), "l"((unsigned long long)map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

// A box from shared to global memory (rows beyond the tensor are left out), in a bulk group.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, unsigned src, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"((unsigned long long)map), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Every box this thread has stored has been read from shared memory.
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Makes this thread's shared-memory writes visible to the async proxy (TMA, tcgen05.mma operands).
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(unsigned bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// One tcgen05.mma (kind::f16, cta_group::1): D[tmem] (+)= A[smem] B[smem]. Both shared-memory
// descriptors are given as (low word, high word): the low word holds the start
// address in 16-byte units, so a K step is one 32-bit add on it; the high word never changes
// for a given operand layout.
__device__ __forceinline__ void tc_mma_bf16_split(unsigned d_tmem, unsigned a_lo, unsigned a_hi, unsigned b_lo,
                                                  unsigned b_hi, unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n.reg .pred p;\n.reg .b64 da, db;\nmov.b64 da, {%1, %2};\nmov.b64 db, {%3, %4};\nsetp.ne.b32 p, %6, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The same with A from TMEM (two bf16 per column). M = 128: lane = row. M = 64: row r of A and of the
// accumulator in lane (r / 16) * 32 + r % 16, or, with 16 added to both lane addresses, 16 lanes behind:
// two such products share their columns.
__device__ __forceinline__ void tc_mma_bf16_ta(unsigned d_tmem, unsigned a_tmem, unsigned b_lo, unsigned b_hi, unsigned idesc,
                                               unsigned accumulate) {
    asm volatile(
        "{\n.reg .pred p;\n.reg .b64 db;\nmov.b64 db, {%2, %3};\nsetp.ne.b32 p, %5, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Two fp32 in a register pair: one instruction for both.
__device__ __forceinline__ unsigned long long pack_u32x2(unsigned a, unsigned b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ unsigned long long pack_f32x2(float a, float b) { return pack_u32x2(__float_as_uint(a), __float_as_uint(b)); }
__device__ __forceinline__ void unpack_f32x2(unsigned long long x, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x));
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <int kColumns = 512>
__device__ __forceinline__ void tmem_alloc(unsigned smem_dst) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(kColumns) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int kColumns = 512>
__device__ __forceinline__ void tmem_dealloc(unsigned tmem_base) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kColumns) : "memory");
}

// 32 lanes x 32 consecutive fp32 columns of TMEM: thread i gets lane (base lane + i). Issue only;
// the registers are valid after tmem_ld_wait().
__device__ __forceinline__ void tmem_ld_32x32_issue(unsigned taddr, unsigned *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// Store 32 consecutive fp32 columns of this thread's TMEM lane (the inverse of the load above).
// Complete for later tcgen05 operations after tmem_st_wait().
__device__ __forceinline__ void tmem_st_32x32_issue(unsigned taddr, const unsigned *r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
          "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
          "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
// The same with 16 columns.
__device__ __forceinline__ void tmem_st_32x16_issue(unsigned taddr, const unsigned *r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_32x8_issue(unsigned taddr, unsigned *r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

// Multiplies fp32 columns of this thread's TMEM lane by f, in place (every lane of the warp
// takes part; lanes that need no change pass f = 1).
template <int kColumns>
__device__ __forceinline__ void rescale_lane(unsigned taddr, float f) {
#pragma unroll 1
    for (int c = 0; c < kColumns / 32; ++c) {
        unsigned r[32];
        tmem_ld_32x32_issue(taddr + c * 32, r);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f);
        tmem_st_32x32_issue(taddr + c * 32, r);
    }
    tmem_st_wait();
}

// Maximum of three in one instruction.
__device__ __forceinline__ float max3(float a, float b, float c) {
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// Maximum of 64 values held in registers: four independent chains of three-input maxima instead of
// one chain of 64 (a quarter of the instructions' latency in a row, half the instructions).
__device__ __forceinline__ float max_of_64(const float *v) {
    float b0 = max3(v[0], v[1], v[2]), b1 = max3(v[3], v[4], v[5]), b2 = max3(v[6], v[7], v[8]), b3 = max3(v[9], v[10], v[11]);
#pragma unroll
    for (int i = 12; i < 60; i += 8) {
        b0 = max3(b0, v[i], v[i + 1]);
        b1 = max3(b1, v[i + 2], v[i + 3]);
        b2 = max3(b2, v[i + 4], v[i + 5]);
        b3 = max3(b3, v[i + 6], v[i + 7]);
    }
    b0 = max3(b0, v[60], v[61]);
    b1 = max3(b1, v[62], v[63]);
    return fmaxf(fmaxf(b0, b1), fmaxf(b2, b3));
}

template <int n>
__device__ __forceinline__ float max_of(const float *v) {
    static_assert(n == 64 || n == 32, "what the kernels read at a time");
    if constexpr (n == 64) {
        return max_of_64(v);
    } else {
        float b0 = max3(v[0], v[1], v[2]), b1 = max3(v[3], v[4], v[5]), b2 = max3(v[6], v[7], v[8]), b3 = max3(v[9], v[10], v[11]);
#pragma unroll
        for (int i = 12; i < 28; i += 8) {
            b0 = max3(b0, v[i], v[i + 1]);
            b1 = max3(b1, v[i + 2], v[i + 3]);
            b2 = max3(b2, v[i + 4], v[i + 5]);
            b3 = max3(b3, v[i + 6], v[i + 7]);
        }
        b0 = max3(b0, v[28], v[29]);
        b1 = max3(b1, v[30], v[31]);
        return fmaxf(fmaxf(b0, b1), fmaxf(b2, b3));
    }
}

__device__ __forceinline__ float warp_max(float x) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}

// Shared-memory matrix descriptor (sm_100 version 1) with 128-byte swizzle. Offsets in bytes.
//   K-major operand (rows of 128 bytes along K): sbo = distance between 8-row groups; lbo unused.
//   MN-major operand (rows of 128 bytes along M/N, one row per K index): sbo = distance between
//   8-K-index groups, lbo = distance between consecutive 64-element chunks along M/N.
// Bits: start address >> 4 in 0..13, lbo >> 4 in 16..29, sbo >> 4 in 32..45, version 1 in 46..47,
// swizzle mode 2 (128 bytes) in 61..63.
// Low and high words of that descriptor; (addr_bytes >> 4) is added to the low word per operand.
__device__ __forceinline__ unsigned desc_lo_sw128(unsigned addr, unsigned lbo) {
    return ((addr >> 4) & 0x3FFF) | (((lbo >> 4) & 0x3FFF) << 16);
}
__host__ __device__ constexpr unsigned desc_hi_sw128(unsigned sbo) { return ((sbo >> 4) & 0x3FFF) | (1u << 14) | (2u << 29); }

// kind::f16 instruction descriptor: D fp32, A and B bf16, A K-major, B K-major or MN-major.
__host__ __device__ constexpr unsigned idesc_bf16(unsigned M, unsigned N, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// Top-k of the (up to) 64 candidates a warp holds two per lane (a node's left and right branch):
// keep the k best by (score descending, candidate index ascending), the candidates numbered
// 2 * lane (left) and 2 * lane + 1 (right); k <= 32.
//
// The k-th largest score is found with a sorting network (a first form counted ranks in one chain of 4096
// comparisons; it is the chain that was slow, see select_topk_counting): the scores become unsigned
// keys of the same order (-0 first brought to +0, so that equal floats give equal keys; an absent
// candidate gets key 0, below every score), the 32 left keys are sorted descending and the 32
// right keys ascending across the lanes (one bitonic network, 15 exchange steps, both registers
// at once), the lane-wise maximum of the two is then the 32 largest keys as a bitonic sequence,
// five more steps sort it, and lane k - 1 holds the threshold. Every candidate above the threshold
// is kept; of those equal to it the first ones in candidate order, as many as are still missing.
struct Keep { bool l, r; };
__device__ __forceinline__ unsigned score_key(bool valid, float s) {
    const unsigned b = __float_as_uint(s + 0.f);
    return valid ? (b ^ ((b & 0x80000000u) ? 0xffffffffu : 0x80000000u)) : 0u;
}
__device__ __forceinline__ Keep select_topk(bool vl, float sl, bool vr, float sr, int k, int lane) {
    const int total = __popc(__ballot_sync(0xffffffffu, vl)) + __popc(__ballot_sync(0xffffffffu, vr));
    if (total <= k) return {vl, vr};
    const unsigned kl = score_key(vl, sl), kr = score_key(vr, sr);
    unsigned a = kl, b = kr;  // a: sorted descending over the lanes, b: ascending
#pragma unroll
    for (int k2 = 2; k2 <= 32; k2 <<= 1) {
#pragma unroll
        for (int j = k2 >> 1; j > 0; j >>= 1) {
            const unsigned oa = __shfl_xor_sync(0xffffffffu, a, j), ob = __shfl_xor_sync(0xffffffffu, b, j);
            // in an ascending network the lower lane of a pair takes the minimum inside an "up" block
            const bool first = (((lane & j) == 0) == ((lane & k2) == 0));
            a = first ? max(a, oa) : min(a, oa);
            b = first ? min(b, ob) : max(b, ob);
        }
    }
    unsigned c = max(a, b);  // the 32 largest of the 64 keys, a bitonic sequence over the lanes
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const unsigned oc = __shfl_xor_sync(0xffffffffu, c, j);
        c = ((lane & j) == 0) ? max(c, oc) : min(c, oc);
    }
    const unsigned thr = __shfl_sync(0xffffffffu, c, k - 1);  // the k-th largest key (with multiplicity)
    const bool gl = kl > thr, gr = kr > thr, el = kl == thr, er = kr == thr;
    const int missing = k - __popc(__ballot_sync(0xffffffffu, gl)) - __popc(__ballot_sync(0xffffffffu, gr));
    const unsigned bel = __ballot_sync(0xffffffffu, el), ber = __ballot_sync(0xffffffffu, er);
    const unsigned lt = (1u << lane) - 1u;
    const int pos_l = __popc(bel & lt) + __popc(ber & lt), pos_r = pos_l + (el ? 1 : 0);
    return {vl && (gl || (el && pos_l < missing)), vr && (gr || (er && pos_r < missing))};
}

// The same of the nodes of lanes 0 .. n - 1, a row's serial way (controller of the block kernel): every lane counts the
// keys above its own two, read four at a time from `room` (64 words of the warp's own, 16-byte aligned). The comparisons do not wait
// for one another; the network's twenty exchanges do, 55 clocks each: 1100 clocks whatever k, this 200 at k = 8.
__device__ __forceinline__ Keep select_topk_counting(bool vl, float sl, bool vr, float sr, int k, int n, int lane, unsigned *room) {
    const int total = __popc(__ballot_sync(0xffffffffu, vl)) + __popc(__ballot_sync(0xffffffffu, vr));
    if (total <= k) return {vl, vr};
    const unsigned kl = score_key(vl, sl), kr = score_key(vr, sr);
    reinterpret_cast<uint2 *>(room)[lane] = make_uint2(kl, kr);
    __syncwarp();
    int above_l = 0, above_r = 0;
#pragma unroll 4
    for (int j = 0; j < (n + 1) / 2; ++j) {
        const uint4 y = reinterpret_cast<const uint4 *>(room)[j];
        above_l += (int)(y.x > kl) + (int)(y.y > kl) + (int)(y.z > kl) + (int)(y.w > kl);
        above_r += (int)(y.x > kr) + (int)(y.y > kr) + (int)(y.z > kr) + (int)(y.w > kr);
    }
    const bool l = above_l < k, r = above_r < k;  // (an absent one has all others above it)
    const unsigned bl = __ballot_sync(0xffffffffu, l), br = __ballot_sync(0xffffffffu, r);
    if (__popc(bl) + __popc(br) == k) return {l, r};
    // equal keys on either side of the line: the lowest that is kept, of those the first in candidate order
    const unsigned thr = __reduce_min_sync(0xffffffffu, min(l ? kl : 0xffffffffu, r ? kr : 0xffffffffu));
    const bool el = l && kl == thr, er = r && kr == thr;
    const unsigned bel = __ballot_sync(0xffffffffu, el), ber = __ballot_sync(0xffffffffu, er);
    const int missing = k - (__popc(bl) + __popc(br) - __popc(bel) - __popc(ber));
    const unsigned lt = (1u << lane) - 1u;
    const int pos_l = __popc(bel & lt) + __popc(ber & lt), pos_r = pos_l + (el ? 1 : 0);
    return {l && (!el || pos_l < missing), r && (!er || pos_r < missing)};
}

// The same for n candidates a lane, numbered n * lane + i: the largest threshold that at least k keys
// reach, bit by bit from the top (it is the k-th largest key), or earlier if exactly k reach it.
template <int n>
__device__ __forceinline__ void select_topk_of(const bool (&have)[n], const float (&score)[n], int k, int lane, bool (&keep)[n]) {
    unsigned key[n], b[n];
    int total = 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
        key[i] = score_key(have[i], score[i]);
        total += __popc(__ballot_sync(0xffffffffu, have[i]));
        keep[i] = have[i];
    }
    if (total <= k) return;
    unsigned thr = 0;
    int above = total;
#pragma unroll 1
    for (unsigned bit = 0x80000000u; bit != 0 && above != k; bit >>= 1) {
        int c = 0;
#pragma unroll
        for (int i = 0; i < n; ++i) c += __popc(__ballot_sync(0xffffffffu, key[i] >= (thr | bit)));
        if (c >= k) { thr |= bit; above = c; }
    }
    int missing = k;
#pragma unroll
    for (int i = 0; i < n; ++i) missing -= __popc(__ballot_sync(0xffffffffu, key[i] > thr));
    int place = 0;
    const unsigned lt = (1u << lane) - 1u;
    if (above == k) missing = 32 * n;  // all that reach it
#pragma unroll
    for (int i = 0; i < n; ++i) {
        b[i] = __ballot_sync(0xffffffffu, have[i] && key[i] == thr);
        place += __popc(b[i] & lt);
    }
#pragma unroll
    for (int i = 0; i < n; ++i) {
        const bool equal = have[i] && key[i] == thr;
        keep[i] = have[i] && (key[i] > thr || (equal && place < missing));
        place += equal ? 1 : 0;
    }
}

// Places of a warp's flags, n of them a lane, in lane order: those before this lane's; all of them.
template <int n>
__device__ __forceinline__ int flags_before(const unsigned (&ballots)[n], unsigned lt) {
    int c = 0;
#pragma unroll
    for (int i = 0; i < n; ++i) c += __popc(ballots[i] & lt);
    return c;
}
template <int n>
__device__ __forceinline__ int flags_all(const unsigned (&ballots)[n]) { return flags_before(ballots, 0xffffffffu); }

// The nodes of a row, kNodes a lane of a warp, before the first level that ranks anything; n of them. q_lim: the row's last allowed
// block, or that of the last of several rows.
// A level with no more than kq allowed candidates keeps them all whatever their scores, so its scores are not waited for:
// its candidates are split on, and what there is to score of them comes with the next level's (a left branch has its
// parent's score), in the one list that all rows of a group share. So it is with the first level of every row that may look at half of
// the blocks at most, the first two where it is a quarter. `splits`: such levels. The last level always has its list. (us, mask build
// with all levels ranked and now: 32 / 8 heads, 4096 tokens, k = 32: 71.4, 50.7; 16384, k = 16: 526, 492; 131072, k = 32: 12050,
// 11620; four layers of 9999, 28 / 4 heads, k = 16: 994, 914; 12 / 2 heads, 10007 tokens in blocks of 32, k = 8: 129.6, 116.7.)
template <int kNodes>
struct FirstNodes {
    int f[kNodes], l[kNodes];  // this lane's (l < f: none)
    int n, splits;
    bool left[kNodes], right[kNodes];  // candidates: first half, second half
    __device__ __forceinline__ FirstNodes(const Geom &g, int kq, int levels, int q_lim, int lane, int *room_f, int *room_l) {
        const unsigned lt = (1u << lane) - 1u;
        unsigned ballots[2 * kNodes];
#pragma unroll
        for (int x = 0; x < kNodes; ++x) {
            const int i = kNodes * lane + x;
            f[x] = (int)(((long long)i * g.N_k) / kq);
            l[x] = i < kq ? (int)(((long long)(i + 1) * g.N_k) / kq) - 1 : f[x] - 1;
        }
        n = kq;
        for (splits = 0;; ++splits) {
#pragma unroll
            for (int x = 0; x < kNodes; ++x) {
                const int m = (f[x] + l[x]) / 2;
                left[x] = f[x] <= l[x] && f[x] <= q_lim;
                right[x] = left[x] && m + 1 <= l[x] && m + 1 <= q_lim;
                ballots[2 * x] = __ballot_sync(0xffffffffu, left[x]);
                ballots[2 * x + 1] = __ballot_sync(0xffffffffu, right[x]);
            }
            const int total = flags_all(ballots);
            if (total > kq || splits + 1 >= levels) return;
            int place = flags_before(ballots, lt);
            __syncwarp();
#pragma unroll
            for (int x = 0; x < kNodes; ++x) {
                const int m = (f[x] + l[x]) / 2;
                if (left[x]) { room_f[place] = f[x]; room_l[place++] = m; }
                if (right[x]) { room_f[place] = m + 1; room_l[place++] = l[x]; }
            }
            __syncwarp();
            n = total;
#pragma unroll
            for (int x = 0; x < kNodes; ++x) {
                const int i = kNodes * lane + x;
                f[x] = i < n ? room_f[i] : 0;
                l[x] = i < n ? room_l[i] : -1;
            }
        }
    }
};

// A CTA's n-th place in an order of items. Every second round runs backwards, so that with items in
// order of falling length every CTA gets about the same sum.
__device__ __forceinline__ int nth_item(int n) {
    return n * (int)gridDim.x + ((n & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
}
constexpr long long kL2KvBytes = 64ll << 20;  // K and V bytes that stay in the 126 MB L2 while items of several heads are walked

// The end of a kernel, of all its threads; `owner`: the warp that has allocated TMEM. After an abort, copies and
// MMAs may still be in flight: they have a bounded time to land before shared memory and TMEM are given back.
template <int kColumns = 512>
__device__ __forceinline__ void leave(const int *abort_flag, unsigned tmem_base, bool owner) {
    if (*(const volatile int *)abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < (1ll << 22)) { }
    }
    tc_fence_before();
    __syncthreads();
    if (owner) {
        tc_fence_after();
        tmem_dealloc<kColumns>(tmem_base);
    }
}

struct Ring {  // position in a ring of barriers with phase tracking
    int idx = 0;
    unsigned phase = 0;
    __device__ void advance(int n) {
        if (++idx == n) { idx = 0; phase ^= 1; }
    }
};

// ----------------------------------------------------------------------------------------------
// Host side
// ----------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

// [batch, heads, T, d] bf16 with element strides -> 4-D map with a box of 64 (or 32) channels x box_rows
// tokens, 128-byte (or 64-byte) swizzle. Rows beyond T read as zeros.
inline stream_status make_map_bf16(CUtensorMap *map, const void *base, long long T, int heads, int batch,
                                   long long s_t, long long s_h, long long s_b, const char *what, int box_rows, int d, int channels = 64) {
    EncodeTiledFn fn = encode_fn();
    if (fn == nullptr) { set_error("cuTensorMapEncodeTiled is not available from this driver"); return STREAM_ERR_CUDA; }
    // extents of 1 may come with arbitrary strides: give them a well-formed one
    if (heads == 1) s_h = s_t * T;
    if (batch == 1) s_b = s_h * heads;
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)T, (cuuint64_t)heads, (cuuint64_t)batch};
    cuuint64_t strides[3] = {(cuuint64_t)s_t * 2, (cuuint64_t)s_h * 2, (cuuint64_t)s_b * 2};
    cuuint32_t box[4] = {(cuuint32_t)channels, (cuuint32_t)box_rows, 1, 1}, estr[4] = {1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, channels == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled(%s) failed with %d", what, (int)r); return STREAM_ERR_CUDA; }
    return STREAM_OK;
}

inline stream_status make_map_bf16_d128(CUtensorMap *map, const void *base, long long T, int heads, int batch,
                                        long long s_t, long long s_h, long long s_b, const char *what, int box_rows = 64) {
    return make_map_bf16(map, base, T, heads, batch, s_t, s_h, s_b, what, box_rows, 128);
}

// The same tensor seen as [batch, heads, channel halves, T, 64]: one box brings a whole
// tile of box_rows tokens x d channels as [half][rows][128 B], the layout of a 128-byte-swizzled
// K-major (or, read along the rows, MN-major) tcgen05 operand.
// Coordinates: (0, token, head, 0, batch) with the half as dimension 3.
inline stream_status make_map5_bf16(CUtensorMap *map, const void *base, long long T, int heads, int batch,
                                    long long s_t, long long s_h, long long s_b, const char *what, int box_rows, int d) {
    EncodeTiledFn fn = encode_fn();
    if (fn == nullptr) { set_error("cuTensorMapEncodeTiled is not available from this driver"); return STREAM_ERR_CUDA; }
    if (heads == 1) s_h = s_t * T;
    if (batch == 1) s_b = s_h * heads;
    cuuint64_t dims[5] = {64, (cuuint64_t)T, (cuuint64_t)heads, (cuuint64_t)(d / 64), (cuuint64_t)batch};
    cuuint64_t strides[4] = {(cuuint64_t)s_t * 2, (cuuint64_t)s_h * 2, 128, (cuuint64_t)s_b * 2};
    cuuint32_t box[5] = {64, (cuuint32_t)box_rows, 1, (cuuint32_t)(d / 64), 1}, estr[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled(%s) failed with %d", what, (int)r); return STREAM_ERR_CUDA; }
    return STREAM_OK;
}

inline bool tma_strides_ok(const Geom &g) {
    auto ok = [](long long s) { return s % 8 == 0; };  // 16-byte multiples
    return ok(g.qs_t) && ok(g.qs_h) && ok(g.qs_b) && ok(g.ks_t) && ok(g.ks_h) && ok(g.ks_b);
}

// kv heads whose groups a mask kernel walks together: as many as have their keys in 32 MB of L2 (there are 126 MB; queries stream by).
// One head after the other, the last one's long groups began when most CTAs were about to finish (us: 28 / 4 heads, 1500 tokens, k = 5:
// 36.1 -> 29.2; 12 / 2 heads, 5000 tokens in blocks of 32, k = 8: 60.7 -> 55.3; three k at 5000 tokens, 28 / 4 heads: 179.6 -> 144.5,
// at 12845, 12 / 2 heads: 288 -> 240; three layers of 11851, 8 / 2 heads, k = 21: 303 -> 271; per token, 32 / 8 heads, 4096 tokens,
// k = 16: 119.5 -> 108.6. With 32 / 8 heads and 16000 tokens or more it makes no difference with one k. With
// three it is the last groups' luck there: k = 5, 10, 20 at 14000 tokens 705 -> 672, 8, 16, 32 at 16000 875 -> 893, 4, 8, 16 at 21000 1183 -> 1136,
// 8, 16, 32 at 32768 2122 -> 2136; 28 / 4 heads, 24000, 1205 -> 1195. Half or a quarter of the 32 MB gives the middle sizes' gain away: 271 -> 299, 164 -> 206).
inline int walked_heads(const Geom &g) {
    const long long fit = (32ll << 20) / (g.T * g.d * 2), all = (long long)g.batch * g.G;
    return (int)(fit < 1 ? 1 : (fit > all ? all : fit));
}

inline int sm_count() {
    static int n_sm = 0;
    if (n_sm == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            n_sm = 0;
    }
    return n_sm;
}

}  // namespace tc
}  // namespace stream
