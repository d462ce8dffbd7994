// Device helpers shared by the tensor-core GETT kernels (tc_gett.cu,
// tc_packed.cu): operand kinds and their conversion, CTA pairs, MMA issue,
// tensor-memory loads, index arithmetic.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "tc_tcgen05.cuh"

namespace tc {
namespace dev {

// (GK_D64: FP64 inputs as exact BF16 digits, tc_packed.cu)
enum GettKind { GK_BF16X3 = 0, GK_BF16 = 1, GK_F16 = 2, GK_TF32 = 3, GK_TF32X3 = 4, GK_E4M3 = 5, GK_D64 = 6 };

// MMA on TF32 words (kind::tf32, 4-byte operand elements)
__host__ __device__ constexpr bool tf32_kind(int k) { return k == GK_TF32 || k == GK_TF32X3; }
// FP32 inputs, converted (or split) by the converter warps
__host__ __device__ constexpr bool float_input(int k) {
    return k == GK_BF16X3 || k == GK_TF32 || k == GK_TF32X3 || k == GK_E4M3;
}

// Named barrier over one warp role that also ORs a predicate across it.
template <int ID, int COUNT>
__device__ __forceinline__ bool role_sync_or(bool pred) {
    uint32_t out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(out)
        : "r"((uint32_t)pred), "n"(ID), "n"(COUNT)
        : "memory");
    return out != 0;
}

// ---- CTA pairs (cta_group::2): two CTAs of a cluster of two share each MMA.
// The pair's MMA is M = 256: each CTA holds 128 rows of A and half of the
// B tile in its own shared memory (at the same offsets), and each CTA's
// tensor memory receives its 128 rows of the accumulator.  One thread of
// the even CTA issues the MMAs; its commits arrive on both CTAs' barriers.
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Every thread of both CTAs: release this CTA's prior writes, acquire the
// peer's.
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The shared::cluster address of the same shared-memory offset in CTA `rank`.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// Arrival on an mbarrier of another CTA of the cluster (release at cluster
// scope: this thread's prior shared-memory writes are visible to a thread
// that acquires the barrier's phase).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait_cl(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait that acquires at cluster scope (barriers other CTAs of the
// pair arrive on); false when the limit expired.
__device__ __forceinline__ bool mbar_wait_cl(uint64_t *bar, uint32_t parity) {
    if (mbar_try_wait_cl(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait_cl(bar, parity)) {
        if (globaltimer() - t0 > kWaitLimitNs) return false;
    }
    return true;
}

__device__ __forceinline__ bool mbar_wait_cl_or(uint64_t *bar, uint32_t parity, volatile int *abort_flag) {
    if (mbar_try_wait_cl(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    while (!mbar_try_wait_cl(bar, parity)) {
        if (*abort_flag || globaltimer() - t0 > kWaitLimitNs) return false;
    }
    return true;
}

// One warp of each CTA of the pair allocates collectively; the address is
// the same in both CTAs.
__device__ __forceinline__ void tmem_alloc2(uint32_t *dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// Commit of the pair's MMAs issued so far by this thread: arrives once on
// the barrier at this shared-memory offset in every CTA of `mask`.
__device__ __forceinline__ void mma_commit2(uint64_t *bar, uint16_t mask) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"(mask)
        : "memory");
}

// A BF16 MMA of several in a row with the same A: the first keeps A in the
// collector buffer (USE 0: fill), the others read it there (1: use, 2: the
// last one) instead of from shared memory.
template <bool PAIR, int USE>
__device__ __forceinline__ void mma_issue_same_a(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                 uint32_t accumulate) {
    if constexpr (PAIR && USE == 0) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (PAIR && USE == 1) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (PAIR && USE == 2) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (!PAIR && USE == 0) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (!PAIR && USE == 1) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (!PAIR && USE == 2) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    }
}

template <int KIND, bool PAIR = false>
__device__ __forceinline__ void mma_issue(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
    if constexpr (PAIR && tf32_kind(KIND)) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (PAIR && KIND == GK_E4M3) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (PAIR) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (tf32_kind(KIND)) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (KIND == GK_E4M3) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    }
}

// 64 consecutive columns of this warp's 32 lanes with one wait: the load
// latency is paid once per 64 columns instead of once per 32.
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t (&r)[64]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Four columns of each of eight accumulators `stride` columns apart, one wait:
// r[4 n + j] is column j of accumulator n.
__device__ __forceinline__ void tmem_ld8x4(uint32_t t, uint32_t stride, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%33];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%34];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%35];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16,%17,%18,%19}, [%36];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20,%21,%22,%23}, [%37];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24,%25,%26,%27}, [%38];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%28,%29,%30,%31}, [%39];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(t), "r"(t + stride), "r"(t + 2 * stride), "r"(t + 3 * stride), "r"(t + 4 * stride), "r"(t + 5 * stride),
          "r"(t + 6 * stride), "r"(t + 7 * stride)
        : "memory");
}

// Two 32-column loads (the split accumulators) and their FP32 sum: both
// loads and the wait in one statement, so no use of the registers can be
// scheduled before the wait.
__device__ __forceinline__ void tmem_ld32_sum(uint32_t ta, uint32_t tb, uint32_t (&r)[32]) {
    uint32_t a[32], b[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%64];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,"
        "%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%65];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]),
          "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]),
          "=r"(a[16]), "=r"(a[17]), "=r"(a[18]), "=r"(a[19]), "=r"(a[20]), "=r"(a[21]), "=r"(a[22]), "=r"(a[23]),
          "=r"(a[24]), "=r"(a[25]), "=r"(a[26]), "=r"(a[27]), "=r"(a[28]), "=r"(a[29]), "=r"(a[30]), "=r"(a[31]),
          "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]),
          "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15]),
          "=r"(b[16]), "=r"(b[17]), "=r"(b[18]), "=r"(b[19]), "=r"(b[20]), "=r"(b[21]), "=r"(b[22]), "=r"(b[23]),
          "=r"(b[24]), "=r"(b[25]), "=r"(b[26]), "=r"(b[27]), "=r"(b[28]), "=r"(b[29]), "=r"(b[30]), "=r"(b[31])
        : "r"(ta), "r"(tb)
        : "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__fadd_rn(__uint_as_float(a[j]), __uint_as_float(b[j])));
}

__device__ __forceinline__ uint32_t f32_to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}



template <int KIND, int BK>
struct KindTraits {
    static constexpr int kElemBytes = tf32_kind(KIND) ? 4 : (KIND == GK_E4M3 ? 1 : 2);  // smem operand element
    static constexpr int kSlices = KIND == GK_BF16X3 ? 3 : (KIND == GK_TF32X3 ? 2 : (KIND == GK_D64 ? 8 : 1));
    static constexpr int kChunk = 16 / kElemBytes;              // K elements per 16-byte row
    static constexpr int kKc = BK / kChunk;                     // core matrices along K per stage
    static constexpr int kKsteps = BK * kElemBytes / 32;        // MMA instructions along K per stage
    // instruction-descriptor operand format: kind::tf32 TF32 = 2; kind::f16
    // F16 = 0, BF16 = 1; kind::f8f6f4 E4M3 = 0
    static constexpr uint32_t kFmt = tf32_kind(KIND) ? 2u : ((KIND == GK_F16 || KIND == GK_E4M3) ? 0u : 1u);
    using In = typename std::conditional<KIND == GK_BF16, __nv_bfloat16,
                                         typename std::conditional<KIND == GK_F16, __half,
                                                                   typename std::conditional<KIND == GK_D64, double, float>::type>::type>::type;
    static constexpr int kInBytes = sizeof(In);
    static constexpr int kVec = 16 / kInBytes;                  // input elements per 16-byte load
};

// x = q * y + r for non-negative x, y > 0: 32-bit division when both fit
// (a 64-bit division is a long dependent instruction sequence, and these
// sit on the per-tile critical path of every role)
__device__ __forceinline__ int64_t divmod(int64_t x, int64_t y, int64_t &r) {
    if (((x | y) >> 31) == 0) {
        const uint32_t q = (uint32_t)x / (uint32_t)y;
        r = x - (int64_t)q * y;
        return q;
    }
    const int64_t q = x / y;
    r = x - q * y;
    return q;
}

__device__ __forceinline__ void decode(int64_t x, int n, const int64_t *ext, const int64_t *s1,
                                       const int64_t *s2, int64_t &o1, int64_t &o2) {
    // first mode fastest
    for (int m = 0; m < n; ++m) {
        int64_t v;
        x = divmod(x, ext[m], v);
        o1 += v * s1[m];
        o2 += v * s2[m];
    }
}

// Converts N (4 or 8) FP32 values into the 16-bit slices or TF32 words
// and stores them at dst (one slice after another, slice_stride apart).
// qs: E4M3 only, the operand's inverse scale (a power of two).
template <int KIND, int N>
__device__ __forceinline__ void store_converted(const float (&x)[N], char *dst, int slice_stride, float qs = 1.0f) {
    if constexpr (KIND == GK_BF16X3) {
        uint32_t w0[N / 2], w1[N / 2], w2[N / 2];
#pragma unroll
        for (int e = 0; e < N; e += 2) split3x2(x[e], x[e + 1], w0[e / 2], w1[e / 2], w2[e / 2]);
        if constexpr (N == 8) {
            *(uint4 *)(dst) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
            *(uint4 *)(dst + slice_stride) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
            *(uint4 *)(dst + 2 * slice_stride) = make_uint4(w2[0], w2[1], w2[2], w2[3]);
        } else {
            *(uint2 *)(dst) = make_uint2(w0[0], w0[1]);
            *(uint2 *)(dst + slice_stride) = make_uint2(w1[0], w1[1]);
            *(uint2 *)(dst + 2 * slice_stride) = make_uint2(w2[0], w2[1]);
        }
    } else if constexpr (KIND == GK_TF32X3) {  // N == 4: x = hi + lo (+ at most 2^-22 |x|)
        uint32_t h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            h[e] = f32_to_tf32(x[e]);
            l[e] = f32_to_tf32(x[e] - __uint_as_float(h[e]));  // the difference is exact
        }
        *(uint4 *)(dst) = make_uint4(h[0], h[1], h[2], h[3]);
        *(uint4 *)(dst + slice_stride) = make_uint4(l[0], l[1], l[2], l[3]);
    } else if constexpr (KIND == GK_E4M3) {  // N == 4 or 16: x * qs rounded to E4M3, saturating
        (void)slice_stride;
        uint32_t w[N / 4];
#pragma unroll
        for (int e = 0; e < N; e += 4) {
            const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(x[e] * qs, x[e + 1] * qs), __NV_SATFINITE, __NV_E4M3);
            const uint32_t hi =
                __nv_cvt_float2_to_fp8x2(make_float2(x[e + 2] * qs, x[e + 3] * qs), __NV_SATFINITE, __NV_E4M3);
            w[e / 4] = lo | (hi << 16);
        }
        if constexpr (N == 16) *(uint4 *)(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        else *(uint32_t *)(dst) = w[0];
    } else {  // TF32: N == 4
        *(uint4 *)(dst) = make_uint4(f32_to_tf32(x[0]), f32_to_tf32(x[1]), f32_to_tf32(x[2]),
                                     f32_to_tf32(x[3]));
    }
}

}  // namespace dev
}  // namespace tc
