// The tensor-core GETT with both inputs pre-converted (no paper
// counterpart).  A pre-pass writes each input once as the stage images the
// MMA reads -- per row tile and K stage the slices in the no-swizzle K-major
// core-matrix layout (8 rows x 16 bytes), zeros past the extents -- and the
// GETT copies them: no input is converted more than once, however many tiles
// of the other input it meets, and any strides cost the GETT nothing.
//
// pack_images_kernel: a block takes 32 rows x 128 K positions through shared
// memory, so that its loads run along the operand's contiguous index (rows or
// K) and its stores are 512-byte runs of an image; one launch for both inputs
// (4096 x 4096 each: BF16 39 us, split-BF16 53 us; one 16-byte chunk per
// thread straight from global memory took 67 and 77 us in two launches).
//
// packed_gett_kernel: persistent and warp-specialised, one CTA per SM or a
// pair of CTAs sharing each MMA (cta_group::2):
//   copy warp 9      one lane streams each stage's two images with
//                    cp.async.bulk.tensor into a ring (both CTAs of a pair
//                    count their bytes on the issuing CTA's barrier);
//   MMA warp 8       one lane issues the stage's slice products;
//   epilogue warps 0-7  drain the accumulators (two warps per 32 lanes,
//                    alternate groups of 32 columns) and store C.
// Why pairs and these widths: an MMA of N columns takes N / 2 clocks and reads
// 4 KB of A and 32 bytes per row of B held here through the shared-memory
// port (128 bytes per clock), next to the copies' writes.  A lone CTA on
// 128 x 256 BF16 tiles would need 192 bytes per clock, a pair, which holds
// half of B each, 128.  The tile width follows the number of waves
// (choose_tile).  ab=aij,jib 4096^2 i=j=64: BF16 78 us on pairs of 256 x 224
// (lone 128 x 256 98 us, pairs of 256 x 256 in four uneven waves 86 us), split-
// BF16 with compensation 462 us on pairs of 256 x 128 (lone 543 us): tensor
// pipe 78-80 % active.  With the MMAs issued under a branch on the lane
// number the same tiles took 178 and 918 us (elect_one).  The compensated
// sums' (hi, lo) in registers leave the tensor memory to two accumulators.
//
// Every wait on an mbarrier is bounded; on expiry the kernel records
// TC_ERROR_TIMEOUT, stops issuing, drains, frees its tensor memory, returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "tc_gett.cuh"
#include "tc_internal.h"

namespace tc {

namespace {

using namespace dev;

constexpr int kRows = 128;                 // accumulator rows per CTA = TMEM lanes
constexpr int kRingBytes = 192 * 1024;     // operand ring
constexpr int kMaxStages = 8;
constexpr int kMaxBn = 256;
constexpr int kEpiWarps = 8;
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kMmaWarp = kEpiWarps, kCopyWarp = kEpiWarps + 1;
constexpr int kThreads = (kCopyWarp + 1) * 32;
constexpr uint32_t kTmemCols = 512;
constexpr int kMapRow = 512;               // bytes per row of an image tensor map

// K positions per stage: about 32-48 KB of images per CTA
template <int KIND>
__host__ __device__ constexpr int stage_k() {
    return KIND == GK_TF32X3 ? 16 : ((KIND == GK_BF16 || KIND == GK_F16 || KIND == GK_E4M3) ? 64 : 32);
}
template <int KIND>
using Traits = KindTraits<KIND, stage_k<KIND>()>;

struct PackedDesc : GettModes {
    const void *A, *B;
    void *C;
    float alpha, beta;
    int init;                   // 1: C = alpha*acc + beta*C, 2: C = alpha*acc
    int64_t tiles_m, tiles_n, num_tiles;
    int bn;                     // columns per tile (a multiple of 16)
    int brows;                  // rows of B per CTA: bn, or bn / 2 in a pair
    int ktiles, chunk;          // K stages; K stages per accumulation unit
    int stages;                 // ring slots
    uint32_t img_a, img_b;      // bytes of a stage image
    int nprod, split;
    int *status;
    const float *qscale;        // E4M3: the inputs' scales
};

// One input's share of the pre-pass.
struct PackJob {
    int op;                     // 0 A, 1 B
    int rows;                   // rows per image tile
    int64_t total_rows;         // rows of all image tiles (past the extent: zeros)
    int rfast;                  // lanes along rows (else along K)
    int64_t blocks;
    char *out;
};

constexpr int kPackRows = 32, kPackK = 128, kPackThreads = 256;

template <int KIND>
__global__ void __launch_bounds__(kPackThreads) pack_images_kernel(const __grid_constant__ PackedDesc d,
                                                                   const PackJob ja, const PackJob jb) {
    using T = Traits<KIND>;
    constexpr int BK = stage_k<KIND>(), CH = T::kChunk;
    constexpr bool kFloatIn = float_input(KIND);
    using L = typename std::conditional<kFloatIn, float, unsigned short>::type;
    // pitches that keep both the store along K and the read along rows free
    // of bank conflicts (an odd number of words)
    constexpr int P = kFloatIn ? kPackRows + 1 : kPackRows + 2;
    __shared__ L tile[kPackK * P];
    __shared__ int64_t koff[kPackK], roff[kPackRows];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool second = blockIdx.x >= ja.blocks;
    const PackJob &J = second ? jb : ja;
    const int64_t blk = second ? (int64_t)blockIdx.x - ja.blocks : (int64_t)blockIdx.x;
    const int64_t kblocks = ((int64_t)d.ktiles * BK + kPackK - 1) / kPackK;
    int64_t kb;
    const int64_t r0 = divmod(blk, kblocks, kb) * kPackRows, k0 = kb * kPackK;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const L *__restrict__ src = (const L *)(J.op == 0 ? d.A : d.B);
    if (tid < kPackK) {
        int64_t k = k0 + tid, o = -1, u = 0;
        if (k < d.K) {
            o = 0;
            const int64_t *ks = J.op == 0 ? d.k_sA : d.k_sB;
            for (int m = d.nk - 1; m >= 0; --m) {
                k = divmod(k, d.k_ext[m], u);
                o += u * ks[m];
            }
        }
        koff[tid] = o;
    } else if (tid < kPackK + kPackRows) {
        int64_t r = r0 + tid - kPackK, o = -1, u = 0;
        if (r < (J.op == 0 ? d.M : d.N)) {
            o = 0;
            if (J.op == 0) decode(r, d.nm, d.m_ext, d.m_sA, d.m_sC, o, u);
            else decode(r, d.nn, d.n_ext, d.n_sB, d.n_sC, o, u);
        }
        roff[tid - kPackK] = o;
    }
    __syncthreads();
    constexpr int NL = kPackK * kPackRows / kPackThreads;  // elements per thread
    L x[NL];
    if (J.rfast) {
        const int64_t ro = roff[lane];
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const int64_t ko = koff[warp + 8 * j];
            x[j] = ro >= 0 && ko >= 0 ? __ldg(src + ro + ko) : L(0);
        }
#pragma unroll
        for (int j = 0; j < NL; ++j) tile[(warp + 8 * j) * P + lane] = x[j];
    } else {
        constexpr int KJ = kPackK / 32;
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const int64_t ro = roff[warp * 4 + j / KJ], ko = koff[lane + 32 * (j % KJ)];
            x[j] = ro >= 0 && ko >= 0 ? __ldg(src + ro + ko) : L(0);
        }
#pragma unroll
        for (int j = 0; j < NL; ++j) tile[(lane + 32 * (j % KJ)) * P + warp * 4 + j / KJ] = x[j];
    }
    __syncthreads();
    const int64_t R = r0 + lane;
    if (R >= J.total_rows) return;
    int64_t rr;
    const int64_t rt = divmod(R, J.rows, rr);
    const int slice = J.rows * BK * T::kElemBytes;
    float qs = 1.0f;
    if constexpr (KIND == GK_E4M3) qs = 1.0f / d.qscale[J.op];
    char *out = J.out + rt * d.ktiles * (int64_t)(T::kSlices * slice) + (rr / 8) * 128 + (rr % 8) * 16;
#pragma unroll
    for (int j = 0; j < kPackK / CH / 8; ++j) {
        const int c = warp + 8 * j;  // chunk of CH K positions
        const int64_t k = k0 + c * CH;
        if (k >= (int64_t)d.ktiles * BK) break;
        const int kc = (int)(k % BK) / CH;
        char *dst = out + (k / BK) * (int64_t)(T::kSlices * slice) + kc * (J.rows / 8) * 128;
        const L *s = tile + c * CH * P + lane;
        if constexpr (kFloatIn) {
            float v[CH];
#pragma unroll
            for (int e = 0; e < CH; ++e) v[e] = s[e * P];
            store_converted<KIND, CH>(v, dst, slice, qs);
        } else {
            uint32_t w[CH / 2];
#pragma unroll
            for (int e = 0; e < CH; e += 2) w[e / 2] = (uint32_t)s[e * P] | ((uint32_t)s[(e + 1) * P] << 16);
            *(uint4 *)dst = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// A box of an image map into shared memory, counted on the barrier at
// shared::cluster address `bar` (a pair: the first CTA's).
template <bool PAIR>
__device__ __forceinline__ void image_load(void *dst, const CUtensorMap *map, uint32_t bar, int32_t row) {
    if constexpr (PAIR)
        asm volatile(
            "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
            "[%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
            "l"((uint64_t)map), "r"(bar), "r"(0), "r"(row)
            : "memory");
    else
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
            "[%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
            "l"((uint64_t)map), "r"(bar), "r"(0), "r"(row)
            : "memory");
}

// Stores 32 accumulator columns c0.. of this thread's row (C offset om, -1:
// none): the columns at on0 + j*lin when lin != 0, else through the table cn
// (-1 past N).  Old values are read eight at a time ahead of the stores.
__device__ __forceinline__ void store_row(const uint32_t (&r)[32], float *__restrict__ C, int64_t om, int c0,
                                          int64_t lin, int64_t on0, int nval, const int64_t *cn, float alpha,
                                          float beta, int init) {
    if (om < 0) return;
    float *p = C + om + on0 + (int64_t)c0 * lin;
    if (lin != 0 && init == 2) {
        if (c0 + 32 <= nval) {
#pragma unroll
            for (int j = 0; j < 32; ++j) p[j * lin] = alpha * __uint_as_float(r[j]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (c0 + j < nval) p[j * lin] = alpha * __uint_as_float(r[j]);
        }
        return;
    }
#pragma unroll
    for (int j0 = 0; j0 < 32; j0 += 8) {
        float *q[8], old[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = c0 + j0 + j;
            q[j] = nullptr;
            if (c < nval) q[j] = lin != 0 ? p + (j0 + j) * lin : C + om + cn[c];
            old[j] = init == 1 && q[j] ? *q[j] : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (!q[j]) continue;
            const float v = alpha * __uint_as_float(r[j0 + j]);
            *q[j] = init == 1 ? fmaf(beta, old[j], v) : v;
        }
    }
}

// COMP: compensated accumulation -- units of d.chunk K stages, double-buffered
// in tensor memory, each folded by TwoSum into a (hi, lo) pair that the
// epilogue threads hold in registers (64 columns each: bn <= 128).  Otherwise
// one unit per tile: one accumulator, or with d.split two (the (0,0) products
// apart); double-buffered where they take at most 256 columns.
template <int KIND, bool COMP, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
packed_gett_kernel(const __grid_constant__ PackedDesc d, const __grid_constant__ CUtensorMap tmA,
                   const __grid_constant__ CUtensorMap tmB) {
    using T = Traits<KIND>;
    constexpr int BK = stage_k<KIND>();
    extern __shared__ __align__(128) char ring[];
    __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], tfull[2], tempty[2], drain;
    __shared__ int64_t cN[2][kMaxBn];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_word;
    volatile int *abort_flag = &abort_word;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    const uint32_t crank = PAIR ? cluster_ctarank() : 0u;
    const int64_t slot0 = PAIR ? (int64_t)(blockIdx.x >> 1) : (int64_t)blockIdx.x;
    const int64_t nslots = PAIR ? (int64_t)(gridDim.x >> 1) : (int64_t)gridDim.x;
    constexpr uint32_t kCtas = PAIR ? 2u : 1u;
    auto bwait = [&](uint64_t *bar, uint32_t parity) -> bool {
        if constexpr (PAIR) return mbar_wait_cl_or(bar, parity, abort_flag);
        else return mbar_wait_or(bar, parity, abort_flag);
    };
    auto give_up = [&]() {
        *abort_flag = 1;
        atomicExch(d.status, (int)TC_ERROR_TIMEOUT);
    };
    const bool split = !COMP && d.split != 0;
    const int nbuf = split && d.bn > 128 ? 1 : 2;
    const uint32_t small_off = split ? (d.bn > 128 ? 256u : 128u) : 0u;  // the smaller products' accumulator
    if (threadIdx.x == 0) {
        for (int s = 0; s < d.stages; ++s) {
            mbar_init(&full[s], 1);   // the issuing CTA's copy lane arms it for every CTA's bytes
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], kEpiWarps * kCtas);
        }
        mbar_init(&drain, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if constexpr (PAIR) {
        // both CTAs run and their barriers are initialised before any copy
        // or arrival crosses the pair or the pair allocates tensor memory
        cluster_sync_all();
        if (warp == kMmaWarp) tmem_alloc2(&tmem_slot, kTmemCols);
    } else {
        if (warp == kMmaWarp) tmem_alloc(&tmem_slot, kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    // launched as a programmatic dependent of the pre-pass: its images are
    // complete from here on
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t stage_bytes = d.img_a + d.img_b;

    if (warp == kCopyWarp) {
        // --------------------------------------------------------- copies
        const int32_t rows_a = (int32_t)(d.img_a / kMapRow), rows_b = (int32_t)(d.img_b / kMapRow);
        int s = 0;
        uint32_t ph = 1;  // parity of the slot's last release (the first round finds it free)
        bool stop = false;
        for (int64_t tile = slot0; tile < d.num_tiles && !stop; tile += nslots) {
            int64_t mt;
            const int64_t nt = divmod(tile, d.tiles_m, mt);
            int32_t ra = (int32_t)((mt * kCtas + crank) * d.ktiles) * rows_a;
            int32_t rb = (int32_t)((nt * kCtas + crank) * d.ktiles) * rows_b;
            for (int kt = 0; kt < d.ktiles; ++kt, ra += rows_a, rb += rows_b) {
                if (!__all_sync(0xffffffffu, bwait(&empty[s], ph))) {
                    stop = true;
                    break;
                }
                if (elect_one()) {
                    uint32_t bar = smem_u32(&full[s]);
                    if constexpr (PAIR) bar = mapa_shared(bar, 0u);
                    if (crank == 0) mbar_arrive_expect_tx(&full[s], kCtas * stage_bytes);
                    char *dst = ring + s * stage_bytes;
                    image_load<PAIR>(dst, &tmA, bar, ra);
                    image_load<PAIR>(dst + d.img_a, &tmB, bar, rb);
                }
                __syncwarp();
                if (++s == d.stages) s = 0, ph ^= 1u;
            }
        }
        if (stop) {
            if (lane == 0) give_up();
            // copies in flight land (microseconds) before the CTA leaves
            const uint64_t t0 = globaltimer();
            while (globaltimer() - t0 < 2000000ull) {
            }
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        // ----------------------------------------------------- MMA issuer
        // The whole warp runs the loops and waits; one elected lane issues
        if (crank == 0) {
            const uint32_t idesc = (1u << 4) | (T::kFmt << 7) | (T::kFmt << 10) | ((uint32_t)(d.bn >> 3) << 17) |
                                   ((uint32_t)((kCtas * kRows) >> 4) << 24);
            constexpr uint32_t lboA = kRows * 16;
            const uint32_t lboB = (uint32_t)d.brows * 16;
            constexpr uint32_t sliceA = kRows * BK * T::kElemBytes;
            const uint32_t sliceB = (uint32_t)(d.brows * BK * T::kElemBytes);
            const uint32_t base = smem_u32(ring);
            // slice pairs in product order (0,0) (0,1) (1,0) (0,2) (1,1) (2,0)
            // (1,2) (2,1) (2,2), one nibble per product
            constexpr uint64_t kPa = 0x221210100ull, kPb = 0x212012010ull;
            // as, bs: descriptors of the stage's slice 0, first K step; the
            // others differ in the address field only (address >> 4)
            auto issue_stage = [&](auto np, uint64_t as, uint64_t bs, uint32_t dt, bool first, int nks) {
                constexpr int NP = decltype(np)::value;
#pragma unroll
                for (int ks = 0; ks < T::kKsteps; ++ks) {
                    if (ks >= nks) break;
#pragma unroll
                    for (int q = 0; q < NP; ++q) {
                        const uint32_t qa = (uint32_t)(kPa >> (4 * q)) & 15u, qb = (uint32_t)(kPb >> (4 * q)) & 15u;
                        const uint64_t ad = as + (uint64_t)((qa * sliceA + ks * 2 * lboA) >> 4);
                        const uint64_t bd = bs + (uint64_t)((qb * sliceB + ks * 2 * lboB) >> 4);
                        // each accumulator starts from zero with its own
                        // first product of the unit
                        const bool fresh = first && ks == 0 && q == (split && q > 0 ? 1 : 0);
                        mma_issue<KIND, PAIR>(q > 0 ? dt + small_off : dt, ad, bd, idesc, !fresh);
                    }
                }
            };
            auto commit = [&](uint64_t *bar) {
                if constexpr (PAIR) mma_commit2(bar, (uint16_t)3);  // both CTAs' barriers
                else mma_commit(bar);
            };
            const int nch = (d.ktiles + d.chunk - 1) / d.chunk;
            int s = 0, buf = 0;
            uint32_t ph = 0, aph = 1;  // parities: stage filled; accumulator drained (free at first)
            bool stop = false;
            for (int64_t tile = slot0; tile < d.num_tiles && !stop; tile += nslots) {
                int64_t left = d.K;  // K positions from this stage on
                for (int c = 0; c < nch && !stop; ++c) {
                    if (!__all_sync(0xffffffffu, bwait(&tempty[buf], aph))) {
                        stop = true;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t dt = tmem + (uint32_t)(buf * 256);
                    const int k1 = min(d.ktiles, (c + 1) * d.chunk);
                    for (int kt = c * d.chunk; kt < k1; ++kt, left -= BK) {
                        if (!__all_sync(0xffffffffu, bwait(&full[s], ph))) {
                            stop = true;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t sa = base + (uint32_t)s * stage_bytes;
                        const uint64_t as = smem_desc(sa, lboA, 128), bs = smem_desc(sa + d.img_a, lboB, 128);
                        const bool first = kt == c * d.chunk;
                        // K steps of the stage that hold K positions
                        const int nks = left >= BK ? T::kKsteps : (int)((left * T::kElemBytes + 31) / 32);
                        if (elect_one()) {
                            if constexpr (KIND == GK_BF16X3) {
                                if (d.nprod == 6) issue_stage(std::integral_constant<int, 6>{}, as, bs, dt, first, nks);
                                else if (d.nprod == 3) issue_stage(std::integral_constant<int, 3>{}, as, bs, dt, first, nks);
                                else issue_stage(std::integral_constant<int, 9>{}, as, bs, dt, first, nks);
                            } else {
                                issue_stage(std::integral_constant<int, KIND == GK_TF32X3 ? 3 : 1>{}, as, bs, dt, first, nks);
                            }
                            commit(&empty[s]);
                            if (kt + 1 == k1) commit(&tfull[buf]);  // arrives when this unit's MMAs are done
                        }
                        __syncwarp();
                        if (++s == d.stages) s = 0, ph ^= 1u;
                    }
                    if (++buf == nbuf) buf = 0, aph ^= 1u;
                }
            }
            if (stop && lane == 0) give_up();
            // nothing issued may still run when the tensor memory is freed
            if (elect_one()) {
                if constexpr (PAIR) mma_commit2(&drain, (uint16_t)1);
                else mma_commit(&drain);
            }
            __syncwarp();
            mbar_wait(&drain, 0);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------- epilogue
        const int et = threadIdx.x, quad = warp % 4, half = warp / 4;
        const int row = quad * 32 + lane;  // accumulator row = TMEM lane
        const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
        float alpha = d.alpha;
        if constexpr (KIND == GK_E4M3) alpha = d.alpha * d.qscale[0] * d.qscale[1];
        float *__restrict__ C = (float *)d.C;
        const int nch = (d.ktiles + d.chunk - 1) / d.chunk;
        int it = 0, buf = 0;
        uint32_t aph = 0;  // parity: accumulator filled
        constexpr int G = COMP ? 2 : 1;
        float hi[G][32], lo[G][32];
        for (int64_t tile = slot0; tile < d.num_tiles; tile += nslots, ++it) {
            int64_t mt, rem, ignored = 0;
            const int64_t nt = divmod(tile, d.tiles_m, mt);
            const int64_t n0 = nt * d.bn, mm = (mt * kCtas + crank) * kRows + row;
            const int nval = (int)min((int64_t)d.bn, d.N - n0);
            // one stride across the tile's columns where C has one
            int64_t lin = 0, on0 = 0, om = -1;
            int64_t *cn = cN[it & 1];
            if (d.nn > 0 && d.n_chain) {
                lin = d.n_sC[0];
                on0 = n0 * lin;
            } else if (d.nn > 0 && (divmod(n0, d.n_ext[0], rem), rem + nval <= d.n_ext[0])) {
                decode(n0, d.nn, d.n_ext, d.n_sB, d.n_sC, ignored, on0);
                lin = d.n_sC[0];
            } else {
                for (int j = et; j < nval; j += kEpiThreads) {
                    int64_t oc = 0;
                    decode(n0 + j, d.nn, d.n_ext, d.n_sB, d.n_sC, ignored, oc);
                    cn[j] = oc;
                }
            }
            if (mm < d.M) {
                om = 0;
                decode(mm, d.nm, d.m_ext, d.m_sA, d.m_sC, ignored, om);
            }
            if (role_sync_or<2, kEpiThreads>(*abort_flag)) break;
            bool aborted = false;
            for (int c = 0; c < nch; ++c) {
                bool ok = bwait(&tfull[buf], aph);
                ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld needs the whole warp
                if (!ok) {
                    give_up();
                    aborted = true;
                    break;  // the next role barrier sees the abort
                }
                tc_fence_after();
                const uint32_t acc = tmem + lane_off + (uint32_t)(buf * 256);
                if constexpr (COMP) {
                    // 16 columns at a time: 128 registers hold (hi, lo)
                    if (c < nch - 1) {
                        if (c == 0) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) hi[0][j] = hi[1][j] = lo[0][j] = lo[1][j] = 0.0f;
                        }
#pragma unroll
                        for (int gj = 0; gj < 4; ++gj) {
                            uint32_t r[16];
                            tmem_ld16(acc + (uint32_t)(half * 32 + gj / 2 * 64 + gj % 2 * 16), r);
#pragma unroll
                            for (int x = 0; x < 16; ++x) {  // (hi, err) = TwoSum(hi, chunk); lo += err
                                const int gi = gj / 2, j = gj % 2 * 16 + x;
                                const float b = __uint_as_float(r[x]), a = hi[gi][j];
                                const float s2 = __fadd_rn(a, b), bb = __fsub_rn(s2, a);
                                hi[gi][j] = s2;
                                lo[gi][j] = __fadd_rn(lo[gi][j], __fadd_rn(__fsub_rn(a, __fsub_rn(s2, bb)), __fsub_rn(b, bb)));
                            }
                        }
                    } else {
#pragma unroll
                        for (int gj = 0; gj < 4; ++gj) {
                            uint32_t r[16];
                            tmem_ld16(acc + (uint32_t)(half * 32 + gj / 2 * 64 + gj % 2 * 16), r);
#pragma unroll
                            for (int x = 0; x < 16; ++x) {  // result = hi + (lo + chunk): one rounding per step
                                const int gi = gj / 2, j = gj % 2 * 16 + x;
                                hi[gi][j] = __fadd_rn(hi[gi][j], __fadd_rn(lo[gi][j], __uint_as_float(r[x])));
                            }
                        }
                    }
                }
                if constexpr (!COMP) {
#pragma unroll 1
                    for (int c0 = half * 32; c0 < d.bn; c0 += 64) {
                        uint32_t r[32];
                        if (split) tmem_ld32_sum(acc + (uint32_t)c0, acc + small_off + (uint32_t)c0, r);
                        else tmem_ld32(acc + (uint32_t)c0, r);
                        store_row(r, C, om, c0, lin, on0, nval, cn, alpha, d.beta, d.init);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (PAIR) mbar_arrive_remote(mapa_shared(smem_u32(&tempty[buf]), 0u));
                    else mbar_arrive(&tempty[buf]);
                }
                if (++buf == nbuf) buf = 0, aph ^= 1u;
            }
            if (aborted) continue;
            if constexpr (COMP) {
                // (the next tile's first chunk accumulates meanwhile)
#pragma unroll
                for (int gi = 0; gi < 2; ++gi) {
                    const int c0 = half * 32 + gi * 64;
                    if (c0 >= d.bn) break;
                    uint32_t r[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(hi[gi][j]);
                    store_row(r, C, om, c0, lin, on0, nval, cn, alpha, d.beta, d.init);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) {
        // neither CTA frees its tensor memory or leaves while the pair's
        // MMAs, copies or arrivals may still reach it
        cluster_sync_all();
        if (warp == kMmaWarp) {
            tc_fence_after();
            tmem_dealloc2(tmem, kTmemCols);
        }
    } else if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

tc_status image_map(CUtensorMap &map, const void *base, int64_t bytes, uint32_t img) {
    if (!g_encode) {
        cudaDriverEntryPointQueryResult q;
        void *fn = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return fail(TC_ERROR_CUDA, "cuTensorMapEncodeTiled not found");
        g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    // the images as rows of 512 bytes; one box is one stage image
    cuuint64_t gdim[2] = {kMapRow / 4, (cuuint64_t)(bytes / kMapRow)}, gstride[1] = {kMapRow};
    cuuint32_t box[2] = {kMapRow / 4, img / kMapRow}, estr[2] = {1, 1};
    const CUresult r = g_encode(&map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<void *>(base), gdim, gstride, box, estr,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TC_SUCCESS : fail(TC_ERROR_CUDA, "tensor map of the stage images");
}

int sm_count() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

struct Tile {
    bool pair;
    int bn;
};

// Pair or lone CTA and the tile width with the least estimated time: waves of
// tiles times the clocks of one tile.  Per 32 bytes of K a product takes
// bn / 2 clocks of the tensor pipe, or what the shared-memory port needs for
// its operands and its share of the copies; 2500 clocks per tile for filling
// the pipeline and draining the last accumulator.
Tile choose_tile(int64_t M, int64_t N, double ksteps, int nprod, int slices, int max_bn, bool single_buffer_past_128) {
    Tile best{false, 128};
    double best_cost = -1;
    for (int pair = 1; pair >= 0; --pair) {
        const int64_t rows = pair ? 2 * kRows : kRows, slots = pair ? sm_count() / 2 : sm_count();
        if (slots < 1) continue;
        for (int bn = max_bn; bn >= 32; bn -= 16) {
            const int brows = pair ? bn / 2 : bn;
            const double port = ((4096.0 + 32.0 * brows) * nprod + 32.0 * (kRows + brows) * slices) / 128.0;
            const double tile = ksteps * std::max(bn / 2.0 * nprod, port) + 2500.0 +
                                (single_buffer_past_128 && bn > 128 ? 10.0 * bn : 0.0);
            const int64_t tiles = ((M + rows - 1) / rows) * ((N + bn - 1) / bn);
            const double cost = (double)((tiles + slots - 1) / slots) * tile;
            if (best_cost < 0 || cost < best_cost) {
                best_cost = cost;
                best = {pair != 0, bn};
            }
        }
    }
    return best;
}

template <int KIND, bool COMP, bool PAIR>
tc_status launch_gett(const PackedDesc &d, const CUtensorMap &ta, const CUtensorMap &tb, cudaStream_t st) {
    auto kern = packed_gett_kernel<KIND, COMP, PAIR>;
    static bool configured = false;
    if (!configured) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes);
        if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
        configured = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kRingBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
    int64_t grid = std::min<int64_t>(d.num_tiles, sm_count());
    if constexpr (PAIR) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = 2;
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = 1;
        ++na;
        grid = 2 * std::min<int64_t>(d.num_tiles, sm_count() / 2);
    }
    cfg.gridDim = dim3((unsigned)grid);
    cfg.attrs = attr;
    cfg.numAttrs = na;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kern, d, ta, tb);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? TC_SUCCESS : fail(TC_ERROR_CUDA, cudaGetErrorString(e));
}

template <int KIND>
tc_status run_packed(Plan &p, PackedDesc &d, bool comp, int64_t comp_k, double fraction, cudaStream_t st) {
    using T = Traits<KIND>;
    constexpr int BK = stage_k<KIND>();
    const int nprod = KIND == GK_BF16X3 ? d.nprod : (KIND == GK_TF32X3 ? 3 : 1);
    int max_bn = comp ? 128 : (p.gett_bn == 128 ? 128 : kMaxBn);
    Tile t = choose_tile(d.M, d.N, (double)((d.K * T::kElemBytes + 31) / 32), nprod, T::kSlices, max_bn, d.split != 0);
    if (p.gett_pair && d.M > kRows) t.pair = true;
    if (fraction < 1.0) d.N = std::min<int64_t>(d.N, std::max<int64_t>(t.bn, (int64_t)(d.N * fraction)));
    d.bn = t.bn;
    d.brows = t.pair ? t.bn / 2 : t.bn;
    const int64_t rows = t.pair ? 2 * kRows : kRows;
    d.tiles_m = (d.M + rows - 1) / rows;
    d.tiles_n = (d.N + d.bn - 1) / d.bn;
    d.num_tiles = d.tiles_m * d.tiles_n;
    d.ktiles = (int)((d.K + BK - 1) / BK);
    d.chunk = comp ? (int)(comp_k / BK) : d.ktiles;
    d.img_a = (uint32_t)(T::kSlices * kRows * BK * T::kElemBytes);
    d.img_b = (uint32_t)(T::kSlices * d.brows * BK * T::kElemBytes);
    d.stages = std::min<int>(kMaxStages, kRingBytes / (int)(d.img_a + d.img_b));
    PackJob ja = {}, jb = {};
    ja.op = 0;
    ja.rows = kRows;
    ja.total_rows = d.tiles_m * rows;
    jb.op = 1;
    jb.rows = d.brows;
    jb.total_rows = d.tiles_n * d.bn;
    const int64_t bytes_a = ja.total_rows / ja.rows * d.ktiles * (int64_t)d.img_a;
    const int64_t bytes_b = jb.total_rows / jb.rows * d.ktiles * (int64_t)d.img_b;
    tc_status s = ensure_device_resources(p, (size_t)packed_bytes(p.dtype, d.M, d.N, d.K));
    if (s != TC_SUCCESS) return s;
    d.status = p.dev_status;
    ja.out = (char *)p.workspace;
    jb.out = ja.out + bytes_a;
    // lanes along whichever of the first row mode and the innermost K mode
    // has the smaller stride
    ja.rfast = d.nm > 0 && (d.nk == 0 || d.m_sA[0] < d.k_sA[d.nk - 1]);
    jb.rfast = d.nn > 0 && (d.nk == 0 || d.n_sB[0] < d.k_sB[d.nk - 1]);
    const int64_t kblocks = ((int64_t)d.ktiles * BK + kPackK - 1) / kPackK;
    ja.blocks = (ja.total_rows + kPackRows - 1) / kPackRows * kblocks;
    jb.blocks = (jb.total_rows + kPackRows - 1) / kPackRows * kblocks;
    if (ja.blocks + jb.blocks > 0x7fffffff) return fail(TC_ERROR_INVALID_EXTENT, "too many blocks for the pre-pass");
    CUtensorMap ta, tb;
    s = image_map(ta, ja.out, bytes_a, d.img_a);
    if (s == TC_SUCCESS) s = image_map(tb, jb.out, bytes_b, d.img_b);
    if (s != TC_SUCCESS) return s;
    pack_images_kernel<KIND><<<(unsigned)(ja.blocks + jb.blocks), kPackThreads, 0, st>>>(d, ja, jb);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
    if constexpr (KIND == GK_BF16X3 || KIND == GK_TF32X3) {
        if (comp) return t.pair ? launch_gett<KIND, true, true>(d, ta, tb, st) : launch_gett<KIND, true, false>(d, ta, tb, st);
    }
    return t.pair ? launch_gett<KIND, false, true>(d, ta, tb, st) : launch_gett<KIND, false, false>(d, ta, tb, st);
}

}  // namespace

int64_t packed_bytes(tc_dtype dt, int64_t M, int64_t N, int64_t K) {
    int img = 6, bk = stage_k<GK_BF16X3>();
    switch (dt) {
    case TC_BF16:
    case TC_F16: img = 2, bk = stage_k<GK_BF16>(); break;
    case TC_TF32: img = 4, bk = stage_k<GK_TF32>(); break;
    case TC_TF32X3: img = 8, bk = stage_k<GK_TF32X3>(); break;
    case TC_E4M3: img = 1, bk = stage_k<GK_E4M3>(); break;
    default: break;
    }
    // A's rows round up to a pair tile, B's to a tile of at most 256, K to a stage
    return (M + N + 512) * ((K + bk - 1) / bk * bk) * img;
}

tc_status exec_packed(Plan &p, const void *alpha, const void *A, const void *B, const void *beta, void *C, void *stream,
                      double fraction, int64_t comp_k, bool split, const float *qscale) {
    PackedDesc d;
    std::memset(&d, 0, sizeof(d));
    tc_status s = describe_modes(p, 3, d);
    if (s != TC_SUCCESS) return s;
    d.A = A;
    d.B = B;
    d.C = C;
    d.alpha = *(const float *)alpha;
    d.beta = *(const float *)beta;
    d.init = d.beta == 0.0f ? 2 : 1;
    d.nprod = p.split_products;
    d.split = split ? 1 : 0;
    d.qscale = qscale;
    const bool comp = comp_k > 0 && d.K > comp_k;
    cudaStream_t st = (cudaStream_t)stream;
    switch (p.dtype) {
    case TC_BF16X3: return run_packed<GK_BF16X3>(p, d, comp, comp_k, fraction, st);
    case TC_BF16: return run_packed<GK_BF16>(p, d, false, 0, fraction, st);
    case TC_F16: return run_packed<GK_F16>(p, d, false, 0, fraction, st);
    case TC_TF32: return run_packed<GK_TF32>(p, d, false, 0, fraction, st);
    case TC_TF32X3: return run_packed<GK_TF32X3>(p, d, comp, comp_k, fraction, st);
    case TC_E4M3: return run_packed<GK_E4M3>(p, d, false, 0, fraction, st);
    default: return fail(TC_ERROR_UNSUPPORTED_DTYPE, "dtype has no pre-converted GETT");
    }
}

}  // namespace tc
