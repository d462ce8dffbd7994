// The tensor-core GETT with both inputs pre-converted (no paper
// counterpart).  A pre-pass writes each input once as the stage images the
// MMA reads -- per row tile and K stage the slices in the no-swizzle K-major
// core-matrix layout (8 rows x 16 bytes), zeros past the extents -- and the
// GETT copies them: no input is converted more than once, however many tiles
// of the other input it meets, and any strides cost the GETT nothing.
//
// pack_images_kernel: a block takes 32 rows x 128 K positions (256 of 16-bit
// inputs) through shared memory, so that its loads run along the operand's
// contiguous index (rows or K) and its stores are 512-byte runs of an image;
// one launch for both inputs (4096 x 4096 each: BF16 36 us, split-BF16 53 us;
// one 16-byte chunk per thread straight from global memory took 67 and 77 us
// in two launches).
//
// packed_gett_kernel: persistent and warp-specialised, one CTA per SM or a
// pair of CTAs sharing each MMA (cta_group::2):
//   copy warp 9      an elected lane streams each stage's two images with
//                    cp.async.bulk.tensor into a ring (both CTAs of a pair
//                    count their bytes on the issuing CTA's barrier);
//   MMA warp 8       an elected lane issues the stage's slice products;
//   epilogue warps 0-7  drain the accumulators and store C (two groups of
//                    four, alternate tiles or alternate 32 columns).
// Why pairs and these widths: an MMA of N columns takes N / 2 clocks and reads
// 4 KB of A and 32 bytes per row of B held here through the shared-memory
// port (128 bytes per clock), next to the copies' writes.  A lone CTA on
// 128 x 256 BF16 tiles would need 192 bytes per clock, a pair, which holds
// half of B each, 128.  The tile width follows the number of waves
// (choose_tile).  ab=aij,jib 4096^2 i=j=64: BF16 78 us on pairs of 256 x 224
// (lone 128 x 256 98 us, pairs of 256 x 256 in four uneven waves 86 us), split-
// BF16 with compensation 462 us on pairs of 256 x 128 (lone 543 us); BF16
// keeps the tensor pipe active 82 % of the SMs' active cycles.  With the MMAs issued under a branch on the lane
// number the same tiles took 178 and 918 us (elect_one).  The compensated
// sums' (hi, lo) in registers leave the tensor memory to two accumulators.
//
// FP64 (GK_D64): digits.  The FP64 unit runs two multiply-adds per SM and
// clock (1.26 TFLOP/s), so a large FP64 GETT is computed from integers on the
// tensor cores (the digit splitting of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication", 2012):
//   * a row of A (column of B) is scaled by the power of two 2^e just above
//     its largest magnitude and cut into 8 balanced base-256 digits d_s,
//     |d| <= 128 (64 for s = 0), x = 2^e sum_s d_s 2^(-6-8s): 62 bits below
//     2^e, exact as BF16 values;
//   * the products d_s d_t with s + t = l < 8 add up in accumulator l.  A sum
//     over 128 K positions stays within 2^24 in magnitude, so every FP32
//     accumulation is exact, in any order; the epilogue adds the levels as
//     64-bit integers (0-3 and 4-7 apart) and rounds the total once.
// What is left out of a term is at most 8.2 x 2^-62 of 2^(eA + eB): 7 products
// of level 8 (2^-62 each) and past it, an entry's rounding to 62 bits (2^-63 of
// either input) and that of level 7 (0.1 x 2^-62 at K = 32).  Two checks keep
// that small:
//   * the pre-pass counts per row the entries below 2^(e-5): where those of a
//     row of A and of a column of B are together at most K / 2, at least K / 2
//     terms of the sum are at least 2^(eA+eB-10), and what is left out is at
//     most 2^-47.9 |A||B|, under the K 2^-53 of a chain of fused multiply-adds
//     from K = 34 on.  Tiles where that does not hold (wide ranges or many
//     zeros along K, infinities, NaN, exponents near the ends) go to a list.
//   * where large terms cancel, |A||B| says little about the result: a chain may
//     be exact where small terms are left beside them.  So a result v is stored
//     only where it is at least 2^-10 2^(eA + eB), the error then at most
//     K 2^-48.9 |v| whatever the terms, and marked otherwise: one of 7000 on
//     uniform entries at K = 256, one of 1300 on normal ones.
// Both are left to the chain (tc_exec.cu, left_kernel).  On uniform and normal
// entries little but the last rounding is lost (5e-17 of the result, 6e-16 in
// the chain).
// B is taken in panels whose images stay in L2.
// abc=iaj,jbic 512^3 i=j=16: 56.7 -> 2.95 ms (18 panels: pre-pass 23 us, GETT
// 137 us each, 128 without the check of the results; left_kernel 60 us.  Of
// the 128, 92 without the drains and conversions; 135 where every product
// reads its digit of A from shared memory, not from the collector buffer, 153
// with a conversion that branches).
//
// FP32 stays on the SIMT tiles.  Four digits (10 products, 0.59 ms against
// 1.83 on the same contraction with uniform entries) hold 30 bits below the
// largest entry of a row, six more than an entry has: where large terms
// cancel, small ones that a chain keeps are lost (7e-5 of the result against
// 2e-7), and the check of every result that would refuse such sums refuses
// about 1 % of ordinary ones.
//
// Every wait on an mbarrier is bounded; on expiry the kernel records
// TC_ERROR_TIMEOUT, stops issuing, drains, frees its tensor memory, returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "tc_gett.cuh"
#include "tc_internal.h"
#include "tc_ring.h"

namespace tc {

namespace {

using namespace dev;

constexpr int kRows = 128;                 // accumulator rows per CTA = TMEM lanes
constexpr int kRingBytes = 192 * 1024;     // operand ring
constexpr int kMaxStages = 8;
constexpr int kMaxBn = 256;
constexpr int kEpiWarps = 8;
constexpr int kMmaWarp = kEpiWarps, kCopyWarp = kEpiWarps + 1;
constexpr int kThreads = (kCopyWarp + 1) * 32;
constexpr uint32_t kTmemCols = 512;
constexpr int kMapRow = 512;               // bytes per row of an image tensor map
constexpr unsigned long long kLandNs = 2000000;  // copies on their way land within this (microseconds)

// K positions per stage: about 32-48 KB of images per CTA
template <int KIND>
__host__ __device__ constexpr int stage_k() {
    return KIND == GK_TF32X3 || KIND == GK_D64 ? 16 : ((KIND == GK_BF16 || KIND == GK_F16 || KIND == GK_E4M3) ? 64 : 32);
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
    int64_t n_begin;            // first column of the panel (N then counts the panel's)
    // digits: scalars in FP64, per row the exponent field of its largest
    // magnitude (0: a row of zeros), per image row tile the most small entries
    // of a row, and the tiles left to SIMT (list[0]: how many, from list[2] on)
    double alpha64, beta64;
    int *exps[2], *small[2];
    int64_t *list;
    // results left to the chain: a bit per column of 32 for each row of A's
    // images, the columns from weak_n0 on
    uint32_t *weak;
    int64_t weak_n0, rows_a, weak_below;
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

constexpr int kPackRows = 32, kPackThreads = 256;
// K positions a block takes: enough loads in flight at two bytes each
template <int KIND>
__host__ __device__ constexpr int pack_k() {
    return KIND == GK_BF16 || KIND == GK_F16 ? 256 : 128;
}

template <int KIND>
__global__ void __launch_bounds__(kPackThreads) pack_images_kernel(const __grid_constant__ PackedDesc d,
                                                                   const PackJob ja, const PackJob jb) {
    using T = Traits<KIND>;
    constexpr int BK = stage_k<KIND>(), CH = T::kChunk, kPackK = pack_k<KIND>();
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
        static_assert(kPackK <= kPackThreads, "one thread per K offset");
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
    }
    if (warp == kPackThreads / 32 - 1) {
        int64_t r = r0 + lane, o = -1, u = 0;
        if (r < (J.op == 0 ? d.M : d.N)) {
            o = 0;
            if (J.op == 0) decode(r, d.nm, d.m_ext, d.m_sA, d.m_sC, o, u);
            else decode(r + d.n_begin, d.nn, d.n_ext, d.n_sB, d.n_sC, o, u);
        }
        roff[lane] = o;
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

// ---- digits
constexpr int kDigitLow = 623, kDigitHigh = 1423;  // exponent fields taken
constexpr int kDigitChunkK = 128;         // K positions per accumulation
constexpr int kDigitBn = 64;              // columns per tile: eight levels fill the tensor memory
// Past it the images of A and of a panel of B hold fewer tiles than SMs, and no
// size is estimated faster than SIMT (the summed levels stay below 2^52).
constexpr int64_t kDigitMaxK = 1 << 15;
constexpr int kRowBad = 1 << 29;
constexpr int kDigitK = 256;  // K positions a block holds at a time

// One input as digit images: a block takes 32 rows; K positions stay in
// registers between the search for the largest magnitudes and the digits (a
// longer K is read twice, the second time mostly from L2).
__global__ void __launch_bounds__(kPackThreads, 2) pack_digits_kernel(const __grid_constant__ PackedDesc d,
                                                                      const PackJob ja, const PackJob jb) {
    constexpr int BK = stage_k<GK_D64>(), S = Traits<GK_D64>::kSlices, P = kPackRows + 1;
    extern __shared__ __align__(16) unsigned char dsm[];
    double *tile = (double *)dsm;  // [kDigitK][P]
    __shared__ int64_t koff[kDigitK], roff[kPackRows];
    __shared__ unsigned emax[kPackRows];
    __shared__ int nlarge[kPackRows];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool second = blockIdx.x >= ja.blocks;
    const PackJob &J = second ? jb : ja;
    const int64_t r0 = (second ? (int64_t)blockIdx.x - ja.blocks : (int64_t)blockIdx.x) * kPackRows;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const double *__restrict__ src = (const double *)(J.op == 0 ? d.A : d.B);
    if (tid < kPackRows) {
        int64_t r = r0 + tid, o = -1, u = 0;
        if (r < (J.op == 0 ? d.M : d.N)) {
            o = 0;
            if (J.op == 0) decode(r, d.nm, d.m_ext, d.m_sA, d.m_sC, o, u);
            else decode(r + d.n_begin, d.nn, d.n_ext, d.n_sB, d.n_sC, o, u);
        }
        roff[tid] = o;
        emax[tid] = 0;
        nlarge[tid] = 0;
    }
    constexpr int NL = kDigitK * kPackRows / kPackThreads, KJ = kDigitK / 32;
    double x[NL];
    auto load = [&](int64_t k0) {  // (a barrier on both sides of the offset table)
        __syncthreads();
        static_assert(kDigitK == kPackThreads, "one thread per K offset");
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
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const int64_t ro = roff[J.rfast ? lane : warp * 4 + j / KJ];
            const int64_t ko = koff[J.rfast ? warp + 8 * j : lane + 32 * (j % KJ)];
            x[j] = ro >= 0 && ko >= 0 ? __ldg(src + ro + ko) : 0.0;
        }
    };
    // largest magnitude: the high word of |x| with a bit for a nonzero low
    // word, ordered as integers
    auto mag = [](double v) -> unsigned {
        const unsigned long long b = __double_as_longlong(v);
        return ((unsigned)(b >> 32) & 0x7fffffffu) | ((unsigned)b != 0 ? 1u : 0u);
    };
    unsigned mx[4] = {0, 0, 0, 0};
    for (int64_t k0 = 0; k0 < d.K; k0 += kDigitK) {
        load(k0);
#pragma unroll
        for (int j = 0; j < NL; ++j) mx[(j / KJ) & 3] = max(mx[(j / KJ) & 3], mag(x[j]));
    }
    if (J.rfast) {
        atomicMax(&emax[lane], max(max(mx[0], mx[1]), max(mx[2], mx[3])));
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned m = __reduce_max_sync(0xffffffffu, mx[i]);
            if (lane == 0) emax[warp * 4 + i] = m;
        }
    }
    __syncthreads();
    const unsigned top = emax[lane];
    const int E = (int)(top >> 20);
    const int64_t R = r0 + lane;
    int64_t rr;
    const int64_t rt = divmod(R, J.rows, rr);
    const int slice = J.rows * BK * 2;
    char *out = J.out + rt * d.ktiles * (int64_t)(S * slice) + (rr / 8) * 128 + (rr % 8) * 16;
    int large = 0;
    const bool once = d.K <= kDigitK;
    for (int64_t k0 = 0; k0 < (int64_t)d.ktiles * BK; k0 += kDigitK) {
        if (!once) load(k0);
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            if (J.rfast) tile[(warp + 8 * j) * P + lane] = x[j];
            else tile[(lane + 32 * (j % KJ)) * P + warp * 4 + j / KJ] = x[j];
        }
        __syncthreads();
#pragma unroll 1
        for (int c = warp; c < kDigitK / 8; c += kPackThreads / 32) {  // chunks of 8 K positions
            const int64_t k = k0 + c * 8;
            if (R >= J.total_rows || k >= (int64_t)d.ktiles * BK) break;
            char *dst = out + (k / BK) * (int64_t)(S * slice) + (int)((k % BK) / 8) * (J.rows / 8) * 128;
            constexpr int kLarge = 4;  // large: exponent field at least the row's minus this
            unsigned long long y[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const unsigned long long b = __double_as_longlong(tile[(c * 8 + e) * P + lane]);
                const unsigned long long frac = b & ((1ull << 52) - 1);
                const int ex = (int)(b >> 52) & 2047;
                const unsigned long long m = ex ? frac | (1ull << 52) : frac;
                const int sh = E - (ex ? ex : 1);
                large += m != 0 && sh <= kLarge;
                // x 2^-e 2^62 = m 2^(9 - sh), rounded where bits fall
                // under the last digit
                unsigned long long w;
                if (sh <= 9) w = m << (9 - sh);
                else w = sh <= 62 ? (m + (1ull << (sh - 10))) >> (sh - 9) : 0ull;
                if (b >> 63) w = 0ull - w;
                y[e] = w + 0x8080808080808080ull;  // bytes: digit + 128
            }
#pragma unroll
            for (int s = 0; s < S; ++s) {
                // 2^23 + byte as FP32 less 2^23 + 128: the digit, whose
                // upper half is its BF16 value
                constexpr unsigned kMagic = 0x4B000000u;
                const int byte = S - 1 - s;
                unsigned q[4];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    float f[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const unsigned word = (unsigned)(y[e + h] >> (byte >= 4 ? 32 : 0));
                        f[h] = __uint_as_float(__byte_perm(word, kMagic, 0x7440 | (byte & 3))) - 8388736.0f;
                    }
                    q[e / 2] = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632);
                }
                *(uint4 *)(dst + (int64_t)s * slice) = make_uint4(q[0], q[1], q[2], q[3]);
            }
        }
    }
    atomicAdd(&nlarge[lane], large);
    __syncthreads();
    if (tid < kPackRows && R < J.total_rows) {  // warp 0: lane = row
        int few = (int)min(d.K, (int64_t)kRowBad) - nlarge[lane];
        if (top == 0) few = 0;  // a row of zeros (or past the extent): exact
        else if (E < kDigitLow || E > kDigitHigh) few = kRowBad;
        d.exps[J.op][R] = E;  // (0: zeros, of a row that is taken)
        if (few > 0) atomicMax(&d.small[J.op][(J.op == 0 ? 0 : d.n_begin / J.rows) + rt], few);
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

// This thread's row of W accumulator columns c0.. (C offset om, -1: none): the
// columns at on0 + j*lin when lin != 0, else through the table cn.
template <int W>
__device__ __forceinline__ void load_old(float (&old)[W], const float *__restrict__ C, int64_t om, int c0, int64_t lin,
                                         int64_t on0, int nval, const int64_t *cn) {
    if (om < 0) return;
    if (lin != 0 && c0 + W <= nval) {
        const float *p = C + om + on0 + (int64_t)c0 * lin;
#pragma unroll
        for (int j = 0; j < W; ++j) old[j] = p[j * lin];
        return;
    }
#pragma unroll
    for (int j = 0; j < W; ++j)
        if (c0 + j < nval) old[j] = C[om + (lin != 0 ? on0 + (int64_t)(c0 + j) * lin : cn[c0 + j])];
}

template <int W>
__device__ __forceinline__ void store_row(const uint32_t (&r)[W], const float (&old)[W], float *__restrict__ C, int64_t om,
                                          int c0, int64_t lin, int64_t on0, int nval, const int64_t *cn, float alpha,
                                          float beta, int init) {
    if (om < 0) return;
    if (lin != 0 && c0 + W <= nval) {  // (no test per column: the common case)
        float *p = C + om + on0 + (int64_t)c0 * lin;
        if (init == 2) {
#pragma unroll
            for (int j = 0; j < W; ++j) p[j * lin] = alpha * __uint_as_float(r[j]);
        } else {
#pragma unroll
            for (int j = 0; j < W; ++j) p[j * lin] = fmaf(beta, old[j], alpha * __uint_as_float(r[j]));
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < W; ++j) {
        if (c0 + j >= nval) continue;
        float v = alpha * __uint_as_float(r[j]);
        if (init == 1) v = fmaf(beta, old[j], v);
        C[om + (lin != 0 ? on0 + (int64_t)(c0 + j) * lin : cn[c0 + j])] = v;
    }
}

// store_row with few registers: old values read eight at a time ahead of the
// stores.
__device__ __forceinline__ void store_row_low(const uint32_t (&r)[32], float *__restrict__ C, int64_t om, int c0,
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

// (hi 2^24 + lo) 2^s rounded to nearest even, |hi| < 2^58; the result is zero
// or a normal number.  Without branches (about 50 integer instructions) and
// without the FP64 unit, which takes 16 clocks for a warp's instruction.
__device__ __forceinline__ double fixed_to_double(int64_t hi, int64_t lo, int s) {
    // the magnitude times 2^8 in three words
    const int64_t h = hi + (lo >> 24);
    const uint32_t sg = (uint32_t)((int32_t)(h >> 32) >> 31);
    uint32_t w0 = ((uint32_t)lo << 8) ^ sg, w1 = (uint32_t)h ^ sg, w2 = (uint32_t)(h >> 32) ^ sg;
    asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;" : "+r"(w0), "+r"(w1), "+r"(w2) : "r"(sg));
    // the leading one to bit 31 of w2
    int e = s + 87 + 1022;
    bool c = w2 == 0;
    w2 = c ? w1 : w2, w1 = c ? w0 : w1, w0 = c ? 0 : w0, e -= c ? 32 : 0;
    c = w2 == 0;
    w2 = c ? w1 : w2, w1 = c ? w0 : w1, e -= c ? 32 : 0;
    const int z = __clz((int)w2);
    const uint32_t top = __funnelshift_l(w1, w2, z), mid = __funnelshift_l(w0, w1, z), end = w0 << z;
    // 53 bits, the rest and a sticky bit
    uint32_t mh = top >> 11, ml = __funnelshift_r(mid, top, 11);
    const uint32_t rest = mid << 21 | (end != 0 ? 1u : 0u);
    const uint32_t up = rest + (ml & 1u) > 0x80000000u ? 1u : 0u;
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(ml), "+r"(mh) : "r"(up));
    mh = (mh + ((uint32_t)(e - z) << 20)) | (sg & 0x80000000u);
    return __hiloint2double((int)(w2 == 0 ? 0u : mh), (int)ml);
}

// COMP: compensated accumulation -- units of d.chunk K stages, double-buffered
// in tensor memory, each folded by TwoSum into a (hi, lo) pair that the
// epilogue threads hold in registers (64 columns each: bn <= 128).  Otherwise
// one unit per tile: one accumulator, or with d.split two (the (0,0) products
// apart; bn <= 128), double-buffered.
template <int KIND, bool COMP, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
packed_gett_kernel(const __grid_constant__ PackedDesc d, const __grid_constant__ CUtensorMap tmA,
                   const __grid_constant__ CUtensorMap tmB) {
    using T = Traits<KIND>;
    constexpr int BK = stage_k<KIND>();
    extern __shared__ __align__(128) char ring[];
    __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], tfull[2], tempty[2], drain;
    // The epilogue: two groups of four warps take alternate tiles, each its
    // own accumulator, so that one tile's index arithmetic, waits and memory
    // latencies overlap the other's stores; where a tile needs every register
    // (compensated) or all of the tensor memory (FP64 digits), the groups
    // share a tile, alternate 32 columns each.
    constexpr bool kAlt = !COMP && KIND != GK_D64;
    constexpr int kGroupWarps = kAlt ? kEpiWarps / 2 : kEpiWarps;
    __shared__ int64_t cN[kAlt ? 4 : 2][kMaxBn];
    constexpr bool DIG = KIND == GK_D64;
    __shared__ int cE[DIG ? 2 : 1][DIG ? kDigitBn : 1];  // digits: exponent fields of the tile's columns
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
    const int nbuf = KIND == GK_D64 ? 1 : 2;
    const uint32_t small_off = split ? 128u : 0u;  // the smaller products' accumulator (bn <= 128)
    if (threadIdx.x == 0) {
        for (int s = 0; s < d.stages; ++s) {
            mbar_init(&full[s], 1);   // the issuing CTA's copy lane arms it for every CTA's bytes
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], kGroupWarps * kCtas);
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
    // digits: a tile with too many small entries is left to SIMT
    auto skip = [&](int64_t mt, int64_t nt) -> bool {
        if constexpr (!DIG) return false;
        const int64_t na = mt * kCtas, nb = d.n_begin / d.brows + nt * kCtas;
        int a = d.small[0][na], b = d.small[1][nb];
        if constexpr (PAIR) {
            a = max(a, d.small[0][na + 1]);
            b = max(b, d.small[1][nb + 1]);
        }
        return 2 * ((int64_t)a + b) > d.K;
    };

    if (warp == kCopyWarp) {
        // --------------------------------------------------------- copies
        const int32_t rows_a = (int32_t)(d.img_a / kMapRow), rows_b = (int32_t)(d.img_b / kMapRow);
        int s = 0;
        uint32_t ph = 1;  // parity of the slot's last release (the first round finds it free)
        int64_t filled = 0;
        bool stop = false;
        for (int64_t tile = slot0; tile < d.num_tiles && !stop; tile += nslots) {
            int64_t mt;
            const int64_t nt = divmod(tile, d.tiles_m, mt);
            if (skip(mt, nt)) continue;
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
                ++filled;
                if (++s == d.stages) s = 0, ph ^= 1u;
            }
        }
        if (stop && lane == 0) give_up();
        // the last copies have landed before the CTA may leave (a pair's arrive
        // on the first CTA's barriers, and neither leaves before both are done)
        if (crank == 0) last_filled(filled, d.stages, [&](int i, uint32_t parity) { mbar_wait(&full[i], parity, kLandNs); });
        // a pair: the first CTA may have stopped before it counted a copy of the
        // second's
        if (PAIR && stop) {
            const uint64_t t0 = globaltimer();
            while (globaltimer() - t0 < kLandNs) {
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
            // digits: product d_s d_t into accumulator s + t
            auto issue_digits = [&](uint64_t as, uint64_t bs, uint32_t dt, bool first, int nks) {
                constexpr int S = T::kSlices;
#pragma unroll
                for (int ks = 0; ks < T::kKsteps; ++ks) {
                    if (ks >= nks) break;
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int t = 0; t < S - s; ++t) {
                            const uint32_t dst = dt + (uint32_t)((s + t) * kDigitBn);
                            const uint64_t ad = as + (uint64_t)((s * sliceA + ks * 2 * lboA) >> 4);
                            const uint64_t bd = bs + (uint64_t)((t * sliceB + ks * 2 * lboB) >> 4);
                            const bool acc = !(first && ks == 0 && s == 0);
                            if (s == S - 1) mma_issue<KIND, PAIR>(dst, ad, bd, idesc, acc);
                            else if (t == 0) mma_issue_same_a<PAIR, 0>(dst, ad, bd, idesc, acc);
                            else if (t == S - s - 1) mma_issue_same_a<PAIR, 2>(dst, ad, bd, idesc, acc);
                            else mma_issue_same_a<PAIR, 1>(dst, ad, bd, idesc, acc);
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
                if constexpr (DIG) {
                    int64_t mt;
                    const int64_t nt = divmod(tile, d.tiles_m, mt);
                    if (skip(mt, nt)) continue;
                }
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
                            if constexpr (DIG) {
                                issue_digits(as, bs, dt, first, nks);
                            } else if constexpr (KIND == GK_BF16X3) {
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
        constexpr int kGroup = kGroupWarps * 32;
        const int et = threadIdx.x % kGroup, quad = warp % 4;
        const int grp = kAlt ? warp / 4 : 0, half = kAlt ? 0 : warp / 4;
        constexpr int kColStep = kAlt ? 32 : 64;
        const int row = quad * 32 + lane;  // accumulator row = TMEM lane
        const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
        float alpha = d.alpha;
        if constexpr (KIND == GK_E4M3) alpha = d.alpha * d.qscale[0] * d.qscale[1];
        float *__restrict__ C = (float *)d.C;
        const int nch = (d.ktiles + d.chunk - 1) / d.chunk;
        int it = 0, buf = kAlt ? grp : 0;
        int64_t seen = 0;  // tiles accumulated
        uint32_t aph = 0;  // parity: accumulator filled
        int64_t dhi[32], dlo[32];  // FP64 digits: levels 0-3 (units of 2^-36) and 4-7 (2^-60), 32 columns
        const bool plain = d.init == 2 && d.alpha64 == 1.0;
        constexpr int G = COMP ? 2 : 1;
        float hi[G][32], lo[G][32];
        for (int64_t tile = slot0; tile < d.num_tiles; tile += nslots) {
            int64_t mt, rem, ignored = 0;
            const int64_t nt = divmod(tile, d.tiles_m, mt);
            if (skip(mt, nt)) {
                if (threadIdx.x == 0 && crank == 0) {
                    const unsigned long long at = atomicAdd((unsigned long long *)d.list, 1ull);
                    d.list[2 + at] = mt + d.tiles_m * (d.n_begin / d.bn + nt);
                }
                continue;
            }
            if (kAlt && (int)(seen++ & 1) != grp) continue;  // the other group's
            ++it;
            const int64_t n0 = d.n_begin + nt * d.bn, mm = (mt * kCtas + crank) * kRows + row;
            const int nval = (int)min((int64_t)d.bn, d.N - nt * d.bn);
            // one stride across the tile's columns where C has one
            int64_t lin = 0, on0 = 0, om = -1;
            const int tab = kAlt ? 2 * grp + (it & 1) : it & 1;
            int64_t *cn = cN[tab];
            if (d.nn > 0 && d.n_chain) {
                lin = d.n_sC[0];
                on0 = n0 * lin;
            } else if (d.nn > 0 && (divmod(n0, d.n_ext[0], rem), rem + nval <= d.n_ext[0])) {
                decode(n0, d.nn, d.n_ext, d.n_sB, d.n_sC, ignored, on0);
                lin = d.n_sC[0];
            } else {
                for (int j = et; j < nval; j += kGroup) {
                    int64_t oc = 0;
                    decode(n0 + j, d.nn, d.n_ext, d.n_sB, d.n_sC, ignored, oc);
                    cn[j] = oc;
                }
            }
            if (mm < d.M) {
                om = 0;
                decode(mm, d.nm, d.m_ext, d.m_sA, d.m_sC, ignored, om);
            }
            int rowE = 0;
            if constexpr (DIG) {
                rowE = d.exps[0][mm];  // (padded rows have one too)
                for (int j = et; j < d.bn; j += kGroup) cE[tab][j] = d.exps[1][nt * d.bn + j];
            }
            const bool quit = grp == 0 ? role_sync_or<2, kGroup>(*abort_flag) : role_sync_or<3, kGroup>(*abort_flag);
            if (quit) break;
            bool aborted = false;
            // the old values of the first columns are on their way before
            // the accumulator is waited for, those of the next ones once the
            // stores have used the last (a column at a time each cost a memory
            // latency: 46 us for 24 MB of C; the compensated form has no
            // registers for it)
            float old[32];
            if (!COMP && KIND != GK_D64 && d.init == 1) load_old(old, C, om, half * 32, lin, on0, nval, cn);
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
                if constexpr (KIND == GK_D64) {
                    if (c == 0) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) dhi[j] = dlo[j] = 0;
                    }
                    // integers from integral FP32 values without conversion
                    // instructions (which run at a few lanes per clock):
                    // adding 1.5 2^23 leaves |v| <= 2^22 in the low bits, a
                    // larger v goes in two halves, v = 256 h + l
                    constexpr float kAdd = 12582912.0f;
                    constexpr unsigned kAddBits = 0x4B400000u;
                    auto small_int = [&](float v) -> int { return (int)(__float_as_uint(__fadd_rn(v, kAdd)) - kAddBits); };
                    auto big_int = [&](float v) -> int {
                        const float h = __fmaf_rn(v, 0.00390625f, kAdd), l = __fmaf_rn(__fsub_rn(h, kAdd), -256.0f, v);
                        return (int)(__float_as_uint(h) * 256u + __float_as_uint(__fadd_rn(l, kAdd)) - kAddBits * 257u);
                    };
#pragma unroll
                    for (int g4 = 0; g4 < 8; ++g4) {  // four columns of every level at a time
                        uint32_t r[32];
                        tmem_ld8x4(tmem + lane_off + (uint32_t)(half * 32 + g4 * 4), kDigitBn, r);
                        auto lev = [&](int n, int j) { return __uint_as_float(r[n * 4 + j]); };
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            // levels 0 to 2: |i| <= 2^22; level 7 joins level
                            // 6 rounded (to at most half its unit)
                            const int i01 = small_int(lev(0, j)) * 256 + small_int(lev(1, j));
                            const int i23 = small_int(lev(2, j)) * 256 + big_int(lev(3, j));
                            dhi[g4 * 4 + j] += (int64_t)i01 * 65536 + i23;
                            dlo[g4 * 4 + j] += (int64_t)big_int(lev(4, j)) * 65536 + (int64_t)big_int(lev(5, j)) * 256 +
                                               big_int(__fmaf_rn(lev(7, j), 0.00390625f, lev(6, j)));
                        }
                    }
                }
                if constexpr (KIND != GK_D64 && !COMP) {
#pragma unroll 1
                    for (int c0 = half * 32; c0 < d.bn; c0 += kColStep) {
                        uint32_t r[32];
                        if (split) tmem_ld32_sum(acc + (uint32_t)c0, acc + small_off + (uint32_t)c0, r);
                        else tmem_ld32(acc + (uint32_t)c0, r);
                        store_row(r, old, C, om, c0, lin, on0, nval, cn, alpha, d.beta, d.init);
                        if (d.init == 1 && c0 + kColStep < d.bn) load_old(old, C, om, c0 + kColStep, lin, on0, nval, cn);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (PAIR) mbar_arrive_remote(mapa_shared(smem_u32(&tempty[buf]), 0u));
                    else mbar_arrive(&tempty[buf]);
                }
                if (kAlt) aph ^= 1u;
                else if (++buf == nbuf) buf = 0, aph ^= 1u;
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
                    store_row_low(r, C, om, c0, lin, on0, nval, cn, alpha, d.beta, d.init);
                }
            }
            if constexpr (KIND == GK_D64) {
                // (the next tile accumulates meanwhile)
                const int *ce = cE[tab];
                uint32_t weak = 0;
                if (om >= 0 && rowE != 0) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if ((uint64_t)(dhi[j] + d.weak_below) < (uint64_t)(2 * d.weak_below) && ce[half * 32 + j] != 0) weak |= 1u << j;
                }
                // a patch of 32 x 32 with many of them is left as a whole
                if (__reduce_add_sync(0xffffffffu, __popc(weak)) > kWeakMax) weak = ~0u;
                d.weak[((n0 - d.weak_n0) / 32 + half) * d.rows_a + mm] = weak;
                if (om >= 0) {
                    double *at = (double *)d.C + om + (lin != 0 ? on0 + half * 32 * lin : 0);
#pragma unroll
                    for (int j = 0; j < 32; ++j, at += lin) {
                        const int cc = half * 32 + j;
                        if (cc >= nval) break;
                        double *q = lin != 0 ? at : at + cn[cc];
                        const double v = fixed_to_double(dhi[j], dlo[j], rowE + ce[cc] - 2104);
                        if (plain) *q = v;
                        else if (d.init == 2) *q = fma(d.alpha64, v, 0.0);  // (+0 where the chain has it)
                        else if (!(weak & 1u << j)) *q = fma(d.alpha64, v, d.beta64 * *q);  // (the chain needs the old value)
                    }
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
Tile choose_tile(int64_t M, int64_t N, double ksteps, int nprod, int slices, int max_bn) {
    Tile best{false, 128};
    double best_cost = -1;
    for (int pair = 1; pair >= 0; --pair) {
        const int64_t rows = pair ? 2 * kRows : kRows, slots = pair ? sm_count() / 2 : sm_count();
        if (slots < 1) continue;
        for (int bn = max_bn; bn >= 32; bn -= 16) {
            const int brows = pair ? bn / 2 : bn;
            const double port = ((4096.0 + 32.0 * brows) * nprod + 32.0 * (kRows + brows) * slices) / 128.0;
            const double tile = ksteps * std::max(bn / 2.0 * nprod, port) + 2500.0;
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
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes);
    if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
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
    e = cudaLaunchKernelEx(&cfg, kern, d, ta, tb);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? TC_SUCCESS : fail(TC_ERROR_CUDA, cudaGetErrorString(e));
}

// Images of one panel of B.  The digit forms read each panel several times
// their own time: half of L2.  The others spend less time per byte, and more
// launches cost more than reading the images from HBM (split-BF16 512^3
// iaj,jbic: 7 panels of 64 MiB 122 us of pre-pass and 290 us of GETT, one of
// 402 MB 102 and 257 us).
constexpr int64_t kDigitPanelBytes = int64_t(64) << 20;  // (a tile takes 32 MiB at most)
constexpr int64_t kPanelBytes = int64_t(512) << 20;
constexpr int64_t kScratchMaxABytes = int64_t(256) << 20;

// Scratch that an execute can do without: taken once, outside a capture, and
// kept.  False: not to be had, the caller runs the form without it, and the
// plan does not ask for as much again.  Another thread's global-mode capture
// is not to fail for it, so the allocation runs in relaxed mode.  A larger one
// keeps the smaller until the plan goes: graphs may hold its address.
bool optional_scratch(Plan &p, int64_t bytes, cudaStream_t st) {
    if (p.scratch_bytes >= (size_t)bytes) return true;
    if ((size_t)bytes >= p.scratch_refused) return false;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    void *mem = nullptr;
    const cudaError_t e = cudaMalloc(&mem, (size_t)bytes);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) {
        cudaGetLastError();
        p.scratch_refused = (size_t)bytes;
        return false;
    }
    if (p.scratch) p.scratch_old.push_back(p.scratch);
    p.scratch = mem;
    p.scratch_bytes = (size_t)bytes;
    return true;
}

// Tiles of B per panel: whole waves where B takes several panels.
int64_t panel_tiles_for(int64_t panel_bytes, int64_t tiles_n, int64_t tiles_m, int64_t tile_bytes, int64_t slots) {
    int64_t pt = std::max<int64_t>(1, panel_bytes / tile_bytes);
    if (pt < tiles_n && pt * tiles_m > slots) pt = std::max<int64_t>(1, pt * tiles_m / slots * slots / tiles_m);
    return std::min(pt, tiles_n);
}

// done == nullptr: the images in the plan's workspace, B as a whole.  Else in
// optional scratch, B in panels; *done tells whether it ran.
template <int KIND>
tc_status run_packed(Plan &p, PackedDesc &d, bool comp, int64_t comp_k, double fraction, cudaStream_t st, bool *done) {
    using T = Traits<KIND>;
    constexpr int BK = stage_k<KIND>();
    const int nprod = KIND == GK_BF16X3 ? d.nprod : (KIND == GK_TF32X3 ? 3 : 1);
    // (split accumulators: 128 columns leave room for two pairs of them, 257
    // against 289 us on 512^3 iaj,jbic)
    const int max_bn = comp || d.split || p.gett_bn == 128 ? 128 : kMaxBn;
    d.ktiles = (int)((d.K + BK - 1) / BK);
    const int64_t col_bytes = (int64_t)d.ktiles * BK * T::kSlices * T::kElemBytes;
    const int64_t panel_n = done ? std::min(d.N, std::max<int64_t>(kMaxBn, kPanelBytes / col_bytes)) : d.N;
    Tile t = choose_tile(d.M, panel_n, (double)((d.K * T::kElemBytes + 31) / 32), nprod, T::kSlices, max_bn);
    if (p.gett_pair && d.M > kRows) t.pair = true;
    const int64_t N = fraction < 1.0 ? std::min<int64_t>(d.N, std::max<int64_t>(t.bn, (int64_t)(d.N * fraction))) : d.N;
    d.bn = t.bn;
    d.brows = t.pair ? t.bn / 2 : t.bn;
    const int64_t rows = t.pair ? 2 * kRows : kRows;
    d.tiles_m = (d.M + rows - 1) / rows;
    d.chunk = comp ? (int)(comp_k / BK) : d.ktiles;
    d.img_a = (uint32_t)(T::kSlices * kRows * BK * T::kElemBytes);
    d.img_b = (uint32_t)(T::kSlices * d.brows * BK * T::kElemBytes);
    d.stages = std::min<int>(kMaxStages, kRingBytes / (int)(d.img_a + d.img_b));
    const int64_t tiles_n = (N + d.bn - 1) / d.bn;
    const int64_t panel = done ? panel_tiles_for(kPanelBytes, (d.N + d.bn - 1) / d.bn, d.tiles_m, d.bn * col_bytes, sm_count() / (t.pair ? 2 : 1))
                               : tiles_n;
    const int64_t bytes_a = d.tiles_m * rows * col_bytes, bytes_b = panel * d.bn * col_bytes;
    tc_status s = ensure_device_resources(p, done ? 0 : (size_t)packed_bytes(p.dtype, d.M, N, d.K));
    if (s != TC_SUCCESS) return s;
    if (done && (bytes_a > kScratchMaxABytes || !optional_scratch(p, bytes_a + bytes_b, st))) return TC_SUCCESS;
    d.status = p.dev_status;
    PackJob ja = {}, jb = {};
    ja.op = 0;
    ja.rows = kRows;
    ja.total_rows = d.tiles_m * rows;
    ja.out = (char *)(done ? p.scratch : p.workspace);
    jb.op = 1;
    jb.rows = d.brows;
    jb.out = ja.out + bytes_a;
    // lanes along whichever of the first row mode and the innermost K mode
    // has the smaller stride
    ja.rfast = d.nm > 0 && (d.nk == 0 || d.m_sA[0] < d.k_sA[d.nk - 1]);
    jb.rfast = d.nn > 0 && (d.nk == 0 || d.n_sB[0] < d.k_sB[d.nk - 1]);
    const int64_t kblocks = ((int64_t)d.ktiles * BK + pack_k<KIND>() - 1) / pack_k<KIND>();
    CUtensorMap ta, tb;
    s = image_map(ta, ja.out, bytes_a, d.img_a);
    if (s == TC_SUCCESS) s = image_map(tb, jb.out, bytes_b, d.img_b);
    if (s != TC_SUCCESS) return s;
    for (int64_t t0 = 0; t0 < tiles_n; t0 += panel) {
        d.n_begin = t0 * d.bn;
        d.tiles_n = std::min(panel, tiles_n - t0);
        d.N = std::min(N - d.n_begin, d.tiles_n * d.bn);
        d.num_tiles = d.tiles_m * d.tiles_n;
        jb.total_rows = d.tiles_n * d.bn;
        ja.blocks = t0 == 0 ? (ja.total_rows + kPackRows - 1) / kPackRows * kblocks : 0;  // A's with the first panel
        jb.blocks = (jb.total_rows + kPackRows - 1) / kPackRows * kblocks;
        if (ja.blocks + jb.blocks > 0x7fffffff) return fail(TC_ERROR_INVALID_EXTENT, "too many blocks for the pre-pass");
        pack_images_kernel<KIND><<<(unsigned)(ja.blocks + jb.blocks), kPackThreads, 0, st>>>(d, ja, jb);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
        bool launched = false;
        if constexpr (KIND == GK_BF16X3 || KIND == GK_TF32X3) {
            if (comp) {
                s = t.pair ? launch_gett<KIND, true, true>(d, ta, tb, st) : launch_gett<KIND, true, false>(d, ta, tb, st);
                launched = true;
            }
        }
        if (!launched) s = t.pair ? launch_gett<KIND, false, true>(d, ta, tb, st) : launch_gett<KIND, false, false>(d, ta, tb, st);
        if (s != TC_SUCCESS) return s;
    }
    if (done) *done = true;
    return TC_SUCCESS;
}

// ---- digits, host side
constexpr int64_t kDigitMinK = 32;       // where the bound of the digits meets the chain's
constexpr int64_t kDigitMaxTiles = int64_t(1) << 22;
constexpr int64_t kWeakBytes = int64_t(32) << 20;

struct DigitPlan {
    bool pair;
    int64_t tiles_m, tiles_n, panel_tiles;  // panel_tiles: columns of tiles per panel of B
    int64_t rows_a, image_a, image_b;       // padded rows of A; bytes of A's images and of a panel's
    int64_t weak_tiles;                     // columns of tiles whose weak results are kept before the chain runs
    int64_t off_b, off_exp_a, off_exp_b, off_weak, off_small_a, off_small_b, off_list, zero_bytes, bytes;
};

// The digit form of an M x N x K product, or false where SIMT is the faster
// estimate or the form does not apply.  Clocks per 16 K positions as
// choose_tile counts them (the shared-memory port), plus what draining the
// levels of a unit costs; SIMT at its measured rate.
bool plan_digits(int64_t M, int64_t N, int64_t K, DigitPlan &P) {
    constexpr int BK = stage_k<GK_D64>(), S = Traits<GK_D64>::kSlices;
    if (K < kDigitMinK || K > kDigitMaxK) return false;
    const int64_t Kp = (K + BK - 1) / BK * BK;
    double best = -1, best_pack = 0;
    for (int pair = 1; pair >= 0; --pair) {
        const int64_t rows = pair ? 2 * kRows : kRows, slots = pair ? sm_count() / 2 : sm_count();
        if (slots < 1) continue;
        DigitPlan q;
        q.pair = pair != 0;
        q.tiles_m = (M + rows - 1) / rows;
        q.tiles_n = (N + kDigitBn - 1) / kDigitBn;
        if (q.tiles_n > kDigitMaxTiles / q.tiles_m) continue;
        q.rows_a = q.tiles_m * rows;
        q.image_a = q.rows_a * Kp * S * 2;
        if (q.image_a > kScratchMaxABytes) continue;
        q.panel_tiles = panel_tiles_for(kDigitPanelBytes, q.tiles_n, q.tiles_m, Kp * S * 2 * kDigitBn, slots);
        const int64_t weak_max = std::max<int64_t>(1, kWeakBytes / (q.rows_a * kDigitBn / 8));
        q.panel_tiles = std::min(q.panel_tiles, weak_max);
        q.weak_tiles = std::min(q.tiles_n, weak_max);
        q.image_b = q.panel_tiles * kDigitBn * Kp * S * 2;
        const int64_t panels = (q.tiles_n + q.panel_tiles - 1) / q.panel_tiles;
        const int brows = pair ? kDigitBn / 2 : kDigitBn, nprod = S * (S + 1) / 2;
        const double port = ((4096.0 + 32.0 * brows) * nprod + 32.0 * (kRows + brows) * S) / 128.0;
        const double tile = (Kp / 16) * std::max(kDigitBn / 2.0 * nprod, port) +
                            (K + kDigitChunkK - 1) / kDigitChunkK * 6000.0 + 3000.0;
        const int64_t waves = (panels - 1) * ((q.panel_tiles * q.tiles_m + slots - 1) / slots) +
                              ((q.tiles_n - (panels - 1) * q.panel_tiles) * q.tiles_m + slots - 1) / slots;
        const double pack = (double)(q.rows_a + q.tiles_n * kDigitBn) * Kp * (8 + S * 2) / 3e12;
        // (left_kernel: a launch and, nearly always, some output's chain, 65 to
        // 105 ns per position)
        const double sec = waves * tile / 1.9e9 + pack + 15e-6 + K * 80e-9 + panels * 6e-6;
        if (best < 0 || sec < best) {
            best = sec;
            best_pack = pack;
            P = q;
        }
    }
    if (best < 0) return false;
    const double simt = 2.0 * (double)M * (double)N * (double)K / 1.24e12;
    if (best > 0.8 * simt) return false;
    // Values that the digits refuse cost the pre-pass and three launches for
    // nothing: where that is much of a small GETT, only for twice the speed
    // (414 x 2622, K = 32, all refused: 99 us, 82 with 64 x 64 SIMT tiles).
    if (best > 0.5 * simt && best_pack + 30e-6 > 0.15 * simt) return false;
    auto up = [](int64_t x) { return (x + 511) / 512 * 512; };
    P.off_b = P.image_a;
    P.off_exp_a = P.off_b + P.image_b;
    P.off_exp_b = P.off_exp_a + up(P.rows_a * 4);
    // zeroed before each execute: the weak results, the row tiles' counts and
    // the list's length
    P.off_weak = P.off_exp_b + up(P.panel_tiles * kDigitBn * 4);
    P.off_small_a = P.off_weak + up(P.weak_tiles * P.rows_a * kDigitBn / 8);
    P.off_small_b = P.off_small_a + up(P.rows_a / kRows * 4);
    P.off_list = P.off_small_b + up(P.tiles_n * 2 * 4);
    P.zero_bytes = P.off_list + 16 - P.off_weak;
    P.bytes = P.off_list + up((P.tiles_m * P.tiles_n + 2) * 8);
    return true;
}

tc_status run_digits(Plan &p, PackedDesc &d, const void *alpha, const void *beta, double fraction, cudaStream_t st,
                     bool *done) {
    constexpr int KIND = GK_D64, BK = stage_k<KIND>(), S = Traits<KIND>::kSlices;
    DigitPlan P;
    if (!plan_digits(d.M, d.N, d.K, P)) return TC_SUCCESS;
    tc_status s = ensure_device_resources(p, 0);
    if (s != TC_SUCCESS) return s;
    if (!optional_scratch(p, P.bytes, st)) return TC_SUCCESS;  // the SIMT tiles run
    char *ws = (char *)p.scratch;
    d.alpha64 = *(const double *)alpha;
    d.beta64 = *(const double *)beta;
    d.init = d.beta64 == 0.0 ? 2 : 1;
    int64_t tiles_n = P.tiles_n;
    const int64_t N = fraction < 1.0 ? std::min<int64_t>(d.N, std::max<int64_t>(kDigitBn, (int64_t)(d.N * fraction))) : d.N;
    tiles_n = (N + kDigitBn - 1) / kDigitBn;
    d.status = p.dev_status;
    d.bn = kDigitBn;
    d.brows = P.pair ? kDigitBn / 2 : kDigitBn;
    d.tiles_m = P.tiles_m;
    d.ktiles = (int)((d.K + BK - 1) / BK);
    d.chunk = std::min(d.ktiles, kDigitChunkK / BK);
    d.img_a = (uint32_t)(S * kRows * BK * 2);
    d.img_b = (uint32_t)(S * d.brows * BK * 2);
    d.stages = std::min<int>(kMaxStages, kRingBytes / (int)(d.img_a + d.img_b));
    d.exps[0] = (int *)(ws + P.off_exp_a);
    d.exps[1] = (int *)(ws + P.off_exp_b);
    d.small[0] = (int *)(ws + P.off_small_a);
    d.small[1] = (int *)(ws + P.off_small_b);
    d.list = (int64_t *)(ws + P.off_list);
    CUtensorMap ta, tb;
    s = image_map(ta, ws, P.image_a, d.img_a);
    if (s == TC_SUCCESS) s = image_map(tb, ws + P.off_b, P.image_b, d.img_b);
    if (s != TC_SUCCESS) return s;
    constexpr int kPackSmem = kDigitK * (kPackRows + 1) * (int)sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(pack_digits_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPackSmem);
    if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
    d.weak = (uint32_t *)(ws + P.off_weak);
    d.rows_a = P.rows_a;
    // 2^-10 in the units of levels 0-3, 2^-36; levels 4-7 add at most 2^8.1 of
    // them per K position
    d.weak_below = (int64_t(1) << 26) + d.K * 512;
    e = cudaMemsetAsync(ws + P.off_weak, 0, (size_t)P.zero_bytes, st);
    if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
    int64_t weak0 = 0;  // first column of tiles of those in d.weak
    auto run_left = [&](int64_t end, int64_t *list) {
        return simt_run_left(p, alpha, d.A, d.B, beta, d.C, d.weak, P.rows_a, weak0 * kDigitBn / 32, end * kDigitBn / 32, list,
                             P.tiles_m, P.pair ? 2 * kRows : kRows, kDigitBn, st);
    };
    for (int64_t t0 = 0; t0 < tiles_n; t0 += P.panel_tiles) {
        d.n_begin = t0 * kDigitBn;
        d.tiles_n = std::min(P.panel_tiles, tiles_n - t0);
        if (t0 + d.tiles_n - weak0 > P.weak_tiles) {
            s = run_left(t0, nullptr);
            if (s != TC_SUCCESS) return s;
            weak0 = t0;
            e = cudaMemsetAsync(d.weak, 0, (size_t)(P.weak_tiles * P.rows_a * kDigitBn / 8), st);
            if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
        }
        d.weak_n0 = weak0 * kDigitBn;
        d.N = std::min<int64_t>(N - d.n_begin, d.tiles_n * kDigitBn);
        d.num_tiles = d.tiles_m * d.tiles_n;
        PackJob ja = {}, jb = {};
        ja.op = 0;
        ja.rows = kRows;
        ja.total_rows = P.rows_a;
        ja.rfast = d.nm > 0 && d.m_sA[0] < d.k_sA[d.nk - 1];
        ja.out = ws;
        ja.blocks = t0 == 0 ? (ja.total_rows + kPackRows - 1) / kPackRows : 0;  // A's with the first panel
        jb.op = 1;
        jb.rows = d.brows;
        jb.total_rows = d.tiles_n * kDigitBn;
        jb.rfast = d.nn > 0 && d.n_sB[0] < d.k_sB[d.nk - 1];
        jb.out = ws + P.off_b;
        jb.blocks = (jb.total_rows + kPackRows - 1) / kPackRows;
        pack_digits_kernel<<<(unsigned)(ja.blocks + jb.blocks), kPackThreads, kPackSmem, st>>>(d, ja, jb);
        e = cudaGetLastError();
        if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
        s = P.pair ? launch_gett<KIND, false, true>(d, ta, tb, st) : launch_gett<KIND, false, false>(d, ta, tb, st);
        if (s != TC_SUCCESS) return s;
    }
    s = run_left(tiles_n, d.list);
    if (s == TC_SUCCESS) *done = true;
    return s;
}

}  // namespace

tc_status exec_digits(Plan &p, const void *alpha, const void *A, const void *B, const void *beta, void *C, void *stream,
                      double fraction, bool *done) {
    *done = false;
    if (p.dtype != TC_F64 || p.gett_pack == 0 || !p.batch.empty() || p.contracted.empty()) return TC_SUCCESS;
    // the chain multiplies A by alpha entry by entry: an infinite one gives NaN
    // beside a zero or opposite signs, which the digits' one product would not
    if (!std::isfinite(*(const double *)alpha)) return TC_SUCCESS;
    PackedDesc d;
    std::memset(&d, 0, sizeof(d));
    tc_status s = describe_modes(p, 3, d);
    if (s != TC_SUCCESS) return s;
    d.A = A;
    d.B = B;
    d.C = C;
    return run_digits(p, d, alpha, beta, fraction, (cudaStream_t)stream, done);
}

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
                      double fraction, int64_t comp_k, bool split, const float *qscale, bool *done) {
    if (done) *done = false;
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
    case TC_BF16X3: return run_packed<GK_BF16X3>(p, d, comp, comp_k, fraction, st, done);
    case TC_BF16: return run_packed<GK_BF16>(p, d, false, 0, fraction, st, done);
    case TC_F16: return run_packed<GK_F16>(p, d, false, 0, fraction, st, done);
    case TC_TF32: return run_packed<GK_TF32>(p, d, false, 0, fraction, st, done);
    case TC_TF32X3: return run_packed<GK_TF32X3>(p, d, comp, comp_k, fraction, st, done);
    case TC_E4M3: return run_packed<GK_E4M3>(p, d, false, 0, fraction, st, done);
    default: return fail(TC_ERROR_UNSUPPORTED_DTYPE, "dtype has no pre-converted GETT");
    }
}

}  // namespace tc
