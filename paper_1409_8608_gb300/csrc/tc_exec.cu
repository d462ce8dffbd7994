// Nest executor: runs one Section 2 algorithm (a loop nest around one BLAS
// kernel) on the GPU, plus the SIMT form of the fused GETT for FP64/FP32.
//
// Reading of the sequential loop nests for a parallel device (the paper
// describes sequential CPU loops only):
//  * Loops keep their nest order.  Iterations of a free loop write disjoint
//    C slices and run concurrently.
//  * A contracted loop that encloses a free loop becomes a device-wide
//    phase: one launch per iteration, in order, C carried through memory.
//  * The remaining contracted loops (those with no free loop inside them)
//    run in order inside each task, C held in registers.
//  * Every C element therefore sees one fixed chain of fused multiply-adds
//    acc = fma(alpha*a, b, acc) over the contracted indices in nest order
//    (phase loops, then in-task loops, then the kernel's own contracted
//    index), starting from beta*C.  Algorithms with the same contracted
//    order give bitwise identical results.
//  * Copies (Section 2: a matrix slice without a unit-stride dimension)
//    materialise the slice into a contiguous workspace at the phase they
//    belong to, once per combination of the loops the slice depends on.
//
// Kernels: dot, axpy, gemv and ger run one thread per output element of a
// kernel call (kernel outputs fastest across threads, then the innermost
// free loop), reading operands straight from L1/L2 -- the BLAS-1/2 shape.
// gemm runs as a shared-memory tiled register-blocked kernel -- the BLAS-3
// shape.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "tc_internal.h"

namespace tc {

struct Dims {
    int n;
    int64_t ext[kMaxModes];
    int64_t sA[kMaxModes], sB[kMaxModes], sC[kMaxModes];
};

struct PhaseDesc {
    Dims out;   // kernel output modes, first fastest
    Dims task;  // free sliced loops, outermost first (innermost fastest)
    Dims red;   // contracted: in-task loops outermost first, kernel index last
    int64_t total;
    const void *A;
    const void *B;
    void *C;
    double alpha, beta;
    int init;       // 0: acc = C, 1: acc = beta*C, 2: acc = 0
    int alpha_one;  // alpha == 1: skip the scaling multiply
};

struct TileDesc {
    Dims m;     // M modes (first fastest): strides sA and sC
    Dims n;     // N modes: strides sB and sC
    Dims red;   // K modes, outermost first
    Dims task;  // tasks: free sliced loops, outermost first
    int64_t M, N, K;
    int64_t tiles_m, tiles_n;
    const void *A;
    const void *B;
    void *C;
    double alpha, beta;
    int init, alpha_one;
    int a_m_fast, b_n_fast;  // load mapping: M (N) contiguous in memory
    int swapped, unused;     // M and N, A and B exchanged (orient): alpha scales B's side
    int64_t tile0;           // batched form: the problem's first tile in the list
    int64_t shape;           // tile shape (simt_rows)
};

struct GatherDesc {
    int n;
    int64_t ext[2 * kMaxModes];
    int64_t ss[2 * kMaxModes];  // source strides
    int64_t sd[2 * kMaxModes];  // destination strides
    int64_t total;
    const void *src;
    void *dst;
};

namespace {

template <typename T>
__device__ __forceinline__ T fma_t(T a, T b, T c);
template <>
__device__ __forceinline__ double fma_t<double>(double a, double b, double c) { return fma(a, b, c); }
template <>
__device__ __forceinline__ float fma_t<float>(float a, float b, float c) { return fmaf(a, b, c); }

// ---------------------------------------------------------------- dot/axpy/gemv/ger
// x = q * y + r for non-negative x, y > 0, in 32 bits when both fit (a
// 64-bit division is a long dependent sequence on every tile's first path)
__device__ __forceinline__ int64_t divmod_pos(int64_t x, int64_t y, int64_t &r) {
    if (((x | y) >> 31) == 0) {
        const uint32_t q = (uint32_t)x / (uint32_t)y;
        r = x - (int64_t)q * y;
        return q;
    }
    const int64_t q = x / y;
    r = x - q * y;
    return q;
}

// AHEAD: four positions' loads in flight at a time, multiplied in order, where
// the innermost index is long (gemv n = 128: 2.03 -> 0.90 ms; on 4 to 32
// positions it costs 4 to 10 %).
template <typename T, bool AHEAD>
__global__ void __launch_bounds__(256) elementwise_kernel(const PhaseDesc d) {
    const T *__restrict__ A = (const T *)d.A;
    const T *__restrict__ B = (const T *)d.B;
    T *__restrict__ C = (T *)d.C;
    const T alpha = (T)d.alpha, beta = (T)d.beta;
    const int nr = d.red.n;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < d.total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e, oA = 0, oB = 0, oC = 0;
        for (int m = 0; m < d.out.n; ++m) {
            const int64_t x = r % d.out.ext[m];
            r /= d.out.ext[m];
            oA += x * d.out.sA[m];
            oB += x * d.out.sB[m];
            oC += x * d.out.sC[m];
        }
        for (int m = d.task.n - 1; m >= 0; --m) {
            const int64_t x = r % d.task.ext[m];
            r /= d.task.ext[m];
            oA += x * d.task.sA[m];
            oB += x * d.task.sB[m];
            oC += x * d.task.sC[m];
        }
        T acc;
        if (d.init == 2) {
            acc = T(0);
        } else {
            acc = C[oC];
            if (d.init == 1) acc = beta * acc;
        }
        if (nr == 0) {
            T a = A[oA];
            if (!d.alpha_one) a = alpha * a;
            acc = fma_t<T>(a, B[oB], acc);
        } else {
            int64_t idx[kMaxModes];
            for (int m = 0; m < nr; ++m) idx[m] = 0;
            const int64_t kext = d.red.ext[nr - 1];
            const int64_t ksA = d.red.sA[nr - 1], ksB = d.red.sB[nr - 1];
            for (;;) {
                int64_t pa = oA, pb = oB;
                for (int m = 0; m < nr - 1; ++m) {
                    pa += idx[m] * d.red.sA[m];
                    pb += idx[m] * d.red.sB[m];
                }
                int64_t k = 0;
                for (; AHEAD && k + 4 <= kext; k += 4) {
                    T a[4], b[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        a[x] = A[pa + x * ksA];
                        b[x] = B[pb + x * ksB];
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) acc = fma_t<T>(d.alpha_one ? a[x] : alpha * a[x], b[x], acc);
                    pa += 4 * ksA;
                    pb += 4 * ksB;
                }
                for (; k < kext; ++k) {
                    T a = A[pa];
                    if (!d.alpha_one) a = alpha * a;
                    acc = fma_t<T>(a, B[pb], acc);
                    pa += ksA;
                    pb += ksB;
                }
                int m = nr - 2;
                while (m >= 0) {
                    if (++idx[m] < d.red.ext[m]) break;
                    idx[m] = 0;
                    --m;
                }
                if (m < 0) break;
            }
        }
        C[oC] = acc;
    }
}

// Cooperative reduction (a phase with few outputs whose innermost contracted
// index has unit stride in an input): a group of G lanes (a power of two,
// 4..32) per kernel output splits that index (red's last mode), so the
// group's loads are contiguous; each lane sums its share over every in-task
// contracted loop, then the group adds the lanes' partial sums with a fixed
// butterfly (the same order every run).
template <typename T, int G>
__global__ void __launch_bounds__(256) coop_reduce_kernel(const PhaseDesc d) {
    const T *__restrict__ A = (const T *)d.A;
    const T *__restrict__ B = (const T *)d.B;
    T *__restrict__ C = (T *)d.C;
    const int gl = threadIdx.x % G;  // lane within the group
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
    const int nr = d.red.n;
    const int64_t kext = d.red.ext[nr - 1], ksA = d.red.sA[nr - 1], ksB = d.red.sB[nr - 1];
    // every lane of a warp runs the same number of rounds (shuffles need the
    // whole warp): the round's output is e = warp's first + the group's
    const int64_t first = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    for (int64_t base = first - (threadIdx.x % 32) / G; base < d.total; base += groups) {
        const int64_t e = base + (threadIdx.x % 32) / G;
        const bool live = e < d.total;
        int64_t r = live ? e : 0, oA = 0, oB = 0, oC = 0;
        for (int m = 0; m < d.out.n; ++m) {
            const int64_t x = r % d.out.ext[m];
            r /= d.out.ext[m];
            oA += x * d.out.sA[m];
            oB += x * d.out.sB[m];
            oC += x * d.out.sC[m];
        }
        for (int m = d.task.n - 1; m >= 0; --m) {
            const int64_t x = r % d.task.ext[m];
            r /= d.task.ext[m];
            oA += x * d.task.sA[m];
            oB += x * d.task.sB[m];
            oC += x * d.task.sC[m];
        }
        T acc = T(0);
        int64_t idx[kMaxModes];
        for (int m = 0; m < nr - 1; ++m) idx[m] = 0;
        for (;;) {
            int64_t pa = oA, pb = oB;
            for (int m = 0; m < nr - 1; ++m) {
                pa += idx[m] * d.red.sA[m];
                pb += idx[m] * d.red.sB[m];
            }
            if (live)
                for (int64_t k = gl; k < kext; k += G) acc = fma_t<T>(A[pa + k * ksA], B[pb + k * ksB], acc);
            int m = nr - 2;
            while (m >= 0) {
                if (++idx[m] < d.red.ext[m]) break;
                idx[m] = 0;
                --m;
            }
            if (m < 0) break;
        }
#pragma unroll
        for (int off = G / 2; off > 0; off /= 2) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (live && gl == 0) {
            T v = d.alpha_one ? acc : (T)d.alpha * acc;
            if (d.init == 0) v += C[oC];
            else if (d.init == 1) v = fma_t<T>((T)d.beta, C[oC], v);
            C[oC] = v;
        }
    }
}

// The same sums, one thread per output: where the index is short and outputs
// are many, the lanes of a group mostly repeat one another's index arithmetic
// (130 k outputs of 9 x 11 positions, FP32: 93-111 us in groups, 24-28 so).
// A thread keeps the G partial sums of a group (kext <= G) and adds them in the
// butterfly's order, so the results are the same bits.
template <typename T, int G>
__global__ void __launch_bounds__(256) lane_sums_kernel(const PhaseDesc d) {
    const T *__restrict__ A = (const T *)d.A;
    const T *__restrict__ B = (const T *)d.B;
    T *__restrict__ C = (T *)d.C;
    const int nr = d.red.n;
    const int kext = (int)d.red.ext[nr - 1];
    const int64_t ksA = d.red.sA[nr - 1], ksB = d.red.sB[nr - 1];
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < d.total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e, oA = 0, oB = 0, oC = 0;
        for (int m = 0; m < d.out.n; ++m) {
            const int64_t x = r % d.out.ext[m];
            r /= d.out.ext[m];
            oA += x * d.out.sA[m];
            oB += x * d.out.sB[m];
            oC += x * d.out.sC[m];
        }
        for (int m = d.task.n - 1; m >= 0; --m) {
            const int64_t x = r % d.task.ext[m];
            r /= d.task.ext[m];
            oA += x * d.task.sA[m];
            oB += x * d.task.sB[m];
            oC += x * d.task.sC[m];
        }
        T acc[G];
#pragma unroll
        for (int l = 0; l < G; ++l) acc[l] = T(0);
        int64_t idx[kMaxModes];
        for (int m = 0; m < nr - 1; ++m) idx[m] = 0;
        for (;;) {
            int64_t pa = oA, pb = oB;
            for (int m = 0; m < nr - 1; ++m) {
                pa += idx[m] * d.red.sA[m];
                pb += idx[m] * d.red.sB[m];
            }
            constexpr int V = 4;  // positions whose loads are in flight together
#pragma unroll
            for (int l0 = 0; l0 < G; l0 += V) {
                if (l0 >= kext) break;
                T a[V], b[V];
#pragma unroll
                for (int l = 0; l < V; ++l) {
                    const bool in = l0 + l < kext;
                    a[l] = in ? A[pa + (l0 + l) * ksA] : T(0);
                    b[l] = in ? B[pb + (l0 + l) * ksB] : T(0);
                }
#pragma unroll
                for (int l = 0; l < V; ++l)
                    if (l0 + l < kext) acc[l0 + l] = fma_t<T>(a[l], b[l], acc[l0 + l]);
            }
            int m = nr - 2;
            while (m >= 0) {
                if (++idx[m] < d.red.ext[m]) break;
                idx[m] = 0;
                --m;
            }
            if (m < 0) break;
        }
#pragma unroll
        for (int off = G / 2; off > 0; off /= 2)
#pragma unroll
            for (int l = 0; l < off; ++l) acc[l] += acc[l + off];
        T v = d.alpha_one ? acc[0] : (T)d.alpha * acc[0];
        if (d.init == 0) v += C[oC];
        else if (d.init == 1) v = fma_t<T>((T)d.beta, C[oC], v);
        C[oC] = v;
    }
}

// ---------------------------------------------------------------- gemm / SIMT GETT
__device__ __forceinline__ uint64_t pack_f2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack_f2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// two independent FP32 fused multiply-adds in one instruction (each rounded
// as fmaf rounds)
__device__ __forceinline__ void fma_f2(uint64_t &c, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

template <typename T, int BM, int BN, int BK>
struct TileSmem {
    // two stage buffers; rows padded by 4 elements so that the K-contiguous
    // store mapping below spreads a warp over all 32 banks
    static constexpr int PAD = 4;
    T As[2][BK][BM + PAD];
    T Bs[2][BK][BN + PAD];
    int64_t offAm[BM], offCm[BM], offBn[BN], offCn[BN];
    int64_t kA[2][BK], kB[2][BK];
};

// One CTA computes a BM x BN tile of one task's C slice; K runs over the
// linearised contracted space in stages of BK through shared memory.  Each
// thread keeps the memory offsets of the rows it copies in registers, so a
// stage's copies read only its K offsets from shared memory (with both read
// per element the offset tables took as many shared-memory cycles as the
// operands: 68 % of the pipe at 37 % of the FMA rate on FP32).  With that,
// paired FP32 multiply-adds and C stored by column runs, FP32 512^3 iaj,jbic
// i=j=16 went from 2.35 to 1.83 ms and the n = 256 gemm nest from 0.287 to
// 0.213 ms; FP64 512^3 from 56.76 to 55.06 ms (the DFMA rate).
template <typename T, int BM, int BN, int BK, int TM, int TN>
__device__ __forceinline__ void tile_body(const TileDesc &d, int64_t bid, TileSmem<T, BM, BN, BK> &sm) {
    // rows across the lanes (TX), so that a warp's stores of one column of C
    // cover a contiguous run of its first index
    constexpr int TX = BM / TM, TY = BN / TN, NT = TX * TY;
    // FP32: a thread owns V consecutive rows per group, V = 2 or 4 (one 8- or
    // 16-byte shared-memory read per group; its rows multiply in pairs with
    // fma.rn.f32x2, which halves the issue slots of the FMAs), and likewise
    // columns; FP64 (V = 1) is bound by the DFMA rate either way
    constexpr bool F32 = sizeof(T) == 4;
    constexpr int V = F32 ? (TM % 4 == 0 && TN % 4 == 0 ? 4 : 2) : 1;
    static_assert(TM % V == 0 && TN % V == 0, "groups of V");
    auto row_of = [](int tx_, int i) { return (i / V) * (TX * V) + tx_ * V + i % V; };
    auto col_of = [](int ty_, int j) { return (j / V) * (TY * V) + ty_ * V + j % V; };
    const T *__restrict__ A = (const T *)d.A;
    const T *__restrict__ B = (const T *)d.B;
    T *__restrict__ C = (T *)d.C;
    const T alpha = (T)d.alpha, beta = (T)d.beta;
    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;

    int64_t tm, tn;
    bid = divmod_pos(bid, d.tiles_m, tm);
    int64_t task = divmod_pos(bid, d.tiles_n, tn);
    int64_t tA = 0, tB = 0, tC = 0;
    for (int m = d.task.n - 1; m >= 0; --m) {
        int64_t x;
        task = divmod_pos(task, d.task.ext[m], x);
        tA += x * d.task.sA[m];
        tB += x * d.task.sB[m];
        tC += x * d.task.sC[m];
    }
    for (int i = tid; i < BM; i += NT) {
        int64_t mm = tm * BM + i;
        int64_t oa = -1, oc = -1;
        if (mm < d.M) {
            oa = tA;
            oc = tC;
            for (int m = 0; m < d.m.n; ++m) {
                int64_t x;
                mm = divmod_pos(mm, d.m.ext[m], x);
                oa += x * d.m.sA[m];
                oc += x * d.m.sC[m];
            }
        }
        sm.offAm[i] = oa;
        sm.offCm[i] = oc;
    }
    for (int j = tid; j < BN; j += NT) {
        int64_t nn = tn * BN + j;
        int64_t ob = -1, oc = -1;
        if (nn < d.N) {
            ob = tB;
            oc = 0;
            for (int m = 0; m < d.n.n; ++m) {
                int64_t x;
                nn = divmod_pos(nn, d.n.ext[m], x);
                ob += x * d.n.sB[m];
                oc += x * d.n.sC[m];
            }
        }
        sm.offBn[j] = ob;
        sm.offCn[j] = oc;
    }
    // K offsets of a stage into table buffer b (threads kk < BK)
    auto k_tables = [&](int64_t k0, int b) {
        if (tid < BK) {
            int64_t k = k0 + tid;
            int64_t oa = -1, ob = -1;
            if (k < d.K) {
                oa = 0;
                ob = 0;
                for (int m = d.red.n - 1; m >= 0; --m) {
                    int64_t x;
                    k = divmod_pos(k, d.red.ext[m], x);
                    oa += x * d.red.sA[m];
                    ob += x * d.red.sB[m];
                }
            }
            sm.kA[b][tid] = oa;
            sm.kB[b][tid] = ob;
        }
    };
    static_assert(NT >= BK, "one thread per K offset");
    k_tables(0, 0);
    if (BK < d.K) k_tables(BK, 1);
    __syncthreads();

    // accumulators: FP32 row pairs (2i, 2i + 1), FP64 one by one
    constexpr int NACC = F32 ? TM / 2 : TM;
    using Acc = typename std::conditional<F32, uint64_t, double>::type;
    Acc acc[NACC][TN];
    if (d.init == 2) {
#pragma unroll
        for (int i = 0; i < NACC; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] = Acc(0);
    } else {
        auto start = [&](int i, int j) {
            const int64_t om = sm.offCm[row_of(tx, i)], on = sm.offCn[col_of(ty, j)];
            T v = T(0);
            if (om >= 0 && on >= 0) {
                v = C[om + on];
                if (d.init == 1) v = beta * v;
            }
            return v;
        };
#pragma unroll
        for (int i = 0; i < NACC; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                if constexpr (F32) acc[i][j] = pack_f2(start(2 * i, j), start(2 * i + 1, j));
                else acc[i][j] = start(i, j);
            }
    }

    // Elements of a stage's R x BK operand tile that a thread copies: with
    // M (N) contiguous in memory (rfast), consecutive threads take
    // consecutive rows and a thread always the same row; otherwise groups of
    // 8 threads take 8 consecutive K positions of one row (32-byte runs in
    // memory; with the padded rows a warp's stores hit 32 distinct banks)
    // and a thread meets at most R / (NT / 8) rows.
    static_assert(BK % 8 == 0 && NT % BM == 0 && NT % BN == 0, "copy mapping");
    constexpr int QA = BM > NT / 8 ? BM / (NT / 8) : 1, QB = BN > NT / 8 ? BN / (NT / 8) : 1;
    constexpr int LA = BM * BK / NT, LB = BN * BK / NT;
    static_assert(LA * NT == BM * BK && LB * NT == BN * BK && LA % QA == 0 && LB % QB == 0, "even split");
    const bool fa = d.a_m_fast != 0, fb = d.b_n_fast != 0;
    const int rA0 = fa ? tid % BM : (tid / 8) % BM, rB0 = fb ? tid % BN : (tid / 8) % BN;
    const int kA0 = fa ? tid / BM : (tid / (8 * BM)) * 8 + tid % 8;
    const int kB0 = fb ? tid / BN : (tid / (8 * BN)) * 8 + tid % 8;
    int64_t roA[QA], roB[QB];
#pragma unroll
    for (int q = 0; q < QA; ++q) roA[q] = sm.offAm[fa ? rA0 : (rA0 + q * (NT / 8)) % BM];
#pragma unroll
    for (int q = 0; q < QB; ++q) roB[q] = sm.offBn[fb ? rB0 : (rB0 + q * (NT / 8)) % BN];
    // element l of the thread: row slot, row and K position
    auto at = [](bool fast, int R, int Q, int l, int r0, int k0, int &q, int &r, int &kk) {
        if (fast) {
            q = 0;
            r = r0;
            kk = k0 + l * (NT / R);
        } else {
            q = l % Q;
            r = r0 + q * (NT / 8);
            // R < NT / 8: the NT threads cover NT / (8R) octets of K per step
            kk = k0 + (l / Q) * (R < NT / 8 ? NT / R : 8);
        }
    };
    // the elements go straight to shared memory with asynchronous copies
    // (zero-filled past the extents)
    auto cp = [](void *dst, const void *src, bool valid) {
        if constexpr (F32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(dst)),
                         "l"(src), "r"(valid ? 4 : 0)
                         : "memory");
        else
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(dst)),
                         "l"(src), "r"(valid ? 8 : 0)
                         : "memory");
    };
    auto async_stage = [&](int b) {
        auto side = [&](auto fast, auto rows, auto Lc, auto Qc, const T *base, const int64_t *ro, const int64_t *kt, int r0,
                        int k0, T *dst, int pitch) {
#pragma unroll
            for (int l = 0; l < decltype(Lc)::value; ++l) {
                int q, r, kk;
                at(decltype(fast)::value, decltype(rows)::value, decltype(Qc)::value, l, r0, k0, q, r, kk);
                const int64_t om = ro[q], ok = kt[kk];
                const bool v = om >= 0 && ok >= 0;
                cp(dst + kk * pitch + r, v ? base + om + ok : base, v);
            }
        };
        using Yes = std::true_type;
        using No = std::false_type;
        if (fa) side(Yes{}, std::integral_constant<int, BM>{}, std::integral_constant<int, LA>{}, std::integral_constant<int, QA>{}, A, roA, sm.kA[b], rA0, kA0, &sm.As[b][0][0], BM + sm.PAD);
        else side(No{}, std::integral_constant<int, BM>{}, std::integral_constant<int, LA>{}, std::integral_constant<int, QA>{}, A, roA, sm.kA[b], rA0, kA0, &sm.As[b][0][0], BM + sm.PAD);
        if (fb) side(Yes{}, std::integral_constant<int, BN>{}, std::integral_constant<int, LB>{}, std::integral_constant<int, QB>{}, B, roB, sm.kB[b], rB0, kB0, &sm.Bs[b][0][0], BN + sm.PAD);
        else side(No{}, std::integral_constant<int, BN>{}, std::integral_constant<int, LB>{}, std::integral_constant<int, QB>{}, B, roB, sm.kB[b], rB0, kB0, &sm.Bs[b][0][0], BN + sm.PAD);
    };
    // the stage's copies have landed; with alpha != 1 each thread scales the
    // elements of A (of B where they are exchanged) that it copied itself
    auto land_stage = [&](int b) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (d.alpha_one) return;
        int q, r, kk;
        if (!d.swapped) {
#pragma unroll
            for (int l = 0; l < LA; ++l) {
                at(fa, BM, QA, l, rA0, kA0, q, r, kk);
                sm.As[b][kk][r] = alpha * sm.As[b][kk][r];
            }
        } else {
#pragma unroll
            for (int l = 0; l < LB; ++l) {
                at(fb, BN, QB, l, rB0, kB0, q, r, kk);
                sm.Bs[b][kk][r] = alpha * sm.Bs[b][kk][r];
            }
        }
    };
    auto step = [&](int sb, int kk) {
        if constexpr (F32) {
            uint64_t a[TM / 2], b[TN];
#pragma unroll
            for (int g = 0; g < TM / V; ++g) {
                if constexpr (V == 4) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&sm.As[sb][kk][row_of(tx, V * g)]);
                    a[2 * g] = v.x;
                    a[2 * g + 1] = v.y;
                } else {
                    a[g] = *reinterpret_cast<const unsigned long long *>(&sm.As[sb][kk][row_of(tx, V * g)]);
                }
            }
#pragma unroll
            for (int g = 0; g < TN / V; ++g) {
                if constexpr (V == 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(&sm.Bs[sb][kk][col_of(ty, V * g)]);
                    b[4 * g] = pack_f2(v.x, v.x);
                    b[4 * g + 1] = pack_f2(v.y, v.y);
                    b[4 * g + 2] = pack_f2(v.z, v.z);
                    b[4 * g + 3] = pack_f2(v.w, v.w);
                } else {
                    const float2 v = *reinterpret_cast<const float2 *>(&sm.Bs[sb][kk][col_of(ty, V * g)]);
                    b[2 * g] = pack_f2(v.x, v.x);
                    b[2 * g + 1] = pack_f2(v.y, v.y);
                }
            }
#pragma unroll
            for (int i = 0; i < TM / 2; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) fma_f2(acc[i][j], a[i], b[j]);
        } else {
            T a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = sm.As[sb][kk][row_of(tx, i)];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = sm.Bs[sb][kk][col_of(ty, j)];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
    };
    // Stage s sits in buffer s & 1 (shared memory and K tables alike).
    // While stage s is multiplied, stage s + 1's copies are in flight into
    // the other buffer, whose last reader (stage s - 1) finished before the
    // barrier that ended the previous iteration; one barrier per stage.
    // Stage s + 2's K tables go to buffer s & 1 right after stage s + 1's
    // copies have read theirs (buffer s & 1 was last read by stage s's
    // copies, before that barrier), so that their integer work overlaps the
    // multiplications.  The last stage stops at K (its padding would cost
    // whole multiplications: K = 8 spent as much as K = 16).
    async_stage(0);
    land_stage(0);
    __syncthreads();
    int sb = 0;
    for (int64_t k0 = 0; k0 < d.K; k0 += BK, sb ^= 1) {
        const bool more = k0 + BK < d.K;
        if (more) async_stage(sb ^ 1);
        if (k0 + 2 * BK < d.K) k_tables(k0 + 2 * BK, sb);
        if (k0 + BK <= d.K) {
#pragma unroll
            for (int kk = 0; kk < BK; ++kk) step(sb, kk);
        } else {
            const int klen = (int)(d.K - k0);
#pragma unroll 1
            for (int kk = 0; kk < klen; ++kk) step(sb, kk);
        }
        if (more) land_stage(sb ^ 1);
        __syncthreads();
    }

#pragma unroll
    for (int g = 0; g < TM / V; ++g) {
        int64_t om[V];
#pragma unroll
        for (int v = 0; v < V; ++v) om[v] = sm.offCm[row_of(tx, V * g + v)];
        const bool run = V > 1 && om[0] >= 0 && om[V - 1] == om[0] + V - 1;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int64_t on = sm.offCn[col_of(ty, j)];
            if (on < 0) continue;
            T x[V];
            if constexpr (F32) {
#pragma unroll
                for (int v = 0; v < V; v += 2) unpack_f2(acc[(V * g + v) / 2][j], x[v], x[v + 1]);
            } else {
                x[0] = acc[g][j];
            }
            T *p = C + om[0] + on;
            // the group's rows are one aligned run of C: one store
            if (run && ((uintptr_t)p % (V * sizeof(T))) == 0) {
                if constexpr (V == 4) *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
                else if constexpr (V == 2) *reinterpret_cast<float2 *>(p) = make_float2(x[0], x[1]);
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (om[v] >= 0) C[om[v] + on] = x[v];
            }
        }
    }
}

// Tile shapes.  The largest keeps the least traffic per multiplication; the
// smaller ones spread small results over the SMs: with the FP64 rate at two
// multiply-adds per SM and clock a 64 x 64 tile of K = 3920 holds one SM for
// 4 ms, and nothing is lost per multiplication down to 16 x 16 (64^3 i = 8:
// 25.9 us with 64 tiles of 64 x 64 and K padded to 16, 10.3 us with 1024
// tiles of 16 x 16 stopping at K; a burst of 24 mixed requests 6.03 -> 2.02
// ms, 5.0 of it one FP64 tile).  The tile does not change any output's chain.
constexpr int kSimtShapes = 3;
constexpr int simt_rows(bool f64, int shape) { return (f64 ? 64 : 128) >> shape; }

// The largest shape whose tiles give two thirds of the SMs one (FP32) or each
// SM eight (FP64), else the smallest.  (FP32 128 x 128 tiles cost less per
// output: 108 of them 140 us and 432 of 64 x 64 147, K = 1000; 117 and 468 632
// and 844 us, K = 4964; 100 and 400 146 and 147.)
int simt_shape(bool f64, int64_t M, int64_t N, int64_t tasks);

template <typename T, int SHAPE>
struct TileOf {
    static constexpr bool F64 = sizeof(T) == 8;
    static constexpr int B = simt_rows(F64, SHAPE);
    static constexpr int TT = B / 16;  // 16 x 16 threads
    // FP32: the smaller tiles take longer stages, whose barriers and copies
    // would otherwise cost more than their multiplications (32 x 128 with K =
    // 5704: 356 stages of 16)
    static constexpr int BK = F64 ? 16 : 16 << SHAPE;
    using Smem = TileSmem<T, B, B, BK>;
    static __device__ __forceinline__ void run(const TileDesc &d, int64_t bid, void *buf) {
        tile_body<T, B, B, BK, TT, TT>(d, bid, *reinterpret_cast<Smem *>(buf));
    }
};

// shared memory that holds any shape's
template <typename T>
__host__ __device__ constexpr size_t tile_smem() {
    size_t m = sizeof(typename TileOf<T, 0>::Smem);
    if (sizeof(typename TileOf<T, 1>::Smem) > m) m = sizeof(typename TileOf<T, 1>::Smem);
    if (sizeof(typename TileOf<T, 2>::Smem) > m) m = sizeof(typename TileOf<T, 2>::Smem);
    return m;
}

template <typename T, int SHAPE>
__global__ void __launch_bounds__(256, 2) tile_kernel(const TileDesc d) {
    __shared__ __align__(16) unsigned char buf[sizeof(typename TileOf<T, SHAPE>::Smem)];
    TileOf<T, SHAPE>::run(d, blockIdx.x, buf);
}

// Batched form of the SIMT GETT (no paper counterpart): CTA t computes tile
// t of the flattened tile list of many problems, each with its own
// descriptor (modes, strides, operands, tile shape); the descriptor of the
// tile's problem is copied to shared memory first.  A problem's tiles
// compute exactly as tile_kernel computes them, whatever else is in the
// batch.
template <typename T>
__global__ void __launch_bounds__(256, 2)
tile_batch_kernel(const TileDesc *__restrict__ descs, const int32_t *__restrict__ tile_prob) {
    constexpr size_t kBytes = tile_smem<T>();
    __shared__ __align__(16) TileDesc sd;
    __shared__ __align__(16) unsigned char buf[kBytes];
    static_assert(kBytes >= sizeof(typename TileOf<T, 1>::Smem) && kBytes >= sizeof(typename TileOf<T, 2>::Smem), "every shape fits");
    static_assert(sizeof(TileDesc) % 8 == 0, "descriptor in 8-byte words");
    constexpr int kWords = sizeof(TileDesc) / 8;
    const int q = tile_prob[blockIdx.x];
    for (int w = threadIdx.x; w < kWords; w += blockDim.x)
        ((int64_t *)&sd)[w] = ((const int64_t *)(descs + q))[w];
    __syncthreads();
    const int64_t bid = (int64_t)blockIdx.x - sd.tile0;
    if (sd.shape == 0) TileOf<T, 0>::run(sd, bid, buf);
    else if (sd.shape == 1) TileOf<T, 1>::run(sd, bid, buf);
    else TileOf<T, 2>::run(sd, bid, buf);
}

// What an FP64 GETT on digits leaves to the chain of fused multiply-adds, with
// the bits that the SIMT GETT gives: single outputs marked in `weak`, one
// thread each; patches of 32 x 32 that are marked as a whole, as tiles; and
// the tiles of a list (list[0] items m + list_m * n from list[2] on, each
// sub_m x sub_n tiles of 64 x 64; list[1] counts the tiles taken).
// 512^3 i=j=16: 60 us for the marks of 4.2 M rows of 32 columns and about 20000
// single outputs.  Tiles refused as a whole: 55.7 ms there; 2148 x 218 x 2150,
// 36 items, 2.28 ms, 4.45 where blocks take fixed tiles of 64 x 64, two on
// some SMs and none on others (the SIMT GETT alone 2.29).
// A block gathers the marks of its patches (8 or 32 at a time, all blocks in
// turn, so that a weak region of C is spread over them) before it computes any.
// Many single outputs are bound by a 32-byte sector per element of A and B; few
// by the chain's K dependent multiply-adds, to which every read of 16 positions
// added its latency: up to kFew of them have their operands brought to shared
// memory by the whole block (500 x 1500, K = 8000: 3.31 -> 2.82 ms; 2000^3 903
// -> 804 us; in two rounds of kFew no faster than a thread each).
struct LeftSingles {
    static constexpr int kCap = 8192, kStep = 32 * kWeakMax;  // places, and the most that one step adds
    static constexpr int kFew = 15;       // outputs computed so, at most,
    static constexpr int kFewK = 128, kFewPitch = 2 * kFewK + 1;  // by so many K positions; their operands
    static constexpr int kFewAt = 64;     // lie in the list from here on
    uint32_t list[kCap];
    int64_t kA[256], kB[256];
};
static_assert((LeftSingles::kCap - LeftSingles::kFewAt) * 4 >= LeftSingles::kFew * LeftSingles::kFewPitch * 8 &&
                  LeftSingles::kFewAt >= LeftSingles::kFew,
              "operands fit");

__global__ void __launch_bounds__(256, 4)
left_kernel(const TileDesc d, const TileDesc patch, const TileDesc small, const uint32_t *__restrict__ weak, int64_t rows, int64_t g0, int64_t g1,
            int64_t *list, int64_t list_m, int sub_m, int sub_n) {
    using Tile = TileOf<double, 0>;
    using Patch = TileOf<double, 1>;
    constexpr int kPatches = 32, kWhole = 256, kAhead = 16;
    constexpr size_t kBytes = sizeof(LeftSingles) > sizeof(Tile::Smem) ? sizeof(LeftSingles) : sizeof(Tile::Smem);
    static_assert(Patch::B == 32, "a patch is a tile");
    __shared__ __align__(16) unsigned char buf[kBytes];
    LeftSingles &sm = *reinterpret_cast<LeftSingles *>(buf);
    __shared__ uint32_t whole[kWhole];
    __shared__ int nlist, nwhole;
    __shared__ int64_t taken;
    const double *__restrict__ A = (const double *)d.A;
    const double *__restrict__ B = (const double *)d.B;
    double *__restrict__ C = (double *)d.C;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int64_t rp = rows / 32, patches = rp * (g1 - g0);
    // patches that a block looks at together: eight where that spreads them
    // over more blocks
    const int group = patches >= (int64_t)gridDim.x * kPatches ? kPatches : 8;
    const int64_t stride = (int64_t)gridDim.x * group;
    // the patch at place x of this block's: rows 32 pm .., columns 32 (g0 + pn) ..
    auto patch_at = [&](int64_t x, int64_t &pm) -> int64_t {
        return divmod_pos((int64_t)blockIdx.x * group + x / group * stride + x % group, rp, pm);
    };
    // operand offsets and C of a listed output
    auto place = [&](uint32_t at, int64_t &oA, int64_t &oB, int64_t &oC) {
        int64_t x, mm, nn = g0 + patch_at(at >> 10, mm);
        mm = mm * 32 + (at >> 5 & 31);
        nn = nn * 32 + (at & 31);
        oA = oB = oC = 0;
        for (int m = 0; m < d.m.n; ++m) {
            mm = divmod_pos(mm, d.m.ext[m], x);
            oA += x * d.m.sA[m];
            oC += x * d.m.sC[m];
        }
        for (int m = 0; m < d.n.n; ++m) {
            nn = divmod_pos(nn, d.n.ext[m], x);
            oB += x * d.n.sB[m];
            oC += x * d.n.sC[m];
        }
    };
    auto k_place = [&](int64_t k, int64_t &a, int64_t &b) {
        int64_t x;
        a = b = 0;
        if (k >= d.K) return;
        for (int m = d.red.n - 1; m >= 0; --m) {
            k = divmod_pos(k, d.red.ext[m], x);
            a += x * d.red.sA[m];
            b += x * d.red.sB[m];
        }
    };
    auto few_singles = [&](int count) {
        constexpr int F = LeftSingles::kFew, K = LeftSingles::kFewK, P = LeftSingles::kFewPitch;
        double *ops = reinterpret_cast<double *>(sm.list + sm.kFewAt);  // output o: K of A, K of B from o P on
        const int pos = tid % K;
        const bool side = tid >= K;
        const bool live = tid < count;  // lanes of one warp: a multiply-add takes the unit as long for one lane
        int64_t oA, oB, oC = 0;
        double acc = 0.0;
        if (live) {
            place(sm.list[tid], oA, oB, oC);
            sm.kA[tid] = oA;
            sm.kB[tid] = oB;
            if (d.init != 2) acc = d.init == 1 ? d.beta * C[oC] : C[oC];
        }
        for (int64_t k0 = 0; k0 < d.K && count > 0; k0 += K) {
            __syncthreads();  // the places are there, the last operands have been read
            int64_t a, b;
            k_place(k0 + pos, a, b);
            const double *src = side ? B + b : A + a;
            const int64_t *at = side ? sm.kB : sm.kA;
            double v[F];
#pragma unroll
            for (int o = 0; o < F; ++o) v[o] = o < count && k0 + pos < d.K ? src[at[o]] : 0.0;
#pragma unroll
            for (int o = 0; o < F; ++o)
                if (o < count) ops[o * P + tid] = side || d.alpha_one ? v[o] : d.alpha * v[o];
            __syncthreads();
            if (!live) continue;
            const int len = (int)min((int64_t)K, d.K - k0);
            const double *q = ops + tid * P;
#pragma unroll 8
            for (int kk = 0; kk < len; ++kk) acc = fma(q[kk], q[K + kk], acc);
        }
        if (live) C[oC] = acc;
    };
    auto singles = [&](int count) {
        for (int e0 = 0; e0 < count; e0 += 256) {
            const bool live = e0 + tid < count;
            int64_t oA = 0, oB = 0, oC = 0;
            if (live) place(sm.list[e0 + tid], oA, oB, oC);
            double acc = 0.0;
            if (live && d.init != 2) acc = d.init == 1 ? d.beta * C[oC] : C[oC];
            for (int64_t k0 = 0; k0 < d.K; k0 += 256) {
                __syncthreads();  // the last offsets have been read
                int64_t a, b;
                k_place(k0 + tid, a, b);
                sm.kA[tid] = a;
                sm.kB[tid] = b;
                __syncthreads();
                if (!live) continue;
                const int len = (int)min((int64_t)256, d.K - k0);
                int kk = 0;
                for (; kk + kAhead <= len; kk += kAhead) {
                    double u[kAhead], v[kAhead];
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) {
                        u[i] = A[oA + sm.kA[kk + i]];
                        v[i] = B[oB + sm.kB[kk + i]];
                    }
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) acc = fma(d.alpha_one ? u[i] : d.alpha * u[i], v[i], acc);
                }
                for (; kk < len; ++kk) {
                    const double u = A[oA + sm.kA[kk]];
                    acc = fma(d.alpha_one ? u : d.alpha * u, B[oB + sm.kB[kk]], acc);
                }
            }
            if (live) C[oC] = acc;
        }
    };
    if (tid == 0) nlist = nwhole = 0;
    __syncthreads();
    int64_t x0 = 0;
    for (int64_t c = (int64_t)blockIdx.x * group; c < patches; c += stride, x0 += group) {
        uint32_t w[kPatches / 8];
#pragma unroll
        for (int i = 0; i < kPatches / 8; ++i) {
            int64_t pm;
            const int64_t pn = divmod_pos(c + warp + 8 * i, rp, pm);
            w[i] = 8 * i < group && c + warp + 8 * i < patches ? weak[pn * rows + pm * 32 + lane] : 0u;
        }
#pragma unroll
        for (int i = 0; i < kPatches / 8; ++i) {
            const uint32_t x = (uint32_t)x0 + warp + 8 * i;
            if (__all_sync(0xffffffffu, w[i] == ~0u)) {
                if (lane == 0) whole[atomicAdd(&nwhole, 1)] = x;
                continue;
            }
            for (uint32_t b = w[i]; b != 0; b &= b - 1) {
                const int at = atomicAdd(&nlist, 1);
                if (at < sm.kCap) sm.list[at] = x << 10 | lane << 5 | (__ffs((int)b) - 1);
            }
        }
        __syncthreads();
        const int count = min(nlist, sm.kCap), tiles = nwhole;
        if (c + stride < patches && count <= sm.kCap - sm.kStep && tiles <= kWhole - kPatches) continue;
        if (count <= sm.kFew) few_singles(count);
        else singles(count);
        __syncthreads();
        for (int i = 0; i < tiles; ++i) {
            int64_t pm;
            const int64_t pn = g0 + patch_at(whole[i], pm);
            if (pm < patch.tiles_m && pn < patch.tiles_n) Patch::run(patch, pm + patch.tiles_m * pn, buf);
            __syncthreads();
        }
        if (tid == 0) nlist = nwhole = 0;
        __syncthreads();
    }
    // the listed tiles, taken in turn: 64 x 64 where every SM gets eight, 32 x 32
    // where it gets four (with the four blocks that fit here 16 x 16 are slower
    // per output: 1024^2, K = 256, 534 against 490 us)
    const int64_t items = list ? list[0] : 0, tiles = items * sub_m * sub_n;
    const int shape = tiles >= 2 * (int64_t)gridDim.x ? 0 : (4 * tiles >= (int64_t)gridDim.x ? 1 : 2);
    const int rows_n = sub_m << shape, per = rows_n * (sub_n << shape);
    while (items > 0) {
        __syncthreads();  // the last tile's tables and number have been read
        if (tid == 0) taken = (int64_t)atomicAdd((unsigned long long *)list + 1, 1ull);
        __syncthreads();
        const int64_t q = taken;
        if (q >= items * per) break;
        const int64_t item = list[2 + q / per];
        const int sub = (int)(q % per);
        const int64_t tm = item % list_m * rows_n + sub % rows_n, tn = item / list_m * (per / rows_n) + sub / rows_n;
        if (shape == 0) {
            if (tm < d.tiles_m && tn < d.tiles_n) Tile::run(d, tm + d.tiles_m * tn, buf);
        } else if (shape == 1) {
            if (tm < patch.tiles_m && tn < patch.tiles_n) Patch::run(patch, tm + patch.tiles_m * tn, buf);
        } else if (tm < small.tiles_m && tn < small.tiles_n) {
            TileOf<double, 2>::run(small, tm + small.tiles_m * tn, buf);
        }
    }
}

// ---------------------------------------------------------------- copy
template <typename T>
__global__ void __launch_bounds__(256) gather_kernel(const GatherDesc g) {
    const T *__restrict__ src = (const T *)g.src;
    T *__restrict__ dst = (T *)g.dst;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < g.total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e, os = 0, od = 0;
        for (int m = 0; m < g.n; ++m) {
            const int64_t x = r % g.ext[m];
            r /= g.ext[m];
            os += x * g.ss[m];
            od += x * g.sd[m];
        }
        dst[od] = src[os];
    }
}

// ---------------------------------------------------------------- host helpers
int g_sm_count = 0;

int sm_count() {
    if (g_sm_count == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sm_count, cudaDevAttrMultiProcessorCount, dev);
        if (g_sm_count <= 0) g_sm_count = 1;
    }
    return g_sm_count;
}

int device_sms() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

int simt_shape(bool f64, int64_t M, int64_t N, int64_t tasks) {
    for (int s = 0; s + 1 < kSimtShapes; ++s) {
        const int64_t b = simt_rows(f64, s);
        if (((M + b - 1) / b) * ((N + b - 1) / b) * tasks >= (f64 ? (int64_t)device_sms() * 8 : (int64_t)device_sms() * 2 / 3)) return s;
    }
    return kSimtShapes - 1;
}

// A warp stores C along M: where C runs along N faster, M and N are exchanged
// (FP32 bca=iaj,jbic, 403 x 18018, K = 12: 44 us along the slower index, 26
// so).  Every product and sum stays the same.
void orient(TileDesc &t) {
    if (t.n.n == 0 || (t.m.n > 0 && t.m.sC[0] <= t.n.sC[0])) return;
    std::swap(t.m, t.n);
    std::swap(t.M, t.N);
    std::swap(t.A, t.B);
    std::swap(t.a_m_fast, t.b_n_fast);
    for (Dims *x : {&t.m, &t.n, &t.red, &t.task}) std::swap(x->sA, x->sB);
    t.swapped = 1;
}

// one launch over the first `tiles` tiles of d's shape
template <typename T>
void launch_tiles(const TileDesc &d, int64_t tiles, cudaStream_t st) {
    if (d.shape == 0) tile_kernel<T, 0><<<(unsigned)tiles, 256, 0, st>>>(d);
    else if (d.shape == 1) tile_kernel<T, 1><<<(unsigned)tiles, 256, 0, st>>>(d);
    else tile_kernel<T, 2><<<(unsigned)tiles, 256, 0, st>>>(d);
}

int64_t grid_for(int64_t total, int per_block) {
    int64_t blocks = (total + per_block - 1) / per_block;
    int64_t cap = (int64_t)sm_count() * 32;
    return std::max<int64_t>(1, std::min(blocks, cap));
}

void add_dim(Dims &d, int64_t ext, int64_t sA, int64_t sB, int64_t sC) {
    d.ext[d.n] = ext;
    d.sA[d.n] = sA;
    d.sB[d.n] = sB;
    d.sC[d.n] = sC;
    ++d.n;
}

// Per-operand addressing for one execution: original or workspace layout.
struct OpView {
    bool copied = false;
    const char *base = nullptr;        // workspace base when copied
    int64_t ws_stride[kMaxIdx] = {};   // workspace stride per index id
    bool ws_has[kMaxIdx] = {};
    // copy description
    std::vector<int> copy_ids;         // kernel modes, then non-phase dependencies
    int64_t elems = 0;
};

struct NestLayout {
    std::vector<int> phase_pos;   // positions of phase loops (contracted, <= q)
    std::vector<int> task_ids;    // free loop index ids, nest order
    std::vector<int> red_ids;     // contracted in-task loops, then kernel k
    std::vector<int> out_ids;     // kernel output modes
    OpView view[3];
    size_t ws_offset[3] = {0, 0, 0};
    size_t ws_bytes = 0;
};

NestLayout layout_for(const Plan &p, const Algorithm &alg) {
    NestLayout L;
    for (int pos = 0; pos < alg.nloops; ++pos) {
        int id = alg.loops[pos];
        if (p.cls[id] == CLS_CONTRACTED) {
            if (pos <= alg.q) L.phase_pos.push_back(pos);
            else L.red_ids.push_back(id);
        } else {
            L.task_ids.push_back(id);
        }
    }
    switch (alg.kernel) {
    case TC_KERNEL_DOT: L.red_ids.push_back(alg.kidx[0]); break;
    case TC_KERNEL_AXPY: L.out_ids.push_back(alg.kidx[0]); break;
    case TC_KERNEL_GEMV:
        L.out_ids.push_back(alg.kidx[0]);
        L.red_ids.push_back(alg.kidx[1]);
        break;
    case TC_KERNEL_GER:
        L.out_ids.push_back(alg.kidx[0]);
        L.out_ids.push_back(alg.kidx[1]);
        break;
    case TC_KERNEL_GEMM:
        L.out_ids.push_back(alg.kidx[0]);
        L.out_ids.push_back(alg.kidx[1]);
        L.red_ids.push_back(alg.kidx[2]);
        break;
    }
    size_t esz[3] = {elem_bytes_ab(p.dtype), elem_bytes_ab(p.dtype), elem_bytes_c(p.dtype)};
    size_t off = 0;
    for (int o = 0; o < 3; ++o) {
        if (alg.copy_level[o] == -2) continue;
        OpView &v = L.view[o];
        v.copied = true;
        const Layout &lay = p.op[o];
        // kernel modes in storage order, then the loops the slice depends on
        // that are not fixed by the phase, in nest order
        for (int m = 0; m < lay.n; ++m)
            for (int r = 0; r < alg.nk; ++r)
                if (lay.idx[m] == alg.kidx[r]) v.copy_ids.push_back(lay.idx[m]);
        for (int pos = 0; pos < alg.nloops; ++pos) {
            int id = alg.loops[pos];
            if (!lay.has(id)) continue;
            bool phase = p.cls[id] == CLS_CONTRACTED && pos <= alg.q;
            if (!phase) v.copy_ids.push_back(id);
        }
        int64_t s = 1;
        for (int id : v.copy_ids) {
            v.ws_stride[id] = s;
            v.ws_has[id] = true;
            s *= p.ext[id];
        }
        v.elems = s;
        L.ws_offset[o] = off;
        off += ((size_t)s * esz[o] + 255) / 256 * 256;
    }
    L.ws_bytes = off;
    return L;
}

template <typename T>
tc_status launch_gather(const GatherDesc &g, cudaStream_t st) {
    int64_t grid = grid_for(g.total, 256);
    gather_kernel<T><<<(unsigned)grid, 256, 0, st>>>(g);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? TC_SUCCESS : fail(TC_ERROR_CUDA, cudaGetErrorString(e));
}

// The gather moves elements of the operand's own size (FP64, FP32, or the
// 16-bit inputs of the BF16 / FP16 forms).
tc_status launch_copy(const Plan &p, int o, const OpView &v, const char *src_base,
                      void *dst, bool scatter, cudaStream_t st, double frac = 1.0) {
    GatherDesc g;
    std::memset(&g, 0, sizeof(g));
    g.n = (int)v.copy_ids.size();
    for (int m = 0; m < g.n; ++m) {
        int id = v.copy_ids[m];
        g.ext[m] = p.ext[id];
        int64_t orig = p.op[o].stride_of(id);
        int64_t ws = v.ws_stride[id];
        g.ss[m] = scatter ? ws : orig;
        g.sd[m] = scatter ? orig : ws;
    }
    g.total = frac >= 1.0 ? v.elems : std::max<int64_t>(1, (int64_t)(v.elems * frac));
    g.src = scatter ? dst : src_base;
    g.dst = scatter ? (void *)src_base : dst;
    const size_t eb = o == OP_C ? elem_bytes_c(p.dtype) : elem_bytes_ab(p.dtype);
    if (eb == 8) return launch_gather<double>(g, st);
    if (eb == 2) return launch_gather<unsigned short>(g, st);
    return launch_gather<float>(g, st);
}

template <typename T>
tc_status run_nest(Plan &p, const Algorithm &alg, T alpha, const T *A, const T *B,
                   T beta, T *C, cudaStream_t st, const Probe *probe) {
    NestLayout L = layout_for(p, alg);
    char *ws = (char *)p.workspace;
    const char *base[3] = {(const char *)A, (const char *)B, (const char *)C};
    const size_t esz = elem_bytes_ab(p.dtype);  // A and B (16 bits for the BF16 / FP16 forms)
    // tensor-core dtypes run their gemm phases on the tensor-core GETT
    const bool tensor = p.dtype != TC_F64 && p.dtype != TC_F32;
    // stride of index id in operand o as the phase kernel sees it
    auto stride_in = [&](int o, int id) -> int64_t {
        if (L.view[o].copied) return L.view[o].ws_has[id] ? L.view[o].ws_stride[id] : 0;
        return p.op[o].stride_of(id);
    };
    auto fill = [&](Dims &d, const std::vector<int> &ids) {
        d.n = 0;
        for (int id : ids)
            add_dim(d, p.ext[id], stride_in(OP_A, id), stride_in(OP_B, id), stride_in(OP_C, id));
    };
    const int init0 = beta == T(0) ? 2 : (beta == T(1) ? 0 : 1);
    const bool alpha_one = alpha == T(1);
    const bool tiled = alg.kernel == TC_KERNEL_GEMM;

    PhaseDesc pd;
    TileDesc td;
    int coop_g = 0;  // lanes per output of coop_reduce_kernel (0: elementwise_kernel)
    bool coop_thread = false;  // its sums in one thread
    std::memset(&pd, 0, sizeof(pd));
    std::memset(&td, 0, sizeof(td));
    int64_t ntasks = 1;
    for (int id : L.task_ids) ntasks *= p.ext[id];
    if (tiled) {
        std::vector<int> mi{L.out_ids[0]}, ni{L.out_ids[1]};
        fill(td.m, mi);
        fill(td.n, ni);
        fill(td.red, L.red_ids);
        fill(td.task, L.task_ids);
        td.M = p.ext[L.out_ids[0]];
        td.N = p.ext[L.out_ids[1]];
        td.K = 1;
        for (int id : L.red_ids) td.K *= p.ext[id];
        td.alpha = alpha;
        td.beta = beta;
        td.alpha_one = alpha_one;
        td.shape = simt_shape(sizeof(T) == 8, td.M, td.N, ntasks);
        // map threads along whichever of M / K is contiguous in memory
        int64_t kinA = td.red.n ? td.red.sA[td.red.n - 1] : 0;
        int64_t kinB = td.red.n ? td.red.sB[td.red.n - 1] : 0;
        td.a_m_fast = td.m.sA[0] <= kinA || kinA == 0;
        td.b_n_fast = td.n.sB[0] <= kinB || kinB == 0;
        if (!tensor) orient(td);
    } else {
        fill(pd.out, L.out_ids);
        fill(pd.task, L.task_ids);
        fill(pd.red, L.red_ids);
        int64_t nout = 1;
        for (int id : L.out_ids) nout *= p.ext[id];
        pd.total = nout * ntasks;
        pd.alpha = alpha;
        pd.beta = beta;
        pd.alpha_one = alpha_one;
        // Access pattern per kernel (Table 1 rows 1-4): one thread per
        // kernel output with consecutive threads along the output mode that
        // is contiguous in C (elementwise_kernel; ger's two output modes are
        // ordered so) -- axpy's vector and gemv's matrix with its free index
        // contiguous are then read coalesced; dot and gemv sum their own
        // contracted index in that thread.  When a phase has fewer outputs
        // than the device holds threads in one wave and its innermost
        // contracted index has unit stride in an input, a group of lanes per
        // output splits that index instead (coop_reduce_kernel, loads
        // contiguous across the group): the reduction, not the output count,
        // then sets the parallelism.  Where that index is short and outputs
        // are not few, one thread computes a group's sums (lane_sums_kernel);
        // a thread's positions follow one another, so with many of them more
        // outputs are needed (FP64, 19200 outputs of 5 x 23: 27 us in groups,
        // 34 so; 9802 of 15 x 10 23 and 30; 27000 of 5 x 4 17 and 14).
        const int kr = pd.red.n - 1;
        if (alg.kernel == TC_KERNEL_GER && pd.out.n == 2 && pd.out.sC[1] < pd.out.sC[0]) {
            std::swap(pd.out.ext[0], pd.out.ext[1]);
            std::swap(pd.out.sA[0], pd.out.sA[1]);
            std::swap(pd.out.sB[0], pd.out.sB[1]);
            std::swap(pd.out.sC[0], pd.out.sC[1]);
        }
        const bool k_unit = kr >= 0 && (pd.red.sA[kr] == 1 || pd.red.sB[kr] == 1);
        if (k_unit && pd.red.ext[kr] > 1 && pd.total < (int64_t)device_sms() * 1024) coop_g = 1;
        if (coop_g) {
            int64_t positions = 1;
            for (int m = 0; m < pd.red.n; ++m) positions *= pd.red.ext[m];
            coop_thread = pd.red.ext[kr] < 32 && pd.total >= (int64_t)device_sms() * (positions <= 64 ? 64 : 256);
            const int64_t kext = pd.red.ext[kr];
            coop_g = kext <= 4 ? 4 : (kext <= 8 ? 8 : (kext <= 16 ? 16 : 32));
        }
    }

    // C copy (reading for a C slice without a unit-stride mode): gather once,
    // run every phase on the workspace, scatter back at the end
    void *Cptr = C;
    tc_status s;
    const bool first_probe = !probe || probe->first;
    const double frac0 = probe ? probe->fraction : 1.0;
    if (L.view[OP_C].copied) {
        Cptr = ws + L.ws_offset[OP_C];
        if (init0 != 2 && first_probe) {
            s = launch_copy(p, OP_C, L.view[OP_C], base[OP_C], Cptr, false, st, frac0);
            if (s != TC_SUCCESS) return s;
        }
    }

    const int nph = (int)L.phase_pos.size();
    // one phase: its copies, then its kernel over `frac` of the work
    auto run_phase = [&](const std::vector<int64_t> &ph, bool first, int changed_from,
                         double frac) -> tc_status {
        // operand bases for this phase: fixed contracted indices applied
        const char *opb[2];
        for (int o = 0; o < 2; ++o) {
            int64_t off = 0;
            for (int k = 0; k < nph; ++k) off += ph[k] * p.op[o].stride_of(alg.loops[L.phase_pos[k]]);
            opb[o] = base[o] + off * (int64_t)esz;
        }
        const void *Aeff = opb[0], *Beff = opb[1];
        for (int o = 0; o < 2; ++o) {
            if (!L.view[o].copied) continue;
            void *dst = ws + L.ws_offset[o];
            int level = alg.copy_level[o];
            bool redo = first || level > alg.q;
            if (!redo) {
                for (int k = changed_from; k < nph; ++k)
                    if (L.phase_pos[k] <= level) redo = true;
            }
            if (redo) {
                tc_status cs = launch_copy(p, o, L.view[o], opb[o], dst, false, st, frac);
                if (cs != TC_SUCCESS) return cs;
            }
            if (o == 0) Aeff = dst;
            else Beff = dst;
        }
        const int init = first ? init0 : 0;
        auto cut = [&](int64_t n) { return frac >= 1.0 ? n : std::max<int64_t>(1, (int64_t)(n * frac)); };
        if (tiled && tensor) {
            NestGemm g;
            std::memset(&g, 0, sizeof(g));
            g.m = {td.m.ext[0], td.m.sA[0], 0, td.m.sC[0]};
            g.n = {td.n.ext[0], 0, td.n.sB[0], td.n.sC[0]};
            g.nk = td.red.n;
            for (int m = 0; m < td.red.n; ++m) g.k[m] = {td.red.ext[m], td.red.sA[m], td.red.sB[m], 0};
            g.nt = td.task.n;  // innermost task loop first (fastest)
            for (int m = 0; m < td.task.n; ++m) {
                const int x = td.task.n - 1 - m;
                g.t[m] = {td.task.ext[x], td.task.sA[x], td.task.sB[x], td.task.sC[x]};
            }
            g.A = Aeff;
            g.B = Beff;
            g.C = Cptr;
            g.alpha = (float)alpha;
            // init 0 (C += alpha acc, the later phases) is beta = 1
            g.init = init == 2 ? 2 : 1;
            g.beta = init == 1 ? (float)beta : 1.0f;
            return gett_launch_nest(p, g, frac, st);
        } else if (tiled) {
            td.A = td.swapped ? Beff : Aeff;
            td.B = td.swapped ? Aeff : Beff;
            td.C = Cptr;
            td.init = init;
            const int64_t b = simt_rows(sizeof(T) == 8, (int)td.shape);
            td.tiles_m = (td.M + b - 1) / b;
            td.tiles_n = (td.N + b - 1) / b;
            launch_tiles<T>(td, cut(td.tiles_m * td.tiles_n * ntasks), st);
        } else {
            PhaseDesc q = pd;
            q.A = Aeff;
            q.B = Beff;
            q.C = Cptr;
            q.init = init;
            q.total = cut(pd.total);
            if (coop_thread) {
                const unsigned grid = (unsigned)grid_for(q.total, 256);
                switch (coop_g) {
                    case 4: lane_sums_kernel<T, 4><<<grid, 256, 0, st>>>(q); break;
                    case 8: lane_sums_kernel<T, 8><<<grid, 256, 0, st>>>(q); break;
                    case 16: lane_sums_kernel<T, 16><<<grid, 256, 0, st>>>(q); break;
                    default: lane_sums_kernel<T, 32><<<grid, 256, 0, st>>>(q); break;
                }
            } else if (coop_g) {
                const int64_t grid = grid_for(q.total * coop_g, 256);
                switch (coop_g) {
                    case 4: coop_reduce_kernel<T, 4><<<(unsigned)grid, 256, 0, st>>>(q); break;
                    case 8: coop_reduce_kernel<T, 8><<<(unsigned)grid, 256, 0, st>>>(q); break;
                    case 16: coop_reduce_kernel<T, 16><<<(unsigned)grid, 256, 0, st>>>(q); break;
                    default: coop_reduce_kernel<T, 32><<<(unsigned)grid, 256, 0, st>>>(q); break;
                }
            } else {
                const unsigned grid = (unsigned)grid_for(q.total, 256);
                if (pd.red.n && pd.red.ext[pd.red.n - 1] >= 64) elementwise_kernel<T, true><<<grid, 256, 0, st>>>(q);
                else elementwise_kernel<T, false><<<grid, 256, 0, st>>>(q);
            }
        }
        cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? TC_SUCCESS : fail(TC_ERROR_CUDA, cudaGetErrorString(e));
    };

    if (probe) {
        std::vector<int64_t> ph(nph, 0);
        for (int k = 0; k < nph && k < (int)probe->phase.size(); ++k)
            ph[k] = std::min<int64_t>(probe->phase[k], p.ext[alg.loops[L.phase_pos[k]]] - 1);
        return run_phase(ph, probe->first, probe->changed_from, probe->fraction);
    }

    std::vector<int64_t> ph(nph, 0);
    bool first = true;
    int changed_from = 0;  // outermost phase digit that changed
    for (;;) {
        s = run_phase(ph, first, changed_from, 1.0);
        if (s != TC_SUCCESS) return s;
        first = false;
        // advance the phase odometer (innermost phase loop fastest)
        int k = nph - 1;
        while (k >= 0) {
            if (++ph[k] < p.ext[alg.loops[L.phase_pos[k]]]) break;
            ph[k] = 0;
            --k;
        }
        if (k < 0) break;
        changed_from = k;
    }
    if (L.view[OP_C].copied) {
        s = launch_copy(p, OP_C, L.view[OP_C], base[OP_C], Cptr, true, st);
        if (s != TC_SUCCESS) return s;
    }
    return TC_SUCCESS;
}

// SIMT GETT: the whole contraction as one tiled kernel, M = free indices
// of A, N = free indices of B, K = contracted indices.
// The SIMT GETT's descriptor: M = free indices of A, N = free indices of B
// (each sorted by their C stride), K = contracted indices with the one
// contiguous in A (or else in B) innermost; the tile shape by simt_shape; with
// `oriented` A's and B's sides exchanged where orient would.
template <typename T>
void describe_gett_simt(const Plan &p, T alpha, const T *A, const T *B, T beta, T *C, TileDesc &td, bool oriented = true) {
    std::memset(&td, 0, sizeof(td));
    auto by_c_stride = [&](std::vector<int> ids) {
        std::stable_sort(ids.begin(), ids.end(), [&](int x, int y) {
            return p.op[OP_C].stride_of(x) < p.op[OP_C].stride_of(y);
        });
        return ids;
    };
    std::vector<int> mi = by_c_stride(p.freeA), ni = by_c_stride(p.freeB);
    // K: the contracted index contiguous in A (or else in B) innermost
    std::vector<int> ki(p.contracted);
    std::stable_sort(ki.begin(), ki.end(), [&](int x, int y) {
        int64_t mx = std::min(p.op[OP_A].stride_of(x), p.op[OP_B].stride_of(x));
        int64_t my = std::min(p.op[OP_A].stride_of(y), p.op[OP_B].stride_of(y));
        return mx > my;
    });
    auto fill = [&](Dims &d, const std::vector<int> &ids) {
        d.n = 0;
        for (int id : ids)
            add_dim(d, p.ext[id], p.op[OP_A].stride_of(id), p.op[OP_B].stride_of(id),
                    p.op[OP_C].stride_of(id));
    };
    fill(td.m, mi);
    fill(td.n, ni);
    fill(td.red, ki);
    fill(td.task, p.batch);  // batch indices: one task per value, all three operands offset
    td.M = td.N = td.K = 1;
    for (int id : mi) td.M *= p.ext[id];
    for (int id : ni) td.N *= p.ext[id];
    for (int id : ki) td.K *= p.ext[id];
    td.A = A;
    td.B = B;
    td.C = C;
    td.alpha = alpha;
    td.beta = beta;
    td.alpha_one = alpha == T(1);
    td.init = beta == T(0) ? 2 : (beta == T(1) ? 0 : 1);
    int64_t kinA = td.red.n ? td.red.sA[td.red.n - 1] : 0;
    int64_t kinB = td.red.n ? td.red.sB[td.red.n - 1] : 0;
    td.a_m_fast = td.m.n ? (td.m.sA[0] <= kinA || kinA == 0) : 0;
    td.b_n_fast = td.n.n ? (td.n.sB[0] <= kinB || kinB == 0) : 0;
    int64_t tasks = 1;
    for (int id : p.batch) tasks *= p.ext[id];
    if (oriented) orient(td);
    td.shape = simt_shape(sizeof(T) == 8, td.M, td.N, tasks);
    const int64_t bm = simt_rows(sizeof(T) == 8, (int)td.shape);
    td.tiles_m = (td.M + bm - 1) / bm;
    td.tiles_n = (td.N + bm - 1) / bm;
}

int64_t task_count(const TileDesc &td) {
    int64_t t = 1;
    for (int m = 0; m < td.task.n; ++m) t *= td.task.ext[m];
    return t;
}

template <typename T>
tc_status run_gett_simt(Plan &p, T alpha, const T *A, const T *B, T beta, T *C,
                        cudaStream_t st, const Probe *probe) {
    TileDesc td;
    describe_gett_simt<T>(p, alpha, A, B, beta, C, td);
    auto cut = [&](int64_t n) {
        return !probe || probe->fraction >= 1.0 ? n : std::max<int64_t>(1, (int64_t)(n * probe->fraction));
    };
    const int64_t tiles = td.tiles_m * td.tiles_n * task_count(td);
    if (tiles > 0x7fffffff) return fail(TC_ERROR_INVALID_EXTENT, "too many tiles for one launch");
    launch_tiles<T>(td, cut(tiles), st);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? TC_SUCCESS
                            : fail(TC_ERROR_CUDA, std::string("GETT tile_kernel launch (") +
                                                      std::to_string(td.tiles_m * td.tiles_n) + " tiles): " +
                                                      cudaGetErrorString(e));
}

}  // namespace

tc_status simt_run_left(Plan &p, const void *alpha, const void *A, const void *B, const void *beta, void *C,
                        const uint32_t *weak, int64_t rows, int64_t g0, int64_t g1, int64_t *list, int64_t list_m,
                        int item_rows, int item_cols, void *stream) {
    TileDesc td;
    describe_gett_simt<double>(p, *(const double *)alpha, (const double *)A, (const double *)B, *(const double *)beta, (double *)C, td, false);
    auto shaped = [&](int shape) {
        TileDesc t = td;
        const int b = simt_rows(true, shape);
        t.shape = shape;
        t.tiles_m = (t.M + b - 1) / b;
        t.tiles_n = (t.N + b - 1) / b;
        return t;
    };
    const int b = simt_rows(true, 0);
    const unsigned grid = (unsigned)device_sms() * 4;
    left_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(shaped(0), shaped(1), shaped(2), weak, rows, g0, g1, list, list_m,
                                                         item_rows / b, item_cols / b);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? TC_SUCCESS : fail(TC_ERROR_CUDA, cudaGetErrorString(e));
}

size_t simt_desc_bytes() { return sizeof(TileDesc); }

int64_t simt_fill_desc(const Plan &p, const void *A, const void *B, void *C, int64_t tile0, void *out) {
    TileDesc td;
    if (p.dtype == TC_F64)
        describe_gett_simt<double>(p, 1.0, (const double *)A, (const double *)B, 0.0, (double *)C, td);
    else
        describe_gett_simt<float>(p, 1.0f, (const float *)A, (const float *)B, 0.0f, (float *)C, td);
    td.tile0 = tile0;
    std::memcpy(out, &td, sizeof(td));
    return td.tiles_m * td.tiles_n * task_count(td);
}

tc_status simt_launch_batch(tc_dtype dt, const void *ddescs, const int32_t *dtile_prob, int64_t ntiles,
                            void *stream) {
    if (ntiles <= 0) return TC_SUCCESS;
    if (ntiles > 0x7fffffff) return fail(TC_ERROR_INVALID_ARGUMENT, "batch has too many tiles");
    cudaStream_t st = (cudaStream_t)stream;
    if (dt == TC_F64)
        tile_batch_kernel<double><<<(unsigned)ntiles, 256, 0, st>>>((const TileDesc *)ddescs, dtile_prob);
    else
        tile_batch_kernel<float><<<(unsigned)ntiles, 256, 0, st>>>((const TileDesc *)ddescs, dtile_prob);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? TC_SUCCESS : fail(TC_ERROR_CUDA, cudaGetErrorString(e));
}

int64_t nest_phase_items(const Plan &p, const Algorithm &alg, bool *tiled) {
    NestLayout L = layout_for(p, alg);
    int64_t ntasks = 1;
    for (int id : L.task_ids) ntasks *= p.ext[id];
    if (alg.kernel == TC_KERNEL_GEMM) {
        *tiled = true;
        const int64_t M = p.ext[L.out_ids[0]], N = p.ext[L.out_ids[1]];
        const bool f64 = p.dtype == TC_F64, simt = f64 || p.dtype == TC_F32;
        const int64_t bm = simt ? simt_rows(f64, simt_shape(f64, M, N, ntasks)) : 128;
        return ((M + bm - 1) / bm) * ((N + bm - 1) / bm) * ntasks;
    }
    *tiled = false;
    int64_t nout = 1;
    for (int id : L.out_ids) nout *= p.ext[id];
    return nout * ntasks;
}

int64_t gett_items(const Plan &p) {
    int64_t M = 1, N = 1, H = 1;
    for (int id : p.freeA) M *= p.ext[id];
    for (int id : p.freeB) N *= p.ext[id];
    for (int id : p.batch) H *= p.ext[id];
    if (p.dtype == TC_F64 || p.dtype == TC_F32) {
        const bool f64 = p.dtype == TC_F64;
        const int64_t b = simt_rows(f64, simt_shape(f64, M, N, H));
        return ((M + b - 1) / b) * ((N + b - 1) / b) * H;
    }
    const int64_t bn = p.gett_bn ? p.gett_bn : (N >= 256 ? 256 : 128);
    return ((M + 127) / 128) * ((N + bn - 1) / bn) * H;
}

size_t nest_workspace_bytes(const Plan &p, const Algorithm &alg) {
    return layout_for(p, alg).ws_bytes;
}

tc_status ensure_device_resources(Plan &p, size_t workspace_bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
    if (p.device < 0) {
        p.device = dev;
    } else if (p.device != dev) {
        return fail(TC_ERROR_INVALID_ARGUMENT, "plan used on a different device than its first execute");
    }
    if (!p.dev_status) {
        e = cudaMalloc((void **)&p.dev_status, sizeof(int) * 4);
        if (e != cudaSuccess) return fail(TC_ERROR_OUT_OF_MEMORY, cudaGetErrorString(e));
        cudaMemset(p.dev_status, 0, sizeof(int) * 4);
    }
    if (workspace_bytes > p.workspace_bytes) {
        if (p.workspace) cudaFree(p.workspace);
        p.workspace = nullptr;
        p.workspace_bytes = 0;
        e = cudaMalloc(&p.workspace, workspace_bytes);
        if (e != cudaSuccess) {
            p.workspace = nullptr;
            return fail(TC_ERROR_OUT_OF_MEMORY, cudaGetErrorString(e));
        }
        p.workspace_bytes = workspace_bytes;
    }
    return TC_SUCCESS;
}

tc_status exec_nest(Plan &p, const Algorithm &alg, const void *alpha, const void *A,
                    const void *B, const void *beta, void *C, void *stream, const Probe *probe) {
    if (p.dtype != TC_F64 && p.dtype != TC_F32 && alg.kernel != TC_KERNEL_GEMM)
        return fail(TC_ERROR_UNSUPPORTED_DTYPE,
                    "at tensor-core dtypes only the gemm loop nests (on the tensor cores) and the GETT run; "
                    "dot / axpy / gemv / ger nests run in FP64 or FP32");
    if (p.dtype == TC_E4M3)
        return fail(TC_ERROR_UNSUPPORTED_DTYPE, "TC_E4M3 runs the fused GETT (algorithm 0) only");
    tc_status s = ensure_device_resources(p, nest_workspace_bytes(p, alg));
    if (s != TC_SUCCESS) return s;
    p.last_stream = stream;
    cudaStream_t st = (cudaStream_t)stream;
    if (p.dtype == TC_F64)
        return run_nest<double>(p, alg, *(const double *)alpha, (const double *)A,
                                (const double *)B, *(const double *)beta, (double *)C, st, probe);
    return run_nest<float>(p, alg, *(const float *)alpha, (const float *)A, (const float *)B,
                           *(const float *)beta, (float *)C, st, probe);
}

tc_status exec_gett_simt(Plan &p, const void *alpha, const void *A, const void *B,
                         const void *beta, void *C, void *stream, const Probe *probe) {
    tc_status s = ensure_device_resources(p, 0);
    if (s != TC_SUCCESS) return s;
    p.last_stream = stream;
    cudaStream_t st = (cudaStream_t)stream;
    if (p.dtype == TC_F64)
        return run_gett_simt<double>(p, *(const double *)alpha, (const double *)A,
                                     (const double *)B, *(const double *)beta, (double *)C, st, probe);
    return run_gett_simt<float>(p, *(const float *)alpha, (const float *)A, (const float *)B,
                                *(const float *)beta, (float *)C, st, probe);
}

}  // namespace tc

// ---------------------------------------------------------------- no-alloc entry point
// A variant of the loop-nest executor whose copy workspace lives in a fixed
// device array instead of memory the plan allocates.  The paper has no
// counterpart; it serves callers that must not allocate device memory.
namespace tc {
namespace {

constexpr size_t kStaticScratchBytes = (size_t)16 << 20;  // 16 MiB per device
constexpr int kMaxDevices = 64;

// One copy per device that loads the library, held until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

std::mutex g_static_mu;
void *g_static_ptr[kMaxDevices] = {};

// Device address of the array on the current device, looked up once per
// device (host code cannot use the symbol itself as a device pointer).
tc_status static_scratch(void **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(TC_ERROR_CUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return fail(TC_ERROR_INVALID_ARGUMENT, "device ordinal too large");
    std::lock_guard<std::mutex> g(g_static_mu);
    if (!g_static_ptr[dev]) {
        void *ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess || !ptr) return fail(TC_ERROR_CUDA, e != cudaSuccess ? cudaGetErrorString(e) : "null symbol address");
        g_static_ptr[dev] = ptr;
    }
    *out = g_static_ptr[dev];
    return TC_SUCCESS;
}

}  // namespace
}  // namespace tc

extern "C" tc_status tc_execute_no_alloc(tc_plan plan, const void *alpha, const void *A, const void *B,
                                         const void *beta, void *C, void *stream) {
    using namespace tc;
    if (!plan) return fail(TC_ERROR_INVALID_ARGUMENT, "plan is NULL");
    if (!alpha || !beta || !A || !B || !C) return fail(TC_ERROR_INVALID_ARGUMENT, "NULL argument");
    Plan &p = plan->p;
    if (p.dtype != TC_F64 && p.dtype != TC_F32)
        return fail(TC_ERROR_UNSUPPORTED_DTYPE, "tc_execute_no_alloc runs the FP64/FP32 loop-nest algorithms");
    const Algorithm &alg = p.algs[p.selected];
    if (alg.kernel == TC_KERNEL_GETT)
        return fail(TC_ERROR_INVALID_ALGORITHM, "tc_execute_no_alloc runs the loop-nest algorithms (ids >= 1)");
    const size_t need = nest_workspace_bytes(p, alg);
    if (need > kStaticScratchBytes)
        return fail(TC_ERROR_INVALID_ARGUMENT,
                    "algorithm needs " + std::to_string(need) + " bytes of copy scratch; the static scratch holds " +
                        std::to_string(kStaticScratchBytes) + " bytes (use tc_execute)");
    void *scratch = nullptr;
    tc_status s = static_scratch(&scratch);
    if (s != TC_SUCCESS) return s;
    // run the same executor with the workspace pointed at the static array
    void *saved = p.workspace;
    const size_t saved_bytes = p.workspace_bytes;
    p.workspace = scratch;
    p.workspace_bytes = kStaticScratchBytes;
    cudaStream_t st = (cudaStream_t)stream;
    if (p.dtype == TC_F64)
        s = run_nest<double>(p, alg, *(const double *)alpha, (const double *)A, (const double *)B,
                             *(const double *)beta, (double *)C, st, nullptr);
    else
        s = run_nest<float>(p, alg, *(const float *)alpha, (const float *)A, (const float *)B,
                            *(const float *)beta, (float *)C, st, nullptr);
    p.workspace = saved;
    p.workspace_bytes = saved_bytes;
    return s;
}
