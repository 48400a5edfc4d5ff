// Device kernels of libtn (sm_103a).
//
//  * cgemm_row / cgemm_tile: one pairwise contraction step (Sec. I, contraction tree;
//    the per-slice work of Sec. I.C) as a batched complex GEMM
//        C[v][bat][m][n] = sum_k A[v][bat][m][k] * B[v][bat][n][k]
//    over versions v (slice assignments of the sliced legs the operands depend on),
//    with the permutation of the result fused into the epilogue: element (bat, m, n)
//    goes to bit-scattered address pos_bat(bat) + pos_m(m) + pos_n(n).
//  * materialize: writes leaf tensors in the layout their consumer reads, fixing the
//    sliced legs (one copy per slice value) and binding closed output legs to the
//    batch pattern (the batch-indexed selector <b_B|).
//  * slice_sum: FP64 sum over the slice set (Sec. I.C step 1), 16 values at a time in slice order;
//    root_slice_sum: the same sum fused with a root step that runs the row kernel.
//  * draw / sampler: Philox4x32-10 draws and the modified frugal rejection step
//    (Sec. II.A), one warp per batch of 64.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "chunk_sum.h"
#include "widen.h"

namespace tnk {

constexpr int kMaxBits = 40;

// Storage formats of a tensor (chosen by the kernel that reads it): interleaved
// complex64, or four planes (re_hi, re_lo, im_hi, im_lo) of bf16 / fp16 with x = hi + lo,
// plane stride = the tensor's element count.  Both use 8 bytes per element.
enum OutFmt { OUT_C64 = 0, OUT_SPLIT_BF16 = 1, OUT_SPLIT_FP16 = 2 };

// A step operand whose closed output legs are selected per batch.  src stores the
// operand with its nq closed legs as the top bits (every value of those legs, shared by
// all batches); dst is the operand as the step reads it: nbits layout bits of which the
// beta bits sit at pos_beta[t] and the other nbits - lb bits are src's low bits in order.
// dst element e of batch beta = src element (sel << (nbits - lb)) | rest(e), where sel
// packs the batch pattern's bits q[0], q[1], ... (closed positions).
struct GatherDesc {
    const char *src;
    char *dst;
    long long nver;              // versions (each: nplanes planes)
    long long src_plane, dst_plane;  // elements per plane
    int nplanes, esize;          // 4 x 2 B (split) or 1 x 8 B / 16 B
    int nbits, lb, nq;
    int vec_log2;                // log2 of elements per 16-byte chunk (0 when runs are shorter)
    int run_log2;                // log2 of chunks per run: dst positions below the lowest beta
                                 // position, where batch and selection stay constant
    int8_t pos_beta[16];         // beta bit t -> dst position, sorted by descending position
    int8_t beta_bit[16];         // ... and which beta bit sits there
    int16_t q[32];
    // byte lookup tables of the same maps (built on the host): for byte j of e and value x,
    // rest_tab[j][x] and beta_tab[j][x] are the contributions of x << 8j to the source's low
    // bits and to the batch index; sel_tab[j][x] that of byte j of the batch pattern
    const uint64_t *rest_tab;    // [5][256]
    const uint32_t *beta_tab;    // [5][256]
    const uint32_t *sel_tab;     // [8][256]
};
constexpr int kGatherTabWords = 5 * 256 + (5 * 256 + 8 * 256) / 2;  // 64-bit words per gather

// Source element of dst element e (a run's first element in the run path).
__device__ __forceinline__ long long gather_src(const GatherDesc &d, long long e, const uint64_t *closed_bits) {
    uint64_t rest = 0;
    uint32_t beta = 0;
#pragma unroll
    for (int j = 0; j < 5; j++) {
        const uint32_t x = (uint32_t)(e >> (8 * j)) & 255u;
        rest |= __ldg(&d.rest_tab[j * 256 + x]);
        beta |= __ldg(&d.beta_tab[j * 256 + x]);
    }
    const uint64_t pat = closed_bits[beta];
    uint64_t sel = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) sel |= __ldg(&d.sel_tab[j * 256 + (uint32_t)((pat >> (8 * j)) & 255u)]);
    return (long long)((sel << (d.nbits - d.lb)) | rest);
}

struct GemmParams {
    const void *const *ptrA;  // per C-version operand base
    const void *const *ptrB;
    void *C;                  // C base (version v at C + v * c_vstride elements)
    long long c_vstride;      // elements
    long long nver;
    int lm, ln, lk, lbat;     // log2 of M, N, K, BAT
    int out_fmt;              // OutFmt of C
    float out_scale;          // multiplier applied before storing
    int swapped;              // operands exchanged (A holds the step's B): keep the step's
                              // operand order inside each complex multiply-add
    // row, tile, long-K and small-step kernels: operands read through their batch gather
    // instead of a gathered copy (null: not gathered); closed_bits are the group's patterns
    const GatherDesc *gA, *gB;
    const uint64_t *closed_bits;
    int *err;                 // long-K kernel: set to 1 if a bounded wait gives up
    int8_t pos_bat[kMaxBits], pos_m[kMaxBits], pos_n[kMaxBits];
};

// Split x into hi + lo in the operand type and store both parts at plane stride.
__device__ __forceinline__ void store_split(void *base, long long plane, long long off, float2 x, bool fp16) {
    if (fp16) {
        __half *h = static_cast<__half *>(base);
        const __half rh = __float2half_rn(x.x), ih = __float2half_rn(x.y);
        h[off] = rh;
        h[plane + off] = __float2half_rn(x.x - __half2float(rh));
        h[2 * plane + off] = ih;
        h[3 * plane + off] = __float2half_rn(x.y - __half2float(ih));
    } else {
        __nv_bfloat16 *h = static_cast<__nv_bfloat16 *>(base);
        const __nv_bfloat16 rh = __float2bfloat16_rn(x.x), ih = __float2bfloat16_rn(x.y);
        h[off] = rh;
        h[plane + off] = __float2bfloat16_rn(x.x - __bfloat162float(rh));
        h[2 * plane + off] = ih;
        h[3 * plane + off] = __float2bfloat16_rn(x.y - __bfloat162float(ih));
    }
}

// Store one complex64 result of version v in C's format.
__device__ __forceinline__ void store_c(const GemmParams &p, long long v, long long off, float2 x) {
    x.x *= p.out_scale;
    x.y *= p.out_scale;
    if (p.out_fmt == OUT_C64) {
        static_cast<float2 *>(p.C)[v * p.c_vstride + off] = x;
    } else {
        unsigned short *base = static_cast<unsigned short *>(p.C) + 4 * v * p.c_vstride;
        store_split(base, p.c_vstride, off, x, p.out_fmt == OUT_SPLIT_FP16);
    }
}
template <typename T> __device__ __forceinline__ void store_c_t(const GemmParams &p, long long v, long long off, T x);
template <> __device__ __forceinline__ void store_c_t<float2>(const GemmParams &p, long long v, long long off, float2 x) {
    store_c(p, v, off, x);
}

__device__ __forceinline__ long long scatter_bits(long long x, const int8_t *pos, int nbits) {
    long long off = 0;
#pragma unroll 4
    for (int i = 0; i < nbits; i++) off |= ((x >> i) & 1LL) << pos[i];
    return off;
}

__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
    c.x = fmaf(a.x, b.x, c.x);
    c.x = fmaf(-a.y, b.y, c.x);
    c.y = fmaf(a.x, b.y, c.y);
    c.y = fmaf(a.y, b.x, c.y);
    return c;
}
template <typename T> __device__ __forceinline__ T czero();
template <> __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }

// One output row (v, bat, m) per thread and call; all N (<= 32) columns in registers.  For the
// gate-absorption steps (small N and K), which are bound by HBM bandwidth.
// Offset of a gathered operand's element e in its shared storage.  Lanes of a warp whose
// elements share the batch and selection (same e >> shift) take the leader's decode.
__device__ __forceinline__ long long gather_src_warp(const GatherDesc &d, long long e, int shift,
                                                     const uint64_t *closed_bits) {
    const unsigned mask = __activemask();
    const int leader = __ffs(mask) - 1;
    const long long e0 = __shfl_sync(mask, e, leader);
    if (__all_sync(mask, (e >> shift) == (e0 >> shift))) {
        long long s0 = 0;
        if ((int)(threadIdx.x & 31) == leader) s0 = gather_src(d, e0, closed_bits);
        s0 = __shfl_sync(mask, s0, leader);
        return s0 + (e - e0);
    }
    return gather_src(d, e, closed_bits);
}

template <typename T, int N>
__device__ __forceinline__ void cgemm_row_one(const GemmParams &p, long long row) {
    const long long M = 1LL << p.lm;
    const long long m = row & (M - 1);
    const long long bat = (row >> p.lm) & ((1LL << p.lbat) - 1);
    const long long v = row >> (p.lm + p.lbat);
    const int K = 1 << p.lk;
    const T *A, *B;
    if (p.gA) {
        const long long e = ((bat << p.lm) | m) << p.lk;
        A = reinterpret_cast<const T *>(p.gA->src) + gather_src_warp(*p.gA, e, p.gA->pos_beta[p.gA->lb - 1], p.closed_bits);
    } else {
        A = static_cast<const T *>(p.ptrA[v]) + (((bat << p.lm) | m) << p.lk);
    }
    if (p.gB) {
        const long long e = bat << (p.ln + p.lk);
        B = reinterpret_cast<const T *>(p.gB->src) + gather_src_warp(*p.gB, e, p.gB->pos_beta[p.gB->lb - 1], p.closed_bits);
    } else {
        B = static_cast<const T *>(p.ptrB[v]) + (bat << (p.ln + p.lk));
    }
    T acc[N];
#pragma unroll
    for (int n = 0; n < N; n++) acc[n] = czero<T>();
    // complex64 rows of even K are read 16 bytes (two elements) at a time; the
    // accumulation order over k is the same either way
    auto step = [&](const T a, int k) {
        if (p.swapped) {
#pragma unroll
            for (int n = 0; n < N; n++) acc[n] = cfma(__ldg(&B[(n << p.lk) + k]), a, acc[n]);
        } else {
#pragma unroll
            for (int n = 0; n < N; n++) acc[n] = cfma(a, __ldg(&B[(n << p.lk) + k]), acc[n]);
        }
    };
    if constexpr (sizeof(T) == 8) {
        if (K >= 2) {
            for (int k = 0; k < K; k += 2) {
                const float4 v = *reinterpret_cast<const float4 *>(A + k);
                step(make_float2(v.x, v.y), k);
                step(make_float2(v.z, v.w), k + 1);
            }
        } else {
            step(A[0], 0);
        }
    } else {
        for (int k = 0; k < K; k++) step(A[k], k);
    }
    const long long cb = scatter_bits(bat, p.pos_bat, p.lbat) + scatter_bits(m, p.pos_m, p.lm);
#pragma unroll
    for (int n = 0; n < N; n++) store_c_t<T>(p, v, cb + scatter_bits(n, p.pos_n, p.ln), acc[n]);
}

// Grid-stride over rows (the grid is bounded by the launch).
template <typename T, int N>
__global__ void __launch_bounds__(256) cgemm_row(GemmParams p) {
    const long long rows = p.nver << (p.lbat + p.lm);
    for (long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
         row += (long long)gridDim.x * blockDim.x)
        cgemm_row_one<T, N>(p, row);
}

// The row kernel with coalesced row reads, for complex64 rows of 16 <= K <= 64: each warp
// copies its 32 rows into shared memory (K/2 lanes per row, 16 bytes each, 64/K rows per
// load instruction), then each lane forms its own row's N outputs exactly as cgemm_row_one
// does (the same k order and multiply-add operand order), so the results are
// bit-identical.  Rows sit kRowPad bytes apart beyond their length, which keeps the lanes'
// 16-byte shared reads free of bank conflicts.
constexpr int kRowWarps = 4;     // warps per block
constexpr int kRowPad = 16;      // bytes between staged rows
template <int N>
__global__ void __launch_bounds__(32 * kRowWarps) cgemm_rowstage(GemmParams p) {
    extern __shared__ __align__(16) unsigned char rowstage_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = 1 << p.lk;
    const int rstride = 8 * K + kRowPad;  // bytes
    unsigned char *stage = rowstage_smem + (size_t)warp * 32 * rstride;
    const long long M = 1LL << p.lm;
    const long long rows = p.nver << (p.lbat + p.lm);
    const int lpr = K >> 1;         // lanes per row (16 bytes = two complex64 each)
    const int rpi = 32 / lpr;       // rows per load instruction
    for (long long r0 = ((long long)blockIdx.x * kRowWarps + warp) * 32; r0 < rows;
         r0 += (long long)gridDim.x * kRowWarps * 32) {
        // this lane's row and its operand bases
        const long long row = r0 + lane;
        const bool live = row < rows;
        const long long m = row & (M - 1);
        const long long bat = (row >> p.lm) & ((1LL << p.lbat) - 1);
        const long long v = row >> (p.lm + p.lbat);
        const float2 *A = nullptr, *B = nullptr;
        if (live) {
            if (p.gA) {
                const long long e = ((bat << p.lm) | m) << p.lk;
                A = reinterpret_cast<const float2 *>(p.gA->src) +
                    gather_src_warp(*p.gA, e, p.gA->pos_beta[p.gA->lb - 1], p.closed_bits);
            } else {
                A = static_cast<const float2 *>(p.ptrA[v]) + (((bat << p.lm) | m) << p.lk);
            }
            if (p.gB) {
                const long long e = bat << (p.ln + p.lk);
                B = reinterpret_cast<const float2 *>(p.gB->src) +
                    gather_src_warp(*p.gB, e, p.gB->pos_beta[p.gB->lb - 1], p.closed_bits);
            } else {
                B = static_cast<const float2 *>(p.ptrB[v]) + (bat << (p.ln + p.lk));
            }
        }
        // stage the warp's rows: in instruction j, lane l copies chunk l % lpr of row
        // j * rpi + l / lpr
        const unsigned long long abase = reinterpret_cast<unsigned long long>(A);
        for (int j = 0; j < 32; j += rpi) {
            const int rr = j + lane / lpr;
            const unsigned long long src = __shfl_sync(0xffffffffu, abase, rr);
            if (r0 + rr < rows) {
                const int c = lane % lpr;
                const float4 x = *reinterpret_cast<const float4 *>(src + 16ull * c);
                *reinterpret_cast<float4 *>(stage + (size_t)rr * rstride + 16 * c) = x;
            }
        }
        __syncwarp();
        if (live) {
            const float2 *a = reinterpret_cast<const float2 *>(stage + (size_t)lane * rstride);
            float2 acc[N];
#pragma unroll
            for (int n = 0; n < N; n++) acc[n] = czero<float2>();
            for (int k = 0; k < K; k += 2) {
                const float4 q = *reinterpret_cast<const float4 *>(a + k);
                const float2 x0 = make_float2(q.x, q.y), x1 = make_float2(q.z, q.w);
                if (p.swapped) {
#pragma unroll
                    for (int n = 0; n < N; n++) acc[n] = cfma(__ldg(&B[(n << p.lk) + k]), x0, acc[n]);
#pragma unroll
                    for (int n = 0; n < N; n++) acc[n] = cfma(__ldg(&B[(n << p.lk) + k + 1]), x1, acc[n]);
                } else {
#pragma unroll
                    for (int n = 0; n < N; n++) acc[n] = cfma(x0, __ldg(&B[(n << p.lk) + k]), acc[n]);
#pragma unroll
                    for (int n = 0; n < N; n++) acc[n] = cfma(x1, __ldg(&B[(n << p.lk) + k + 1]), acc[n]);
                }
            }
            const long long cb = scatter_bits(bat, p.pos_bat, p.lbat) + scatter_bits(m, p.pos_m, p.lm);
#pragma unroll
            for (int n = 0; n < N; n++) store_c_t<float2>(p, v, cb + scatter_bits(n, p.pos_n, p.ln), acc[n]);
        }
        __syncwarp();  // the stage is rewritten by the next iteration
    }
}

// Small steps, several to a launch: the steps of one launch have all their operands ready
// and write disjoint results.  Block b computes outputs [blocks[b].y, blocks[b].y + 128) of
// step descs[blocks[b].x], one per thread, accumulated as cgemm_row_one does (k ascending,
// the step's operand order), so the bits are those of a launch of its own.  Bound by launch
// latency: a 12-qubit circuit's 33 steps took 3.6 us each, nearly all of it the launch and
// the wait for the step before.  Gathered operands are decoded per row if a row is
// contiguous in the stored form, else per element.  Whole calls: that circuit 127 -> 86 us,
// 20 qubits in split bf16 (92 steps) 501 -> 264 us.
constexpr int kSmallBlock = 128;
// One output of a small step: what can be worked out before the operands exist.
struct SmallWork {
    const float2 *A, *B;  // the operands' rows (null: no output, or elements decoded one by one)
    long long o, off;     // output, its position in C
    long long v;
    bool any;
};
__device__ __forceinline__ SmallWork small_prepare(const GemmParams &p, long long o, const uint64_t *closed_bits) {
    SmallWork w = {nullptr, nullptr, o, 0, 0, o < p.nver << (p.lbat + p.lm + p.ln)};
    if (!w.any) return w;
    const long long n = o & ((1LL << p.ln) - 1), m = (o >> p.ln) & ((1LL << p.lm) - 1);
    const long long bat = (o >> (p.ln + p.lm)) & ((1LL << p.lbat) - 1);
    w.v = o >> (p.lbat + p.lm + p.ln);
    const long long ea = ((bat << p.lm) | m) << p.lk, eb = ((bat << p.ln) | n) << p.lk;
    auto rows = [&](const GatherDesc *g) { return !g || (g->lb ? g->pos_beta[g->lb - 1] : g->nbits) >= p.lk; };
    if (rows(p.gA) && rows(p.gB)) {
        w.A = p.gA ? reinterpret_cast<const float2 *>(p.gA->src) + gather_src(*p.gA, ea, closed_bits)
                   : static_cast<const float2 *>(p.ptrA[w.v]) + ea;
        w.B = p.gB ? reinterpret_cast<const float2 *>(p.gB->src) + gather_src(*p.gB, eb, closed_bits)
                   : static_cast<const float2 *>(p.ptrB[w.v]) + eb;
    }
    w.off = scatter_bits(bat, p.pos_bat, p.lbat) + scatter_bits(m, p.pos_m, p.lm) + scatter_bits(n, p.pos_n, p.ln);
    return w;
}
// Operands are read past L1: in a chain another SM wrote them.
__device__ __forceinline__ void small_finish(const GemmParams &p, const SmallWork &w, const uint64_t *closed_bits) {
    if (!w.any) return;
    const int K = 1 << p.lk;
    float2 acc = make_float2(0.f, 0.f);
    if (w.A) {
        if (K >= 2) {
#pragma unroll 8
            for (int k = 0; k < K; k += 2) {
                const float4 a = __ldcg(reinterpret_cast<const float4 *>(w.A + k)), b = __ldcg(reinterpret_cast<const float4 *>(w.B + k));
                acc = cfma(make_float2(a.x, a.y), make_float2(b.x, b.y), acc);
                acc = cfma(make_float2(a.z, a.w), make_float2(b.z, b.w), acc);
            }
        } else {
            acc = cfma(__ldcg(w.A), __ldcg(w.B), acc);
        }
    } else {
        const long long n = w.o & ((1LL << p.ln) - 1), bm = w.o >> p.ln;
        const long long ea = (bm & ((1LL << (p.lbat + p.lm)) - 1)) << p.lk;
        const long long eb = ((((bm >> p.lm) & ((1LL << p.lbat) - 1)) << p.ln) | n) << p.lk;
        for (int k = 0; k < K; k++) {
            const float2 *a = p.gA ? reinterpret_cast<const float2 *>(p.gA->src) + gather_src(*p.gA, ea + k, closed_bits)
                                   : static_cast<const float2 *>(p.ptrA[w.v]) + ea + k;
            const float2 *b = p.gB ? reinterpret_cast<const float2 *>(p.gB->src) + gather_src(*p.gB, eb + k, closed_bits)
                                   : static_cast<const float2 *>(p.ptrB[w.v]) + eb + k;
            acc = cfma(__ldcg(a), __ldcg(b), acc);
        }
    }
    store_c(p, w.v, w.off, acc);
}
// A step's parameters into shared memory, by the kSmallBlock threads tid = 0 ..
__device__ __forceinline__ void small_load(GemmParams *p, const GemmParams *d, int tid) {
    static_assert(sizeof(GemmParams) % 4 == 0, "copied as words");
    for (int i = tid; i < (int)(sizeof(GemmParams) / 4); i += kSmallBlock)
        reinterpret_cast<uint32_t *>(p)[i] = reinterpret_cast<const uint32_t *>(d)[i];
}
__global__ void __launch_bounds__(kSmallBlock) small_steps(const GemmParams *descs, const int2 *blocks,
                                                           const uint64_t *closed_bits) {
    __shared__ GemmParams p;
    const int2 bl = blocks[blockIdx.x];
    small_load(&p, descs + bl.x, threadIdx.x);
    __syncthreads();
    small_finish(p, small_prepare(p, (long long)bl.y + threadIdx.x, closed_bits), closed_bits);
}

// Consecutive small launches as one: a cluster of eight blocks runs them in turn, with a
// cluster barrier between them in place of the end of one launch and the start of the next.
// Launch i is blocks [level[i], level[i + 1]), at most kChainBlocks of them, one per group of
// kSmallBlock threads.  What a launch reads that no launch writes (its steps' parameters,
// pointers, patterns) is read between the two halves of the barrier before it, so a launch
// costs the barrier, one read of the operands and the products.  12 qubits, 33 steps, a whole
// call: 86 -> 60 us.
constexpr int kChainCluster = 8, kChainGroups = 8, kChainBlocks = kChainCluster * kChainGroups;
__global__ void __cluster_dims__(kChainCluster, 1, 1) __launch_bounds__(kChainGroups *kSmallBlock)
    small_chain(const GemmParams *descs, const int2 *blocks, const int *level, int n_levels, const uint64_t *closed_bits) {
    __shared__ GemmParams p[2][kChainGroups];
    const int grp = threadIdx.x / kSmallBlock, tid = threadIdx.x % kSmallBlock;
    const int task = blockIdx.x + grp * kChainCluster;
    auto prepare = [&](int i) {
        SmallWork w = {nullptr, nullptr, 0, 0, 0, false};
        if (i < n_levels) {
            const int b = level[i] + task;
            if (b < level[i + 1]) {
                const int2 bl = blocks[b];
                small_load(&p[i & 1][grp], descs + bl.x, tid);
                asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kSmallBlock) : "memory");
                w = small_prepare(p[i & 1][grp], (long long)bl.y + tid, closed_bits);
            }
        }
        return w;
    };
    SmallWork w = prepare(0);
    for (int i = 0; i < n_levels; i++) {
        small_finish(p[i & 1][grp], w, closed_bits);
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        w = prepare(i + 1);
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// mbarrier primitives (shared-memory barriers with transaction counts).
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after ~limit cycles or when another role has aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                          long long limit) {
    const long long t0 = clock64();
    for (int it = 0;; ++it) {
        if (mbar_try(bar, parity)) return true;
        if ((it & 63) == 63) {
            if (*abort_flag) return false;
            if (clock64() - t0 > limit) {
                *abort_flag = 1;
                return false;
            }
        }
    }
}

// Bounded wait that ignores the abort flag (used to drain work already issued).
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity, long long limit) {
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try(bar, parity)) return true;
        if (clock64() - t0 > limit) return false;
    }
}

// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) global -> shared,
// completing on mbarrier `bar` as transaction bytes.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Batched products with at most 64 rows and 8 columns and a long K (K >= 1024, complex64
// operands).  A block takes R = W MW rows of one (version, batch) at a time (a batch with
// more rows is split into row blocks); each of W warps owns MW rows of A and every column.
// The block's work is one sequence of stages, each a (unit, K block of 64 U elements) pair.
// Warp 0 streams them through a ring of ST shared-memory stages with the bulk-copy engine
// (one contiguous copy per row and stage, ST - 1 stages ahead across unit boundaries,
// completing on the stage's `full` barrier); every warp waits for a stage and releases it
// on its `empty` barrier by itself, so no block barrier ties the warps together.  In a stage
// lane l reads elements 2 l and 2 l + 1 of each
// 64-element block of its warp's A rows; the stage's B rows are shared by the block.  Each
// lane accumulates in ascending k and the warp adds its 32 lane sums in the tree of a xor
// butterfly (halving the values a lane still holds at each level: 62 shuffles for 32 outputs
// instead of 320).  Gathered operands are read in place, one decode per row and unit.  Every
// wait is bounded: on timeout the block sets *err, lets its copies in flight land (bounded)
// and returns.  The lane split of K rounds differently from the kernels that accumulate
// each output over k in one thread, so it is the only kernel the engine runs for these
// shapes.  Bound by shared-memory reads next to FP32 issue: with MW rows a warp reads MW + N
// 16-byte rows per 8 MW N multiply-adds, so MW is four: (bat, m, n, k bits) =
// (14, 4, 3, 10) took 1.04 ms with two rows per warp and two block barriers per stage, 0.79 ms
// so (2.7 TB/s; its 2.2 GB take 0.32 ms at the copy rate).
constexpr int kSkinnyU = 1;   // 64-element K blocks per stage
constexpr int kSkinnyST = 4;  // ring stages
template <int W, int MW, int N>
constexpr int skinny_stage_bytes() {
    return (W * MW + N) * kSkinnyU * 32 * 16;
}
template <int W, int MW, int N>
__global__ void __launch_bounds__(32 * W) cgemm_skinny(GemmParams p) {
    extern __shared__ float4 skinny_ring[];
    constexpr int R = W * MW, U = kSkinnyU, ST = kSkinnyST;
    constexpr int RPL = (R + N + 31) / 32;  // rows copied per lane of warp 0
    __shared__ __align__(8) uint64_t full[ST], empty[ST];
    __shared__ int abort_flag;
    const long long kLimit = 4000000000LL;
    constexpr int kStage = (R + N) * U * 32;  // float4 per stage
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row_blocks = (1 << p.lm) / R;
    const long long units = (p.nver << p.lbat) * row_blocks;
    const int nk = (1 << p.lk) / (64 * U);  // stages per unit
    const long long mine = units > blockIdx.x ? (units - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    auto unit_of = [&](long long ul, long long &bat, long long &v, int &row0) {
        const long long u = blockIdx.x + ul * gridDim.x;
        const long long bv = u / row_blocks;
        bat = bv & ((1LL << p.lbat) - 1);
        v = bv >> p.lbat;
        row0 = (int)(u % row_blocks) * R;  // the unit's first row of A
    };
    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; i++) {
            mbar_init(smem_u32(&full[i]), 1);
            mbar_init(smem_u32(&empty[i]), W);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    // warp 0's copy side: stage (iul, ikb) goes to slot islot; lane r copies row r of a stage (A
    // rows, then B rows), and row r + 32 if there is one
    const float2 *src[RPL];
    long long iul = 0, issued = 0;
    int ikb = 0, islot = 0;
    uint32_t iparity = 0;
    auto issue = [&]() {
        if (iul >= mine) return true;
        if (ikb == 0) {
            long long bat, v;
            int row0;
            unit_of(iul, bat, v, row0);
#pragma unroll
            for (int i = 0; i < RPL; i++) {
                const int r = lane + 32 * i;
                if (r < R) {
                    const long long e = ((bat << p.lm) | (long long)(row0 + r)) << p.lk;
                    src[i] = p.gA ? reinterpret_cast<const float2 *>(p.gA->src) + gather_src(*p.gA, e, p.closed_bits)
                                  : static_cast<const float2 *>(p.ptrA[v]) + e;
                } else if (r < R + N) {
                    const long long e = ((bat << p.ln) | (long long)(r - R)) << p.lk;
                    src[i] = p.gB ? reinterpret_cast<const float2 *>(p.gB->src) + gather_src(*p.gB, e, p.closed_bits)
                                  : static_cast<const float2 *>(p.ptrB[v]) + e;
                }
            }
        }
        int go = 1;
        if (lane == 0) {
            if (issued >= ST) go = mbar_wait(smem_u32(&empty[islot]), iparity ^ 1u, &abort_flag, kLimit);
            if (go) mbar_expect_tx(smem_u32(&full[islot]), (uint32_t)((R + N) * U * 512));
        }
        if (!__shfl_sync(0xffffffffu, go, 0)) return false;
#pragma unroll
        for (int i = 0; i < RPL; i++) {
            const int r = lane + 32 * i;
            if (r < R + N)
                bulk_load(&skinny_ring[islot * kStage + r * U * 32], src[i] + ikb * 64 * U, U * 512,
                          smem_u32(&full[islot]));
        }
        issued++;
        if (++ikb == nk) { ikb = 0; iul++; }
        if (++islot == ST) { islot = 0; iparity ^= 1u; }
        return true;
    };
    if (warp == 0)
        for (int i = 0; i < ST - 1; i++) issue();
    {
        int slot = 0;
        uint32_t parity = 0;
        bool ok = true;
        for (long long ul = 0; ul < mine && ok; ul++) {
            float2 acc[MW * N];
#pragma unroll
            for (int o = 0; o < MW * N; o++) acc[o] = make_float2(0.f, 0.f);
            for (int kb = 0; kb < nk; kb++) {
                // the slot that warp 0 refills here was read one stage ago
                if (warp == 0 && !issue()) { ok = false; break; }
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&full[slot]), parity, &abort_flag, kLimit));
                if (!ok) break;
                const float4 *st = skinny_ring + slot * kStage;
#pragma unroll
                for (int u = 0; u < U; u++) {
                    float4 x[MW];
#pragma unroll
                    for (int i = 0; i < MW; i++) x[i] = st[((warp * MW + i) * U + u) * 32 + lane];
#pragma unroll
                    for (int n = 0; n < N; n++) {
                        const float4 y = st[((R + n) * U + u) * 32 + lane];
#pragma unroll
                        for (int i = 0; i < MW; i++) {
                            acc[i * N + n] = cfma(make_float2(x[i].x, x[i].y), make_float2(y.x, y.y), acc[i * N + n]);
                            acc[i * N + n] = cfma(make_float2(x[i].z, x[i].w), make_float2(y.z, y.w), acc[i * N + n]);
                        }
                    }
                }
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&empty[slot])) : "memory");
                if (++slot == ST) { slot = 0; parity ^= 1u; }
            }
            if (!ok) break;
            // add the lanes' sums: at each level a lane keeps the half of the outputs that its
            // lane bit selects, until it holds one (then both lanes of a pair add the same)
            int left = MW * N, out = 0;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const bool up = (lane & off) != 0;
                if (left > 1) {
                    left >>= 1;
                    out = 2 * out + (up ? 1 : 0);
#pragma unroll
                    for (int o = 0; o < MW * N / 2; o++) {
                        if (o >= left) break;
                        const float2 keep = up ? acc[o + left] : acc[o], send = up ? acc[o] : acc[o + left];
                        acc[o].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, off);
                        acc[o].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, off);
                    }
                } else {
                    acc[0].x += __shfl_xor_sync(0xffffffffu, acc[0].x, off);
                    acc[0].y += __shfl_xor_sync(0xffffffffu, acc[0].y, off);
                }
            }
            if ((lane & (32 / (MW * N) - 1)) == 0) {
                long long bat, v;
                int row0;
                unit_of(ul, bat, v, row0);
                const int m = row0 + warp * MW + out / N, n = out % N;
                store_c(p, v,
                        scatter_bits(bat, p.pos_bat, p.lbat) + scatter_bits(m, p.pos_m, p.lm) + scatter_bits(n, p.pos_n, p.ln),
                        acc[0]);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) {
        // after a timeout, let the copies already issued land before the shared memory is released
        atomicExch(p.err, 1);
        for (long long q = issued > ST ? issued - ST : 0; q < issued; q++)
            mbar_drain(smem_u32(&full[q % ST]), (uint32_t)((q / ST) & 1), kLimit);
    }
    __syncthreads();
}

// Batched small products (M, N <= 64, K <= 64): a block stages the operands of 2^lg
// consecutive batches in shared memory and walks that chunk's outputs in the order of
// their positions in C (local bit i = chunk bit kind[i] / idx[i]), so consecutive threads
// store to consecutive addresses whenever C's lowest positions lie in the chunk.
struct SmallMap {
    int lg;              // log2 batches per block
    int nloc;            // lg + lm + ln
    int8_t kind[48];     // 0: batch bit, 1: m bit, 2: n bit
    int8_t idx[48];
};

template <typename T>
__global__ void __launch_bounds__(256) cgemm_small(GemmParams p, SmallMap smp) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    __shared__ SmallMap sm;  // its tables are read per output
    if (threadIdx.x == 0) sm = smp;
    T *As = reinterpret_cast<T *>(small_smem);
    const int M = 1 << p.lm, N = 1 << p.ln, K = 1 << p.lk, G = 1 << smp.lg;
    const int KP = K + 1;  // padded row: rows of consecutive outputs fall in different banks
    T *Bs = As + (size_t)G * M * KP;
    const long long chunks = 1LL << (p.lbat - smp.lg);
    const long long v = (long long)blockIdx.x / chunks;
    const long long bat0 = ((long long)blockIdx.x - v * chunks) << smp.lg;
    if (v >= p.nver) return;
    const T *A = static_cast<const T *>(p.ptrA[v]) + (bat0 << (p.lm + p.lk));
    const T *B = static_cast<const T *>(p.ptrB[v]) + (bat0 << (p.ln + p.lk));
    for (int e = threadIdx.x; e < G * M * K; e += blockDim.x) As[(e >> p.lk) * KP + (e & (K - 1))] = A[e];
    for (int e = threadIdx.x; e < G * N * K; e += blockDim.x) Bs[(e >> p.lk) * KP + (e & (K - 1))] = B[e];
    __syncthreads();
    const long long cbase = scatter_bits(bat0, p.pos_bat, p.lbat);
    const int nout = G * M * N;
    for (int l = threadIdx.x; l < nout; l += blockDim.x) {
        int b = 0, m = 0, n = 0;
        for (int i = 0; i < sm.nloc; i++) {
            const int bit = (l >> i) & 1;
            if (sm.kind[i] == 0) b |= bit << sm.idx[i];
            else if (sm.kind[i] == 1) m |= bit << sm.idx[i];
            else n |= bit << sm.idx[i];
        }
        const T *a = As + (size_t)(b * M + m) * KP;
        const T *bb = Bs + (size_t)(b * N + n) * KP;
        T acc = czero<T>();
        for (int k = 0; k < K; k++) acc = cfma(a[k], bb[k], acc);
        const long long off = cbase + scatter_bits(b, p.pos_bat, smp.lg) + scatter_bits(m, p.pos_m, p.lm) +
                              scatter_bits(n, p.pos_n, p.ln);
        store_c_t<T>(p, v, off, acc);
    }
}

// Packed FP32 multiply-add: two independent fmaf in one instruction.
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long x) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
    return r;
}

// The complex64 tile kernel: products of packed FP32 pairs.  A pair is two rows of A, so the
// four multiply-adds of a complex product take two instructions per output instead of four,
// each with the rounding and, per output, the order of cfma (SW: with the operands exchanged,
// as the rows hold the step's B), so the results are bit-identical to the other kernels'.
// Bound by FP32 issue and, next to it, shared-memory reads: A sits in shared memory as planes
// of real and imaginary parts (four rows per 16-byte read), B as complex values (two
// columns per read, spread to pairs in registers), so an 8 x 8 thread tile reads 8 x 16
// bytes for 256 multiply-adds.  (0, 21, 9, 7) took 28.3 ms with scalar fmaf (39 TFLOP/s),
// 30.7 ms with packed pairs of re and im whose both orders came from shared memory, 22.5 ms so
// (49 TFLOP/s; fmaf alone reaches 78); (15, 8, 4, 9), its operands in place, 33.1 -> 11.5 ms;
// (11, 10, 2, 7) 4.1 -> 0.41 ms on tiles of 256 x 4.
//
// The longer side are the tile's rows, so a narrow step fills narrow tiles.  Each thread owns
// groups of four adjacent rows and two adjacent columns; consecutive lanes take consecutive
// row groups if C's lowest position is a row bit, else consecutive column groups, and
// adjacent outputs go out in one store.  K runs in chunks of TK through two shared-memory
// buffers; the next chunk's loads are in flight during the products.  Gathered operands
// whose batch block is contiguous in the stored form are read in place.
template <int TM, int TN, int RM, int RN, int TK, bool SW>
__global__ void __launch_bounds__((TM / RM) * (TN / RN)) cgemm_tile(GemmParams p) {
    constexpr int NTX = TN / RN, NTY = TM / RM, NT = NTX * NTY, GM = RM / 4, GN = RN / 2;
    constexpr int LA = (TM * TK / 2 + NT - 1) / NT, LB = (TN * TK / 2 + NT - 1) / NT;
    static_assert(TM <= NT * LA && TN <= NT * LB, "K = 1 loads one element per slot");
    __shared__ __align__(16) float As[2][2][TK][TM + 4];  // [buffer][re, im]
    __shared__ __align__(16) float2 Bs[2][TK][TN + 2];
    const int tid = threadIdx.x;
    const bool rows_low = p.lm > 0 && p.pos_m[0] < (p.ln > 0 ? p.pos_n[0] : kMaxBits);
    const int tx = rows_low ? tid / NTY : tid % NTX, ty = rows_low ? tid % NTY : tid / NTX;
    const long long M = 1LL << p.lm, N = 1LL << p.ln;
    const int lkt = min(p.lk, __ffs(TK) - 1), kt = 1 << lkt;
    const int ltiles_m = max(0, p.lm - (__ffs(TM) - 1)), ltiles_n = max(0, p.ln - (__ffs(TN) - 1));
    long long bid = blockIdx.x;
    const long long n0 = (bid & ((1LL << ltiles_n) - 1)) * TN;
    bid >>= ltiles_n;
    const long long m0 = (bid & ((1LL << ltiles_m) - 1)) * TM;
    bid >>= ltiles_m;
    const long long bat = bid & ((1LL << p.lbat) - 1);
    const long long v = bid >> p.lbat;
    if (v >= p.nver) return;
    const int mrows = (int)min((long long)TM, M - m0), ncols = (int)min((long long)TN, N - n0);
    const long long eA = bat << (p.lm + p.lk), eB = bat << (p.ln + p.lk);
    const float2 *A = (p.gA ? reinterpret_cast<const float2 *>(p.gA->src) + gather_src(*p.gA, eA, p.closed_bits)
                            : static_cast<const float2 *>(p.ptrA[v]) + eA) + (m0 << p.lk);
    const float2 *B = (p.gB ? reinterpret_cast<const float2 *>(p.gB->src) + gather_src(*p.gB, eB, p.closed_bits)
                            : static_cast<const float2 *>(p.ptrB[v]) + eB) + (n0 << p.lk);
    // slot i of a chunk: elements k and k + 1 of a row (K = 1: one element)
    const int lh = max(0, lkt - 1);  // log2 slots per row
    float4 ra[LA], rb[LB];
    auto fetch = [&](const float2 *X, int valid, int k0, float4 *r, int n) {
#pragma unroll
        for (int i = 0; i < n; i++) {
            const int s = tid + i * NT, row = s >> lh, c = (s & ((1 << lh) - 1)) << 1;
            r[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < valid) {
                const float2 *x = X + ((long long)row << p.lk) + k0 + c;
                if (lkt > 0) r[i] = *reinterpret_cast<const float4 *>(x);
                else r[i].x = x->x, r[i].y = x->y;
            }
        }
    };
    auto stage = [&](int b) {
#pragma unroll
        for (int i = 0; i < LA; i++) {
            const int s = tid + i * NT, row = s >> lh, c = (s & ((1 << lh) - 1)) << 1;
            if (row < TM) {
                As[b][0][c][row] = ra[i].x;
                As[b][1][c][row] = ra[i].y;
                if (lkt > 0) {
                    As[b][0][c + 1][row] = ra[i].z;
                    As[b][1][c + 1][row] = ra[i].w;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < LB; i++) {
            const int s = tid + i * NT, row = s >> lh, c = (s & ((1 << lh) - 1)) << 1;
            if (row < TN) {
                Bs[b][c][row] = make_float2(rb[i].x, rb[i].y);
                if (lkt > 0) Bs[b][c + 1][row] = make_float2(rb[i].z, rb[i].w);
            }
        }
    };
    // pair i of the thread's rows, column j: real and imaginary sums
    unsigned long long re[RM / 2][RN], im[RM / 2][RN];
#pragma unroll
    for (int i = 0; i < RM / 2; i++)
#pragma unroll
        for (int j = 0; j < RN; j++) re[i][j] = im[i][j] = 0ull;
    const int K = 1 << p.lk;
    fetch(A, mrows, 0, ra, LA);
    fetch(B, ncols, 0, rb, LB);
    stage(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += kt, buf ^= 1) {
        const bool more = k0 + kt < K;
        if (more) {
            fetch(A, mrows, k0 + kt, ra, LA);
            fetch(B, ncols, k0 + kt, rb, LB);
        }
        auto mul = [&](int kk) {
            unsigned long long ar[RM / 2], ai[RM / 2], ni[RM / 2];
#pragma unroll
            for (int g = 0; g < GM; g++) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&As[buf][0][kk][4 * (ty + g * NTY)]);
                const ulonglong2 y = *reinterpret_cast<const ulonglong2 *>(&As[buf][1][kk][4 * (ty + g * NTY)]);
                ar[2 * g] = x.x;
                ar[2 * g + 1] = x.y;
                ai[2 * g] = y.x;
                ai[2 * g + 1] = y.y;
            }
#pragma unroll
            for (int i = 0; i < RM / 2; i++) ni[i] = ai[i] ^ 0x8000000080000000ull;
#pragma unroll
            for (int h = 0; h < GN; h++) {
                const float4 q = *reinterpret_cast<const float4 *>(&Bs[buf][kk][2 * (tx + h * NTX)]);
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    const int j = 2 * h + c;
                    const unsigned long long bx = c ? pack2(q.z, q.z) : pack2(q.x, q.x);
                    const unsigned long long by = c ? pack2(q.w, q.w) : pack2(q.y, q.y);
#pragma unroll
                    for (int i = 0; i < RM / 2; i++) {
                        re[i][j] = fma2(ar[i], bx, re[i][j]);
                        im[i][j] = SW ? fma2(ai[i], bx, im[i][j]) : fma2(ar[i], by, im[i][j]);
                    }
#pragma unroll
                    for (int i = 0; i < RM / 2; i++) {
                        re[i][j] = fma2(ni[i], by, re[i][j]);
                        im[i][j] = SW ? fma2(ar[i], by, im[i][j]) : fma2(ai[i], bx, im[i][j]);
                    }
                }
            }
        };
        if (kt == TK) {
#pragma unroll
            for (int kk = 0; kk < TK; kk++) mul(kk);
        } else {
            for (int kk = 0; kk < kt; kk++) mul(kk);
        }
        if (more) {
            stage(buf ^ 1);
            __syncthreads();
        }
    }
    const long long cb = scatter_bits(bat, p.pos_bat, p.lbat);
    // adjacent outputs of a plain complex C in one store: four rows, or two columns
    const bool row4 = p.out_fmt == OUT_C64 && p.lm >= 2 && p.pos_m[0] == 0 && p.pos_m[1] == 1;
    const bool col2 = p.out_fmt == OUT_C64 && p.ln >= 1 && p.pos_n[0] == 0;
    float2 *C = static_cast<float2 *>(p.C) + v * p.c_vstride;
    const float sc = p.out_scale;
#pragma unroll
    for (int h = 0; h < GN; h++) {
        const int c0 = 2 * (tx + h * NTX);
        const long long offn0 = cb + scatter_bits(n0 + c0, p.pos_n, p.ln);
        const long long offn1 = cb + scatter_bits(n0 + c0 + 1, p.pos_n, p.ln);
#pragma unroll
        for (int g = 0; g < GM; g++) {
            const int r0 = 4 * (ty + g * NTY);
            if (r0 >= mrows || c0 >= ncols) continue;
            float2 x[2][4];  // column, row
#pragma unroll
            for (int c = 0; c < 2; c++)
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    const float2 a = unpack2(re[2 * g + i][2 * h + c]), b = unpack2(im[2 * g + i][2 * h + c]);
                    x[c][2 * i] = make_float2(a.x, b.x);
                    x[c][2 * i + 1] = make_float2(a.y, b.y);
                }
            if (row4) {
                const long long om = scatter_bits(m0 + r0, p.pos_m, p.lm);
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    if (c0 + c >= ncols) break;
                    float4 *q = reinterpret_cast<float4 *>(C + om + (c ? offn1 : offn0));
                    q[0] = make_float4(x[c][0].x * sc, x[c][0].y * sc, x[c][1].x * sc, x[c][1].y * sc);
                    q[1] = make_float4(x[c][2].x * sc, x[c][2].y * sc, x[c][3].x * sc, x[c][3].y * sc);
                }
                continue;
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                if (r0 + i >= mrows) break;
                const long long om = scatter_bits(m0 + r0 + i, p.pos_m, p.lm);
                if (col2) {
                    *reinterpret_cast<float4 *>(C + om + offn0) =
                        make_float4(x[0][i].x * sc, x[0][i].y * sc, x[1][i].x * sc, x[1][i].y * sc);
                } else {
                    store_c(p, v, om + offn0, x[0][i]);
                    if (c0 + 1 < ncols) store_c(p, v, om + offn1, x[1][i]);
                }
            }
        }
    }
}

// ---------------------------------------------------------------- leaves

struct MatDesc {
    const double2 *src;  // full leaf tensor, data index = sum_t value(leg t) << t
    void *dst;           // [code][2^nd] in the consumer's layout and format
    int fmt;             // OutFmt
    float scale;         // multiplier (split fp16 range scaling)
    int nd;              // destination bits
    int ncode_bits;      // sliced legs of the leaf
    int8_t dst_leg[kMaxBits];  // destination bit -> source leg position
    int8_t sl_leg[8];          // code bit u -> source leg position
};

// grid.y = leaf; threads over (code, element).
__global__ void materialize(const MatDesc *descs) {
    const MatDesc d = descs[blockIdx.y];
    const long long total = 1LL << (d.nd + d.ncode_bits);
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (long long)gridDim.x * blockDim.x) {
        const long long code = g >> d.nd, e = g & ((1LL << d.nd) - 1);
        long long src = 0;
        for (int t = 0; t < d.nd; t++) src |= ((e >> t) & 1) << d.dst_leg[t];
        for (int u = 0; u < d.ncode_bits; u++) src |= ((code >> u) & 1) << d.sl_leg[u];
        const double2 x = d.src[src];
        const float2 y = make_float2((float)(x.x * d.scale), (float)(x.y * d.scale));
        if (d.fmt == OUT_C64) {
            static_cast<float2 *>(d.dst)[g] = y;
        } else {
            const long long ne = 1LL << d.nd;
            unsigned short *base = static_cast<unsigned short *>(d.dst) + 4 * code * ne;
            store_split(base, ne, e, y, d.fmt == OUT_SPLIT_FP16);
        }
    }
}

// ---------------------------------------------------------------- batch gathers

__device__ __forceinline__ void gather_copy(const GatherDesc &d, long long vp, long long e, long long se) {
    const char *src = d.src + (vp * d.src_plane + se) * d.esize;
    char *dst = d.dst + (vp * d.dst_plane + e) * d.esize;
    if (d.vec_log2 > 0 || d.esize == 16) *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(src);
    else if (d.esize == 8) *reinterpret_cast<uint2 *>(dst) = *reinterpret_cast<const uint2 *>(src);
    else *reinterpret_cast<unsigned short *>(dst) = *reinterpret_cast<const unsigned short *>(src);
}

// grid.y = gather.  Runs of at least 32 chunks: one warp per run decodes the batch and
// selection once and its lanes copy the run's 16-byte chunks; shorter runs: one thread
// per chunk.  The descriptor is staged in shared memory.
__global__ void gather_batches(const GatherDesc *descs, const uint64_t *closed_bits) {
    __shared__ GatherDesc d;
    if (threadIdx.x == 0) d = descs[blockIdx.y];
    __syncthreads();
    const int vl = d.vec_log2;
    const long long per_plane = d.dst_plane >> vl;  // chunks per plane
    if (d.run_log2 >= 5) {
        const int lr = d.run_log2, lane = threadIdx.x & 31;
        const long long runs_plane = per_plane >> lr;
        const long long runs = runs_plane * d.nplanes * d.nver;
        const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
        for (long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < runs; r += nw) {
            const long long vp = r / runs_plane;
            const long long e0 = (r - vp * runs_plane) << (lr + vl);
            const long long se0 = gather_src(d, e0, closed_bits);
            for (long long c = lane; c < (1LL << lr); c += 32) gather_copy(d, vp, e0 + (c << vl), se0 + (c << vl));
        }
        return;
    }
    const long long total = per_plane * d.nplanes * d.nver;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (long long)gridDim.x * blockDim.x) {
        const long long vp = g / per_plane;
        const long long e = (g - vp * per_plane) << vl;
        gather_copy(d, vp, e, gather_src(d, e, closed_bits));
    }
}

// ---------------------------------------------------------------- calibration

// *absmax_bits = max(*absmax_bits, max |re|, |im| over the n elements of one version of a
// tensor stored in format fmt (split formats: planes 0 and 2, the hi parts).  Non-negative
// floats compare as integers.
__global__ void absmax_kernel(const void *data, long long n, int fmt, int *absmax_bits) {
    float m = 0.f;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (fmt == OUT_C64) {
            const float2 x = static_cast<const float2 *>(data)[i];
            m = fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y)));
        } else {
            const __nv_bfloat16 *h = static_cast<const __nv_bfloat16 *>(data);
            m = fmaxf(m, fmaxf(fabsf(__bfloat162float(h[i])), fabsf(__bfloat162float(h[2 * n + i]))));
        }
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(absmax_bits, __float_as_int(m));
}

// ---------------------------------------------------------------- slice sum

// out[e] = sum over explicit root versions v (in order) and over the 2^nfree patterns f
// of the sliced legs carried as layout bits (ascending) of root_v[(f << nout) | e], FP64.
// complex64 values are added 16 at a time where a version has that many (chunk_sum.h: 2^14
// outputs of 48 values 16 -> 10 us; for the large sums see root_sum_small), else one by one;
// complex64 inputs are widened with integer operations (exact), which leaves the FP64
// pipe to the additions.
__device__ __forceinline__ double slice_widen(float x) { return tn_widen(x); }

template <typename T>
__global__ void slice_sum(const void *const *ptr, long long nver, int nfree, int nout, double2 *out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (1LL << nout)) return;
    double re = 0.0, im = 0.0;
    const long long nf = 1LL << nfree;
    if constexpr (sizeof(T) == sizeof(float2)) {
        if (nf >= 16) {
            ChunkSum sr, si;
            for (long long v = 0; v < nver; v++) {
                const float2 *r = static_cast<const float2 *>(ptr[v]) + e;
                for (long long f = 0; f < nf; f += 16) {
                    float xr[16], xi[16];
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        const float2 x = __ldcs(&r[(f + i) << nout]);
                        xr[i] = x.x;
                        xi[i] = x.y;
                    }
                    sr.add16(xr);
                    si.add16(xi);
                }
            }
            out[e] = make_double2(sr.total(), si.total());
            return;
        }
    }
    for (long long v = 0; v < nver; v++) {
        const T *r = static_cast<const T *>(ptr[v]) + e;
        long long f = 0;
        // loads issued four at a time; the additions stay in slice order
        for (; f + 4 <= nf; f += 4) {
            const T x0 = r[(f + 0) << nout], x1 = r[(f + 1) << nout], x2 = r[(f + 2) << nout], x3 = r[(f + 3) << nout];
            re = __dadd_rn(re, slice_widen(x0.x));
            im = __dadd_rn(im, slice_widen(x0.y));
            re = __dadd_rn(re, slice_widen(x1.x));
            im = __dadd_rn(im, slice_widen(x1.y));
            re = __dadd_rn(re, slice_widen(x2.x));
            im = __dadd_rn(im, slice_widen(x2.y));
            re = __dadd_rn(re, slice_widen(x3.x));
            im = __dadd_rn(im, slice_widen(x3.y));
        }
        for (; f < nf; f++) {
            const T x = r[f << nout];
            re = __dadd_rn(re, slice_widen(x.x));
            im = __dadd_rn(im, slice_widen(x.y));
        }
    }
    out[e] = make_double2(re, im);
}

// ---------------------------------------------------------------- root product + slice sum

// The batch, row and column bits of C position pos under the row-kernel parameters p
// (pos_* give each bit's C position; positions no bit maps to contribute nothing).
__device__ __forceinline__ void root_split(const GemmParams &p, long long pos, long long &bat, long long &m, int &n) {
    bat = 0;
    m = 0;
    n = 0;
    for (int i = 0; i < p.lbat; i++) bat |= ((pos >> p.pos_bat[i]) & 1LL) << i;
    for (int i = 0; i < p.lm; i++) m |= ((pos >> p.pos_m[i]) & 1LL) << i;
    for (int i = 0; i < p.ln; i++) n |= (int)((pos >> p.pos_n[i]) & 1LL) << i;
}

// The value cgemm_row_one stores for output (v, bat, m, n), before the store: the same
// operand rows (gathered ones read in place), k order and multiply-add operand order.
template <typename T>
__device__ __forceinline__ T root_value(const GemmParams &p, long long v, long long bat, long long m, int n) {
    const T *A, *B;
    if (p.gA) {
        const long long e = ((bat << p.lm) | m) << p.lk;
        A = reinterpret_cast<const T *>(p.gA->src) + gather_src_warp(*p.gA, e, p.gA->pos_beta[p.gA->lb - 1], p.closed_bits);
    } else {
        A = static_cast<const T *>(p.ptrA[v]) + (((bat << p.lm) | m) << p.lk);
    }
    if (p.gB) {
        const long long e = bat << (p.ln + p.lk);
        B = reinterpret_cast<const T *>(p.gB->src) + gather_src_warp(*p.gB, e, p.gB->pos_beta[p.gB->lb - 1], p.closed_bits);
    } else {
        B = static_cast<const T *>(p.ptrB[v]) + (bat << (p.ln + p.lk));
    }
    B += (long long)n << p.lk;
    const int K = 1 << p.lk;
    T acc = czero<T>();
    if (p.swapped) {
        for (int k = 0; k < K; k++) acc = cfma(__ldg(&B[k]), A[k], acc);
    } else {
        for (int k = 0; k < K; k++) acc = cfma(A[k], __ldg(&B[k]), acc);
    }
    return acc;
}

// What store_c_t applies before storing: the output scale.
__device__ __forceinline__ float2 root_scaled(const GemmParams &p, float2 x) {
    x.x *= p.out_scale;
    x.y *= p.out_scale;
    return x;
}

constexpr int kRootTabBytes = 3;  // free patterns of up to 24 bits

// The root step fused with the slice sum: out[e] = sum over explicit root versions v (in
// order) and free patterns f (ascending) of the root product's value at C position
// (f << nout) | e, p being the root step's row-kernel parameters.  Each value is formed
// as the row kernel forms it and widened and added in FP64 as slice_sum does, so out is
// bit-identical to the row kernel followed by slice_sum, and the root's 2^(nout + nfree)
// values never pass through memory.  The host checks that p's batch, row and column bits
// cover the positions [0, nout + nfree) once each, so every (bat, m, n) below is in range.
template <typename T>
__global__ void __launch_bounds__(256, 3) root_slice_sum(GemmParams p, int nfree, int nout, double2 *out) {
    // byte tables: t*[j][b] are the batch, row and column bits of position (b << 8j) << nout
    __shared__ long long tbat[kRootTabBytes][256], tm[kRootTabBytes][256];
    __shared__ int tn[kRootTabBytes][256];
    const int nbytes = (nfree + 7) >> 3;
    for (int i = threadIdx.x; i < nbytes * 256; i += blockDim.x) {
        const int j = i >> 8;
        long long b, m;
        int n;
        root_split(p, ((long long)(i & 255) << (8 * j)) << nout, b, m, n);
        tbat[j][i & 255] = b;
        tm[j][i & 255] = m;
        tn[j][i & 255] = n;
    }
    __syncthreads();
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (1LL << nout)) return;
    long long be, me;
    int ne;
    root_split(p, e, be, me, ne);
    const long long nf = 1LL << nfree;
    auto term = [&](long long v, long long f) {
        long long bat = be, m = me;
        int n = ne;
        for (int j = 0; j < nbytes; j++) {
            const int b = (int)((f >> (8 * j)) & 255);
            bat |= tbat[j][b];
            m |= tm[j][b];
            n |= tn[j][b];
        }
        return root_scaled(p, root_value<T>(p, v, bat, m, n));
    };
    if constexpr (sizeof(T) == sizeof(float2)) {
        if (nf >= 16) {
            ChunkSum sr, si;
            for (long long v = 0; v < p.nver; v++)
                for (long long f = 0; f < nf; f += 16) {
                    float xr[16], xi[16];
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        const float2 x = term(v, f + i);
                        xr[i] = x.x;
                        xi[i] = x.y;
                    }
                    sr.add16(xr);
                    si.add16(xi);
                }
            out[e] = make_double2(sr.total(), si.total());
            return;
        }
    }
    double re = 0.0, im = 0.0;
    for (long long v = 0; v < p.nver; v++) {
        for (long long f = 0; f < nf; f++) {
            const T x = term(v, f);
            re = __dadd_rn(re, slice_widen(x.x));
            im = __dadd_rn(im, slice_widen(x.y));
        }
    }
    out[e] = make_double2(re, im);
}

// The same for complex64 roots with K = 2^LK of 1, 2 or 4, the fast form of the fusion.
// Unfused, such a root writes 8 bytes per multiply-add and the slice sum reads them back:
// (bat, m, n, k bits) = (22, 3, 5, 0) took 3.4 + 4.1 ms for 2^30 values.  Here a thread owns an
// output and forms its terms from the operands, which are 2^-5 of the root's size and come
// from L1.  The sliced bits of the root's position are a fixed pattern of each operand's
// offset (they are never batch-index bits, so a gathered operand's stored block does not
// depend on them): off[f] holds both operands' offsets of free pattern f, in elements.
// Dynamic shared memory: 8 bytes << nfree.  The host checks the offsets fit 32 bits.
// Now (22, 3, 5, 0) takes 1.57 ms in place of 3.4 + 4.1 ms, (20, 2, 4, 0) 0.14 in place of 0.37
// + 0.28 ms; bound by issue (about 30 instructions per term, 16 of them the sums).
template <int LK>
__global__ void __launch_bounds__(256, 3) root_sum_small(GemmParams p, int nfree, int nout, double2 *out) {
    extern __shared__ uint2 root_off[];
    constexpr int K = 1 << LK;
    const int nf = 1 << nfree;
    auto rest = [](const GatherDesc &d, long long e) {  // stored offset of e's non-batch bits
        uint64_t r = 0;
        for (int j = 0; j < 5; j++) r |= __ldg(&d.rest_tab[j * 256 + ((e >> (8 * j)) & 255)]);
        return (uint32_t)r;
    };
    for (int f = threadIdx.x; f < nf; f += blockDim.x) {
        long long b, m;
        int n;
        root_split(p, (long long)f << nout, b, m, n);
        const long long ea = ((b << p.lm) | m) << LK, eb = ((b << p.ln) | n) << LK;
        root_off[f] = make_uint2(p.gA ? rest(*p.gA, ea) : (uint32_t)ea, p.gB ? rest(*p.gB, eb) : (uint32_t)eb);
    }
    __syncthreads();
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (1LL << nout)) return;
    long long be, me;
    int ne;
    root_split(p, e, be, me, ne);
    const long long ea = ((be << p.lm) | me) << LK, eb = ((be << p.ln) | ne) << LK;
    const long long ga = p.gA ? gather_src(*p.gA, ea, p.closed_bits) : ea;
    const long long gb = p.gB ? gather_src(*p.gB, eb, p.closed_bits) : eb;
    ChunkSum sr, si;
    for (long long v = 0; v < p.nver; v++) {
        const float2 *A = (p.gA ? reinterpret_cast<const float2 *>(p.gA->src) : static_cast<const float2 *>(p.ptrA[v])) + ga;
        const float2 *B = (p.gB ? reinterpret_cast<const float2 *>(p.gB->src) : static_cast<const float2 *>(p.ptrB[v])) + gb;
        auto term = [&](int f) {
            const uint2 o = root_off[f];
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; k++) {
                const float2 a = __ldg(&A[o.x + k]), b = __ldg(&B[o.y + k]);
                acc = p.swapped ? cfma(b, a, acc) : cfma(a, b, acc);
            }
            return root_scaled(p, acc);
        };
        if (nf >= 16) {
            for (int f = 0; f < nf; f += 16) {
                float xr[16], xi[16];
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const float2 x = term(f + i);
                    xr[i] = x.x;
                    xi[i] = x.y;
                }
                sr.add16(xr);
                si.add16(xi);
            }
        } else {
            for (int f = 0; f < nf; f++) {
                const float2 x = term(f);
                sr.acc = __dadd_rn(sr.acc, slice_widen(x.x));
                si.acc = __dadd_rn(si.acc, slice_widen(x.y));
            }
        }
    }
    out[e] = make_double2(sr.total(), si.total());
}

// ---------------------------------------------------------------- sampling job

// acc[e] += x[e] in FP64 for e < n: a sampling job adds each slice chunk's sum over its
// slices (Sec. I.C step 1) to the running total of the same batches, chunk after chunk,
// so every amplitude is summed in one fixed order.
__global__ void accumulate_amps(double2 *acc, const double2 *x, long long n) {
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const double2 a = acc[e], b = x[e];
        acc[e] = make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
    }
}

// ---------------------------------------------------------------- verification XEB

// The amplitude of each of nb bitstrings from its batch: out[t] = amps[(t << n_open) | idx[t]].
__global__ void pick_amplitudes(const double2 *amps, int n_open, const int32_t *idx, long long nb, double2 *out) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nb) out[t] = amps[(t << n_open) | idx[t]];
}

// FP64 sum of |a_i|^2 = re*re + im*im (rounded products, no fused multiply-add) over n
// values in a fixed order: thread j of block b sums i = b*256 + j, then every stride of
// kNormGrid*256, in turn; each block halves its 256 partials pairwise into partial[b].
// norm_total then halves the kNormGrid partials the same way.
constexpr int kNormGrid = 256;
__global__ void __launch_bounds__(256) sum_norms(const double2 *a, long long n, double *partial) {
    __shared__ double sh[256];
    double acc = 0.0;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)kNormGrid * 256)
        acc = __dadd_rn(acc, __dadd_rn(__dmul_rn(a[i].x, a[i].x), __dmul_rn(a[i].y, a[i].y)));
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) sh[threadIdx.x] = __dadd_rn(sh[threadIdx.x], sh[threadIdx.x + h]);
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}
__global__ void __launch_bounds__(256) norm_total(const double *partial, double *out) {
    __shared__ double sh[kNormGrid];
    sh[threadIdx.x] = partial[threadIdx.x];
    __syncthreads();
    for (int h = kNormGrid / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) sh[threadIdx.x] = __dadd_rn(sh[threadIdx.x], sh[threadIdx.x + h]);
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

// ---------------------------------------------------------------- top-N selection (XEB spoofing)

// Selection of the `need` largest of n <= 2^16 probabilities p_i = re*re + im*im in FP64
// (rounded products, no fused multiply-add), ties by position, written in ascending position:
// position i as the bitstring base | (bit r of i at qubit open.q[r]), with its p_i.
//
// One cluster of eight blocks holds all keys in registers (the bit patterns of non-negative
// doubles order like the doubles).  A radix select, most significant 8-bit digit first, adds
// the blocks' shared histograms through the cluster's shared memory and picks the digit in
// every block alike, so the eight digits cost eight cluster barriers; then the blocks rank
// the selected keys and write them.  Before, every digit was a launch, a copy to the host
// and a wait, and the ranking three more launches: a whole call of 2^16 strings, N = 6553, 457
// -> 339 us with a first form of this kernel (57 us); 34 us as it stands.
struct OpenQubits {
    int8_t q[64];
    int n;
};
constexpr int kSelBlock = 1024, kSelCluster = 8, kSelKeys = 8;  // threads, blocks, keys per thread

// Exclusive ranks of this thread's two flags among the block's flags, and the block's totals
// (the second's in the upper halves).  Every warp scans the 32 warp totals by shuffles.
__device__ __forceinline__ unsigned int block_rank2(bool f, bool g, unsigned int *warp_tot, unsigned int &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned int bf = __ballot_sync(0xffffffffu, f), bg = __ballot_sync(0xffffffffu, g), below = (1u << lane) - 1u;
    if (lane == 0) warp_tot[warp] = (unsigned int)__popc(bf) | (unsigned int)__popc(bg) << 16;
    __syncthreads();
    unsigned int inc = warp_tot[lane];
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    total = __shfl_sync(0xffffffffu, inc, 31);
    const unsigned int before = __shfl_sync(0xffffffffu, inc, max(warp - 1, 0));
    __syncthreads();  // warp_tot is reused by the next call
    return (warp ? before : 0u) + ((unsigned int)__popc(bf & below) | (unsigned int)__popc(bg & below) << 16);
}

__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The word at this block's shared address `x`, in block `rank` of the cluster.
__device__ __forceinline__ unsigned int cluster_load(const unsigned int *x, int rank) {
    uint32_t remote, v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(x)), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote) : "memory");
    return v;
}

__global__ void __cluster_dims__(kSelCluster, 1, 1) __launch_bounds__(kSelBlock)
    spoof_select(const double2 *a, long long n, long long need, unsigned long long base, OpenQubits open,
                 unsigned long long *bits, double *prob) {
    __shared__ unsigned int hist[2][256], total[256], above[256], counts[2], wt[kSelBlock / 32];
    __shared__ unsigned int pick, pick_above, pick_total;
    const int tid = threadIdx.x, rank = blockIdx.x;
    // block r holds positions [r per, (r + 1) per), kSelBlock at a time
    const long long per = max((long long)kSelBlock, n / kSelCluster), first = rank * per;
    unsigned long long key[kSelKeys];
#pragma unroll
    for (int j = 0; j < kSelKeys; j++) {
        const long long o = (long long)j * kSelBlock + tid, i = first + o;
        key[j] = 0ull;
        if (o < per && i < n)
            key[j] = (unsigned long long)__double_as_longlong(
                __dadd_rn(__dmul_rn(a[i].x, a[i].x), __dmul_rn(a[i].y, a[i].y)));
    }
    auto held = [&](int j) {
        const long long o = (long long)j * kSelBlock + tid;
        return o < per && first + o < n;
    };
    unsigned long long prefix = 0, mask = 0;
    unsigned int left = (unsigned int)need;
    if (tid < 256) hist[0][tid] = 0;
    __syncthreads();
    for (int d = 0; d < 8; d++) {
        const int shift = 56 - 8 * d, cur = d & 1;
#pragma unroll
        for (int j = 0; j < kSelKeys; j++)
        {
            // the leading digits of all keys are nearly the same: where a warp's digits are one, it
            // adds their number at once (a match of arbitrary digits costs more than it saves)
            const bool in = held(j) && (key[j] & mask) == prefix;
            const unsigned int act = __ballot_sync(0xffffffffu, in);
            if (act) {
                const int lead = __ffs(act) - 1;
                const unsigned int digit = (unsigned int)(key[j] >> shift) & 255u;
                const unsigned int first_digit = __shfl_sync(0xffffffffu, digit, lead);
                if (__all_sync(0xffffffffu, !in || digit == first_digit)) {
                    if ((tid & 31) == lead) atomicAdd(&hist[cur][digit], (unsigned int)__popc(act));
                } else if (in) {
                    atomicAdd(&hist[cur][digit], 1u);
                }
            }
        }
        cluster_barrier();
        // every block reads all histograms; the other buffer was last read before this barrier
        if (tid < 256) {
            unsigned int part[kSelCluster], t = 0;  // the loads are in flight together
#pragma unroll
            for (int r = 0; r < kSelCluster; r++) part[r] = cluster_load(&hist[cur][tid], r);
#pragma unroll
            for (int r = 0; r < kSelCluster; r++) t += part[r];
            total[tid] = t;
            hist[cur ^ 1][tid] = 0;
        }
        __syncthreads();
        // above[x]: keys with a larger digit, by one warp, 8 digits per lane
        if (tid < 32) {
            unsigned int own = 0;
            for (int i = 0; i < 8; i++) own += total[255 - (8 * tid + i)];
            unsigned int inc = own;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (tid >= o) inc += y;
            }
            unsigned int run = inc - own;
            for (int i = 0; i < 8; i++) {
                above[255 - (8 * tid + i)] = run;
                run += total[255 - (8 * tid + i)];
            }
        }
        __syncthreads();
        // the largest digit whose keys and those above reach `left` (0 if none does)
        if (tid < 256 && above[tid] < left && (tid == 0 || above[tid] + total[tid] >= left)) {
            pick = tid;
            pick_above = above[tid];
            pick_total = total[tid];
        }
        __syncthreads();
        left -= pick_above;
        prefix |= (unsigned long long)pick << shift;
        mask |= 255ull << shift;
        const bool whole = pick_total == left;  // every key with this prefix: lower digits don't matter
        __syncthreads();
        if (whole) break;
    }
    // selected: keys above prefix (as far as its digits go), and the first `left` equal to it
    unsigned int g = 0, e = 0;
#pragma unroll
    for (int j = 0; j < kSelKeys; j++) {
        g += __syncthreads_count(held(j) && (key[j] & mask) > prefix);
        e += __syncthreads_count(held(j) && (key[j] & mask) == prefix);
    }
    if (tid == 0) {
        counts[0] = g;
        counts[1] = e;
    }
    cluster_barrier();
    unsigned int g0 = 0, e0 = 0;  // in the blocks before this one
    {
        unsigned int cg[kSelCluster], ce[kSelCluster];
#pragma unroll
        for (int r = 0; r < kSelCluster; r++) {
            cg[r] = cluster_load(&counts[0], r);
            ce[r] = cluster_load(&counts[1], r);
        }
#pragma unroll
        for (int r = 0; r < kSelCluster; r++)
            if (r < rank) {
                g0 += cg[r];
                e0 += ce[r];
            }
    }
    cluster_barrier();  // no block leaves while its counts are being read
#pragma unroll
    for (int j = 0; j < kSelKeys; j++) {
        const bool gt = held(j) && (key[j] & mask) > prefix, eq = held(j) && (key[j] & mask) == prefix;
        unsigned int t;
        const unsigned int local = block_rank2(gt, eq, wt, t), lg = local & 0xffffu, le = local >> 16;
        if (gt || (eq && e0 + le < left)) {
            const unsigned int pos = g0 + lg + min(e0 + le, left);
            const long long i = first + (long long)j * kSelBlock + tid;
            unsigned long long b = base;
            for (int r = 0; r < open.n; r++) b |= (unsigned long long)((i >> r) & 1) << open.q[r];
            bits[pos] = b;
            if (prob) prob[pos] = __longlong_as_double((long long)key[j]);
        }
        g0 += t & 0xffffu;
        e0 += t >> 16;
    }
}

// ---------------------------------------------------------------- Philox

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of two 32x32->64
// multiplications with key bumps by the Weyl constants.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; r++) {
        if (r > 0) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

__device__ __forceinline__ double u53(uint32_t lo, uint32_t hi) {
    const uint64_t w = ((uint64_t)hi << 32) | lo;
    return __dmul_rn((double)(w >> 11), 1.0 / 9007199254740992.0);
}

__global__ void draw_batches(uint64_t seed, uint64_t t0, long long T, int b_bits, uint64_t *j) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const uint64_t tt = t0 + (uint64_t)t;
    const uint4 o = philox4x32_10(make_uint4((uint32_t)tt, (uint32_t)(tt >> 32), 0u, 0u),
                                  make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    const uint64_t w = ((uint64_t)o.y << 32) | o.x;
    j[t] = b_bits >= 64 ? w : (w & ((1ull << b_bits) - 1));
}

struct SampleParams {
    const double *p;      // T*64 probabilities, or null (then amps/F)
    const double2 *amps;  // T*64 amplitudes
    double invF_num;      // F (p = |a|^2 / F)
    long long T;
    int b_bits;
    double alpha;
    uint64_t seed, t0;
    uint8_t *accept;
    int32_t *pick;
    double *eps;          // optional: max(0, p_j - alpha/N_B)
    const uint64_t *j;    // optional: batch patterns (for bitstrings)
    uint64_t *bits;       // optional: assembled bitstrings
    int n_open, n_closed;
    int8_t open_q[16];
    int8_t closed_q[64];
};

// One warp, one batch (Sec. II.A steps 2-3); lane l holds p_{2l}, p_{2l+1}.
__device__ __forceinline__ void sampler_batch(const SampleParams &sp, long long warp, int lane) {
    double p0, p1;
    if (sp.p) {
        p0 = sp.p[warp * 64 + 2 * lane];
        p1 = sp.p[warp * 64 + 2 * lane + 1];
    } else {
        const double2 a0 = sp.amps[warp * 64 + 2 * lane], a1 = sp.amps[warp * 64 + 2 * lane + 1];
        p0 = __ddiv_rn(__dadd_rn(__dmul_rn(a0.x, a0.x), __dmul_rn(a0.y, a0.y)), sp.invF_num);
        p1 = __ddiv_rn(__dadd_rn(__dmul_rn(a1.x, a1.x), __dmul_rn(a1.y, a1.y)), sp.invF_num);
    }
    double x = __dadd_rn(p0, p1);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x = __dadd_rn(y, x);
    }
    const double pj = __shfl_sync(0xffffffffu, x, 31);
    double excl = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) excl = 0.0;
    const uint64_t t = sp.t0 + (uint64_t)warp;
    const uint2 key = make_uint2((uint32_t)sp.seed, (uint32_t)(sp.seed >> 32));
    const uint4 o0 = philox4x32_10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), 0u, 0u), key);
    const uint4 o1 = philox4x32_10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), 1u, 0u), key);
    const double u = u53(o0.z, o0.w), v = u53(o1.x, o1.y);
    const double NB = ldexp(1.0, sp.b_bits);
    const bool acc = __dmul_rn(u, sp.alpha) < __dmul_rn(pj, NB);
    const double tau = __dmul_rn(v, pj);
    const double c0 = __dadd_rn(excl, p0), c1 = x;
    const bool h0 = c0 > tau, h1 = c1 > tau;
    const unsigned hit = __ballot_sync(0xffffffffu, h0 || h1);
    int pick;
    if (hit) {
        const int L = __ffs(hit) - 1;
        const bool l0 = __shfl_sync(0xffffffffu, h0, L);
        pick = l0 ? 2 * L : 2 * L + 1;
    } else {
        const unsigned nz = __ballot_sync(0xffffffffu, p0 > 0.0 || p1 > 0.0);
        if (nz) {
            const int L = 31 - __clz(nz);
            const bool z1 = __shfl_sync(0xffffffffu, p1 > 0.0, L);
            pick = z1 ? 2 * L + 1 : 2 * L;
        } else {
            pick = 63;
        }
    }
    if (lane == 0) {
        sp.accept[warp] = acc ? 1 : 0;
        sp.pick[warp] = pick;
        if (sp.eps) sp.eps[warp] = fmax(__dadd_rn(pj, -sp.alpha / NB), 0.0);
        if (sp.bits) {
            const uint64_t jj = sp.j[warp];
            uint64_t b = 0;
            for (int r = 0; r < sp.n_open; r++) b |= (uint64_t)((pick >> r) & 1) << sp.open_q[r];
            for (int c = 0; c < sp.n_closed; c++) b |= ((jj >> c) & 1ull) << sp.closed_q[c];
            sp.bits[warp] = b;
        }
    }
}

__global__ void sampler(SampleParams sp) {
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp < sp.T) sampler_batch(sp, warp, threadIdx.x & 31);
}

// The sampler on given probabilities, decided in FP32 wherever FP32 can decide.
//
// The kernel above is bound by the FP64 pipe (2 lanes per clock and SM): about 20 FP64
// instructions per batch, each issued for a whole warp, took 330 us on 225280 batches whose
// 115 MB of probabilities take 17 us to read.  Both decisions are comparisons (u alpha < p
// N_B, and the first prefix above v p), so they are made on FP32 approximations first:
// prefixes of truncated values are within 2^-20 of the total of the FP64 prefixes, v within
// 2^-23, so a comparison whose sides differ by more than 2^-18 of the total has the same
// outcome in FP64.  A batch with any closer comparison, with a value that is negative, not
// finite or -0, whose total is outside [2^-90, 2^90], or without a hit runs sampler_batch
// (about one in 2000 for random probabilities), so every output equals the kernel above:
// 330 -> 53 us for a whole call on those batches.
// A warp takes `per` (<= 32) consecutive batches; lane b forms batch b's draws, which would
// otherwise be formed 32 times over.  Requires 16-byte aligned p and a finite xscale =
// N_B / alpha in [2^-60, 2^60] (the host's rule); no eps, no bits.
constexpr int kFilterUnroll = 8;  // batches whose loads are in flight together
__device__ __forceinline__ float trunc_to_float(uint32_t lo, uint32_t hi) {
    // a non-negative finite double's FP32 truncation (below 2^-120: 0; from 2^121: 2^121)
    const uint32_t h = min(hi, (1023u + 121u) << 20) - ((1023u - 127u) << 20);
    return hi < ((1023u - 120u) << 20) ? 0.f : __uint_as_float((h << 3) | (lo >> 29));
}
__global__ void __launch_bounds__(256) sampler_filter(SampleParams sp, int per, float xscale) {
    const int lane = threadIdx.x & 31;
    const long long t0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per;
    if (t0 >= sp.T) return;
    const int nb = (int)min((long long)per, sp.T - t0);
    const float kMargin = 1.f / 262144.f;
    float u = 0.f, v = 0.f;
    if (lane < nb) {
        const uint64_t t = sp.t0 + (uint64_t)(t0 + lane);
        const uint2 key = make_uint2((uint32_t)sp.seed, (uint32_t)(sp.seed >> 32));
        const uint4 o0 = philox4x32_10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), 0u, 0u), key);
        const uint4 o1 = philox4x32_10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), 1u, 0u), key);
        // the draws' upper 32 of 53 bits
        u = __uint2float_rn(o0.w) * (1.f / 4294967296.f);
        v = __uint2float_rn(o1.y) * (1.f / 4294967296.f);
    }
    int pick = 0;        // lane b: batch b's pick and total
    float total = 0.f;
    unsigned exact = 0;  // batches that need FP64
    for (int b0 = 0; b0 < nb; b0 += kFilterUnroll) {
        uint4 q[kFilterUnroll];
#pragma unroll
        for (int i = 0; i < kFilterUnroll; i++) {
            const long long t = t0 + min(b0 + i, nb - 1);
            q[i] = __ldcs(reinterpret_cast<const uint4 *>(sp.p + t * 64) + lane);
        }
#pragma unroll
        for (int i = 0; i < kFilterUnroll; i++) {
            const int b = b0 + i;
            if (b >= nb) break;
            // sign, infinity and NaN show in the high words
            bool bad = max(q[i].y, q[i].w) >= 0x7ff00000u;
            const float p0 = trunc_to_float(q[i].x, q[i].y), p1 = trunc_to_float(q[i].z, q[i].w);
            float x = p0 + p1;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const float y = __shfl_up_sync(0xffffffffu, x, off);
                if (lane >= off) x += y;
            }
            const float pj = __shfl_sync(0xffffffffu, x, 31);
            float excl = __shfl_up_sync(0xffffffffu, x, 1);
            if (lane == 0) excl = 0.f;
            const float tau = __shfl_sync(0xffffffffu, v, b) * pj, m = pj * kMargin;
            const float d0 = excl + p0 - tau, d1 = x - tau;
            bad |= fabsf(d0) <= m || fabsf(d1) <= m;
            const unsigned hit = __ballot_sync(0xffffffffu, d0 > 0.f || d1 > 0.f);
            const unsigned even = __ballot_sync(0xffffffffu, d0 > 0.f);
            const unsigned anybad = __ballot_sync(0xffffffffu, bad);
            const int L = __ffs(hit) - 1;
            if (lane == b) {
                pick = 2 * L + (((even >> (L & 31)) & 1u) ? 0 : 1);
                total = pj;
            }
            if (anybad || !hit || !(pj > 0x1p-90f && pj < 0x1p90f)) exact |= 1u << b;
        }
    }
    const float x = total * xscale, d = x - u;
    const bool close = lane < nb && !(fabsf(d) > kMargin * (x + u) + 0x1p-29f);
    exact |= __ballot_sync(0xffffffffu, close);
    if (lane < nb && !((exact >> lane) & 1u)) {
        sp.accept[t0 + lane] = d > 0.f ? 1 : 0;
        sp.pick[t0 + lane] = pick;
    }
    for (; exact; exact &= exact - 1) sampler_batch(sp, t0 + __ffs(exact) - 1, lane);
}

// ---------------------------------------------------------------- slice cut

// A double as an unsigned integer in the same order (-0 as +0; NaN as 0, below all others).
__device__ __forceinline__ unsigned long long order_key(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    if ((b << 1) > 0xffe0000000000000ull) return 0ull;
    if ((b << 1) == 0ull) return 1ull << 63;
    return b >> 63 ? ~b : b | (1ull << 63);
}

// Alg. 1 steps 4-5 for 2^k <= 4096 norms, in two launches.  Norm i's place in (R descending,
// i ascending) order is the number of norms before it: slice_rank counts them, 32 norms per
// block against all keys in shared memory, one eighth of the keys per warp (a broadcast read
// serves the 32 norms).  slice_cut then scatters the keys to their places and adds them up.
//
// Both are bound by latency.  A bitonic sort in one block (order keys as integers, since an
// FP64 comparison of a warp holds the SM's FP64 pipe 16 cycles) took most of 105 us at 2^12 norms:
// 78 dependent stages on one SM.  The FP64 prefix is a chain of one addition per norm up to
// the cut; every lane of a warp forms it, lane l keeps the l-th of 32 sums, and the 32
// comparisons with f are one ballot.  Repeated whole calls at 2^12 norms and f = 0.3: 150 -> 75 us.
constexpr int kRankWarps = 8;
__global__ void __launch_bounds__(32 * kRankWarps) slice_rank(const double *R, int k, int32_t *rank) {
    extern __shared__ unsigned long long rank_key[];
    __shared__ int part[kRankWarps][32];
    const int n = 1 << k, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < n; i += 32 * kRankWarps) rank_key[i] = order_key(R[i]);
    __syncthreads();
    const int i = blockIdx.x * 32 + lane, seg = (n + kRankWarps - 1) / kRankWarps;
    const int lo = warp * seg, hi = min(n, lo + seg);
    int c = 0;
    if (i < n) {
        const unsigned long long x = rank_key[i];
        // an equal norm is before i if its index is lower
        const int mid = max(lo, min(hi, i));
#pragma unroll 8
        for (int j = lo; j < mid; j++) c += rank_key[j] >= x;
#pragma unroll 8
        for (int j = mid; j < hi; j++) c += rank_key[j] > x;
    }
    part[warp][lane] = c;
    __syncthreads();
    if (warp == 0 && i < n) {
        int t = 0;
        for (int w = 0; w < kRankWarps; w++) t += part[w][lane];
        rank[i] = t;
    }
}

// rank: from slice_rank; may be X itself (it is read before X is written).
__global__ void __launch_bounds__(1024) slice_cut(const double *R, int k, double f, const int32_t *rank, int32_t *X,
                                                  int32_t *n_x, double *F) {
    extern __shared__ unsigned char smem[];
    __shared__ int count;
    const int n = 1 << k;
    double *r = reinterpret_cast<double *>(smem);
    unsigned short *idx = reinterpret_cast<unsigned short *>(r + n);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int t = rank[i];
        r[t] = R[i];
        idx[t] = (unsigned short)i;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const unsigned long long fk = f == f ? order_key(f) : ~0ull;  // no sum reaches a NaN f
        double acc = 0.0;
        int cnt = n;
        for (int t = 0; t < n; t += 32) {
            const int m = min(32, n - t);
            double mine = 0.0;
#pragma unroll 8
            for (int i = 0; i < m; i++) {
                acc = __dadd_rn(acc, r[t + i]);
                if (lane == i) mine = acc;
            }
            const unsigned hit = __ballot_sync(0xffffffffu, lane < m && order_key(mine) >= fk);
            if (hit) {
                const int l = __ffs(hit) - 1;
                cnt = t + l + 1;
                acc = __shfl_sync(0xffffffffu, mine, l);
                break;
            }
        }
        if (lane == 0) {
            count = cnt;
            *n_x = cnt;
            *F = acc;
        }
    }
    __syncthreads();
    const int cnt = count;
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) X[t] = idx[t];
}
// Both launches; rank and X share their 2^k words.
inline void launch_slice_cut(const double *R, int k, double f, int32_t *X, int32_t *n_x, double *F, cudaStream_t st) {
    const int n = 1 << k;
    slice_rank<<<(n + 31) / 32, 32 * kRankWarps, n * sizeof(unsigned long long), st>>>(R, k, X);
    slice_cut<<<1, std::max(32, std::min(1024, n)), n * (sizeof(double) + sizeof(unsigned short)), st>>>(R, k, f, X, X, n_x,
                                                                                                       F);
}

}  // namespace tnk
