// tcgen05 split-precision complex GEMM (sm_103a) for the contraction steps.
//
// C[bat][m][n] = sum_k A[bat][m][k] * B[bat][n][k] with A and B stored as four planes
// (re_hi, re_lo, im_hi, im_lo) of bf16 or fp16, plane-major: plane p of batch b is the
// row-major [rows][K] matrix at plane index p * BAT + b.  With x = hi + lo the complex
// product keeps hi*hi + hi*lo + lo*hi of each real product:
//   Cr = Ar Br - Ai Bi,  Ci = Ar Bi + Ai Br,
// i.e. 12 tensor-core MMAs per K slice accumulated in FP32 in two TMEM accumulators
// (Cr, Ci); the subtracted products use the descriptor's negate-A bit.
//
// One CTA computes a 128 x BN tile: warp 0 / lane 0 streams the 8 operand plane tiles
// of each 32-wide K slice with 4-D TMA (64-byte swizzle) into a ring of stages, warp 1 /
// lane 0 issues the MMAs and releases ring slots with tcgen05.commit, and eight epilogue
// warps read the accumulators back with tcgen05.ld (warp w owns TMEM lanes
// 32 (w % 4) .. 32 (w % 4) + 31, i.e. tile rows, and half of the columns) and store in the
// consumer's format through the bit-scatter epilogue.
// Every mbarrier wait is bounded: on timeout the CTA sets *err, stops, waits (bounded)
// for work it already issued, frees its TMEM and returns.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "kernels.cuh"

namespace tnk {

constexpr int kTcBM = 128;
constexpr int kTcBK = 32;      // K elements per ring slot (64 bytes per row: 64B swizzle)

// An operand read in place from its stored form instead of a per-batch gathered copy.
// The stored form is the read layout [K][rows][non-beta batch bits] with the operand's
// closed legs on top; a tile of batch `bat` reads plane coordinate (non-beta bits of bat)
// | (the batch pattern's bits q[0..nq) packed) << nnb, the pattern being the group's
// closed_bits[beta index of bat].
struct TcGather {
    const uint64_t *closed;  // null: the operand is read as laid out (no gather)
    uint32_t beta_mask;      // bits of bat that are beta (batch-index) bits
    int8_t beta_t[24];       // for such bit i: which bit of the batch index it is
    int nnb;                 // non-beta bits of bat
    int nq;
    int8_t q[32];            // closed positions of the pattern bits, lowest first
};

// The stored block a batch pattern selects: its bits at the closed positions q[].
__device__ __forceinline__ int tc_gather_sel(const TcGather &g, uint64_t pat) {
    int sel = 0;
    for (int t = 0; t < g.nq; t++) sel |= (int)((pat >> g.q[t]) & 1ull) << t;
    return sel;
}

__device__ __forceinline__ int tc_gather_plane(const TcGather &g, int lbat, int bat) {
    int beta = 0, nonb = 0, j = 0;
    for (int i = 0; i < lbat; i++) {
        const int bit = (bat >> i) & 1;
        if ((g.beta_mask >> i) & 1) beta |= bit << g.beta_t[i];
        else nonb |= bit << j++;
    }
    return nonb | (tc_gather_sel(g, g.closed[beta]) << g.nnb);
}

// The batch index whose beta bits are `beta` and whose other bits are `nonb` (lowest first).
__device__ __forceinline__ int tc_compose_bat(const TcGather &g, int lbat, int nonb, int beta) {
    int bat = 0, j = 0;
    for (int i = 0; i < lbat; i++) {
        const int bit = ((g.beta_mask >> i) & 1) ? (beta >> g.beta_t[i]) & 1 : (nonb >> j++) & 1;
        bat |= bit << i;
    }
    return bat;
}

// Stacked tiles.  The batches of a group whose patterns select the same stored block of
// the in-place operand A multiply the same A matrix; a stacked tile takes up to S of them
// (S = BN / N) and puts their B rows side by side in its BN columns, so the A panel is
// loaded once for S batches and one MMA of BN columns serves them all.  The stack list is
// built on the device per group (tc_stack_build): word 0 the number of stacks, then S + 1
// words per stack: the selected block, then S batch indices (beta), -1 in unused slots
// (the valid ones first).
constexpr int kTcMaxStack = 4;

// Sorts the group's T = 2^nbeta batch indices by (selected block, beta) with a bitonic
// sort in shared memory (deterministic), then cuts each block's run into stacks of S.
// One block of 1024 threads; dynamic shared memory 8 T bytes.
__global__ void __launch_bounds__(1024) tc_stack_build(TcGather g, int nbeta, int S, int *out) {
    extern __shared__ unsigned long long keys[];
    __shared__ int scan[1024];
    const int T = 1 << nbeta, nt = blockDim.x, tid = threadIdx.x;
    for (int b = tid; b < T; b += nt)
        keys[b] = ((unsigned long long)(unsigned)tc_gather_sel(g, g.closed[b]) << 32) | (unsigned)b;
    for (int i = tid; i < T * (S + 1); i += nt) out[1 + i] = -1;
    __syncthreads();
    // a thread owns pair t of a stage, so stages with j <= 32 stay inside a warp's 64 keys
    for (int k = 2; k <= T; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = tid; t < T / 2; t += nt) {
                const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1)), l = i | j;
                const unsigned long long x = keys[i], y = keys[l];
                if ((x > y) == ((i & k) == 0)) {
                    keys[i] = y;
                    keys[l] = x;
                }
            }
            if (j > 32 || (j == 1 && k > 32)) __syncthreads();
            else __syncwarp();
        }
    }
    __syncthreads();
    // thread tid walks positions [lo, hi) of the sorted list; a run starts where the block
    // changes, and a stack at every S-th position of a run
    const int E = (T + nt - 1) / nt, lo = min(T, tid * E), hi = min(T, lo + E);
    auto head = [&](int i) { return i == 0 || (keys[i] >> 32) != (keys[i - 1] >> 32); };
    int last = -1;
    for (int i = lo; i < hi; i++)
        if (head(i)) last = i;
    scan[tid] = last;  // inclusive max-scan: the last run start at or before the chunk's end
    __syncthreads();
    for (int d = 1; d < nt; d <<= 1) {
        const int v = tid >= d ? scan[tid - d] : -1;
        __syncthreads();
        scan[tid] = max(scan[tid], v);
        __syncthreads();
    }
    const int run0 = tid > 0 ? scan[tid - 1] : -1;
    __syncthreads();
    int starts = 0;
    last = run0;
    for (int i = lo; i < hi; i++) {
        if (head(i)) last = i;
        starts += (i - last) % S == 0;
    }
    scan[tid] = starts;  // inclusive sum-scan of the stack starts
    __syncthreads();
    for (int d = 1; d < nt; d <<= 1) {
        const int v = tid >= d ? scan[tid - d] : 0;
        __syncthreads();
        scan[tid] += v;
        __syncthreads();
    }
    int id = scan[tid] - starts - 1;  // stacks started before this chunk, minus one
    last = run0;
    for (int i = lo; i < hi; i++) {
        if (head(i)) last = i;
        const int pos = (i - last) % S;
        int *e = out + 1 + (id + (pos == 0)) * (S + 1);
        if (pos == 0) {
            id++;
            e[0] = (int)(keys[i] >> 32);
        }
        e[1 + pos] = (int)(keys[i] & 0xffffffffu);
    }
    if (tid == nt - 1) out[0] = scan[tid];
}

// Row products over the stack list: C[bat][m][n] = sum_k A[bat][m][k] B[bat][n][k] for a long
// row side read in place from stored blocks, N <= 4 columns and K <= 16.  The row kernel reads
// every batch's block anew (16384 batches of 1 MB each from 4096 stored blocks: 17 GB through
// L1, 16 bytes of 32 rows per instruction; (bat, m, n, k bits) = (14, 13, 0, 4) took 5.4 ms);
// here a block of threads takes up to 2048 rows of a stored block, 256 at a time, each thread
// one row in registers (staged through padded shared memory with coalesced loads), and
// applies them to the stack's batches; the addresses are decoded once per 2048 rows.  Each output's products and order are the row kernel's.  The same step: 5.4 -> 1.46 ms
// (3.1 ms with an item per 256 rows, whose decode then took as long as its rows).
constexpr int kRowStackRows = 256, kRowStackChunks = 8;  // rows per pass, passes per item
template <int N, int K>
__global__ void __launch_bounds__(kRowStackRows) cgemm_rowstack(GemmParams p, TcGather g, const int *stack, int S) {
    constexpr int kPitch = 8 * K + 16;  // bytes between staged rows: 16-byte reads without conflicts
    __shared__ __align__(16) unsigned char stage[kRowStackRows * kPitch];
    __shared__ __align__(16) float2 vec[kTcMaxStack][N * K];
    __shared__ long long cbase[kTcMaxStack];
    __shared__ const float2 *src[1 + kTcMaxStack];  // the block, the batches' columns
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int passes = min(kRowStackChunks, 1 << (p.lm - 8)), groups = (1 << (p.lm - 8)) / passes;
    const long long items = (long long)stack[0] * groups << g.nnb;
    unsigned char *mine = stage + warp * 32 * kPitch;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        const long long q = it / groups;
        const int row0 = (int)(it - q * groups) * passes * kRowStackRows, nonb = (int)(q & ((1 << g.nnb) - 1));
        const int *e = stack + 1 + (q >> g.nnb) * (S + 1);
        __syncthreads();  // the shared words of the previous item
        // one thread per address: the block's, then the batches'
        if (tid <= S) {
            const int beta = e[max(1, tid)];
            src[tid] = nullptr;
            if (beta >= 0) {
                const long long bat = tc_compose_bat(g, p.lbat, nonb, beta);
                if (tid == 0) {
                    src[0] = reinterpret_cast<const float2 *>(p.gA->src) +
                             gather_src(*p.gA, bat << (p.lm + p.lk), p.closed_bits);
                } else {
                    const long long eb = bat << (p.ln + p.lk);
                    src[tid] = p.gB ? reinterpret_cast<const float2 *>(p.gB->src) + gather_src(*p.gB, eb, p.closed_bits)
                                    : static_cast<const float2 *>(p.ptrB[0]) + eb;
                    cbase[tid - 1] = scatter_bits(bat, p.pos_bat, p.lbat);
                }
            }
        }
        __syncthreads();
        // the warp's 32 rows of a pass: 16 K float4, consecutive lanes consecutive addresses
        const float4 *A = reinterpret_cast<const float4 *>(src[0] + ((long long)(row0 + warp * 32) << p.lk)) + lane;
        float4 in[K / 2];
#pragma unroll
        for (int i = 0; i < K / 2; i++) in[i] = __ldg(A + i * 32);
        int cnt = 0;
        while (cnt < S && src[1 + cnt]) cnt++;
        for (int i = tid; i < cnt * N * K; i += kRowStackRows) vec[i / (N * K)][i % (N * K)] = __ldg(src[1 + i / (N * K)] + i % (N * K));
        __syncthreads();
        for (int c = 0; c < passes; c++) {
#pragma unroll
            for (int i = 0; i < K / 2; i++) {
                const int o = i * 32 + lane;
                *reinterpret_cast<float4 *>(mine + (o / (K / 2)) * kPitch + 16 * (o % (K / 2))) = in[i];
            }
            __syncwarp();
            float2 a[K];
#pragma unroll
            for (int i = 0; i < K / 2; i++) {
                const float4 x = *reinterpret_cast<const float4 *>(mine + lane * kPitch + 16 * i);
                a[2 * i] = make_float2(x.x, x.y);
                a[2 * i + 1] = make_float2(x.z, x.w);
            }
            __syncwarp();
            if (c + 1 < passes) {  // the next pass's rows are in flight during this one's products
                A += kRowStackRows * K / 2;
#pragma unroll
                for (int i = 0; i < K / 2; i++) in[i] = __ldg(A + i * 32);
            }
            const long long offm = scatter_bits(row0 + c * kRowStackRows + tid, p.pos_m, p.lm);
            for (int j = 0; j < cnt; j++) {
#pragma unroll
                for (int n = 0; n < N; n++) {
                    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < K / 2; i++) {
                        const float4 y = *reinterpret_cast<const float4 *>(&vec[j][n * K + 2 * i]);
                        const float2 y0 = make_float2(y.x, y.y), y1 = make_float2(y.z, y.w);
                        acc = p.swapped ? cfma(y0, a[2 * i], acc) : cfma(a[2 * i], y0, acc);
                        acc = p.swapped ? cfma(y1, a[2 * i + 1], acc) : cfma(a[2 * i + 1], y1, acc);
                    }
                    store_c(p, 0, cbase[j] + offm + scatter_bits(n, p.pos_n, p.ln), acc);
                }
            }
        }
    }
}

struct TcParams {
    void *C;                 // output base (version 0); version v at C + 8 * v * c_plane bytes
    long long c_plane;       // elements per version (= split plane stride)
    const int *vidx;         // [v]: A version index, [nver + v]: B version index
    int nver;                // explicit versions of C (power of two not required)
    int fold;                // 0: versions are tiles; 1: versions folded into M; 2: into N
    int lm, ln, lk, lbat;
    int out_fmt;
    int in_fp16;             // operands are fp16 (else bf16)
    float out_scale;         // multiply results by this before storing
    int *err;                // set to 1 if a bounded wait gives up
    int group_m;             // m tiles per raster group (>= 1): see tc_tile
    long long stall_cycles;  // > 0 (tests only): the MMA warp first waits this long on a
                             // barrier nothing arrives on, so the bounded-wait path runs
    TcGather ga, gb;         // operands read in place through their batch gather
    const int *stack;        // non-null: stacked tiles over this stack list (tc_stack_build)
    int stack_S;             // batches per stacked tile (BN >> ln)
    int8_t pos_bat[kMaxBits], pos_m[kMaxBits], pos_n[kMaxBits];
};

// Tile t of a launch: (batch, version) outermost; inside, groups of group_m m tiles are
// walked n tile by n tile with the m tiles of the group fastest, so the CTAs running
// together share a few operand panels of both A and B in L2 (with group_m = 1 this is
// the plain n-fastest order).
struct TcTile {
    int tn_i, tm_i, bat;
    int v;
};

// Stacked tile t: m tiles fastest, then stacks (sorted by block: the stacks of one block
// run back to back and share its panels in L2), then the non-beta batch bits, then version.
// Tile counts fit 32 bits (the host checks), which keeps the divisions short: the producer
// forms them between copies.
struct TcStackTile {
    int tm_i, stack, nonb;
    int v;
};
__device__ __forceinline__ TcStackTile tc_stack_tile(uint32_t t, uint32_t tiles_m, uint32_t n_stacks, int nnb) {
    TcStackTile r;
    uint32_t q = t / tiles_m;
    r.tm_i = (int)(t - q * tiles_m);
    const uint32_t z = q / n_stacks;
    r.stack = (int)(q - z * n_stacks);
    r.nonb = (int)(z & ((1u << nnb) - 1));
    r.v = (int)(z >> nnb);
    return r;
}

__device__ __forceinline__ TcTile tc_tile(uint32_t t, uint32_t tiles_m, uint32_t tiles_n, int lbat, uint32_t group_m) {
    const uint32_t per_bat = tiles_m * tiles_n;
    const uint32_t bv = t / per_bat, tl = t - bv * per_bat;
    TcTile r;
    r.bat = (int)(bv & ((1u << lbat) - 1));
    r.v = (int)(bv >> lbat);
    const uint32_t gsz = group_m * tiles_n;
    const uint32_t g = tl / gsz, rr = tl - g * gsz;
    const uint32_t gm = min(group_m, tiles_m - g * group_m);
    const uint32_t n = rr / gm;
    r.tn_i = (int)n;
    r.tm_i = (int)(g * group_m + rr - n * gm);
    return r;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor: K-major tile, 64-byte swizzle, 8-row groups 512 B
// apart (rows are 64 bytes), start address advanced by 32 B per 16-element K step.
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;            // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(512 >> 4) << 32;   // stride byte offset: 8 rows x 64 B
    d |= (uint64_t)1 << 46;            // descriptor version
    d |= (uint64_t)4 << 61;            // 64-byte swizzle
    return d;
}

// Instruction descriptor, kind::f16: D = F32, A/B = BF16 (1) or F16 (0), K-major both,
// N >> 3 at bit 17, M >> 4 at bit 24, optional negation of A.
__device__ __forceinline__ uint32_t idesc_f16(int n, bool fp16, bool neg_a) {
    uint32_t ab = fp16 ? 0u : 1u;
    return (1u << 4) | (ab << 7) | (ab << 10) | ((neg_a ? 1u : 0u) << 13) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(kTcBM >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

// Both accumulators' 16 columns (Cr, Ci) with one wait for the two loads.
__device__ __forceinline__ void tmem_ld16x2(uint32_t ta, uint32_t tb, float *va, float *vb) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(ta), "r"(tb)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) {
        va[i] = __uint_as_float(r[i]);
        vb[i] = __uint_as_float(r[16 + i]);
    }
}

template <int BN, int STAGES>
struct TcSmem {
    static constexpr int kAPlane = kTcBM * kTcBK * 2;  // bytes per A plane tile
    static constexpr int kBPlane = BN * kTcBK * 2;
    static constexpr int kStage = 4 * kAPlane + 4 * kBPlane;
    static constexpr int kBytes = STAGES * kStage + 1024 /*barriers*/ + 1024 /*alignment*/;
};

// 32 bytes (a whole sector) in one store instruction; dst 32-byte aligned.
__device__ __forceinline__ void st_global_32(void *dst, const uint32_t *w) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                 "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}

// hi and lo parts of two values as packed 16-bit pairs (the roundings of store_split).
__device__ __forceinline__ void split_pack2(float a, float b, bool fp16, uint32_t &hi, uint32_t &lo) {
    if (fp16) {
        const __half2 h = __floats2half2_rn(a, b);
        const float2 f = __half22float2(h);
        const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
        hi = *reinterpret_cast<const uint32_t *>(&h);
        lo = *reinterpret_cast<const uint32_t *>(&l);
    } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        hi = *reinterpret_cast<const uint32_t *>(&h);
        const __nv_bfloat162 l =
            __floats2bfloat162_rn(a - __uint_as_float(hi << 16), b - __uint_as_float(hi & 0xffff0000u));
        lo = *reinterpret_cast<const uint32_t *>(&l);
    }
}

// How the epilogue's lanes (one tile row each) and their 16 columns lie in C.
struct TcStorePlan {
    int nrun;    // 2^nrun columns are adjacent (the columns' lowest bits are C's lowest)
    bool mpair;  // rows 2 i and 2 i + 1 are adjacent (the rows' lowest bit is C's lowest)
    bool odd;    // this lane's row is odd
};

// Store 16 results of one tile row, column j at off0 + lo[j] (elements), if ok; every lane of
// the warp calls it.  The stores, not the products, set the pace of the tiles with small
// K: a lane that holds one row of a C with n lowest touches 32 separate sectors per store
// instruction whatever its width, so its adjacent columns go out together, up to 32 bytes at
// a time; with m lowest and split planes a 2-byte store per lane fills only 64 bytes per
// instruction, so neighbouring lanes exchange columns and store two rows of one column as
// 4 bytes.  (bat, m, n, k bits) = (12, 11, 5, 8), stacked, n lowest, complex64: 2.3 -> 1.95
// ms; (0, 21, 11, 7), m lowest, split: 15.5 -> 12.1 ms; (0, 23, 7, 5): 3.7 -> 2.75 ms.
__device__ __forceinline__ void tc_store16(const TcParams &p, void *Cv, long long off0, const long long (&lo)[16],
                                           const TcStorePlan sp, bool ok, const float (&re)[16], const float (&im)[16]) {
    const float sc = p.out_scale;
    if (p.out_fmt == OUT_C64) {
        if (!ok) return;
        float2 *c = static_cast<float2 *>(Cv) + off0;
        if (sp.nrun >= 2) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                uint32_t w[8];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    w[2 * i] = __float_as_uint(re[j + i] * sc);
                    w[2 * i + 1] = __float_as_uint(im[j + i] * sc);
                }
                st_global_32(c + lo[j], w);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 16; j++) c[lo[j]] = make_float2(re[j] * sc, im[j] * sc);
        }
        return;
    }
    const bool fp16 = p.out_fmt == OUT_SPLIT_FP16;
    unsigned short *h = static_cast<unsigned short *>(Cv) + off0;
#pragma unroll
    for (int ri = 0; ri < 2; ri++) {
        unsigned short *ph = h + 2 * ri * p.c_plane, *pl = ph + p.c_plane;
        uint32_t hi[8], lw[8];
#pragma unroll
        for (int j = 0; j < 16; j += 2)
            split_pack2((ri ? im[j] : re[j]) * sc, (ri ? im[j + 1] : re[j + 1]) * sc, fp16, hi[j / 2], lw[j / 2]);
        if (sp.mpair) {
            // an even lane keeps column j, its odd neighbour column j + 1
            const uint32_t sel = sp.odd ? 0x3276u : 0x5410u;
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
                const uint32_t oh = __shfl_xor_sync(0xffffffffu, hi[j / 2], 1);
                const uint32_t ol = __shfl_xor_sync(0xffffffffu, lw[j / 2], 1);
                const long long o = sp.odd ? lo[j + 1] - 1 : lo[j];
                if (ok) {
                    *reinterpret_cast<uint32_t *>(ph + o) = __byte_perm(hi[j / 2], oh, sel);
                    *reinterpret_cast<uint32_t *>(pl + o) = __byte_perm(lw[j / 2], ol, sel);
                }
            }
        } else if (!ok) {
            continue;
        } else if (sp.nrun >= 4) {
            st_global_32(ph, hi);
            st_global_32(pl, lw);
        } else if (sp.nrun >= 2) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                *reinterpret_cast<uint2 *>(ph + lo[j]) = make_uint2(hi[j / 2], hi[j / 2 + 1]);
                *reinterpret_cast<uint2 *>(pl + lo[j]) = make_uint2(lw[j / 2], lw[j / 2 + 1]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
                ph[lo[j]] = (unsigned short)hi[j / 2];
                ph[lo[j + 1]] = (unsigned short)(hi[j / 2] >> 16);
                pl[lo[j]] = (unsigned short)lw[j / 2];
                pl[lo[j + 1]] = (unsigned short)(lw[j / 2] >> 16);
            }
        }
    }
}

constexpr int kTcEpiWarps = 8;   // two per TMEM lane quarter, each owning half the tile's columns
constexpr int kTcThreads = 64 + 32 * kTcEpiWarps;  // warp 0: TMA, warp 1: MMA, warps 2-9: epilogue

// Persistent kernel: CTA c processes tiles c, c + gridDim.x, ...  Tile order: N tiles
// fastest, then M tiles, then batch, then explicit version (CTAs running together share
// the A row panel).  Operand maps are 4-D: [version][4 * BAT planes][rows][K].
// TMEM holds two accumulator pairs (Cr | Ci for BN columns each) so the epilogue of
// one tile overlaps the MMAs of the next.
// SW: the operands are exchanged (A holds the step's B, p.vidx's halves as for the step): the
// planes of each product swap sides and the products keep their order, so the bits are the
// same.  The engine exchanges them where C is split with m lowest, which puts 16 adjacent
// outputs into one lane (its rule, with both sides measured, stands at the launch).
template <int BN, int STAGES, bool SW = false>
__global__ void __launch_bounds__(kTcThreads, 1)
    tc_cgemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, TcParams p) {
    using L = TcSmem<BN, STAGES>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *ctl = smem + STAGES * L::kStage;
    uint64_t *full = reinterpret_cast<uint64_t *>(ctl);
    uint64_t *empty = full + STAGES;
    uint64_t *acc_full = empty + STAGES;  // [2]: MMA -> epilogue
    uint64_t *acc_empty = acc_full + 2;   // [2]: epilogue -> MMA
    uint64_t *never = acc_empty + 2;      // test stall: initialised, never arrived on
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(never + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *slot_cols = abort_flag + 1;  // [STAGES]: a stacked tile's MMA width

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Tiles: (n tile, m tile, batch, version) without folding.  With folding the rows
    // (fold 1) or columns (fold 2) of all versions form one axis: versions are stacked,
    // 128/M (or BN/N) per tile, and the operand's map box spans that many versions.
    const int ltm = min(p.lm, 7), ltn = min(p.ln, __ffs(BN) - 1);
    const int vm = p.fold == 1 ? (kTcBM >> p.lm) : 1;  // versions per m tile
    const int vn = p.fold == 2 ? (BN >> p.ln) : 1;      // versions per n tile
    const uint32_t tiles_m = p.fold == 1 ? (p.nver + vm - 1) / vm : (1u << (p.lm - ltm));
    const uint32_t tiles_n = p.fold == 2 ? (p.nver + vn - 1) / vn : (1u << (p.ln - ltn));
    const uint32_t tiles_v = p.fold ? 1 : p.nver;
    // stacked: (version, non-beta bits, stack, m tile); the host guarantees one n tile
    const bool stk = p.stack != nullptr;
    const int S = p.stack_S, n_stacks = stk ? p.stack[0] : 0;
    const uint32_t ntiles = (stk ? (tiles_m * n_stacks << p.ga.nnb) : (tiles_m * tiles_n << p.lbat)) * tiles_v;
    const int BAT = 1 << p.lbat;
    const int K = 1 << p.lk;
    const int nkb = (K + kTcBK - 1) / kTcBK;
    constexpr uint32_t kCols = 4 * BN;  // two accumulator pairs
    const long long kLimit = 4000000000LL;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; s++) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_empty[b]), kTcEpiWarps);  // one arrive per epilogue warp
        }
        mbar_init(smem_u32(never), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    long long issued = 0;  // producer: ring slots issued
    if (warp == 0) {
        const int sza = p.ga.closed ? 1 << (p.ga.nnb + p.ga.nq) : BAT;
        const int szb = p.gb.closed ? 1 << (p.gb.nnb + p.gb.nq) : BAT;
        int s = 0;
        uint32_t par = 1;  // of the empty barrier the next slot waits for
        bool ok = true;
        if (!stk && lane == 0) {
            for (uint32_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                const TcTile tt = tc_tile(t, tiles_m, tiles_n, p.lbat, p.group_m);
                const int tn_i = tt.tn_i, tm_i = tt.tm_i, bat = tt.bat, v = tt.v;
                const int *va = p.vidx + (SW ? p.nver : 0), *vb = p.vidx + (SW ? 0 : p.nver);
                const int ia = p.fold == 1 ? va[0] + tm_i * vm : va[p.fold == 2 ? 0 : v];
                const int ib = p.fold == 2 ? vb[0] + tn_i * vn : vb[p.fold == 1 ? 0 : v];
                const int rowA = p.fold == 1 ? 0 : tm_i * kTcBM, rowB = p.fold == 2 ? 0 : tn_i * BN;
                // plane coordinates: plane pl of batch bat, or of its stored pattern block
                const int pza = p.ga.closed ? tc_gather_plane(p.ga, p.lbat, bat) : bat;
                const int pzb = p.gb.closed ? tc_gather_plane(p.gb, p.lbat, bat) : bat;
                for (int kb = 0; kb < nkb; kb++) {
                    if (issued >= STAGES && !mbar_wait(smem_u32(&empty[s]), par, abort_flag, kLimit)) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = smem_u32(&full[s]);
                    mbar_expect_tx(fb, L::kStage);
                    unsigned char *st = smem + s * L::kStage;
                    for (int pl = 0; pl < 4; pl++) {
                        tma_load_4d(smem_u32(st + pl * L::kAPlane), &tmA, kb * kTcBK, rowA, pl * sza + pza, ia, fb);
                        tma_load_4d(smem_u32(st + 4 * L::kAPlane + pl * L::kBPlane), &tmB, kb * kTcBK, rowB,
                                    pl * szb + pzb, ib, fb);
                    }
                    issued++;
                    if (++s == STAGES) {
                        s = 0;
                        par ^= 1u;
                    }
                }
            }
        }
        // Stacked tiles: one A panel, then one (1 << ln)-row B box per batch of the stack (its
        // valid slots come first); every slot tells the MMA thread its width.  Decoding a tile
        // takes a chain of loads (stack entry, batch patterns) and divisions as long as several
        // ring slots, so the warp decodes the next tile, one lane per batch, right after it has
        // issued the first slot of this one, while the ring is full: (12, 11, 5, 8) 1.95 ->
        // 1.80 ms.  (The same for unstacked tiles, whose decode is short, made them 10% slower.)
        struct Dec {
            int pza, pzb, rowA, ia, ib, nbox;
        };
        auto decode = [&](uint32_t t) {
            Dec d;
            const TcStackTile tt = tc_stack_tile(t, tiles_m, n_stacks, p.ga.nnb);
            const int *e = p.stack + 1 + (long long)tt.stack * (S + 1);
            const int beta = lane < S ? e[1 + lane] : -1;
            d.pza = tt.nonb | (e[0] << p.ga.nnb);  // the block the stack selects
            d.pzb = 0;
            if (beta >= 0) {
                const int bat = tc_compose_bat(p.ga, p.lbat, tt.nonb, beta);
                d.pzb = p.gb.closed ? tc_gather_plane(p.gb, p.lbat, bat) : bat;
            }
            d.nbox = __popc(__ballot_sync(0xffffffffu, beta >= 0));
            d.rowA = tt.tm_i * kTcBM;
            d.ia = p.vidx[tt.v];
            d.ib = p.vidx[p.nver + tt.v];
            return d;
        };
        const int bbox = (kTcBK * 2) << p.ln;  // bytes per B box
        Dec next = {0, 0, 0, 0, 0, 0};
        if (stk && blockIdx.x < ntiles) next = decode(blockIdx.x);
        for (uint32_t t = blockIdx.x; t < ntiles && ok && stk; t += gridDim.x) {
            const Dec d = next;
            int pzb[kTcMaxStack];
#pragma unroll
            for (int j = 0; j < kTcMaxStack; j++) pzb[j] = __shfl_sync(0xffffffffu, d.pzb, j);
            for (int kb = 0; kb < nkb; kb++) {
                if (lane == 0) {
                    if (issued >= STAGES) ok = mbar_wait(smem_u32(&empty[s]), par, abort_flag, kLimit);
                    if (ok) {
                        slot_cols[s] = d.nbox << p.ln;  // published by the arrive below
                        const uint32_t fb = smem_u32(&full[s]);
                        mbar_expect_tx(fb, (uint32_t)(4 * L::kAPlane + 4 * d.nbox * bbox));
                        unsigned char *st = smem + s * L::kStage;
#pragma unroll
                        for (int pl = 0; pl < 4; pl++) {
                            tma_load_4d(smem_u32(st + pl * L::kAPlane), &tmA, kb * kTcBK, d.rowA, pl * sza + d.pza, d.ia, fb);
#pragma unroll
                            for (int j = 0; j < kTcMaxStack; j++)
                                if (j < d.nbox)
                                    tma_load_4d(smem_u32(st + 4 * L::kAPlane + pl * L::kBPlane + j * bbox), &tmB,
                                                kb * kTcBK, 0, pl * szb + pzb[j], d.ib, fb);
                        }
                    }
                }
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                if (!ok) break;
                issued++;
                if (++s == STAGES) {
                    s = 0;
                    par ^= 1u;
                }
                if (kb == 0 && t + gridDim.x < ntiles) next = decode(t + gridDim.x);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // products (A plane, B plane, accumulator 0 = Cr / 1 = Ci, negate A);
            // planes: 0 re_hi, 1 re_lo, 2 im_hi, 3 im_lo
            const int8_t p0[12] = {0, 0, 1, 2, 2, 3, 0, 0, 1, 2, 2, 3};
            const int8_t p1[12] = {0, 1, 0, 2, 3, 2, 2, 3, 2, 0, 1, 0};
            const int8_t(&pa)[12] = SW ? p1 : p0, (&pb)[12] = SW ? p0 : p1;
            const int8_t acc[12] = {0, 0, 0, 0, 0, 0, 1, 1, 1, 1, 1, 1};
            const int8_t neg[12] = {0, 0, 0, 1, 1, 1, 0, 0, 0, 0, 0, 0};
            uint32_t id_pos = idesc_f16(BN, p.in_fp16, false), id_neg = idesc_f16(BN, p.in_fp16, true);
            long long slot = 0;
            int it = 0, last_b = -1;
            uint32_t last_par = 0;
            bool ok = true;
            // test hook: a wait that runs out before any MMA is issued
            if (p.stall_cycles > 0) ok = mbar_wait(smem_u32(never), 0u, abort_flag, p.stall_cycles);
            for (uint32_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x, it++) {
                const int b = it & 1;
                if (it >= 2 &&
                    !mbar_wait(smem_u32(&acc_empty[b]), (uint32_t)(((it >> 1) & 1) ^ 1), abort_flag, kLimit)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t dcol = tmem + (uint32_t)(b * 2 * BN);
                for (int kb = 0; kb < nkb; kb++, slot++) {
                    const int s = (int)(slot % STAGES);
                    if (!mbar_wait(smem_u32(&full[s]), (uint32_t)((slot / STAGES) & 1), abort_flag, kLimit)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (stk && kb == 0) {
                        // a stacked tile multiplies only its valid batches' columns (the
                        // valid slots come first): N = count << ln, a multiple of 32
                        const int n = slot_cols[s];
                        id_pos = idesc_f16(n, p.in_fp16, false);
                        id_neg = idesc_f16(n, p.in_fp16, true);
                    }
                    const uint32_t st = smem_u32(smem + s * L::kStage);
#pragma unroll
                    for (int kk = 0; kk < kTcBK / 16; kk++) {
#pragma unroll
                        for (int q = 0; q < 12; q++) {
                            const uint64_t ad = smem_desc_sw64(st + pa[q] * L::kAPlane + kk * 32);
                            const uint64_t bd = smem_desc_sw64(st + 4 * L::kAPlane + pb[q] * L::kBPlane + kk * 32);
                            const uint32_t accum = (kb == 0 && kk == 0 && (q == 0 || q == 6)) ? 0u : 1u;
                            mma_f16(dcol + (acc[q] ? BN : 0), ad, bd, neg[q] ? id_neg : id_pos, accum);
                        }
                    }
                    mma_commit(smem_u32(&empty[s]));
                }
                mma_commit(smem_u32(&acc_full[b]));  // also after an abort: flushes issued MMAs
                last_b = b;
                last_par = (uint32_t)((it >> 1) & 1);
            }
            // after an abort, MMAs may still be running: drain them before TMEM is freed
            if (*abort_flag && last_b >= 0) mbar_drain(smem_u32(&acc_full[last_b]), last_par, kLimit);
        }
    } else {
        // epilogue warps 2..9: TMEM lane quarter = warp % 4 = tile rows 32*(warp%4)..; warps
        // 2-5 store columns [0, BN/2) of the tile, warps 6-9 columns [BN/2, BN)
        const int quarter = warp & 3;
        const int c_begin = ((warp - 2) >> 2) * (BN / 2), c_end = c_begin + BN / 2;
        const int row = 32 * quarter + lane;
        const long long M = 1LL << p.lm, N = 1LL << p.ln;
        // scatter(n0 + c0 + j) = scatter(n0 + c0) + scatter(j) for j < 16 (disjoint bits)
        const int lo_bits = min(p.ln, 4);
        long long lo[16];
#pragma unroll
        for (int j = 0; j < 16; j++) lo[j] = scatter_bits(j, p.pos_n, lo_bits);
        TcStorePlan plan = {0, p.lm > 0 && p.pos_m[0] == 0, (row & 1) != 0};
        while (plan.nrun < lo_bits && p.pos_n[plan.nrun] == plan.nrun) plan.nrun++;
        int it = 0;
        for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x, it++) {
            const int b = it & 1;
            // the tile's coordinates and output bases first: their loads and bit scatters
            // overlap the wait for the accumulator
            TcTile tt;
            const int *sb = nullptr;  // stacked: this tile's batch indices
            int nonb = 0;
            if (stk) {
                const TcStackTile ts = tc_stack_tile(t, tiles_m, n_stacks, p.ga.nnb);
                tt.tn_i = 0;
                tt.tm_i = ts.tm_i;
                tt.v = ts.v;
                tt.bat = 0;
                sb = p.stack + 2 + (long long)ts.stack * (S + 1);  // the stack's batch indices
                nonb = ts.nonb;
            } else {
                tt = tc_tile(t, tiles_m, tiles_n, p.lbat, p.group_m);
            }
            const int tn_i = tt.tn_i, tm_i = tt.tm_i, bat = tt.bat;
            long long vrow = tt.v;  // this row's version
            long long m;
            if (p.fold == 1) {
                vrow = (long long)tm_i * vm + (row >> p.lm);
                m = row & (M - 1);
            } else {
                m = (long long)tm_i * kTcBM + row;
            }
            const bool row_ok = m < M && vrow < p.nver;
            const long long mbase = row_ok ? scatter_bits(m, p.pos_m, p.lm) : 0;
            long long cbase = scatter_bits(bat, p.pos_bat, p.lbat) + mbase;
            // stacked: this warp's columns cover the stack's batches j0 and (if BN / 2 > N)
            // j0 + 1; their indices (-1: empty) and output bases
            const int j0 = c_begin >> p.ln;
            int be0 = -1, be1 = -1;
            long long cb0 = 0, cb1 = 0;
            if (stk) {
                be0 = j0 < S ? sb[j0] : -1;
                be1 = (j0 + 1 < S && ((j0 + 1) << p.ln) < c_end) ? sb[j0 + 1] : -1;
                if (be0 >= 0) cb0 = scatter_bits(tc_compose_bat(p.ga, p.lbat, nonb, be0), p.pos_bat, p.lbat) + mbase;
                if (be1 >= 0) cb1 = scatter_bits(tc_compose_bat(p.ga, p.lbat, nonb, be1), p.pos_bat, p.lbat) + mbase;
            }
            if (!mbar_wait(smem_u32(&acc_full[b]), (uint32_t)((it >> 1) & 1), abort_flag, kLimit)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t lane_addr = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(b * 2 * BN);
            for (int c0 = c_begin; c0 < c_end; c0 += 16) {
                float re[16], im[16];
                // stacked: columns [j N, (j + 1) N) belong to the stack's batch j (N >= 32);
                // an empty slot's columns were not computed (warp-uniform skip)
                const bool first = (c0 >> p.ln) == j0;
                const int be = stk ? (first ? be0 : be1) : 0;
                if (be < 0) continue;
                __syncwarp();
                tmem_ld16x2(lane_addr + c0, lane_addr + BN + c0, re, im);
                if (p.ln < 4) {
                    if (!row_ok) continue;
                    // fewer than 16 columns per version: versions folded into N, column by
                    // column (c0 + j is column n of version v)
#pragma unroll
                    for (int j = 0; j < 16; j++) {
                        const long long col = (long long)tn_i * BN + c0 + j;
                        const long long v = vrow + (col >> p.ln), n = col & (N - 1);
                        if (v < p.nver && (p.fold == 2 || col < N)) {
                            void *Cv = static_cast<char *>(p.C) + 8 * v * p.c_plane;
                            const long long off = cbase + scatter_bits(n, p.pos_n, p.ln);
                            const float2 x = make_float2(re[j] * p.out_scale, im[j] * p.out_scale);
                            if (p.out_fmt == OUT_C64) static_cast<float2 *>(Cv)[off] = x;
                            else store_split(Cv, p.c_plane, off, x, p.out_fmt == OUT_SPLIT_FP16);
                        }
                    }
                    continue;
                }
                // 16 columns of one batch and version: column nb + j at hi + lo[j]
                const long long col = (long long)tn_i * BN + c0;
                long long v = vrow, nb = col, hi = cbase;
                if (stk) {
                    hi = first ? cb0 : cb1;
                    nb = c0 & (N - 1);
                } else if (p.fold == 2) {
                    v = col >> p.ln;
                    nb = col & (N - 1);
                }
                tc_store16(p, static_cast<char *>(p.C) + 8 * v * p.c_plane,
                           hi + scatter_bits(nb >> 4, p.pos_n + 4, p.ln - 4), lo, plan, row_ok && nb < N && v < p.nver,
                           re, im);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[b])) : "memory");
        }
    }
    __syncwarp();
    if (*abort_flag && threadIdx.x == 0) {
        atomicExch(p.err, 1);
        // let copies already issued land before the shared memory is released
        for (long long k = 0; k < issued && k < STAGES; k++) {
            const long long slot = issued - 1 - k;
            mbar_drain(smem_u32(&full[slot % STAGES]), (uint32_t)((slot / STAGES) & 1), kLimit);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

}  // namespace tnk
