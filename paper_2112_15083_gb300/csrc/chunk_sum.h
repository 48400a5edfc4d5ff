// The FP64 sum of FP32 values, 16 at a time: what the slice sum of a contraction adds up.
// Host and device code share this header (the CPU tests run it on the host).
//
// The GPU's FP64 pipe takes 2 lanes per clock and SM, so one addition per value bounds the sum
// (2^20 outputs of 1024 complex values: 4.1 ms, 2.1 TB/s).  Here 16 values are first added in
// FP32 without loss, split at powers of two (e: exponent of the largest |x|):
// hi = (s + x) - s with s = 1.5 * 2^(e + 4) is a multiple of 2^(e - 19), so the 16 hi parts
// add exactly; lo = x - hi is at most 2^(e - 20), and the lo parts add exactly if the smallest
// |x| is within 2^17 of the largest.  The chunk's sum is then two FP32 sums, exact in FP64, and
// takes one rounding to join the running sum.
//
// Otherwise (a gate entry such as cos(pi / 2) = 6e-17 makes terms 2^-54 of the others) lo is
// split 20 bits lower, and what is left twice more, from its own largest value down: four exact
// FP32 sums, the two upper ones joined into one FP64 value, the two lower ones into another.
// Each has a running sum of its own (acc, low) and is added where the exponents show that
// neither addition rounds.  Where one might, or the values reach further down than the splits,
// acc and low are joined and the chunk is added one value after the other.  So a chunk is added
// exactly, or with one rounding, or with those of the plain sum; and where FP64 additions one
// by one would not round at all, cancellation included, the result is theirs.  Values that FP32
// cannot split (infinite, NaN, or a largest one outside 2^-80 .. 2^100) are added one by one.
//
// With what is left of lo added in rounded FP32 instead, ahead of the larger parts, a small
// residual of values that cancel was lost; 20 qubits in split bf16, whose chunks all take the
// four splits, took 206 us a call so and take 215 us now; 24 qubits in split fp16 880 and 868 us.
#pragma once

#include <math.h>
#include <string.h>

#include "widen.h"

#ifdef __CUDACC__
#define TN_HD_MEMBER __host__ __device__ __forceinline__
#else
#define TN_HD_MEMBER inline
#endif

namespace tnk {

TN_HD uint32_t float_bits(float x) {
    uint32_t u;
    memcpy(&u, &x, 4);
    return u;
}
TN_HD float bits_float(uint32_t u) {
    float x;
    memcpy(&x, &u, 4);
    return x;
}
TN_HD uint64_t double_bits(double x) {
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
}
TN_HD double chunk_widen(float x) {
#ifdef __CUDA_ARCH__
    return tn_widen(x);
#else
    return (double)x;
#endif
}

// Biased exponent of a double.
TN_HD int exponent_of(double x) { return (int)((double_bits(x) >> 52) & 2047u); }
// Zeros are told by their bits: a comparison would go to the FP64 pipe.  None here is -0.
TN_HD bool not_zero(double x) { return double_bits(x) != 0; }
TN_HD int min_of(int a, int b) { return a < b ? a : b; }

struct ChunkSum {
    double acc = 0.0, low = 0.0;          // the sum is acc + low
    int acc_bit = 4096, low_bit = 4096;   // biased exponents that no set bit of theirs lies below
    TN_HD_MEMBER double total() const { return not_zero(low) ? acc + low : acc; }
    TN_HD_MEMBER void join() {
        acc = total();
        low = 0.0;
        acc_bit = min_of(acc_bit, low_bit);
        low_bit = 4096;
    }
    // 1.5 * 2^e for a biased e
    static TN_HD_MEMBER float split_at(int e) { return bits_float(((uint32_t)e << 23) | 0x400000u); }
    TN_HD_MEMBER void add16(const float (&x)[16]) {
        float mx = 0.f;
        uint32_t mn = 0xffffffffu;  // smallest 2 |bits| - 1: zeros, which add nothing, come last
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const uint32_t u = 2u * float_bits(x[i]) - 1u;
            mx = fmaxf(mx, fabsf(x[i]));
            mn = u < mn ? u : mn;
        }
        if (mn == 0xffffffffu) return;  // all zero
        // biased by 127; en is the exponent of the smallest value, or one less
        const int ex = (int)(float_bits(mx) >> 23), en = (int)(mn >> 24);
        const int bit = en - 23 + 1023 - 127;  // of the values' lowest bits, as a double's exponent
        const float s1 = split_at(ex + 4);
        float sh = 0.f, sl = 0.f;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            const float hi = (s1 + x[i]) - s1;
            sl += x[i] - hi;
            sh += hi;
        }
        bool plain = !(ex >= 47 && ex <= 227 && sh == sh);
        double lower = 0.0;
        int upper_bit = bit;
        if (!plain && ex - en > 17) {
            // sl: the values' next 20 bits; r: what is left of them
            const float s2 = split_at(ex - 16);
            float r[16], ml = 0.f;
            sl = 0.f;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const float lo = x[i] - ((s1 + x[i]) - s1), h = (s2 + lo) - s2;
                sl += h;
                r[i] = lo - h;
                ml = fmaxf(ml, fabsf(r[i]));
            }
            const int el = (int)(float_bits(ml) >> 23);
            plain = ml > 0.f && (el < 24 || el - en > 17);
            const float s3 = split_at(el + 4);
            float rh = 0.f, rl = 0.f;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const float h = (s3 + r[i]) - s3;
                rl += r[i] - h;
                rh += h;
            }
            lower = chunk_widen(rh) + chunk_widen(rl);
            upper_bit = ex - 39 + 1023 - 127;
        }
        const double upper = chunk_widen(sh) + chunk_widen(sl);
        if (!plain && (not_zero(lower) || not_zero(low))) {
            // an addition is exact if the 53 bits of its result reach down to both lowest bits
            const double a = acc + upper, l = low + lower;
            const int ab = min_of(acc_bit, upper_bit), lb = min_of(low_bit, bit);
            if (exponent_of(a) - 52 <= ab && exponent_of(l) - 52 <= lb) {
                acc = a;
                low = l;
                acc_bit = ab;
                low_bit = lb;
                return;
            }
            join();
            plain = not_zero(lower);
        }
        if (plain) {
            join();
#pragma unroll
            for (int i = 0; i < 16; i++) acc += chunk_widen(x[i]);
        } else {
            acc += upper;
        }
        acc_bit = min_of(acc_bit, bit);
    }
};

}  // namespace tnk
