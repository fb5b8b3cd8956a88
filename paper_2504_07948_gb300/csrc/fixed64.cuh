// FP64 dot products on the integer pipe.
//
// GB300 issues one FP64 instruction per 16 SM cycles and a 32 x 32 + 64 bit
// integer multiply-add (IMAD.WIDE) per cycle (measured: 15.7 and 1.06 cycles
// per warp instruction), so a dot product of doubles is cheaper in fixed
// point: each operand row is scaled by its own power of two to integers of
// at most kFxQ = 57 bits, held as two signed limbs of 29 bits, and
//   sum_k a_k b_k = 2^58 sum hi hi + 2^29 sum (hi lo + lo hi) (+ sum lo lo)
// takes three multiply-adds per term, exact in 64 bits for kFxBlock = 32
// terms (|hi|, |lo| <= 2^28).  The lo lo terms (below 2^-58 of the product of
// the two row maxima per term) are dropped: against the exact value a dot
// product of k terms is off by about sqrt(k) 2^-59 of max|a| max|b|, where
// an FP64 chain is off by some sqrt(k) 2^-54 of its partial sums.  So it is the
// better of the two where the sum's terms come near the product of the maxima, and
// the worse where they lie far below it: its users compare the two (kFxSlack).
// On water clusters of 1 to 14 waters E_L and the ionic derivatives from these
// products are 20 to 40 % closer to extended precision than from FP64 chains,
// in the mean over walkers as over the worst of them.  This is the splitting
// of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012) with integer
// digits.  Non-finite rows give NaN (fx_scale); rows below 2^-994 count as
// zero.
#pragma once

#include <cuda_runtime.h>
#include <string.h>

namespace qmc {

constexpr int kFxQ = 57;
constexpr int kFxLimb = 29;
constexpr int kFxBlock = 32;

// Bits by which the product of two rows' largest entries may exceed the largest
// product of their entries before a fixed-point dot product of them gives way to
// FP64: its error is some 2^-59 sqrt(k) of the former, that of an FP64 chain some
// 2^-54 sqrt(k) of the latter (k_wavefunction.cu, sweep64.cuh, k_force.cu).
constexpr int kFxSlack = 6;

// Biased exponent of x (2047: infinity or NaN).
__host__ __device__ __forceinline__ long long fx_bits(double x) {
    long long b;
    memcpy(&b, &x, sizeof(b));
    return b;
}
__host__ __device__ __forceinline__ double fx_double(long long b) {
    double x;
    memcpy(&x, &b, sizeof(x));
    return x;
}
__host__ __device__ __forceinline__ int fx_expo(double x) { return (int)((fx_bits(x) >> 52) & 0x7ff); }

// Limbs (x: high, y: low) of v in a row whose largest exponent is emax.
__host__ __device__ __forceinline__ int2 fx_limbs(double v, int emax) {
    const long long b = fx_bits(v);
    const int e = (int)((b >> 52) & 0x7ff);
    const long long m = e ? ((b & 0xfffffffffffffLL) | (1LL << 52)) : 0;   // |v| = m 2^(e - 1075)
    const int sh = e - emax + (kFxQ - 53);
    long long q = sh >= 0 ? m << sh : sh > -54 ? (m + (1LL << (-sh - 1))) >> -sh : 0;
    if (b < 0) q = -q;
    const int lo = ((int)(q & ((1 << kFxLimb) - 1)) ^ (1 << (kFxLimb - 1))) - (1 << (kFxLimb - 1));
    return make_int2((int)((q - lo) >> kFxLimb), lo);
}

// Power of two of a row: the product of two rows' scales turns the integer
// sum of FxDot into the dot product.
__host__ __device__ __forceinline__ double fx_scale(int emax) {
    if (emax >= 2047) return fx_double(0x7ff8000000000000LL);
    return emax >= 28 ? fx_double((long long)(emax - 27) << 52) : 0.0;
}

// Accumulator of one dot product.  add() at most kFxBlock times between
// calls of fold(); at most 2^30 folds.
struct FxDot {
    long long hh = 0, mid = 0;
    __device__ __forceinline__ void add(int2 a, int2 b) {
        hh += (long long)a.x * b.x;
        mid += (long long)a.x * b.y;
        mid += (long long)a.y * b.x;
    }
};

// Sum of blocks, exact (the order of the terms does not matter): units of
// 2^58 split in 32-bit halves, and the part below.
struct FxSum {
    long long hi = 0, lo = 0, rem = 0;
    __device__ __forceinline__ void fold(FxDot& d) {
        const long long v = d.hh + (d.mid >> kFxLimb);   // below 2^62 in magnitude
        hi += v >> 32;
        lo += v & 0xffffffffLL;
        rem += d.mid & ((1LL << kFxLimb) - 1);
        d.hh = 0;
        d.mid = 0;
    }
    __device__ __forceinline__ double value() const {
        const long long t = lo + ((rem + (1LL << (kFxLimb - 1))) >> kFxLimb);
        const long long h = hi + (t >> 32), l = t & 0xffffffffLL;
        if (h == (long long)(int)h) return (double)(long long)(((unsigned long long)h << 32) | (unsigned long long)l);
        return (double)h * 4294967296.0 + (double)l;
    }
};

__device__ __forceinline__ int warp_max_u(int v) { return (int)__reduce_max_sync(0xffffffffu, (unsigned)v); }

}  // namespace qmc
