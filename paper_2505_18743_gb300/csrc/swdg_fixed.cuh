// swdg_fixed.cuh -- block fixed-point arithmetic of the 1D contractions.
//
// GB300 issues one FP64 warp instruction per SM every 16 clocks, and one
// 32 x 32 -> 64-bit integer multiply-add (mad.wide) every 0.55 (measured:
// 64 lanes per clock).  A contraction with a constant table is a sum of
// products of numbers of one size, so it needs no floating point: the values
// of one field on one cell share an exponent (the block's), each is a 61-bit
// integer, and the sum is formed exactly by integer multiply-adds, three per
// term.
//
// Format: value = X 2^(eb - 1022 - FB), |X| <= 2^FB, eb the block's biased
// exponent (the largest IEEE exponent field among its values, so that
// |value| < 2^(eb - 1022)).  X = hi 2^LB + lo with lo in [-2^(LB-1), 2^(LB-1)):
// the digit pair that the multiply-adds take.  Tables are held the same way,
// T = Tint 2^(tb - FB), where 2^tb bounds every row's sum of |T|, so a
// contraction of |X| <= 2^FB gives |X| <= 2^FB again, with exponent eb + tb.
// A block far below its bound may be moved up within it (headroom).  What is split
// or multiplied is below 2^60.9 (the digit pair wraps from 2^61 - 2^29 on).
//
// Rounding: a conversion rounds at 2^-60 of the block's largest value, a
// contraction leaves out lo lo (at most a quarter of a unit of 2^-60 per term)
// and rounds the table to 2^-61 of its row bound: together about a unit of
// 2^-60 of the bound of the result, against 2^-53 of each partial sum in FP64
// arithmetic (the row bounds of two or four contractions in a row exceed the
// values by a few bits, so the room is used).  What this gives up is the relative
// accuracy of a value far below the largest of its block: no loss in a sum that
// the large value is part of, but one in a sum that leaves it out.  So a block
// holds only values that meet in the same sums (the pixels' land, which no sum
// takes, is kept out of theirs).
//
// Room: the sums hold up to 13 terms (hi Tlo and lo Thi are below 2^59 each).  Two
// sums of the residual take a second table at the first one's scale: |X| <= 1.75
// 2^FB there, which the joint rows are checked for where the tables are built.
//
// A block that holds an infinity or a NaN takes the exponent POISON; every
// value converted back from it is NaN.  Values below 2^-1018 are zero.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace swdg {
namespace fx {

constexpr int FB = 60;
constexpr int LB = 30;
constexpr int EMIN = 5;        // smallest block exponent: values below 2^(EMIN - 1023) read as 0
constexpr int POISON = 4096;   // block exponent of a block with an infinity or a NaN
constexpr int POISON_MIN = 3072; // any exponent derived from POISON by table exponents is above

__host__ __device__ __forceinline__ int clz64(unsigned long long a) {
#ifdef __CUDA_ARCH__
    const unsigned h = (unsigned)(a >> 32);
    return h ? __clz((int)h) : 32 + __clz((int)(unsigned)a);
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}
__host__ __device__ __forceinline__ unsigned long long dbits(double v) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long b;
    __builtin_memcpy(&b, &v, 8);
    return b;
#endif
}
__host__ __device__ __forceinline__ double bitsd(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    __builtin_memcpy(&v, &b, 8);
    return v;
#endif
}
__host__ __device__ __forceinline__ unsigned fbits(float v) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(v);
#else
    unsigned b;
    __builtin_memcpy(&b, &v, 4);
    return b;
#endif
}
__host__ __device__ __forceinline__ float bitsf(unsigned b) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float v;
    __builtin_memcpy(&v, &b, 4);
    return v;
#endif
}

__host__ __device__ __forceinline__ long long to_int(double v) { // |v| < 2^62, to nearest
#ifdef __CUDA_ARCH__
    return __double2ll_rn(v);
#else
    return (long long)__builtin_rint(v);
#endif
}
// digit pair {hi, lo} of X, |X| < 2^60.9
__host__ __device__ __forceinline__ int2 split(long long X) {
    int2 d;
    d.y = (int)((unsigned)X << (32 - LB)) >> (32 - LB);
    d.x = (int)((X + (1ll << (LB - 1))) >> LB);
    return d;
}
__host__ __device__ __forceinline__ long long join(int2 d) {
    return (long long)d.x * (1ll << LB) + d.y;
}

// exact sum of table x value products, without lo x lo
struct Acc {
    long long a1, a2, a3; // a3 apart from a2: two chains of dependent additions
    // a2 starts at half a unit of the final shift (round to nearest)
    __host__ __device__ __forceinline__ Acc() : a1(0), a2(1ll << (FB - LB - 1)), a3(0) {}
    __host__ __device__ __forceinline__ void mac(int2 t, int2 v) {
        a1 += (long long)t.x * v.x;
        a2 += (long long)t.x * v.y;
        a3 += (long long)t.y * v.x;
    }
    __host__ __device__ __forceinline__ long long get() const { // X: (a1 2^(2 LB) + (a2 + a3) 2^LB) 2^-FB
        return (a1 << (2 * LB - FB)) + ((a2 + a3) >> (FB - LB));
    }
};
static_assert(2 * LB >= FB, "scale of a1");

// the exponent that a double contributes to its block's (from its high word),
// and the block's exponent from the largest of them
__host__ __device__ __forceinline__ unsigned mag(double v) {
    return (unsigned)(dbits(v) >> 32) & 0x7fffffffu;
}
__host__ __device__ __forceinline__ int block_exp(unsigned maxmag) {
    const int e = (int)(maxmag >> 20);
    return e == 0x7ff ? POISON : (e < EMIN ? EMIN : e);
}
// X of v in a block of exponent eb, rounded to nearest, and the value of X,
// rounded to nearest (below the normal range 0, above it infinity).  Each is one
// conversion instruction with the exponent moved by integer additions: 17 clocks
// of the FP64 pipe, against 16 and 38 integer instructions.  The kernels' hot
// code exceeds the 32 KB that the instruction cache holds, so its size decides
// (while the FP64 pipe was the bound, the integer forms were 10 % faster).
__host__ __device__ __forceinline__ long long from_double(double v, int eb) {
    const unsigned long long b = dbits(v);
    const int s = FB + 1022 - eb;
    const int least = s > 1 - EMIN ? EMIN - 1 : -s; // below the block's last place (or poisoned)
    if (((int)(b >> 52) & 0x7ff) <= least) return 0;
    return to_int(bitsd(b + ((unsigned long long)(long long)s << 52)));
}
// to_double at the ends of the exponent range (rare; not inlined: the callers'
// code stays small)
__host__ __device__ __noinline__ inline double out_of_range(long long X, int eb) {
    if (eb >= POISON_MIN) return bitsd(0x7ff8000000000000ull);
    const unsigned long long b = dbits((double)X);
    const int E = ((int)(b >> 52) & 0x7ff) + eb - (FB + 1022);
    if (X == 0 || E <= 0) return 0.0;
    if (E >= 2047) return bitsd((b & 0x8000000000000000ull) | 0x7ff0000000000000ull);
    return bitsd(b + ((unsigned long long)(long long)(eb - (FB + 1022)) << 52));
}
__host__ __device__ __forceinline__ double to_double(long long X, int eb) {
    if ((unsigned)(eb - 128) >= 1792u) return out_of_range(X, eb);
    const unsigned long long b = dbits((double)X);
    return bitsd(X == 0 ? 0ull : b + ((unsigned long long)(long long)(eb - (FB + 1022)) << 52));
}
// how far a block moves up, m = the largest high word of its |X|, for |X| < 2^FB
// (|X| = 2^FB itself stays)
__host__ __device__ __forceinline__ int headroom(unsigned m) {
    const int s = clz64((unsigned long long)m << 32 | 0xffffffffu) - (64 - FB);
    return s < 0 ? 0 : s;
}
// high word of |X|
__host__ __device__ __forceinline__ unsigned high(long long X) {
    return (unsigned)((unsigned long long)(X < 0 ? -X : X) >> 32);
}
// product of two block values: X of exponent product_exp(e1, e2)
__host__ __device__ __forceinline__ long long product(int2 a, int2 b) {
    Acc s;
    s.mac(a, b);
    return s.get();
}
__host__ __device__ __forceinline__ int product_exp(int e1, int e2) { return e1 + e2 - 1022; }

// the same for FP32 values: the block exponent (in the double's bias) from the
// largest bit pattern of the magnitudes, X of a value, the value of an X
// (FP32 subnormals count as zero)
__host__ __device__ __forceinline__ int block_exp_f(unsigned maxbits) {
    const int e = (int)(maxbits >> 23);
    return e == 0xff ? POISON : e + 896;
}
__host__ __device__ __forceinline__ long long from_float(float v, int eb) {
    const unsigned b = fbits(v);
    const int ef = (int)(b >> 23) & 0xff;
    unsigned d = (unsigned)(eb - (ef + 896));
    d = ef == 0 ? 63u : (d < 63u ? d : 63u);
    const unsigned long long m = (unsigned long long)((b & 0x7fffffu) | 0x800000u) << (FB - 24);
    const long long X = (long long)((m + ((1ull << d) >> 1)) >> d); // to nearest
    return (int)b < 0 ? -X : X;
}
__host__ __device__ __forceinline__ float to_float(long long X, int eb) {
    const unsigned long long a = (unsigned long long)(X < 0 ? -X : X);
    const int lz = clz64(a);
    const unsigned long long m = a << (lz & 63);
    const int E = eb + (64 - FB) - lz - 896;
    unsigned r = ((unsigned)(E - 1) << 23) + (unsigned)(m >> 40) + ((unsigned)(m >> 39) & 1u);
    if (a == 0 || E <= 0) r = 0u;
    if (E >= 255) r = 0x7f800000u;
    if (eb >= POISON_MIN) r = 0x7fc00000u;
    return bitsf(r | ((unsigned)((unsigned long long)X >> 32) & 0x80000000u));
}

} // namespace fx
} // namespace swdg
