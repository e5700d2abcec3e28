// Modular arithmetic for primes next to a power of two.
//
// A chain's primes lie next to powers of two: q_0 and the special primes are the largest below theirs,
// the scaling primes the nearest to the scale.  So
//     2^K = e (mod q),   e = 2^K - q,   |e| < 2^26,
// and the part of a number above bit K is brought back ("folded") by one multiplication by a
// 32-bit constant.  hostmath::fold_consts says which primes qualify: 33 to 60 bits but not 57, and |e| small
// enough for one fold to make any value of a transform canonical, which is the tighter bound at 33 to 42 bits
// (|e| below about 2^24.5 at 42 bits, 2^22.7 at 40, 2^18.5 at 36) and lets every |e| < 2^26 through from 43 bits on
// (2^25 at 58).  The chains of the named parameter sets qualify.  A long chain of primes
// at 42 bits or less does not: the primes run away from 2^K (N = 2^16, 24 limbs of 42 bits: 7 of 32
// refused; none at 45 or 48 bits), and one refused prime puts the whole context on Shoup products.  Values are signed 64-bit words that are only congruent to the residue.  A
// product with a constant w is taken as
//     x w = x0 W0 + x1 W1 (mod q),   x = x1 2^32 + x0,  W0 = w,  W1 = w 2^32 mod q,
// with W0, W1 the representatives in [-q/2, q/2] and every low half (x0, the low halves of W0 and
// W1) taken as a signed 32-bit digit.  The sum S of the four 32 x 32 products then needs no
// carries between its partial sums and stays below 2^(K+31), so its part H above bit K is a
// signed 32-bit word, and S = H 2^K + L = L + H e takes one more product: five wide multiplies
// against the six wide and four narrow ones of a Shoup product (10 against 16 lane-cycles of the
// integer-multiply pipe), and about half its instructions with the additions of the butterfly,
// since signed values need no offsets and no comparisons.  The result lies in
//     (-2^31 |e|, 2^K + 2^31 |e|),
// within R = 2^K + 2^31 |e|: a 42- or 48-bit prime (R < 2^57) has room for all sixteen stages
// of a forward transform, a 60-bit prime (R < 1.02 2^60) is folded every four.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FOLD_HD __host__ __device__ __forceinline__
#else
#define FOLD_HD inline
#endif

// constants of one prime (hostmath::fold_consts); all zero when the prime does not qualify
struct FoldMod {
    unsigned kc, mask;   // K - 32, 2^(K-32) - 1
    int e;               // 2^K - q
    unsigned big;        // 60-bit class: values are folded every four stages
    // first fold of a 128-bit sum, at bit K, or at 64 in the 60-bit class: position - 32, the mask of
    // the word that bit lies in, 2^position mod q (nearest to 0)
    unsigned kr, maskr;
    int er;
};

// a b + c, signed 32 x 32 -> 64 (one wide multiply-add)
FOLD_HD int64_t mad_wide(int a, int b, int64_t c) {
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (int64_t)a * b + c;
#endif
}
FOLD_HD int64_t mul_wide(int a, int b) {
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
#else
    return (int64_t)a * b;
#endif
}

// x w (mod q) for a constant packed by hostmath::ntt_pair: w0, w1 hold the signed low digit of W0 / W1
// in their low half and the matching high digit in their high half
FOLD_HD int64_t fold_mul(int64_t x, uint64_t w0, uint64_t w1, const FoldMod& f) {
    const int x0 = (int)x, x1 = (int)(x >> 32) + (int)((unsigned)x >> 31);
    const int64_t a = mad_wide(x1, (int)w1, mul_wide(x0, (int)w0));
    // a's high half is added last: as the addend of the first product it would cost a register move
    const int64_t c = mad_wide(x1, (int)(w1 >> 32), mul_wide(x0, (int)(w0 >> 32))) + (a >> 32);
#ifdef __CUDA_ARCH__
    const int h = (int)__funnelshift_r((unsigned)c, (unsigned)(c >> 32), f.kc);
#else
    const int h = (int)(c >> f.kc);
#endif
    return mad_wide(h, f.e, (int64_t)(((uint64_t)((unsigned)c & f.mask) << 32) | (unsigned)a));
}

// any word folded once: into [0, 2^K) + (v >> K) e
FOLD_HD int64_t fold_word(int64_t v, const FoldMod& f) {
    const int hi = (int)(v >> 32);
    return mad_wide(hi >> f.kc, f.e, (int64_t)(((uint64_t)((unsigned)hi & f.mask) << 32) | (unsigned)v));
}

// the canonical residue of a word whose fold lies in (-q, 2 q)
FOLD_HD uint64_t fold_canon(int64_t v, uint64_t q, const FoldMod& f) {
    int64_t s = fold_word(v, f);
    if (s < 0) s += (int64_t)q;
    const int64_t t = s - (int64_t)q;
    return (uint64_t)(t < 0 ? s : t);
}

#ifdef __CUDACC__
// the canonical residue of hi 2^64 + lo, a sum of at most 40 products of two residues.  With
// s = kr + 32: T = H 2^s + L = L + H e_r (H below 2^62, two signed digits: two wide multiplies) is
// below 2^(K+31), its fold at K within R, and the fold of that canonical up to one q: four wide
// multiplies, against about twenty for a Shoup reduction of each half.
__device__ __forceinline__ unsigned long long fold_128(unsigned long long hi, unsigned long long lo,
                                                       unsigned long long q, const FoldMod& f) {
    const unsigned v1 = (unsigned)(lo >> 32), v2 = (unsigned)hi, v3 = (unsigned)(hi >> 32);
    const unsigned h0 = __funnelshift_rc(v1, v2, f.kr), h1 = __funnelshift_rc(v2, v3, f.kr);
    const int64_t a = mul_wide((int)h0, f.er), b = mul_wide((int)h1 + (int)(h0 >> 31), f.er);
    unsigned t0, t1, t2;
    asm("add.cc.u32  %0, %3, %4;\n\t"
        "addc.cc.u32 %1, %5, %6;\n\t"
        "addc.u32    %2, %7, %8;\n\t"
        "add.cc.u32  %1, %1, %9;\n\t"
        "addc.u32    %2, %2, 0;"
        : "=&r"(t0), "=&r"(t1), "=&r"(t2)
        : "r"((unsigned)lo), "r"((unsigned)a), "r"(v1 & f.maskr), "r"((unsigned)(a >> 32)),
          "r"((unsigned)(a >> 63)), "r"((unsigned)(b >> 32)), "r"((unsigned)b));
    const int h = (int)__funnelshift_r(t1, t2, f.kc);
    return fold_canon(mad_wide(h, f.e, (int64_t)(((uint64_t)(t1 & f.mask) << 32) | t0)), q, f);
}
#endif
