// sf_arith.cuh -- 64-bit modular arithmetic for moduli q < 2^51.
//
// Residues live in uint64 words.  Three published reductions are used:
//  * Shoup (1996) / Harvey (2014) multiplication by a fixed operand w with the
//    precomputed companion w' = floor(w * 2^64 / q): for any x < 2^64,
//    x*w - floor(x*w'/2^64)*q lies in [0, 2q).
//  * Montgomery (1985) REDC with R = 2^64 for products of two variable
//    residues: for T < q*2^64, (T + m q)/2^64 with m = T * (-q^-1) mod 2^64
//    lies in [0, 2q) and equals T * 2^-64 mod q.
// The lazy products and butterflies of the transforms are in sf_reg.cuh.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define SF_HD __host__ __device__ __forceinline__
#else
#define SF_HD inline
#endif

typedef uint64_t u64;

SF_HD u64 sf_mulhi(u64 a, u64 b)
{
#if defined(__CUDA_ARCH__)
    return __umul64hi(a, b);
#else
    return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}

// x*w mod q in [0, 2q) for any x < 2^64; w < q, wp = floor(w 2^64 / q).
SF_HD u64 sf_mul_shoup_lazy(u64 x, u64 w, u64 wp, u64 q)
{
    u64 qhat = sf_mulhi(x, wp);
    return x * w - qhat * q;
}

SF_HD u64 sf_mul_shoup(u64 x, u64 w, u64 wp, u64 q)
{
    u64 r = sf_mul_shoup_lazy(x, w, wp, q);
    return r >= q ? r - q : r;
}

SF_HD u64 sf_csub(u64 x, u64 q) { return x >= q ? x - q : x; }

SF_HD u64 sf_add(u64 a, u64 b, u64 q) { return sf_csub(a + b, q); }

SF_HD u64 sf_sub(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// Montgomery REDC: returns T * 2^-64 mod q in [0, 2q) for T = hi*2^64 + lo < q*2^64.
// qinv_neg = -q^-1 mod 2^64.
SF_HD u64 sf_redc_lazy(u64 hi, u64 lo, u64 q, u64 qinv_neg)
{
    u64 m = lo * qinv_neg;
    u64 mq_hi = sf_mulhi(m, q);
    // lo + (m*q mod 2^64) == 0 mod 2^64, with a carry out exactly when lo != 0
    return hi + mq_hi + (lo != 0 ? 1 : 0);
}

SF_HD u64 sf_redc(u64 hi, u64 lo, u64 q, u64 qinv_neg)
{
    return sf_csub(sf_redc_lazy(hi, lo, q, qinv_neg), q);
}

// a * b_mont * 2^-64 mod q: with b_mont = b * 2^64 mod q this is a*b mod q.
SF_HD u64 sf_mul_mont(u64 a, u64 b_mont, u64 q, u64 qinv_neg)
{
    return sf_redc(sf_mulhi(a, b_mont), a * b_mont, q, qinv_neg);
}

// High 64 bits of a*b from three of the four 32 x 32-bit partial products:
// the low x low product and the carries out of the two cross products are
// dropped, so the result is the exact high part minus 0, 1 or 2.
SF_HD u64 sf_mulhi_trunc(u64 a, u64 b)
{
#if defined(__CUDA_ARCH__)
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    return (u64)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
#else
    const u64 al = (uint32_t)a, ah = a >> 32, bl = (uint32_t)b, bh = b >> 32;
    return ah * bh + ((ah * bl) >> 32) + ((al * bh) >> 32);
#endif
}

// Reduce any x < 2^64 to [0, q): Shoup multiplication by 1 (one_p =
// floor(2^64 / q)) lands in [0, 2q), then one conditional subtraction.
SF_HD u64 sf_reduce(u64 x, u64 q, u64 one_p)
{
    return sf_csub(x - sf_mulhi(x, one_p) * q, q);
}
