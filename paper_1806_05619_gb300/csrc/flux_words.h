// The refinement residual r = 1 - c sum_f k_f (u_P - u_f) of one cell (FP32
// faces, FP64 values) in three FP32 words per number, on host and device.
//
// A difference d of two FP64 values has 53 bits: 24 + 24 + 5. Its product with
// a face is two error-free FP32 products (each product and its error by one
// FMA) and a last one whose rounding is 2^-72 of the flux; the four fluxes and
// the scaling by c keep every rounding error of the first two words by TwoSum
// and add only third words in plain FP32. What is left beyond the rounding of
// the differences themselves, which the FP64 form has too, is below 2^-62 of
// c sum_f |k_f d_f|, where the FP64 form's own products and sums leave up to
// 2^-51; the value that comes back is rounded to 2^-46 of itself.
#pragma once

#include <cstdint>
#include <cstring>
#ifndef __CUDACC__
#include <cmath>
#define MLQMC_WORDS inline
#else
#define MLQMC_WORDS __host__ __device__ __forceinline__
#endif

namespace mlqmc_words {

// One rounding each, never contracted (host code that uses them is compiled with -ffp-contract=off).
#ifdef __CUDA_ARCH__
MLQMC_WORDS float add(float a, float b) { return __fadd_rn(a, b); }
MLQMC_WORDS float sub(float a, float b) { return __fsub_rn(a, b); }
MLQMC_WORDS float mul(float a, float b) { return __fmul_rn(a, b); }
MLQMC_WORDS float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
MLQMC_WORDS uint32_t hi_word(double d) { return static_cast<uint32_t>(__double2hiint(d)); }
MLQMC_WORDS uint32_t lo_word(double d) { return static_cast<uint32_t>(__double2loint(d)); }
MLQMC_WORDS float as_float(uint32_t b) { return __uint_as_float(b); }
MLQMC_WORDS uint32_t as_bits(float f) { return __float_as_uint(f); }
#else
MLQMC_WORDS float add(float a, float b) { return a + b; }
MLQMC_WORDS float sub(float a, float b) { return a - b; }
MLQMC_WORDS float mul(float a, float b) { return a * b; }
MLQMC_WORDS float fma_rn(float a, float b, float c) { return fmaf(a, b, c); }
MLQMC_WORDS uint64_t bits_of(double d)
{
    uint64_t b;
    memcpy(&b, &d, 8);
    return b;
}
MLQMC_WORDS uint32_t hi_word(double d) { return static_cast<uint32_t>(bits_of(d) >> 32); }
MLQMC_WORDS uint32_t lo_word(double d) { return static_cast<uint32_t>(bits_of(d)); }
MLQMC_WORDS float as_float(uint32_t b)
{
    float f;
    memcpy(&f, &b, 4);
    return f;
}
MLQMC_WORDS uint32_t as_bits(float f)
{
    uint32_t b;
    memcpy(&b, &f, 4);
    return b;
}
#endif

// a + b = s + e (Knuth)
MLQMC_WORDS void two_sum(float a, float b, float& s, float& e)
{
    s = add(a, b);
    const float bb = sub(s, a);
    e = add(sub(a, sub(s, bb)), sub(b, bb));
}

struct Words {
    float h, m, l;  // h + m + l
};

// By the conversion instructions: magnitudes below 2^-74 or from 2^128 on, infinities, NaN.
#ifdef __CUDACC__
static __host__ __device__ __noinline__ Words split_rare(double d)
#else
static Words split_rare(double d)
#endif
{
    Words w = {static_cast<float>(d), 0.0f, 0.0f};
    if (w.h - w.h != 0.0f) return w;
    const double r = d - static_cast<double>(w.h);
    w.m = static_cast<float>(r);
    w.l = static_cast<float>(r - static_cast<double>(w.m));
    return w;
}

// d = h + m + l exactly, for magnitudes from 2^-74 to 2^128 by bit operations:
// the 29 significand bits below FP32's are rounded off h (half up), as a signed
// number; its last five are rounded off m in the same way and make up l.
MLQMC_WORDS Words split(double d)
{
    const uint32_t hi = hi_word(d), lo = lo_word(d);
    const uint32_t e = (hi >> 20) & 0x7FFu;
    if (e - 949u > 201u) {
        if (((hi << 1) | lo) == 0u) return Words{0.0f, 0.0f, 0.0f};
        return split_rare(d);
    }
    const uint32_t sgn = hi & 0x80000000u;
    const uint64_t r = ((static_cast<uint64_t>(hi) << 32) | lo) + 0x10000000ull;
    const uint32_t mag = static_cast<uint32_t>(r >> 29) - 0xC0000000u;
    const int low = static_cast<int>(static_cast<uint32_t>(r) & 0x1FFFFFFFu) - 0x10000000;
    const int mid = (low + 16) & ~31;  // |mid| <= 2^28 in steps of 32: an FP32 number
    const float unit = as_float(((e - 948u) << 23) | sgn);  // the last bit of d, with d's sign
    Words w;
    w.h = as_float((mag & 0x7FFFFFFFu) | sgn);
    w.m = mul(static_cast<float>(mid), unit);
    // |low - mid| <= 16 as a float: the integer added to the bits of 1.5 x 2^23
    w.l = mul(sub(as_float(0x4B400000u + static_cast<uint32_t>(low - mid)), 12582912.0f), unit);
    return w;
}

// k (a - b)
MLQMC_WORDS Words flux(float k, double a, double b)
{
    const Words d = split(a - b);
    Words f;
    f.h = mul(k, d.h);
    const float p = mul(k, d.m);
    float g;
    two_sum(fma_rn(k, d.h, -f.h), p, f.m, g);
    f.l = fma_rn(k, d.l, add(fma_rn(k, d.m, -p), g));
    return f;
}

// r = 1 - c (west - east + south - north) = b + rem, b rounded to FP32.
MLQMC_WORDS void residual(float c, const Words& w, const Words& e, const Words& s, const Words& n, float& b, float& rem)
{
    // in pairs, not one after the other: the chains are what a warp waits for
    float h1, h2, h, x1, x2, x3, m1, m2, m3, m4, m5, m, t1, t2, t3, t4, t5, t6;
    two_sum(w.h, -e.h, h1, x1);
    two_sum(s.h, -n.h, h2, x2);
    two_sum(h1, h2, h, x3);
    two_sum(w.m, -e.m, m1, t1);
    two_sum(s.m, -n.m, m2, t2);
    two_sum(m1, m2, m3, t3);
    two_sum(x1, x2, m4, t4);
    two_sum(m4, x3, m5, t5);
    two_sum(m3, m5, m, t6);
    const float l = add(add(add(sub(w.l, e.l), sub(s.l, n.l)), add(t1, t2)), add(add(t3, t4), add(t5, t6)));
    // 1 - c (h + m + l)
    const float ah = mul(c, h), bh = mul(c, m);
    float x, y, z, tx, tz;
    two_sum(1.0f, -ah, x, y);
    two_sum(fma_rn(c, h, -ah), bh, z, tz);
    two_sum(x, -z, x, tx);
    const float tail = fma_rn(c, l, add(fma_rn(c, m, -bh), tz));
    two_sum(x, sub(add(y, tx), tail), b, rem);
}

}  // namespace mlqmc_words
