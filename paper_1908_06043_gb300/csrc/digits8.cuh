// Seven balanced 8-bit digits of an FP64 value as FP16 MMA operands, and the sum of the seven
// accumulators of their products, in integer instructions: FP64 instructions and conversions run at
// 2 a clock and SM on this GPU.
//
// Cutting.  With |x| < 2^E, y = round(x 2^(55 - E)) has x = 2^(E - 7) sum_p q_p 2^(-8p) with the
// balanced digits q_0 .. q_6, |q_p| <= 128.  y + 0x80..80 has the digits, biased by 128, as its bytes;
// a byte u is the FP16 number (0x6400 | u) - 1152: one byte permutation, one logic operation and
// one packed subtraction for two digits.
// Summing.  a_d is the sum of the digit products p + q = d over 64 terms, |a_d| <= (d + 1) 2^20.  The
// product is (a_0 2^48 + .. + a_5 2^8 + a_6) 2^(E_a + E_b - 62); it is formed as one 64-bit integer T in
// units of 2^(E_a + E_b - 56), kTUnit, and packed into an FP64 by shifts.  (Units of 2^-52, which is
// where the dropped products p + q > 6 lie, already cost a factorisation near an eigenvalue a
// factor of two in accuracy.)
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "tc_ptx.cuh"

namespace sstc {

constexpr int kFtSlices = 7;
constexpr int kTUnit = 56;                          // T counts 2^(E_a + E_b - kTUnit)
constexpr int kFtNan = 1 << 20;                     // "exponent" of a non-finite value
constexpr int kFtZero = -(1 << 20);                 // "exponent" of zero

// biased exponent of v plus sh (1 plus sh for a denormal, whose leading bit is not implicit); kFtZero for
// zero, kFtNan
__device__ __forceinline__ int ft_exp(double v, int sh) {
    const uint32_t lo = (uint32_t)__double2loint(v), hi = (uint32_t)__double2hiint(v) & 0x7fffffffu;
    const int ex = (int)(hi >> 20), e = (hi | lo) == 0 ? kFtZero : max(ex, 1) + sh;
    return ex == 0x7ff ? kFtNan : e;
}

// round(x 2^(55 - E)) + 0x80808080808080 for |x| < 2^E; em = E + 1022 >= ex, the exponents as from
// ft_exp
__device__ __forceinline__ unsigned long long ft_biased(double v, int ex, int em) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const uint32_t hi = (uint32_t)(bits >> 32);
    const uint32_t mh = (hi & 0xfffffu) | ((hi & 0x7ff00000u) != 0 ? 0x100000u : 0u);     // 0 for zero
    unsigned long long m = ((unsigned long long)mh << 32) | (uint32_t)bits;
    m = (((m << 3) >> min(em - ex, 60)) + 1) >> 1;  // 4 m 2^(ex - em), rounded
    const unsigned long long s = (unsigned long long)((long long)bits >> 63);
    return ((m ^ s) - s) + 0x80808080808080ull;
}

// the 7 digits of 8 values (biased as above) as FP16, 16 bytes to each slice
__device__ __forceinline__ void ft_store8(const unsigned long long (&z)[8], unsigned char *dst, uint32_t stride) {
    const __half2 bias = __half2half2(__ushort_as_half((unsigned short)0x6480));    // 1152
#pragma unroll
    for (int p = 0; p < kFtSlices; ++p) {
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const unsigned long long z0 = z[2 * e], z1 = z[2 * e + 1];
            uint32_t h;
            if (p == 0) {                           // the top digit is 0 .. 256: both bytes
                h = __byte_perm((uint32_t)(z0 >> 32), (uint32_t)(z1 >> 32), 0x7632) | 0x64006400u;
            } else {
                const int byte = 6 - p;             // of the 8 bytes of z
                const uint32_t w0 = (uint32_t)(byte >= 4 ? z0 >> 32 : z0), w1 = (uint32_t)(byte >= 4 ? z1 >> 32 : z1);
                const uint32_t b = byte & 3;
                h = (__byte_perm(w0, w1, b | (b << 4) | ((4 + b) << 8) | ((4 + b) << 12)) & 0x00ff00ffu) | 0x64006400u;
            }
            const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&h), bias);
            o[e] = *reinterpret_cast<const uint32_t *>(&d);
        }
        *reinterpret_cast<uint4 *>(dst + p * stride) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// 16 columns of one accumulator; the values are there after ft_tmem_wait on the same registers
__device__ __forceinline__ void ft_tmem_ld(uint32_t t, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(t)
        : "memory");
}
__device__ __forceinline__ void ft_tmem_wait(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// integer-valued |a| <= 2^22 plus 0x4B400000 as an integer: the bits of a + 1.5 2^23
constexpr long long kFtMagic = 0x4B400000ll;
__device__ __forceinline__ long long ft_int22(uint32_t a) {
    return (long long)__float_as_int(__uint_as_float(a) + 12582912.0f);
}
// integer-valued |a| < 2^23 as int
__device__ __forceinline__ int ft_int23(uint32_t a) {
    const int b = (int)a, s = b >> 31;
    const int m = __float_as_int(__uint_as_float(a) + __int_as_float((b & (int)0x80000000) | 0x4B000000)) & 0x7fffff;
    return (m ^ s) - s;
}

// bits of T 2^E, rounded to nearest (ties away), by shifts and an integer addition: no branch, for
// |T| < 2^63 and results in the normal range (or T = 0)
__device__ __forceinline__ unsigned long long ft_pack(long long T, int E) {
    const unsigned long long s = (unsigned long long)(T >> 63);
    unsigned long long u = ((unsigned long long)T ^ s) - s;
    const int lz = __clzll((long long)u);           // 64 for T = 0: u stays 0
    u <<= (lz & 63);
    const unsigned long long bits = ((unsigned long long)(uint32_t)(1023 + 62 - lz + E) << 52) + (u >> 11) + ((u >> 10) & 1);
    return T == 0 ? 0ull : (bits | (s & (1ull << 63)));
}

// T of 16 consecutive columns of the thread's lane, accumulator d at taddr + 64 d:
// T = a_0 2^42 + a_1 2^34 + a_2 2^26 + a_3 2^18 + a_4 2^10 + a_5 2^2 + a_6 2^-6, the last term rounded;
// the magic numbers' share is taken off once
__device__ __forceinline__ void ft_sum(uint32_t taddr, long long (&T)[16]) {
    uint32_t r[16];
    auto load = [&](int d) {
        ft_tmem_ld(taddr + (uint32_t)d * 64, r);
        ft_tmem_wait(r);
    };
    load(6);
#pragma unroll
    for (int e = 0; e < 16; ++e) T[e] = __float_as_int(fmaf(__uint_as_float(r[e]), 1.0f / 64.0f, 12582912.0f));
    load(5);
#pragma unroll
    for (int e = 0; e < 16; ++e) T[e] += (long long)ft_int23(r[e]) * 4;
    load(4);
#pragma unroll
    for (int e = 0; e < 16; ++e) T[e] += (long long)ft_int23(r[e]) * (1 << 10);
    load(3);
#pragma unroll
    for (int e = 0; e < 16; ++e) T[e] += ft_int22(r[e]) * (1 << 18);
    load(2);
#pragma unroll
    for (int e = 0; e < 16; ++e) T[e] += ft_int22(r[e]) * (1 << 26);
    load(1);
#pragma unroll
    for (int e = 0; e < 16; ++e) T[e] += ft_int22(r[e]) << 34;
    load(0);
    constexpr long long kAll =
        (long long)((unsigned long long)kFtMagic * (1ull + (1ull << 18) + (1ull << 26) + (1ull << 34) + (1ull << 42)));
#pragma unroll
    for (int e = 0; e < 16; ++e)
        T[e] = (long long)((unsigned long long)T[e] + ((unsigned long long)ft_int22(r[e]) << 42)) - kAll;
}

}  // namespace sstc
