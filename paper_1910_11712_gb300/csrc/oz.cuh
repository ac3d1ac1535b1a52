// FP64 products from 8-bit digits on the tensor core (Ozaki's scheme).
//
// FP64 issues at 1/64 of FP32 on this part, so a contraction is faster as exact integer products:
//   * every row of the left and every column of the right operand is scaled by a power of two to |x| < 1 and
//     rounded to 62 bits, v = sum_t d_t 2^(8t) with d_t in [-128, 127]: the bytes of v + 0x8080808080808080,
//     less 128;
//   * digits are exact in FP16, their products (at most 2^14) and the sums of all products with the
//     same weight 2^(8(ta+tb)) over 128 terms (at most 8 * 128 * 2^14 = 2^24) are exact in FP32, whatever the order
//     in which the tensor core adds them;
//   * the eight weights ta + tb = 14 .. 7 are kept (36 of 64 products) and put together in 64-bit integers;
//     one FP64 addition then rounds once.
// What is dropped: with A and B the powers of two that scale the row and the column, digits of weight 6 and less
// are at most 2^-59.2 A B of a real product and the roundings to 62 bits 2^-62 A B, so n complex terms lose at most
// n 2^-58 A B in each component. The n terms' bound in FP64 is 2 n 2^-53 sum |a||b|, whatever the operands' scales.
// The digits stay within it where sum |a||b| >= 2^-6 A B, which evenly scaled operands meet and
// terms of opposite scale (1e3 against 1e-3) do not. Hence the guard: one more MMA step per 8 terms on the leading 6
// bits of max(|re|, |im|), rounded down, gives sum |a||b| from below as an integer of 2^-12 A B; results
// with less than GUARD of it are summed in FP64.
// Complex operands in real form: rows Re, Im of a row [c.re, -c.im], [c.im, c.re] against columns [y.re; y.im],
// so 64 complex terms fill the 128.
#pragma once
#include "nep_common.cuh"

namespace nep {
namespace oz {
constexpr int S = 8;              // digits
constexpr int CH = 64;            // complex terms per exact accumulation
constexpr int EXP_LO = 623, EXP_HI = 1423;  // exponent fields taken (2^-400 .. 2^400)
constexpr int E_ZERO = EXP_HI + 1;          // stands for the exponent of a row or column of zeros
constexpr float GUARD = 64.0f;              // 2^-6 A B in units of 2^-12 A B

// exponent field of x, 1 for subnormal numbers and 0 for zero alone
__device__ __forceinline__ int exp_field(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) << 1;
    return max((int)(b >> 53), b != 0 ? 1 : 0);
}
__device__ __forceinline__ int exp_field(zd c) { return max(exp_field(c.re), exp_field(c.im)); }

// x as digits + 128 in the bytes of the result, E the exponent field that scales it
__device__ __forceinline__ unsigned long long fixed62(double x, int E) {
    const unsigned long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff, d = E - e;
    unsigned long long v = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 9;
    if (d > 0) v = d < 63 ? (v + (1ull << (d - 1))) >> d : 0ull;
    if (e == 0) v = 0ull;
    if ((long long)b < 0) v = 0ull - v;
    return v + 0x8080808080808080ull;
}
// digit t of two numbers (bytes b.t) as two halves
__device__ __forceinline__ unsigned digits2(unsigned long long a, unsigned long long b, int t) {
    const unsigned wa = t < 4 ? (unsigned)a : (unsigned)(a >> 32), wb = t < 4 ? (unsigned)b : (unsigned)(b >> 32);
    unsigned h = __byte_perm(wa, wb, (t & 3) | ((4 + (t & 3)) << 8));  // bytes 0 and 2
    h = (h & 0x00ff00ffu) | 0x64006400u;                               // 1024 + byte
    unsigned r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0x64806480u));  // - 1152
    return r;
}
// max(|re|, |im|) of c in 64ths of the power of two above the scale E, rounded down (0 .. 63)
__device__ __forceinline__ unsigned lead(zd c, int E) {
    const unsigned h = max((unsigned)__double2hiint(c.re) & 0x7fffffffu, (unsigned)__double2hiint(c.im) & 0x7fffffffu);
    const int d = E - (int)(h >> 20);
    return d < 6 ? ((h & 0xfffffu) | 0x100000u) >> (15 + d) : 0u;
}
// (f, 0) as two halves
__device__ __forceinline__ unsigned lead2(unsigned f) {
    unsigned r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(0x64006400u | f), "r"(0x64006400u));  // 1024 + f - 1024
    return r;
}
// The results that the guard rejects, summed in FP64 by the warp, four at a time with eight lanes each: lane l's
// result is the sum over k < n of (conj of, where cj) pa[(l / 4) ra + k ka] times pb[(l % 4) rb + k kb], for the lanes
// in todo.
__device__ __noinline__ static zd fp64_sums(unsigned todo, int n, const zd* pa, int64_t ra, int64_t ka, bool cj,
                                            const zd* pb, int64_t rb, int64_t kb) {
    const int lane = threadIdx.x & 31;
    zd s = mk(0.0, 0.0);
    while (todo) {
        unsigned m = todo;
        for (int i = lane >> 3; i > 0; --i) m &= m - 1;
        const int l = m ? __ffs(m) - 1 : -1;  // this group's result
        zd t = mk(0.0, 0.0);
        if (l >= 0) {
            const zd *a = pa + (l >> 2) * ra, *b = pb + (l & 3) * rb;
#pragma unroll 4
            for (int k = lane & 7; k < n; k += 8) {
                const zd x = a[k * ka];
                t = fma_(t, cj ? conj(x) : x, b[k * kb]);
            }
        }
        for (int o = 4; o > 0; o >>= 1) {
            t.re += __shfl_xor_sync(0xffffffffu, t.re, o);
            t.im += __shfl_xor_sync(0xffffffffu, t.im, o);
        }
        for (int i = 0; i < 4; ++i) {
            const zd v = mk(__shfl_sync(0xffffffffu, t.re, 8 * i), __shfl_sync(0xffffffffu, t.im, 8 * i));
            if (__shfl_sync(0xffffffffu, l, 8 * i) == lane) s = v;
            todo &= todo - 1;
        }
    }
    return s;
}
__device__ __forceinline__ void mma16816(float (&d)[4], uint4 a, unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
// exact conversion of |h| < 2^51
__device__ __forceinline__ double to_double(long long h) {
    return __longlong_as_double(0x4338000000000000ll + h) - 6755399441055744.0;
}

// the eight level sums of one result, scaled by 2^(ex): E fields ea, eb of its row and column
__device__ __forceinline__ double combine(const float (&D)[S][4], int q, int ea, int eb) {
    long long h = 0, l = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        h = h * 256 + __float2int_rn(D[t][q]);
        l = l * 256 + __float2int_rn(D[4 + t][q]);
    }
    // x = v 2^(E - 1084); the level sums carry 2^56 beside the two integers
    return fma(to_double(h), 4294967296.0, to_double(l)) * __longlong_as_double((long long)(1023 + ea + eb - 2112) << 52);
}
}  // namespace oz
}  // namespace nep
