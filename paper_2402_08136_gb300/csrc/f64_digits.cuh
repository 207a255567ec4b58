// FP64 values as signed base-256 digits and back (dense_f64.cu, dense_f64_tc.cu).
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include <cmath>

namespace qsim {
namespace f64 {

constexpr int kDigits = 8;
constexpr int kMinExp = 200, kMaxExp = 1900;  // biased exponents of a group's largest value that take the split

__device__ __forceinline__ unsigned mag_bits(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// x as a 62-bit integer relative to 2^(E + 1) (E: a biased exponent not below x's), plus 128 in
// every byte: byte i is digit i + 128 of the signed base-256 form, -128 <= digit <= 127
__device__ __forceinline__ unsigned long long fixed_bytes(double x, int E) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int s = E - (int)((hi >> 20) & 0x7ffu);
    const unsigned mh = (__funnelshift_l(lo, hi, 9) & 0x1fffffffu) | 0x20000000u;
    unsigned long long v = ((unsigned long long)mh << 32) | (lo << 9);
    asm("shr.u64 %0, %0, %1;" : "+l"(v) : "r"(s));  // 0 from 64 on
    const long long sg = (long long)((int)hi >> 31);
    return (v ^ (unsigned long long)sg) + (0x8080808080808080ull - (unsigned long long)sg);
}

// The digits of two reals as FP16 pairs: out[i] = (digit i of a, digit i of b), i = 0 the highest.
// A byte under 0x64 is FP16 1024 + byte.
__device__ __forceinline__ void digit_pairs(unsigned long long a, unsigned long long b, unsigned (&out)[kDigits]) {
    const __half2 off = __floats2half2_rn(1152.f, 1152.f);
#pragma unroll
    for (int w = 0; w < 2; w++) {
        const unsigned x = w ? (unsigned)a : (unsigned)(a >> 32), y = w ? (unsigned)b : (unsigned)(b >> 32);
        const unsigned t[2] = {__byte_perm(x, y, 0x7362), __byte_perm(x, y, 0x5140)};  // bytes 2, 3 and 0, 1
#pragma unroll
        for (int i = 0; i < 4; i++) {  // digit 4 w + i is byte 3 - i of the word
            const unsigned h = __byte_perm(t[i >> 1], 0x64646464u, (i & 1) ? 0x4140 : 0x4342);
            const __half2 r = __hsub2(*reinterpret_cast<const __half2 *>(&h), off);
            out[4 * w + i] = *reinterpret_cast<const unsigned *>(&r);
        }
    }
}

constexpr float kBiasF = 12582912.0f;  // 1.5 2^23: an FP32 sum started there has its integer in its low bits

// sum_t acc[t] 2^(8 (7 - t)) / 2^SH, rounded to FP64, times 2^ex (0 for a zero sum)
template <bool BIAS, int SH>
__device__ __forceinline__ double join(const float (&acc)[kDigits], int ex) {
    long long T;
    if constexpr (BIAS) {
        int h[4];
#pragma unroll
        for (int p = 0; p < 4; p++)
            h[p] = (int)((__float_as_uint(acc[2 * p]) << 8) + __float_as_uint(acc[2 * p + 1]) - 257u * 0x4B400000u +
                         (p == 3 ? 1u << (SH - 1) : 0u));
        T = (long long)h[2] * (1 << (16 - SH)) + (long long)(h[3] >> SH);
        T += (long long)h[1] * (1 << (32 - SH));
        T += (long long)((unsigned long long)(unsigned)(h[0] << (16 - SH)) << 32);
    } else {
        long long p[2];
#pragma unroll
        for (int w = 0; w < 2; w++) {
            p[w] = (long long)__float2int_rn(acc[4 * w]) * (1 << 24) + (long long)__float2int_rn(acc[4 * w + 1]) * (1 << 16);
            p[w] += (long long)__float2int_rn(acc[4 * w + 2]) * (1 << 8) + (long long)__float2int_rn(acc[4 * w + 3]);
        }
        T = (p[0] << (32 - SH)) + ((p[1] + (1 << (SH - 1))) >> SH);
    }
    const double d = (double)T;
    const int hi = __double2hiint(d);
    return __hiloint2double(hi ? hi + (ex << 20) : 0, __double2loint(d));
}

// u scale (an integer below 2^62) as signed base-256 digits, -127 <= digit <= 128 (so that no product of a
// digit with one of the state's reaches +2^14): byte i is digit i + 127
inline unsigned long long digit_bytes(double u, double scale) {
    return (unsigned long long)std::llrint(u * scale) + 0x7F7F7F7F7F7F7F7Full;
}
// digit d (0 the highest) as an FP16 bit pattern
struct HalfTable {
    unsigned short bits[256];  // of -127 .. 128
};
constexpr HalfTable make_half_table() {
    HalfTable t{};
    for (int i = 0; i < 256; i++) {
        const int v = i - 127, m = v < 0 ? -v : v;
        int e = 0;
        while ((m >> e) > 1) e++;
        t.bits[i] = (unsigned short)(m == 0 ? 0 : (v < 0 ? 0x8000 : 0) | ((e + 15) << 10) | (((m << 10) >> e) & 0x3ff));
    }
    return t;
}
constexpr HalfTable kHalf = make_half_table();
inline unsigned short half_digit(unsigned long long bytes, int d) { return kHalf.bits[(bytes >> (8 * (kDigits - 1 - d))) & 255]; }

}  // namespace f64
}  // namespace qsim
