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

// Bits dropped from a sum of RED products at most: what keeps the quotient in 62 bits.  A constant for short sums, whose
// kernels wait for issue slots (as a variable it cost gates of up to 3 targets a fifth of their rate); for longer ones
// the gate's own f64_sh, which its row sums allow to be 2 or 3 bits less.
constexpr int kept_shift(int RED) { return RED <= 16 ? 10 : RED <= 32 ? 11 : RED <= 64 ? 12 : 13; }

// sum_t acc[t] 2^(8 (7 - t)) / 2^sh (7 <= sh <= 13, the quotient below 2^63), rounded to FP64, times 2^ex (0 for a zero sum).
// BIAS > 0: the sums started at kBiasF, and sh is BIAS.
template <int BIAS>
__device__ __forceinline__ double join(const float (&acc)[kDigits], int sh, int ex) {
    long long T;
    if constexpr (BIAS > 0) {
        int h[4];
#pragma unroll
        for (int p = 0; p < 4; p++)
            h[p] = (int)((__float_as_uint(acc[2 * p]) << 8) + __float_as_uint(acc[2 * p + 1]) - 257u * 0x4B400000u +
                         (p == 3 ? 1u << (BIAS - 1) : 0u));
        T = (long long)h[2] * (1 << (16 - BIAS)) + (long long)(h[3] >> BIAS);
        T += (long long)h[1] * (1 << (32 - BIAS));
        T += (long long)((unsigned long long)(unsigned)(h[0] << (16 - BIAS)) << 32);
    } else {
        long long p[2];
#pragma unroll
        for (int w = 0; w < 2; w++) {
            p[w] = (long long)__float2int_rn(acc[4 * w]) * (1 << 24) + (long long)__float2int_rn(acc[4 * w + 1]) * (1 << 16);
            p[w] += (long long)__float2int_rn(acc[4 * w + 2]) * (1 << 8) + (long long)__float2int_rn(acc[4 * w + 3]);
        }
        T = (long long)((unsigned long long)p[0] << (32 - sh)) + ((p[1] + (1 << (sh - 1))) >> sh);
    }
    const double d = (double)T;
    const int hi = __double2hiint(d);
    return __hiloint2double(hi ? hi + (ex << 20) : 0, __double2loint(d));
}

// A group's sums are as good as FP64 ones when every row's sum |u| |x| is not too far below the group's scale (see
// dense_f64_plan).  That sum from below, in bytes: |x| as 2^-8 of the group's scale and |u| of U's, rounded down.
// m: the high word, without sign, of an amplitude's larger part; E: the group's exponent.
__device__ __forceinline__ unsigned mag_byte(unsigned m, int E) {
    unsigned v = (m & 0xfffffu) | 0x100000u;
    asm("shr.u32 %0, %0, %1;" : "+r"(v) : "r"(E - (int)(m >> 20) + 13));  // 0 from 32 on
    return v;
}
template <int N>
__device__ __forceinline__ unsigned dot_bytes(const unsigned *u, const unsigned (&w)[N], unsigned s) {
    unsigned v[N];
    if constexpr (N == 4) {
        const uint4 t = *reinterpret_cast<const uint4 *>(u);
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else if constexpr (N == 2) {
        const uint2 t = *reinterpret_cast<const uint2 *>(u);
        v[0] = t.x, v[1] = t.y;
    } else {
        v[0] = *u;
    }
#pragma unroll
    for (int i = 0; i < N; i++) s = __dp4a(v[i], w[i], s);
    return s;
}
// Whether the rows q, q + 4, .. of the lane's group reach their thresholds; the four lanes of a group (q = 0..3, `near`
// and `far` apart) hold its columns q + 4 e as byte e of w.  safe: bit e for row q + 4 e, safe by itself; zero: the
// group is.  rows: U's bytes, row by row the columns of lane 0, 1, ..; behind them the thresholds, those of lane 0's rows
// first.  By half of the columns first: that is enough for most states.
template <int D>
__device__ __forceinline__ bool rows_fit(const unsigned (&w)[D / 16], unsigned safe, bool zero, int q, int near, int far,
                                         const unsigned char *rows) {
    constexpr int N = D / 16;
    const uint4 *thr = reinterpret_cast<const uint4 *>(rows + D * D) + q * (D / 16);
    const unsigned char *mine = rows + q * D;
    unsigned o[3][N];
    auto fetch = [&](int d, int mask) {
#pragma unroll
        for (int i = 0; i < N; i++) o[d][i] = __shfl_xor_sync(~0u, w[i], mask);
    };
    unsigned low;  // rows below their thresholds
    auto test = [&](auto sum) {
        low = 0;
#pragma unroll 1
        for (int g = 0; g < D / 16; g++) {
            const uint4 t = thr[g];
            const unsigned *u = reinterpret_cast<const unsigned *>(mine + 16 * g * D);
            unsigned l = 0;
            if (sum(u) < t.x) l |= 1u;
            if (sum(u + D) < t.y) l |= 2u;
            if (sum(u + 2 * D) < t.z) l |= 4u;
            if (sum(u + 3 * D) < t.w) l |= 8u;
            low |= l << (4 * g);
        }
    };
    fetch(0, near);
    auto half = [&](const unsigned *u) { return dot_bytes<N>(u + (q ^ 1) * N, o[0], dot_bytes<N>(u + q * N, w, 0u)); };
    test(half);
    if (__all_sync(~0u, (low & ~safe) == 0 || zero)) return true;
    fetch(1, far);
    fetch(2, near | far);
    test([&](const unsigned *u) { return dot_bytes<N>(u + (q ^ 3) * N, o[2], dot_bytes<N>(u + (q ^ 2) * N, o[1], half(u))); });
    return (low & ~safe) == 0 || zero;
}
// bytes, thresholds, and for rows with a scaled amplitude the exponent of that amplitude, above the group's, from
// which on they are safe
constexpr int rows_bytes(int D) { return D * D + 8 * D; }

// The same for a lane's amplitudes as high words of their larger parts, out of line.  diag: rows with a diagonal entry
// multiplied in FP64.
template <int D, int NEAR, int FAR>
__device__ __noinline__ bool rows_fit_of(const unsigned (&m)[D / 4], int E, bool zero, int q, unsigned long long diag,
                                         const unsigned char *rows) {
    const int *from = reinterpret_cast<const int *>(rows + D * D + 4 * D);
    unsigned w[D / 16], safe = 0;
#pragma unroll
    for (int e = 0; e < D / 4; e++) {
        w[e / 4] = (e % 4 ? w[e / 4] : 0u) | mag_byte(m[e], E) << (8 * (e % 4));
        if (((diag >> (q + 4 * e)) & 1ull) && (int)(m[e] >> 20) >= max(E + from[q + 4 * e], 1)) safe |= 1u << e;
    }
    return rows_fit<D>(w, safe, zero, q, NEAR, FAR, rows);
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
