// Dense k-qubit gates on a complex128 state (sm_103a) as exact fixed-point products on the
// tensor cores.
//
// What bounds the plain form: FP64 runs at 2 fused multiply-adds per clock and SM on this GPU, so
// the 4 2^k of them that a complex128 amplitude needs take 2 2^k clocks per SM, against 1.5 clocks
// for its 32 bytes of HBM traffic: every width from k = 1 up is bound by the FP64 pipe, by a factor
// of 80 at k = 6.  The split used here (Ozaki, Ogita, Oishi & Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and its applications",
// Numerical Algorithms 2012) moves the products to the tensor cores without giving up precision:
//   - the reals of a group (the 2^k amplitudes that differ in the target bits) are written as
//     62-bit integers relative to the group's largest exponent, and those as eight signed base-256
//     digits; U's entries likewise, relative to its largest entry (on the host, once);
//   - a digit is exact in FP16, a product of two has 15 bits, and the FP32 accumulator of the MMA
//     adds up to 2^10 of them exactly (all sums stay integers of at most 2^24): the 36 digit pairs
//     (i, j) with i + j <= 7 go to the eight accumulators i + j;
//   - the eight sums are put together in 64-bit integer arithmetic and rounded once to FP64.
// What is left out (pairs with i + j > 7, bits below 2^-62 of the group's largest value) is below
// 2^-57 of the largest product; the plain form rounds after every one of its 2 2^k additions.
// All of it is integer and tensor work; the FP64 pipe only does the final conversion.
//
// A warp owns 8 groups (the N columns of m16n8k16; 4 groups x {re, im} for a real U).  The MMA's B
// fragment wants, per lane, a pair of rows of one column, and which amplitude is which row is free,
// so every lane loads its amplitudes straight from HBM into the fragment's place: there is no
// shared-memory stage, no barrier and no exchange but the quad's maximum.  The accumulator's rows
// are output amplitudes, written back in place.  U's digits sit in shared memory in fragment order.
// Group bits are the lowest free qubits, so a warp's load covers whole 128-byte lines.
//
// Not all gates take this form (dense_f64_applies): those with mostly zero rows keep the FP64
// kernels, which are exact on permutations; rows that only scale their own amplitude (the padding of
// an eigenvector matrix, a controlled gate written as a dense one) are computed in FP64 on the way out, and
// neither those amplitudes nor their entries count in the scales of the others.
// A tile with a group that is not finite, or whose largest exponent is far from 1, is computed in
// the plain FP64 form by the same warp (plain_tile).
//
// 26 qubits, FP64 form -> this one, TB/s: k = 1 2.26 -> 3.83, 2 1.17 -> 3.8, 3 0.62 -> 3.8, 4 0.31 -> 2.45, 5 0.16 -> 1.35,
// 6 0.072 -> 0.76 (from 4 targets on, large states take dense_f64_tc.cu).  k <= 3 is bound by issue slots (splitting and
// joining the digits), wider gates by the MMAs.  Error against long double 4.6e-17 of the largest amplitude
// (FP64 form 7e-17 to 3.5e-16).
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.h"
#include "f64_digits.cuh"

namespace qsim {
namespace f64 {

constexpr int kMaxFix = 40;

struct Args {
    void *psi;
    const uint4 *dig;            // U's digits in fragment order (pack_digits)
    const double2 *Ut;           // U transposed, FP64 (plain_tile)
    long long ntasks;
    unsigned long long cmask;
    unsigned long long diag;     // bit r set: row and column r are zero off the diagonal (computed in FP64)
    int su;                      // U = (integers) 2^(su - 62)
    int k;                       // the gate's own targets (below 3: the rest of the 8 amplitudes are group bits)
    int real_u;
    int nfix;
    int fix[kMaxFix];            // ascending: targets, controls, group bits inside a task
    long long amp[128];          // byte offset of amplitude a of a group
    long long col[8];            // byte offset of group column 0..7 (0..3 for a real U)
    long long tile[4];           // byte offset of the task's tiles
};

template <int K, bool REALU, int TBITS = -1>
struct Cfg {
    static constexpr int D = 1 << K;                   // amplitudes per group
    static constexpr bool RF = K == 3 && !REALU;       // real form: one m-tile of (re, im) rows
    static constexpr int MT = RF ? 1 : D / 16;         // m-tiles
    static constexpr int KS = RF ? 1 : D / 16;         // k-steps
    static constexpr int TABS = RF || REALU ? 1 : 3;   // U | Re U, Im U, -Im U
    static constexpr int TAB = MT * KS * kDigits * 32; // uint4 per table
    static constexpr int GB = REALU ? 2 : 3;           // group bits of a tile
    static constexpr int RED = REALU ? D : 2 * D;      // terms of a sum
    static constexpr bool BIAS = RED <= 32;            // sums below 2^22: read back without a conversion
    static constexpr int SH = RED > 64 ? 13 : 12;      // bits dropped from the 2^-68 sum
    // tiles per task: up to 8 amplitudes (16 reals) per lane in flight; states with too few tasks for
    // the warps of the chip take one tile per task
    static constexpr int TBMAX = REALU ? (K == 4 ? 2 : K == 5 ? 1 : 0) : (K == 3 ? 2 : K == 4 ? 1 : 0);
    static constexpr int TB = TBITS < 0 ? TBMAX : TBITS;
    static constexpr int NT = 1 << TB;
    static constexpr int EPL = REALU ? D / 4 : D / 2;  // reals per lane and tile
    static constexpr bool PREFETCH = EPL * NT <= 16;
    static constexpr int THREADS = K == 6 && !REALU ? 256 : (K >= 5 ? 384 : 512);
    static constexpr int SMEM = TABS * TAB * 16;
};

__device__ __forceinline__ void mma(float (&d)[4], const uint4 &a, unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// One tile in the plain FP64 form, U's columns in order as the plain kernels add them.
template <int K, bool REALU>
__device__ __noinline__ void plain_tile(const Args &a, char *base, int lane) {
    constexpr int D = 1 << K, GB = Cfg<K, REALU>::GB;
    constexpr int LPG = 32 >> GB, OUT = D / LPG;  // lanes per group, outputs per lane
    char *p = base + a.col[lane / LPG];
    const int D0 = 1 << a.k;  // bits from a.k on are group bits
    double2 y[OUT];
#pragma unroll 1
    for (int o = 0; o < OUT; o++) {
        const int row = lane % LPG + o * LPG, r = row & (D0 - 1);
        double2 s = make_double2(0.0, 0.0);
#pragma unroll 1
        for (int c = 0; c < D0; c++) {
            const double2 x = *reinterpret_cast<const double2 *>(p + a.amp[(row & ~(D0 - 1)) | c]);
            const double2 u = a.Ut[c * D0 + r];
            s.x = fma(u.x, x.x, s.x);
            if (!a.real_u) s.x = fma(-u.y, x.y, s.x);
            s.y = fma(u.x, x.y, s.y);
            if (!a.real_u) s.y = fma(u.y, x.x, s.y);
        }
        y[o] = s;
    }
    __syncwarp();  // every output of the tile is computed before any is stored
#pragma unroll 1
    for (int o = 0; o < OUT; o++) {
        *reinterpret_cast<double2 *>(p + a.amp[lane % LPG + o * LPG]) = y[o];
    }
    __syncwarp();
}

// The result y of amplitude `row` into its place: for a diagonal row, U's entry times the value there.
template <int K>
__device__ __forceinline__ void put(const Args &a, int row, char *at, double2 y) {
    double2 *p = reinterpret_cast<double2 *>(at);
    if ((a.diag >> row) & 1ull) {
        const int r = row & ((1 << a.k) - 1);
        const double2 u = __ldg(a.Ut + (r << a.k) + r), x = *p;
        y.x = u.x * x.x;
        y.y = u.x * x.y;
        if (!a.real_u) {
            y.x = fma(-u.y, x.y, y.x);
            y.y = fma(u.y, x.x, y.y);
        }
    }
    __stcs(p, y);
}

template <int K, bool REALU, int TBITS>
__global__ void __launch_bounds__(Cfg<K, REALU>::THREADS, 1) dense_f64_kernel(const __grid_constant__ Args a) {
    using C = Cfg<K, REALU, TBITS>;
    constexpr int NT = C::NT, EPL = C::EPL, KS = C::KS;
    extern __shared__ __align__(16) uint4 tabs[];  // [TABS][MT][KS][digit][lane]
    const int tid = threadIdx.x, lane = tid & 31, q = lane & 3, n = lane >> 2;
    for (int i = tid; i < C::TAB * (C::TABS == 3 ? 2 : 1); i += blockDim.x) {
        uint4 v = a.dig[i];
        tabs[i] = v;
        if (C::TABS == 3 && i >= C::TAB) {  // -Im U
            v.x ^= 0x80008000u;
            v.y ^= 0x80008000u;
            v.z ^= 0x80008000u;
            v.w ^= 0x80008000u;
            tabs[i + C::TAB] = v;
        }
    }
    __syncthreads();
    const int wpc = blockDim.x / 32;
    const long long warps = (long long)gridDim.x * wpc;
    // B column n: group (n mod 2) 4 + n / 2 (the store of one accumulator column then covers the
    // lowest group bits), or re / im of group n / 2 for a real U
    const long long in_off = REALU ? a.col[n >> 1] + 8 * (n & 1) : a.col[(n & 1) * 4 + (n >> 1)];
    const long long in_lane = in_off + a.amp[q], out_lane = a.amp[n] + a.col[q];
    char *psi = static_cast<char *>(a.psi);

    double x[NT][EPL];  // this lane's reals: EPL / 2 amplitudes of one group, or EPL parts for a real U
    auto task_base = [&](long long t) -> char * {
        unsigned long long g = (unsigned long long)t;
        for (int i = 0; i < a.nfix; i++) {
            const int p = a.fix[i];
            g = ((g >> p) << (p + 1)) | (g & ((1ull << p) - 1ull));
        }
        return psi + 16 * (g | a.cmask);
    };
    auto load = [&](long long t, double(&v)[NT][EPL]) {
        const char *p = task_base(t) + in_lane;
#pragma unroll
        for (int i = 0; i < NT; i++)
            if constexpr (REALU) {
#pragma unroll
                for (int e = 0; e < EPL; e++) v[i][e] = __ldcs(reinterpret_cast<const double *>(p + a.tile[i] + a.amp[4 * e]));
            } else {
#pragma unroll
                for (int e = 0; e < EPL / 2; e++) {
                    const double2 z = __ldcs(reinterpret_cast<const double2 *>(p + a.tile[i] + a.amp[4 * e]));
                    v[i][2 * e] = z.x;
                    v[i][2 * e + 1] = z.y;
                }
            }
    };
    long long t = (long long)blockIdx.x * wpc + (tid >> 5);
    if (C::PREFETCH && t < a.ntasks) load(t, x);
    for (; t < a.ntasks; t += warps) {
        if (!C::PREFETCH) load(t, x);
        char *base = task_base(t);
#pragma unroll
        for (int i = 0; i < NT; i++) {
            char *tb = base + a.tile[i], *ob = tb + out_lane;
            bool finite = true;
            if (a.diag) {  // amplitudes that are only scaled take no part in the products or in their scale
                const unsigned long long mine = a.diag >> q;
#pragma unroll
                for (int e = 0; e < EPL; e++)
                    if ((mine >> (4 * (REALU ? e : e / 2))) & 1ull) {
                        finite = finite && mag_bits(x[i][e]) < 0x7ff00000u;
                        x[i][e] = 0.0;
                    }
            }
            // exponent of each column's largest value: over the quad, or for narrow gates (RF, k < 3)
            // over the amplitudes that share the bits from k on
            unsigned m0 = 0, m1 = 0;
            if constexpr (C::RF) {
                m0 = max(mag_bits(x[i][0]), mag_bits(x[i][1]));
                m1 = max(mag_bits(x[i][2]), mag_bits(x[i][3]));
                m0 = max(m0, __shfl_xor_sync(~0u, m0, 1));
                m1 = max(m1, __shfl_xor_sync(~0u, m1, 1));
                if (a.k >= 2) {
                    m0 = max(m0, __shfl_xor_sync(~0u, m0, 2));
                    m1 = max(m1, __shfl_xor_sync(~0u, m1, 2));
                }
                if (a.k >= 3) m0 = m1 = max(m0, m1);
            } else {
#pragma unroll
                for (int e = 0; e < EPL; e++) m0 = max(m0, mag_bits(x[i][e]));
                m0 = max(m0, __shfl_xor_sync(~0u, m0, 1));
                m0 = max(m0, __shfl_xor_sync(~0u, m0, 2));
                m1 = m0;
            }
            const int E0 = m0 ? (int)(m0 >> 20) : 1023, E1 = m1 ? (int)(m1 >> 20) : 1023;
            bool fits = finite && E0 >= kMinExp && E0 <= kMaxExp && E1 >= kMinExp && E1 <= kMaxExp;
            if (m0 == 0 || m1 == 0) {  // all zero, or denormals whose high words are 0
                unsigned low = 0;
#pragma unroll
                for (int e = 0; e < EPL; e++) low |= (unsigned)__double2loint(x[i][e]) & (mag_bits(x[i][e]) ? 0u : ~0u);
                fits = fits && low == 0;
            }
            unsigned br[KS][2][kDigits], bi[REALU || C::RF ? 1 : KS][2][kDigits];
            if constexpr (C::RF) {
                digit_pairs(fixed_bytes(x[i][0], E0), fixed_bytes(x[i][1], E0), br[0][0]);
                digit_pairs(fixed_bytes(x[i][2], E1), fixed_bytes(x[i][3], E1), br[0][1]);
            } else {
#pragma unroll
                for (int s = 0; s < KS; s++)
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int e = 4 * s + 2 * h;  // this lane's entries e, e + 1 of the k-step
                        if constexpr (REALU) {
                            digit_pairs(fixed_bytes(x[i][e], E0), fixed_bytes(x[i][e + 1], E0), br[s][h]);
                        } else {
                            digit_pairs(fixed_bytes(x[i][2 * e], E0), fixed_bytes(x[i][2 * e + 2], E0), br[s][h]);
                            digit_pairs(fixed_bytes(x[i][2 * e + 1], E0), fixed_bytes(x[i][2 * e + 3], E0), bi[s][h]);
                        }
                    }
            }
            if (C::PREFETCH && i == NT - 1 && t + warps < a.ntasks) load(t + warps, x);
            if (!__all_sync(~0u, fits)) {
                plain_tile<K, REALU>(a, tb, lane);
                continue;
            }
            // result exponents of this lane's two accumulator columns 2 q, 2 q + 1 (and row n)
            const int ep = E0 | (E1 << 16);
            const int src = 8 * q + (C::RF && a.k < 2 ? (n & 2) : 0);
            int ex[2];
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const int v = __shfl_sync(~0u, ep, src + 4 * j);
                ex[j] = (C::RF && n >= 4 ? v >> 16 : v & 0xffff) - 1022 + a.su - (68 - C::SH);
            }
            float acc[4][kDigits];
            auto clear = [&] {
#pragma unroll
                for (int c = 0; c < 4; c++)
#pragma unroll
                    for (int d = 0; d < kDigits; d++) acc[c][d] = C::BIAS ? kBiasF : 0.f;
            };
            auto step = [&](const uint4 *tab, const unsigned(&b)[2][kDigits]) {
#pragma unroll
                for (int j = 0; j < kDigits; j++) {
                    const uint4 u = tab[j * 32 + lane];
#pragma unroll
                    for (int d = 0; d + j < kDigits; d++) {
                        float v[4] = {acc[0][d + j], acc[1][d + j], acc[2][d + j], acc[3][d + j]};
                        mma(v, u, b[0][d], b[1][d]);
#pragma unroll
                        for (int c = 0; c < 4; c++) acc[c][d + j] = v[c];
                    }
                }
            };
            if constexpr (C::RF) {
                clear();
                step(tabs, br[0]);
#pragma unroll
                for (int j = 0; j < 2; j++) {  // amplitude n of group q + 4 j
                    const double2 y = make_double2(join<C::BIAS, C::SH>(acc[j], ex[j]), join<C::BIAS, C::SH>(acc[2 + j], ex[j]));
                    put<K>(a, n, ob + a.col[4 * j], y);
                }
            } else {
#pragma unroll 1
                for (int mt = 0; mt < C::MT; mt++) {
                    const uint4 *tu = tabs + mt * KS * kDigits * 32;
                    if constexpr (REALU) {
                        clear();
#pragma unroll
                        for (int s = 0; s < KS; s++) step(tu + s * kDigits * 32, br[s]);
#pragma unroll
                        for (int h = 0; h < 2; h++) {  // amplitudes n and n + 8 of group q
                            const int row = 16 * mt + 8 * h + n;
                            const double2 y = make_double2(join<C::BIAS, C::SH>(acc[2 * h], ex[0]), join<C::BIAS, C::SH>(acc[2 * h + 1], ex[1]));
                            put<K>(a, row, ob + a.amp[16 * mt + 8 * h], y);
                        }
                    } else {
                        double re[4];
                        clear();
#pragma unroll
                        for (int s = 0; s < KS; s++) {
                            step(tu + s * kDigits * 32, br[s]);
                            step(tu + 2 * C::TAB + s * kDigits * 32, bi[s]);
                        }
#pragma unroll
                        for (int c = 0; c < 4; c++) re[c] = join<C::BIAS, C::SH>(acc[c], ex[c & 1]);
                        clear();
#pragma unroll
                        for (int s = 0; s < KS; s++) {
                            step(tu + C::TAB + s * kDigits * 32, br[s]);
                            step(tu + s * kDigits * 32, bi[s]);
                        }
#pragma unroll
                        for (int c = 0; c < 4; c++) {  // amplitudes n and n + 8 of groups q and q + 4
                            const int row = 16 * mt + 8 * (c >> 1) + n;
                            const double2 y = make_double2(re[c], join<C::BIAS, C::SH>(acc[c], ex[c & 1]));
                            put<K>(a, row, ob + a.col[4 * (c & 1)] + a.amp[16 * mt + 8 * (c >> 1)], y);
                        }
                    }
                }
            }
        }
    }
}

// kernel width of a gate: at least 3 targets, 4 for a real U
static int width_of(const Op &op) {
    const int k = (int)op.targets.size();
    return k <= 3 ? 3 : k;
}
static bool real_form(const Op &op) { return op.real_u && op.targets.size() >= 4; }

template <int K, bool REALU>
static void pack_digits(const Op &op, int su, unsigned char *out) {
    using C = Cfg<K, REALU>;
    const int k = (int)op.targets.size(), D0 = 1 << k;
    unsigned short *o = reinterpret_cast<unsigned short *>(out);
    auto entry = [&](int r, int c) -> cd {  // group bits from k on: identity
        if ((r >> k) != (c >> k) || ((op.f64_diag >> (r & (D0 - 1))) & 1ull)) return cd(0.0, 0.0);
        return op.U[(size_t)(r & (D0 - 1)) * D0 + (c & (D0 - 1))];
    };
    const int tabs = C::TABS == 3 ? 2 : 1;
    const double scale = std::ldexp(1.0, 62 - su);
    for (int tab = 0; tab < tabs; tab++)
        for (int mt = 0; mt < C::MT; mt++)
            for (int ks = 0; ks < C::KS; ks++)
                for (int lane = 0; lane < 32; lane++)
                    for (int e = 0; e < 8; e++) {
                        // A fragment half e: register e / 2 (row + 8 for 1, 3; column + 8 for 2, 3)
                        const int row = (lane >> 2) + 8 * ((e >> 1) & 1);
                        const int kp = 2 * (lane & 3) + (e & 1) + 8 * (e >> 2);
                        double u;
                        if (C::RF) {  // rows: re of amplitude 0..7, then im; columns: (re, im) pairs
                            const cd z = entry(row & 7, kp >> 1);
                            if (row < 8) u = (kp & 1) ? -z.imag() : z.real();
                            else u = (kp & 1) ? z.real() : z.imag();
                        } else {  // column kp: amplitude (q + 4 (e + 2 h)) of the k-step
                            const int c = 16 * ks + ((kp & 7) >> 1) + 4 * ((kp & 1) + 2 * (kp >> 3));
                            const cd z = entry(16 * mt + row, c);
                            u = tab ? z.imag() : z.real();
                        }
                        const unsigned long long dg = digit_bytes(u, scale);
                        for (int j = 0; j < kDigits; j++)
                            o[((((size_t)(tab * C::MT + mt) * C::KS + ks) * kDigits + j) * 32 + lane) * 8 + e] = half_digit(dg, j);
                    }
}

template <int K, bool REALU, int TBITS>
static void launch(const Args &a, int sms, cudaStream_t st) {
    using C = Cfg<K, REALU, TBITS>;
    auto kern = dense_f64_kernel<K, REALU, TBITS>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
        if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("dense_f64_kernel attribute: ") + cudaGetErrorString(e));
        attr = true;
    }
    // a state with fewer tasks than the chip has warps is spread over the SMs: full blocks would leave most of them
    // idle (16 qubits, 4 targets: 512 tasks, 32 blocks of 16 warps 7.0 us, 256 of 2 warps 4.1 us); not where a block
    // loads 192 KB of digits first (6 targets complex at 17 qubits: 29 us in full blocks, 45 us with one warp each)
    int wpc = C::THREADS / 32;
    while (C::SMEM <= 64 * 1024 && wpc > 1 && a.ntasks < (long long)sms * wpc) wpc /= 2;
    const int threads = wpc * 32;
    const int per_sm = occupancy_cached(reinterpret_cast<const void *>(kern), threads, C::SMEM);
    QSIM_REQUIRE(per_sm > 0, "dense_f64_kernel does not fit on an SM");
    const long long grid = std::min<long long>((a.ntasks + wpc - 1) / wpc, (long long)sms * per_sm);
    kern<<<(int)grid, threads, C::SMEM, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("dense_f64_kernel: ") + cudaGetErrorString(e));
    note_launches(1, QSIM_KERNEL_DENSE_TC);
}

#define QSIM_F64_SWITCH(op, CALL)                            \
    switch (f64::width_of(op) + (f64::real_form(op) ? 10 : 0)) { \
        case 3: CALL(3, false); break;                       \
        case 4: CALL(4, false); break;                       \
        case 5: CALL(5, false); break;                       \
        case 6: CALL(6, false); break;                       \
        case 14: CALL(4, true); break;                       \
        case 15: CALL(5, true); break;                       \
        case 16: CALL(6, true); break;                       \
        default: break;                                      \
    }

}  // namespace f64

// Rows that, with their columns, are zero off the diagonal.
static unsigned long long diagonal_rows(const Op &op) {
    const int D = 1 << (int)op.targets.size();
    unsigned long long diag = 0;
    for (int r = 0; r < D; r++) {
        bool d = true;
        for (int c = 0; c < D && d; c++)
            d = c == r || (op.U[(size_t)r * D + c] == cd(0.0, 0.0) && op.U[(size_t)c * D + r] == cd(0.0, 0.0));
        if (d) diag |= 1ull << r;
    }
    return diag;
}

// Gates of 1..6 targets with mostly nonzero rows.  A sum of a few terms that misses the group's largest value
// is more exact in FP64 than relative to that value (a permutation is exact), so a gate with a row of at most half
// its entries nonzero (diagonal rows and columns apart) stays in FP64 where the row form makes that cheap
// (sparse_width).  A gate that mixes such rows with full ones, a quarter of its entries nonzero at least, comes here
// all the same: the plain kernel would multiply all of its zeros (the eigenvectors of a grid that falls apart
// without its slack bus, 64 x 64 in blocks of 63 and 1: 30.8 ms in FP64 on 2^27 amplitudes, 1.5 ms here).  The error
// of its short rows is then 2^-57 of the group's largest value, as that of the full ones.
bool dense_f64_applies(const Op &op) {
    const int k = (int)op.targets.size();
    if (op.kind != OP_DENSE || k < 1 || k > 6) return false;
    const int D = 1 << k;
    const unsigned long long diag = diagonal_rows(op);
    double top = 0.0;
    int live = 0, all = 0;
    bool short_rows = false;
    for (int r = 0; r < D; r++) live += !((diag >> r) & 1ull);
    for (int r = 0; r < D; r++) {
        if ((diag >> r) & 1ull) continue;
        int nz = 0;
        for (int c = 0; c < D; c++) {
            const cd u = op.U[(size_t)r * D + c];
            top = std::max(top, std::max(std::fabs(u.real()), std::fabs(u.imag())));
            if (!((diag >> c) & 1ull)) nz += u != cd(0.0, 0.0);
        }
        short_rows = short_rows || 2 * nz <= live;
        all += nz;
    }
    if (short_rows && (sparse_width(op) > 0 || 4 * all < live * live)) return false;
    return live > 0 && top > std::ldexp(1.0, -100) && top < std::ldexp(1.0, 100);
}

size_t dense_f64_blob_bytes(const Op &op) {
    size_t n = 0;
#define QSIM_F64_BYTES(K, R) n = (size_t)f64::Cfg<K, R>::TAB * 16 * (f64::Cfg<K, R>::TABS == 3 ? 2 : 1)
    QSIM_F64_SWITCH(op, QSIM_F64_BYTES)
#undef QSIM_F64_BYTES
    return n;
}

// f64_su: exponent of U's scale, every entry of a row that is not only scaled is below 2^su in magnitude
void dense_f64_scale(Op &op) {
    const int D = 1 << (int)op.targets.size();
    op.f64_diag = diagonal_rows(op);
    double top = 0.0;
    for (int r = 0; r < D; r++)
        for (int c = 0; c < D && !((op.f64_diag >> r) & 1ull); c++) {
            const cd &u = op.U[(size_t)r * D + c];
            top = std::max(top, std::max(std::fabs(u.real()), std::fabs(u.imag())));
        }
    std::frexp(top, &op.f64_su);  // top = f 2^su, f in [1/2, 1)
}

void dense_f64_pack(const Op &op, unsigned char *out) {
#define QSIM_F64_PACK(K, R) f64::pack_digits<K, R>(op, op.f64_su, out)
    QSIM_F64_SWITCH(op, QSIM_F64_PACK)
#undef QSIM_F64_PACK
}

// Returns false when the state is too small for the kernel's tiles (the plain kernels take it).
bool launch_dense_f64(void *state, int n, const Op &op, const void *dig, const void *Ut, int sms, cudaStream_t st) {
    const int k = (int)op.targets.size(), K = f64::width_of(op);
    int tb = 0, gb = 0, warps = 0;  // warps: of a full chip
#define QSIM_F64_BITS(KK, R) tb = f64::Cfg<KK, R>::TB, gb = f64::Cfg<KK, R>::GB, warps = sms * f64::Cfg<KK, R>::THREADS / 32
    QSIM_F64_SWITCH(op, QSIM_F64_BITS)
#undef QSIM_F64_BITS
    unsigned long long used = 0, cmask = 0;
    for (int q : op.targets) used |= 1ull << q;
    for (int q : op.controls) used |= 1ull << q, cmask |= 1ull << q;
    std::vector<int> fr;  // free qubits ascending: columns, then the amplitude bits from k on, then tiles
    for (int q = 0; q < n; q++)
        if (!((used >> q) & 1ull)) fr.push_back(q);
    const int groups = (int)fr.size() - gb - (K - k);  // tiles, log2
    if (groups < tb || (1ll << (groups - tb)) < 2 * warps) tb = 0;
    const int inside = gb + (K - k) + tb;
    if ((int)fr.size() < inside || (int)(op.targets.size() + op.controls.size()) + inside > f64::kMaxFix) return false;
    f64::Args a;
    std::memset(&a, 0, sizeof(a));
    a.psi = state;
    a.dig = static_cast<const uint4 *>(dig);
    a.Ut = static_cast<const double2 *>(Ut);
    a.ntasks = 1ll << ((int)fr.size() - inside);
    a.cmask = cmask;
    a.su = op.f64_su;
    a.k = k;
    a.real_u = op.real_u ? 1 : 0;
    for (int r = 0; r < (1 << K); r++)
        if ((op.f64_diag >> (r & ((1 << k) - 1))) & 1ull) a.diag |= 1ull << r;
    std::vector<int> amp(op.targets), fix(op.targets);
    std::sort(amp.begin(), amp.end());
    for (int j = 0; j < K - k; j++) amp.push_back(fr[gb + j]);
    for (int v = 0; v < (1 << K); v++)
        for (int b = 0; b < K; b++)
            if ((v >> b) & 1) a.amp[v] += 16ll << amp[b];
    for (int v = 0; v < (1 << gb); v++)
        for (int b = 0; b < gb; b++)
            if ((v >> b) & 1) a.col[v] += 16ll << fr[b];
    for (int v = 0; v < (1 << tb); v++)
        for (int b = 0; b < tb; b++)
            if ((v >> b) & 1) a.tile[v] += 16ll << fr[gb + K - k + b];
    fix.insert(fix.end(), op.controls.begin(), op.controls.end());
    fix.insert(fix.end(), fr.begin(), fr.begin() + inside);
    std::sort(fix.begin(), fix.end());
    a.nfix = (int)fix.size();
    for (int i = 0; i < a.nfix; i++) a.fix[i] = fix[i];
#define QSIM_F64_LAUNCH(KK, R)                                                                  \
    do {                                                                                        \
        if (tb) f64::launch<KK, R, f64::Cfg<KK, R>::TBMAX>(a, sms, st);                         \
        else f64::launch<KK, R, 0>(a, sms, st);                                                 \
    } while (0)
    QSIM_F64_SWITCH(op, QSIM_F64_LAUNCH)
#undef QSIM_F64_LAUNCH
    return true;
}

}  // namespace qsim
