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
// What is left out (the pairs with i + j > 7, bits below the last kept one) is relative to the largest value of the group
// and of U, not to a sum's own terms.  dense_f64_plan says when that is within the bound of an FP64 sum of the same terms;
// where it is not, the group's tile runs in FP64, so that small outputs next to large ones keep their bits.
// All of it is integer and tensor work; the FP64 pipe only does the final conversion.
//
// A warp owns 8 groups (the N columns of m16n8k16; 4 groups x {re, im} for a real U).  The MMA's B
// fragment wants, per lane, a pair of rows of one column, and which amplitude is which row is free,
// so every lane loads its amplitudes straight from HBM into the fragment's place: there is no
// shared-memory stage, no barrier and no exchange but the quad's maximum.  The accumulator's rows
// are output amplitudes, written back in place.  U's digits sit in shared memory in fragment order.
// Group bits are the lowest free qubits, so a warp's load covers whole 128-byte lines.
//
// Not all gates take this form (dense_f64_plan): those with mostly zero rows keep the FP64 kernels, which are exact on
// permutations.  Entries that stand (almost) alone in their row and column (the padding of an eigenvector matrix, a
// controlled gate written as a dense one, the diagonal of a gate close to the identity) are multiplied in FP64 on the way
// out, and neither they nor their amplitudes count in the scales of the rest.
// A tile with a group that is not finite, whose largest exponent is far from 1, or whose sums would lose more than FP64
// ones is computed in the plain FP64 form by the same warp (plain_tile; from 4 targets on and where the groups are tested,
// that group alone: plain_groups).
//
// 26 qubits, FP64 form -> this one, TB/s: k = 1 2.26 -> 3.83, 2 1.17 -> 3.8, 3 0.62 -> 3.8, 4 0.31 -> 2.45, 5 0.16 -> 1.35,
// 6 0.072 -> 0.76 (from 4 targets on, large states take dense_f64_tc.cu).  k <= 3 is bound by issue slots (splitting and
// joining the digits), wider gates by the MMAs.  Gates with small entries, whose groups are tested, 25 qubits: real 2, 4
// and 5 targets 295 -> 340, 291 -> 379, 432 -> 488 us (Haar), 1 target close to the identity 288 -> 346 us (FP64 485 us).  Error against long
// double 4.6e-17 of the largest amplitude (FP64 form 7e-17 to 3.5e-16).
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <climits>
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
    unsigned long long diag;     // bit r set: entry (r, r) is multiplied in FP64
    unsigned long long beside;   // ... and its row or column has other entries
    const double2 *vw;           // by row and column r of those: what amplitude r and sum r are multiplied by for the digits
    int su, sh;                  // U = (integers) 2^(su - 62); bits dropped from the 2^-68 sum
    int check;                   // test every group: by what each lane of it holds (reach, see dense_f64_plan), else rows_fit
    int reach;
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
    static constexpr int BIAS = RED <= 32 ? kept_shift(RED) : 0;  // sums below 2^22: read back without a conversion
    // tiles per task: up to 8 amplitudes (16 reals) per lane in flight; states with too few tasks for
    // the warps of the chip take one tile per task
    static constexpr int TBMAX = REALU ? (K == 4 ? 2 : K == 5 ? 1 : 0) : (K == 3 ? 2 : K == 4 ? 1 : 0);
    static constexpr int TB = TBITS < 0 ? TBMAX : TBITS;
    static constexpr int NT = 1 << TB;
    static constexpr int EPL = REALU ? D / 4 : D / 2;  // reals per lane and tile
    static constexpr bool PREFETCH = EPL * NT <= 16;
    static constexpr int THREADS = K == 6 && !REALU ? 256 : (K >= 5 ? 384 : 512);
    static constexpr int ROWS = rows_bytes(D);         // the rows' bytes and thresholds, behind the tables
    static constexpr int SMEM = TABS * TAB * 16 + ROWS;
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
#pragma unroll 4
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

// The groups of a tile in mask gm in FP64 (K >= 4), a warp per group (two with 4 targets): a lane loads its amplitudes and
// has their rows, U's columns come in order, the column's amplitude from its lane.
template <int K, bool REALU>
__device__ __noinline__ void plain_groups(const Args &a, char *base, unsigned gm, int lane) {
    constexpr int D = 1 << K, L = D < 32 ? D : 32, ROWS = D / L;  // lanes per group, rows per lane
    const int r = lane % L;
    while (gm) {
        int g = __ffs(gm) - 1;
        bool mine = true;
        gm &= gm - 1;
        if (L < 32 && lane >= L) {
            mine = gm != 0;
            if (mine) g = __ffs(gm) - 1;
        }
        if (L < 32) gm &= gm - 1;
        char *p = base + a.col[g];
        double2 x[ROWS], y[ROWS];
#pragma unroll
        for (int o = 0; o < ROWS; o++) {
            x[o] = *reinterpret_cast<const double2 *>(p + a.amp[r + 32 * o]);
            y[o] = make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int h = 0; h < ROWS; h++)
#pragma unroll 4
            for (int c = 0; c < L; c++) {
                const double zx = __shfl_sync(~0u, x[h].x, c, L), zy = __shfl_sync(~0u, x[h].y, c, L);
#pragma unroll
                for (int o = 0; o < ROWS; o++) {
                    const double2 *w = a.Ut + (c + 32 * h) * D + r + 32 * o;
                    const double2 u = REALU ? make_double2(__ldg(&w->x), 0.0) : __ldg(w);
                    y[o].x = fma(u.x, zx, y[o].x);
                    if (!REALU) y[o].x = fma(-u.y, zy, y[o].x);
                    y[o].y = fma(u.x, zy, y[o].y);
                    if (!REALU) y[o].y = fma(u.y, zx, y[o].y);
                }
            }
        __syncwarp();  // every output of a group is computed before any is stored
        if (mine)
#pragma unroll
            for (int o = 0; o < ROWS; o++) *reinterpret_cast<double2 *>(p + a.amp[r + 32 * o]) = y[o];
    }
    __syncwarp();
}

// The result y of amplitude `row` into its place; where a diagonal entry is left to FP64, its product with the value there
// is added.
template <int K, bool SPEC>
__device__ __forceinline__ void put(const Args &a, int row, char *at, double2 y) {
    double2 *p = reinterpret_cast<double2 *>(at);
    if (SPEC && ((a.diag >> row) & 1ull)) {
        const int r = row & ((1 << a.k) - 1);
        const double2 u = __ldg(a.Ut + (r << a.k) + r), x = *p;
        if (K >= 4 && ((a.beside >> row) & 1ull)) {
            const double w = __ldg(a.vw + r).y;
            y.x *= w;
            y.y *= w;
        }
        y.x = fma(u.x, x.x, y.x);  // without other entries in the row the sum is 0
        y.y = fma(u.x, x.y, y.y);
        if (!a.real_u) {
            y.x = fma(-u.y, x.y, y.x);
            y.y = fma(u.y, x.x, y.y);
        }
    }
    __stcs(p, y);
}

// SPEC: gates with diagonal entries multiplied in FP64, or whose groups are tested.  Forms of their own: as branches of the
// one kernel they cost gates of up to 3 targets a fifth of their rate.
template <int K, bool REALU, int TBITS, bool SPEC>
__global__ void __launch_bounds__(Cfg<K, REALU>::THREADS, 1) dense_f64_kernel(const __grid_constant__ Args a) {
    using C = Cfg<K, REALU, TBITS>;
    constexpr int NT = C::NT, EPL = C::EPL, KS = C::KS;
    extern __shared__ __align__(16) uint4 tabs[];  // [TABS][MT][KS][digit][lane]
    const int tid = threadIdx.x, lane = tid & 31, q = lane & 3, n = lane >> 2;
    constexpr int IN = C::TAB * (C::TABS == 3 ? 2 : 1);  // tables in memory, the rows' bytes behind them
    for (int i = tid; i < IN + (SPEC && a.check ? C::ROWS / 16 : 0); i += blockDim.x) {
        uint4 v = a.dig[i];
        tabs[i < IN ? i : i - IN + C::TABS * C::TAB] = v;
        if (C::TABS == 3 && i >= C::TAB && i < IN) {  // -Im U
            v.x ^= 0x80008000u;
            v.y ^= 0x80008000u;
            v.z ^= 0x80008000u;
            v.w ^= 0x80008000u;
            tabs[i + C::TAB] = v;
        }
    }
    const unsigned char *rows = reinterpret_cast<const unsigned char *>(tabs + C::TABS * C::TAB);
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
            if (SPEC && K >= 4 && a.beside) {  // amplitudes with a diagonal entry of their own, scaled to the rest of their column
#pragma unroll
                for (int e = 0; e < EPL; e++) {
                    const int c = q + 4 * (REALU ? e : e / 2);
                    if ((a.beside >> c) & 1ull) x[i][e] *= __ldg(a.vw + c).x;
                }
            }
            // amplitudes without such a rest do not count: U's digits are 0 in their columns, whatever theirs are
            const unsigned long long alone = SPEC ? (a.diag & ~a.beside) >> q : 0ull;
            unsigned all = 0;
            auto mag = [&](int e) -> unsigned {
                const unsigned m = mag_bits(x[i][e]);
                all = max(all, m);
                return SPEC && ((alone >> (4 * (REALU ? e : e / 2))) & 1ull) ? 0u : m;
            };
            // exponent of each column's largest value: over the quad, or for narrow gates (RF, k < 3)
            // over the amplitudes that share the bits from k on
            unsigned m0 = 0, m1 = 0, l0 = 0, l1 = 0;  // l0, l1: of this lane
            if constexpr (C::RF) {
                m0 = l0 = max(mag(0), mag(1));
                m1 = l1 = max(mag(2), mag(3));
                m0 = max(m0, __shfl_xor_sync(~0u, m0, 1));
                m1 = max(m1, __shfl_xor_sync(~0u, m1, 1));
                if (a.k >= 2) {
                    m0 = max(m0, __shfl_xor_sync(~0u, m0, 2));
                    m1 = max(m1, __shfl_xor_sync(~0u, m1, 2));
                }
                if (a.k >= 3) m0 = m1 = max(m0, m1);
            } else {
#pragma unroll
                for (int e = 0; e < EPL; e++) m0 = max(m0, mag(e));
                l0 = m0;
                m0 = max(m0, __shfl_xor_sync(~0u, m0, 1));
                m0 = max(m0, __shfl_xor_sync(~0u, m0, 2));
                m1 = m0;
            }
            const int E0 = m0 ? (int)(m0 >> 20) : 1023, E1 = m1 ? (int)(m1 >> 20) : 1023;
            bool fits = (!SPEC || all < 0x7ff00000u) && E0 >= kMinExp && E0 <= kMaxExp && E1 >= kMinExp && E1 <= kMaxExp;
            if (m0 == 0 || m1 == 0) {  // all zero, or denormals whose high words are 0
                unsigned low = 0;
#pragma unroll
                for (int e = 0; e < EPL; e++) low |= (unsigned)__double2loint(x[i][e]) & (mag_bits(x[i][e]) ? 0u : ~0u);
                fits = fits && low == 0;
            }
            if (SPEC && a.check) {
                if constexpr (C::RF) {  // rows q and q + 4; the quad's amplitudes as bytes of two words
                    unsigned w[2] = {mag_byte(l0, E0) << (8 * q), mag_byte(l1, E1) << (8 * q)};
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        w[h] |= __shfl_xor_sync(~0u, w[h], 1);
                        w[h] |= __shfl_xor_sync(~0u, w[h], 2);
                    }
                    const unsigned *u = reinterpret_cast<const unsigned *>(rows), *thr = u + 16;
                    fits = fits && (m0 == 0 || dot_bytes<2>(u + 2 * q, w, 0u) >= thr[q]) &&
                           (m1 == 0 || dot_bytes<2>(u + 2 * q + 8, w, 0u) >= thr[q + 4]);
                } else {
                    if (!__all_sync(~0u, (int)(l0 >> 20) >= E0 - a.reach || m0 == 0)) {
                        unsigned m[C::D / 4];
#pragma unroll
                        for (int e = 0; e < C::D / 4; e++)
                            m[e] = REALU ? mag(e) : max(mag(2 * e), mag(2 * e + 1));
                        fits = rows_fit_of<C::D, 1, 2>(m, E0, m0 == 0, q, a.diag, rows) && fits;
                    }
                }
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
            unsigned gm = 0;  // groups in FP64
            if (!__all_sync(~0u, fits)) {
                if constexpr (SPEC && !C::RF) {
                    gm = __reduce_or_sync(~0u, fits ? 0u : 1u << (REALU ? n >> 1 : (n & 1) * 4 + (n >> 1)));
                    plain_groups<K, REALU>(a, tb, gm, lane);
                    if (gm == (1u << (1 << C::GB)) - 1u) continue;
                } else {
                    plain_tile<K, REALU>(a, tb, lane);
                    continue;
                }
            }
            // result exponents of this lane's two accumulator columns 2 q, 2 q + 1 (and row n)
            const int ep = E0 | (E1 << 16);
            const int src = 8 * q + (C::RF && a.k < 2 ? (n & 2) : 0);
            int ex[2];
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const int v = __shfl_sync(~0u, ep, src + 4 * j);
                ex[j] = (C::RF && n >= 4 ? v >> 16 : v & 0xffff) - 1022 + a.su - 68 + a.sh;
            }
            float acc[4][kDigits];
            auto clear = [&] {
#pragma unroll
                for (int c = 0; c < 4; c++)
#pragma unroll
                    for (int d = 0; d < kDigits; d++) acc[c][d] = C::BIAS > 0 ? kBiasF : 0.f;
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
                    const double2 y = make_double2(join<C::BIAS>(acc[j], a.sh, ex[j]), join<C::BIAS>(acc[2 + j], a.sh, ex[j]));
                    put<K, SPEC>(a, n, ob + a.col[4 * j], y);
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
                            const double2 y = make_double2(join<C::BIAS>(acc[2 * h], a.sh, ex[0]), join<C::BIAS>(acc[2 * h + 1], a.sh, ex[1]));
                            if (!SPEC || !((gm >> q) & 1u)) put<K, SPEC>(a, row, ob + a.amp[16 * mt + 8 * h], y);
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
                        for (int c = 0; c < 4; c++) re[c] = join<C::BIAS>(acc[c], a.sh, ex[c & 1]);
                        clear();
#pragma unroll
                        for (int s = 0; s < KS; s++) {
                            step(tu + C::TAB + s * kDigits * 32, br[s]);
                            step(tu + s * kDigits * 32, bi[s]);
                        }
#pragma unroll
                        for (int c = 0; c < 4; c++) {  // amplitudes n and n + 8 of groups q and q + 4
                            const int row = 16 * mt + 8 * (c >> 1) + n;
                            const double2 y = make_double2(re[c], join<C::BIAS>(acc[c], a.sh, ex[c & 1]));
                            if (!SPEC || !((gm >> (q + 4 * (c & 1))) & 1u))
                                put<K, SPEC>(a, row, ob + a.col[4 * (c & 1)] + a.amp[16 * mt + 8 * (c >> 1)], y);
                        }
                    }
                }
            }
        }
    }
}

// A few outputs of every group exchanged (launch_dense_f64_moves).
constexpr int kMaxMoves = 16;
struct MoveArgs {
    double2 *psi;
    long long groups;
    unsigned long long cmask;
    int nfix, count;
    int fix[kMaxFix];
    long long to[kMaxMoves], from[kMaxMoves];
};
__global__ void __launch_bounds__(256) move_kernel(const __grid_constant__ MoveArgs a) {
    for (long long t = blockIdx.x * 256ll + threadIdx.x; t < a.groups; t += gridDim.x * 256ll) {
        unsigned long long g = (unsigned long long)t;
        for (int i = 0; i < a.nfix; i++) {
            const int p = a.fix[i];
            g = ((g >> p) << (p + 1)) | (g & ((1ull << p) - 1ull));
        }
        double2 *p = a.psi + (g | a.cmask), y[kMaxMoves];
#pragma unroll
        for (int i = 0; i < kMaxMoves; i++)
            if (i < a.count) y[i] = p[a.from[i]];
#pragma unroll
        for (int i = 0; i < kMaxMoves; i++)
            if (i < a.count) p[a.to[i]] = y[i];
    }
}

// kernel width of a gate: at least 3 targets, 4 for a real U
static int width_of(const Op &op) {
    const int k = (int)op.targets.size();
    return k <= 3 ? 3 : k;
}
static bool real_form(const Op &op) { return op.real_u && op.targets.size() >= 4; }

// the matrix that is multiplied
static const std::vector<cd> &matrix(const Op &op) { return op.f64_U.empty() ? op.U : op.f64_U; }

template <int K, bool REALU>
static void pack_digits(const Op &op, int su, unsigned char *out) {
    using C = Cfg<K, REALU>;
    const int k = (int)op.targets.size(), D0 = 1 << k;
    unsigned short *o = reinterpret_cast<unsigned short *>(out);
    auto entry = [&](int r, int c) -> cd {  // group bits from k on: identity
        return (r >> k) == (c >> k) ? op.f64_left[(size_t)(r & (D0 - 1)) * D0 + (c & (D0 - 1))] : cd(0.0, 0.0);
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
    out += (size_t)tabs * C::TAB * 16;
    std::memcpy(out, op.f64_rows.data(), C::ROWS);
    dense_f64_pack_scales(op, out + C::ROWS);
}

template <int K, bool REALU, int TBITS, bool SPEC>
static void launch(const Args &a, int sms, cudaStream_t st) {
    using C = Cfg<K, REALU, TBITS>;
    auto kern = dense_f64_kernel<K, REALU, TBITS, SPEC>;
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
static unsigned long long diagonal_rows(const std::vector<cd> &U, int D) {
    unsigned long long diag = 0;
    for (int r = 0; r < D; r++) {
        bool d = true;
        for (int c = 0; c < D && d; c++)
            d = c == r || (U[(size_t)r * D + c] == cd(0.0, 0.0) && U[(size_t)c * D + r] == cd(0.0, 0.0));
        if (d) diag |= 1ull << r;
    }
    return diag;
}

// Gates of 1..6 targets with mostly nonzero rows.  A gate with a row of at most half its entries nonzero (diagonal
// rows and columns apart) stays in FP64 where the row form makes that cheap (sparse_width).  A gate that mixes such
// rows with full ones, a quarter of its entries nonzero at least, is a candidate all the same: the plain kernel would
// multiply all of its zeros (the eigenvectors of a grid that falls apart without its slack bus, 64 x 64 in blocks
// of 63 and 1: 30.8 ms in FP64 on 2^27 amplitudes).
static bool digit_candidate(const Op &op) {
    const int k = (int)op.targets.size();
    if (op.kind != OP_DENSE || k < 1 || k > 6) return false;
    const int D = 1 << k;
    const unsigned long long diag = diagonal_rows(op.U, D);
    int live = 0, all = 0;
    bool short_rows = false;
    for (int r = 0; r < D; r++) live += !((diag >> r) & 1ull);
    for (int r = 0; r < D; r++) {
        int nz = 0;
        for (int c = 0; c < D; c++) {
            const cd u = op.U[(size_t)r * D + c];
            if (!std::isfinite(u.real()) || !std::isfinite(u.imag())) return false;  // products of fused gates can overflow
            if (!((diag >> c) & 1ull)) nz += u != cd(0.0, 0.0);
        }
        if ((diag >> r) & 1ull) continue;
        short_rows = short_rows || 2 * nz <= live;
        all += nz;
    }
    return live > 0 && !(short_rows && (sparse_width(op) > 0 || 4 * all < live * live));
}

static double size_of(const cd &u) { return std::max(std::fabs(u.real()), std::fabs(u.imag())); }
static constexpr int kNoEntries = INT_MIN;

// The largest entry off (r, c) in its row and its column.
static double beside(const std::vector<cd> &U, int D, int r, int c) {
    double m = 0.0;
    for (int j = 0; j < D; j++) {
        if (j != c) m = std::max(m, size_of(U[(size_t)r * D + j]));
        if (j != r) m = std::max(m, size_of(U[(size_t)j * D + c]));
    }
    return m;
}

// Rows that hardly mix with the others: one entry, and beside it in its row and column only zeros or, from 4 targets on,
// values 2^7 times smaller (a bus without a line but to the slack bus: the eigensolver leaves 1e-17 and less there).
// That entry alone would set the scale of row and column, so it is multiplied in FP64 and the rest is scaled up (all
// entries on the diagonal of a gate close to the identity).  Off
// the diagonal it is brought there first: U = P U2 with such a row r of U as row c of U2; P moves a few outputs.
static void separate(Op &op) {
    const int k = (int)op.targets.size(), D = 1 << k;
    op.f64_U.clear();
    op.f64_moves.clear();
    op.f64_diag = 0;
    std::vector<int> at(D);  // row r of U is row at[r] of U2
    for (int r = 0; r < D; r++) at[r] = r;
    for (int r = 0; r < D; r++) {
        int c = 0;
        for (int j = 1; j < D; j++)
            if (size_of(op.U[(size_t)r * D + j]) > size_of(op.U[(size_t)r * D + c])) c = j;
        const double one = size_of(op.U[(size_t)r * D + c]), rest = beside(op.U, D, r, c);
        if (one == 0.0) {
            c = r;  // a row of zeros is one with its own column if that is zero too
            if (beside(op.U, D, r, r) != 0.0) continue;
        } else if (rest > (k >= 4 ? std::ldexp(one, -7) : 0.0)) {
            continue;
        }
        op.f64_diag |= 1ull << c;
        std::swap(at[r], *std::find(at.begin(), at.end(), c));
    }
    for (int r = 0; r < D; r++)
        if (at[r] != r) op.f64_moves.emplace_back(r, at[r]);
    if (op.f64_moves.empty()) return;
    op.f64_U.resize(op.U.size());
    for (int r = 0; r < D; r++) std::copy_n(op.U.begin() + (size_t)r * D, D, op.f64_U.begin() + (size_t)at[r] * D);
}

// Exponents that bring what is left of the separated rows and columns to the scale of the others (below 2^f64_su).
static bool scale(Op &op) {
    const int D = 1 << (int)op.targets.size();
    const std::vector<cd> &U = f64::matrix(op);
    auto own = [&](int r) { return (op.f64_diag >> r) & 1ull; };
    auto left = [&](int r, int c) { return r == c && own(r) ? 0.0 : size_of(U[(size_t)r * D + c]); };
    auto exponent = [](double v) {
        int e = 0;
        std::frexp(v, &e);  // v = f 2^e, f in [1/2, 1)
        return e;
    };
    double top = 0.0;
    for (int pass = 0; pass < 2 && top == 0.0; pass++)  // of the rows and columns that mix; of all when none does
        for (int r = 0; r < D; r++)
            for (int c = 0; c < D; c++)
                if (pass || (!own(r) && !own(c))) top = std::max(top, left(r, c));
    if (!(top > std::ldexp(1.0, -100) && top < std::ldexp(1.0, 100))) return false;
    op.f64_su = exponent(top);
    op.f64_row.assign(D, 0);
    op.f64_col.assign(D, 0);
    bool all = true;
    for (int r = 0; r < D; r++) all = all && own(r);
    // by the entries in the rows and columns that mix
    for (int i = 0; i < D; i++) {
        if (!own(i)) continue;
        double in_row = 0.0, in_col = 0.0;
        for (int j = 0; j < D; j++)
            if (all || !own(j)) in_row = std::max(in_row, left(i, j)), in_col = std::max(in_col, left(j, i));
        op.f64_row[i] = in_row == 0.0 ? kNoEntries : exponent(in_row) - op.f64_su;
        op.f64_col[i] = in_col == 0.0 ? kNoEntries : all ? 0 : exponent(in_col) - op.f64_su;
    }
    // an entry between two separated ones that is above both scales' product raises them alike
    for (int r = 0; r < D; r++)
        for (int c = 0; c < D; c++) {
            if (r == c || !own(r) || !own(c) || left(r, c) == 0.0) continue;
            int &er = op.f64_row[r], &ec = op.f64_col[c];
            const int e = exponent(left(r, c)) - op.f64_su;
            if (er == kNoEntries && ec == kNoEntries) ec = 0;
            if (er == kNoEntries) er = e - ec;
            else if (ec == kNoEntries) ec = e - er;
            else if (e > er + ec) {
                const int d = e - er - ec;
                er += d - d / 2;
                ec += d / 2;
            }
        }
    for (int i = 0; i < D; i++)  // far from 1: the products by these powers would leave the range of FP64
        if ((op.f64_row[i] != kNoEntries && std::abs(op.f64_row[i]) > 400) || (op.f64_col[i] != kNoEntries && std::abs(op.f64_col[i]) > 400))
            return false;
    return true;
}

unsigned long long dense_f64_beside(const Op &op) {
    unsigned long long m = 0;
    for (size_t i = 0; i < op.f64_row.size(); i++)
        if (((op.f64_diag >> i) & 1ull) && (op.f64_row[i] != kNoEntries || op.f64_col[i] != kNoEntries)) m |= 1ull << i;
    return m;
}

void dense_f64_pack_scales(const Op &op, unsigned char *out) {
    double *vw = reinterpret_cast<double *>(out);
    for (size_t i = 0; i < op.f64_row.size(); i++) {
        vw[2 * i] = op.f64_col[i] == kNoEntries ? 0.0 : std::ldexp(1.0, op.f64_col[i]);
        vw[2 * i + 1] = op.f64_row[i] == kNoEntries ? 0.0 : std::ldexp(1.0, op.f64_row[i]);
    }
}

// Whether and how a gate takes the digit form.  What is left out of a sum is relative to the group's scale (2^su times
// the power of two above its largest amplitude), an FP64 sum's error to its own terms: n products in any order are
// within n 2^-53 S of the exact value, S = sum |u_rc| |x_c| over the row.  The digit form keeps to the same bound:
//   - the last kept bit is 2^(sh - 68) of the scale, rounded; sh as kept_shift says, or as small as the largest row sum of U allows;
//   - the digit pairs left out, 7 per product and below 2^-62 of the scale each, add up like random numbers: 21.4
//     sqrt(7 n) units of 2^-68 in the mean square (digits spread evenly over -128..127); four times that is allowed for;
//   - so a row is safe while S >= (2^sh + 453 sqrt(n)) / n units of 2^-16 of the scale: thr, compared with a sum of
//     bytes that is never above S (f64_digits.cuh, rows_fit).  A row with an entry multiplied in FP64 is safe too
//     while that product alone bounds the error of the rest: from an exponent of its amplitude on (`from`).
// A group has an amplitude of 128 units at least, so a U without small entries is safe for every state (most Haar
// gates of up to 3 targets).  With others every group is tested, and one that fails runs in FP64 (up to 3 targets its
// tile).  The four lanes that hold a group look at their own largest amplitudes first: with one of 2^(7 - reach) units
// in each, whichever columns they are in, a row has at least its smallest entry of every lane's columns times that.  A
// gate with rows that fail even where all amplitudes are within a factor of two of each other stays in FP64 as a whole.
bool dense_f64_plan(Op &op) {
    if (!digit_candidate(op)) return false;
    const int k = (int)op.targets.size(), D = 1 << k;
    separate(op);
    if (op.f64_moves.size() > f64::kMaxMoves || !scale(op)) return false;
    op.f64_left = f64::matrix(op);  // as it is split into digits
    double sum = 0.0;
    for (int r = 0; r < D; r++) {
        double s = 0.0;
        for (int c = 0; c < D; c++) {
            cd &u = op.f64_left[(size_t)r * D + c];
            if (r == c && ((op.f64_diag >> r) & 1ull)) u = 0.0;
            const int er = op.f64_row[r], ec = op.f64_col[c];
            if ((er != 0 || ec != 0) && u != cd(0.0, 0.0)) u = cd(std::ldexp(u.real(), -er - ec), std::ldexp(u.imag(), -er - ec));
            s += std::fabs(u.real()) + std::fabs(u.imag());
        }
        sum = std::max(sum, s);
    }
    const int RED = op.real_u && k >= 4 ? D : 2 * std::max(D, 8);
    op.f64_sh = f64::kept_shift(RED);
    if (RED > 32) op.f64_sh = std::min(op.f64_sh, std::max(7, 6 + (int)std::ceil(std::log2(std::ldexp(sum, -op.f64_su)))));
    op.f64_check = false;
    op.f64_reach = 3;
    const int DK = std::max(D, 8);  // of the kernel: below 3 targets the group bits from k on are rows too
    op.f64_rows.assign(f64::rows_bytes(DK), 0);
    unsigned *at = reinterpret_cast<unsigned *>(op.f64_rows.data() + DK * DK);
    int *from = reinterpret_cast<int *>(at + DK);
    const double units = std::ldexp(1.0, 8 - op.f64_su);
    for (int r = 0; r < D; r++) {
        if (op.f64_row[r] == kNoEntries) continue;
        int nz = 0;
        unsigned least = 255, even = 0;
        unsigned lane[4] = {255, 255, 255, 255};
        for (int c = 0; c < D; c++) {
            if (op.f64_col[c] == kNoEntries) continue;
            const cd u = op.f64_left[(size_t)r * D + c];
            const unsigned b = (unsigned)(size_of(u) * units);
            if (k >= 4) op.f64_rows[(size_t)r * D + (c & 3) * (D / 4) + (c >> 2)] = (unsigned char)b;
            for (int g = 0; k <= 3 && g < 8; g += D) op.f64_rows[(size_t)(g + r) * 8 + g + c] = (unsigned char)b;
            nz += u != cd(0.0, 0.0);
            least = std::min(least, b);
            even += 64 * b;
            lane[c & 3] = std::min(lane[c & 3], b);
        }
        const double n = std::max(1, op.real_u ? nz : 2 * nz), lost = std::ldexp(1.0, op.f64_sh) + 453.0 * std::sqrt(n);
        const unsigned thr = (unsigned)std::ceil(lost / n);
        if (k >= 4) at[(r & 3) * (D / 4) + (r >> 2)] = thr;
        for (int g = 0; k <= 3 && g < 8; g += D) at[g + r] = thr;
        op.f64_check = op.f64_check || 128 * least < thr;
        while (op.f64_reach > 0 && (lane[0] + lane[1] + lane[2] + lane[3]) << (7 - op.f64_reach) < thr) op.f64_reach--;
        const bool own = (op.f64_diag >> r) & 1ull;
        if (!own && even < thr) return false;
        // |u_rr x_r| n 2^-53 >= (lost / 2) 2^-68 2^(su + 1) 2^E 2^row, x_r = (the scaled amplitude) 2^-col
        if (own)
            from[r] = (int)std::ceil(std::log2(lost / n / size_of(f64::matrix(op)[(size_t)r * D + r])) - 15.0) + op.f64_su + op.f64_row[r] +
                      (op.f64_col[r] == kNoEntries ? 0 : op.f64_col[r]);
    }
    if (op.f64_reach == 0) op.f64_reach = -1;  // no such rule: never reached
    return true;
}

size_t dense_f64_blob_bytes(const Op &op) {
    size_t n = 0;
#define QSIM_F64_BYTES(K, R) \
    n = (size_t)f64::Cfg<K, R>::TAB * 16 * (f64::Cfg<K, R>::TABS == 3 ? 2 : 1) + f64::Cfg<K, R>::ROWS
    QSIM_F64_SWITCH(op, QSIM_F64_BYTES)
#undef QSIM_F64_BYTES
    return n + 16 * op.f64_row.size();
}

void dense_f64_pack(const Op &op, unsigned char *out) {
#define QSIM_F64_PACK(K, R) f64::pack_digits<K, R>(op, op.f64_su, out)
    QSIM_F64_SWITCH(op, QSIM_F64_PACK)
#undef QSIM_F64_PACK
}

// Outputs of a group to their places: y[r] = y2[s] for the pairs (r, s) of f64_moves, a thread per group.
void launch_dense_f64_moves(void *state, int n, const Op &op, int sms, cudaStream_t st) {
    f64::MoveArgs a;
    std::memset(&a, 0, sizeof(a));
    a.psi = static_cast<double2 *>(state);
    std::vector<int> fix(op.targets);
    for (int q : op.controls) {
        fix.push_back(q);
        a.cmask |= 1ull << q;
    }
    std::sort(fix.begin(), fix.end());
    QSIM_REQUIRE((int)fix.size() <= f64::kMaxFix, "too many fixed qubits");
    a.groups = 1ll << (n - (int)fix.size());
    a.nfix = (int)fix.size();
    for (int i = 0; i < a.nfix; i++) a.fix[i] = fix[i];
    a.count = (int)op.f64_moves.size();
    for (int i = 0; i < a.count; i++)
        for (size_t b = 0; b < op.targets.size(); b++) {
            a.to[i] |= (long long)((op.f64_moves[i].first >> b) & 1) << op.targets[b];
            a.from[i] |= (long long)((op.f64_moves[i].second >> b) & 1) << op.targets[b];
        }
    const long long grid = std::min<long long>((a.groups + 255) / 256, (long long)sms * 8);
    f64::move_kernel<<<(int)grid, 256, 0, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("move_kernel: ") + cudaGetErrorString(e));
    note_launches(1, QSIM_KERNEL_DENSE_SIMT);
}

// Returns false when the state is too small for the kernel's tiles, or for a real 1-target gate (Hadamard, RY) on 2^18
// amplitudes or more: its 2 multiply-adds a real cost FP64 less than splitting and joining cost here (25 qubits 260 us
// there, 288 here; 27 qubits 1000, 1115; 18 qubits 9.8, 11.4; below, 16 qubits, 9.9, 8.8).  The plain kernels take both.
bool launch_dense_f64(void *state, int n, const Op &op, const void *dig, const void *Ut, int sms, cudaStream_t st) {
    const int k = (int)op.targets.size(), K = f64::width_of(op);
    if (k == 1 && op.real_u && n - (int)op.controls.size() >= 18) return false;
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
    a.vw = reinterpret_cast<const double2 *>(static_cast<const unsigned char *>(dig) + dense_f64_blob_bytes(op) - 16 * op.f64_row.size());
    a.ntasks = 1ll << ((int)fr.size() - inside);
    a.cmask = cmask;
    a.su = op.f64_su;
    a.sh = op.f64_sh;
    a.check = op.f64_check ? 1 : 0;
    a.reach = op.f64_reach;
    a.k = k;
    a.real_u = op.real_u ? 1 : 0;
    for (int r = 0; r < (1 << K); r++)
        if ((op.f64_diag >> (r & ((1 << k) - 1))) & 1ull) a.diag |= 1ull << r;
    a.beside = dense_f64_beside(op);
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
        const bool spec = a.diag || a.check;                                                    \
        if (tb && spec) f64::launch<KK, R, f64::Cfg<KK, R>::TBMAX, true>(a, sms, st);           \
        else if (tb) f64::launch<KK, R, f64::Cfg<KK, R>::TBMAX, false>(a, sms, st);             \
        else if (spec) f64::launch<KK, R, 0, true>(a, sms, st);                                 \
        else f64::launch<KK, R, 0, false>(a, sms, st);                                          \
    } while (0)
    QSIM_F64_SWITCH(op, QSIM_F64_LAUNCH)
#undef QSIM_F64_LAUNCH
    return true;
}

}  // namespace qsim
