// Wide complex128 gates as exact digit products on the 5th-generation tensor cores (sm_103a):
// tcgen05.mma kind::f16, eight FP32 accumulators per output in tensor memory.
//
// The digits and sums are dense_f64.cu's (see there for the split and its error).  Its warp-level MMAs run at
// 1024 products per clock and SM, which bounds gates of 4 targets and more (36 2^(k+1) products a real);
// tcgen05 runs four times as fast, and the accumulators leave the registers.
//
// A tile is 128 rows: 128 groups of a complex gate of 4 or 5 targets (a row holds the group's reals), or 64
// groups times {re, im} of a 6-target gate.  Digit i of the rows is one MMA operand (A, 128 x 16 per K-step), and
// the digits 0..7-i of U, stacked along N, are the other one: with accumulator t for the digit pairs i + j = t in
// columns 32 t .. 32 t + 31, one MMA of N = 32 (8 - i) columns adds digit i's products with all of them to
// accumulators i..7, and a K-step is 8 MMAs.  A unit is 32 output reals of a row, 256 columns; two units
// alternate, so the sums of one are put together while the MMAs fill the other.
//   4 targets            K = 32 reals,  1 unit
//   5 targets            K = 64,        2 units (the rows' digits stay in shared memory for the second)
//   6 targets, real U    K = 64,        2 units (rows (group, re or im))
//   6 targets            K = 128: the row's own part times Re U, then the other part (negated for re) times
//                        Im U; 2 units at once (U's digits leave room for two K-steps only)
//
// 17 warps: 8 load amplitudes (each thread 8 or 16 of them, the next tile's into the same registers as they are
// used up), write their digits to a ring of K-steps and release it; one lane issues the MMAs; 8 read finished
// units, put the sums together, and pass the amplitudes through shared memory so that a warp's store covers
// 4 amplitudes of 8 groups (the lowest targets and free qubits: whole lines).  Roles meet at mbarriers only,
// every wait is bounded, tensor memory is freed after the last MMA has completed (as in dense_tc.cu).
// Groups outside the fixed-point range, or whose sums would lose more than an FP64 sum (dense_f64_plan), are marked and
// computed in FP64 by the reading warps (plain_groups).
//
// 26 qubits, dense_f64.cu's form -> this one, TB/s: 4 targets 2.42 -> 3.54, 5 1.40 -> 2.9, 6 0.77 -> 1.63, 6 with a real U
// 1.57 -> 2.8.  What bounds it: issue slots for splitting and joining the digits (0.59 instructions a clock and
// scheduler at 4 targets, 0.50 at 5; the tensor pipe at 21 to 39 %); at 6 complex targets the MMAs and the joining take turns, as tensor
// memory holds one tile's two units and no more.  The FP64 pipe is at 17 to 37 %: its last
// conversion only, apart from rows with an entry left to FP64, which have a function of their own (with them in the
// main path the pipe was 69 % busy).  Testing the groups of an eigenvector matrix with many small entries, and marking
// them one by one, costs a 27-qubit solve 13.27 -> 13.67 ms (with tiles marked as a whole some systems took 17 ms and more).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.h"
#include "f64_digits.cuh"
#include "tc_ptx.cuh"

namespace qsim {

__device__ unsigned int g_f64_error = 0;

namespace f64tc {

using namespace f64;
using namespace tc;

constexpr int kMaxFix = 40;
constexpr int kProdWarps = 8, kEpiWarps = 8, kMmaWarp = kProdWarps + kEpiWarps;
constexpr int kThreads = (kMmaWarp + 4) * 32;  // the issuing warp's group of four is filled up for setmaxnreg
// registers a thread: launched with 96 (640 threads), 61440 in all; 256 x 112 + 256 x 96 + 128 x 64 = 61440 after the split.
// The reading warps keep the 96 that a function they call may use (with 80 for them and 128 for the loading ones: 4, 5, 6
// real, 6 targets at 25 qubits 308 356 391 670 us instead of 289 345 384 674).
constexpr int kProdRegs = 112, kEpiRegs = 96, kMmaRegs = 64;
constexpr int kSlot = kDigits * 4096;  // one K-step of a tile: 8 digits x 128 rows x 16 FP16
constexpr int kBlock = 8192;           // U's digits of one unit and K-step: 256 rows x 16 FP16
// Slots of what the loading warps tell the reading ones about a tile (exponents, marked groups).  Tile t is written once
// its first K-step has a ring slot, so the MMAs of the K-step SLOTS before it are complete, and they had waited for
// the unit two before theirs to be read: tile t - 4 with 4 targets (2 tiles in the ring, 2 in tensor memory), tile
// t - 2 in the other modes.  Every earlier tile has been read when slot t mod 4 is written.
constexpr int kTiles = 4;

enum Mode { C4 = 0, C5 = 1, R6 = 2, C6 = 3 };

template <int MODE>
struct Cfg {
    static constexpr int K = MODE == C4 ? 4 : MODE == C5 ? 5 : 6, D = 1 << K;
    static constexpr bool PARTS = MODE >= R6;             // rows are (group, re or im)
    static constexpr int GB = PARTS ? 6 : 7;              // group bits of a tile
    static constexpr int KS = MODE == C4 ? 2 : MODE == C6 ? 8 : 4;  // K-steps
    static constexpr int UNITS = MODE == C4 ? 1 : 2;
    static constexpr int SLOTS = MODE == C6 ? 2 : 4;
    static constexpr int ITEMS = PARTS ? 1 : 2;           // rows per loading thread
    static constexpr int EPT = MODE == C4 ? 4 : MODE == C5 ? 8 : 16;  // amplitudes per item: every fourth
    static constexpr int STEP = PARTS ? 4 : 2;            // amplitudes per item and K-step
    static constexpr int RED = MODE == C4 ? 32 : MODE == C6 ? 128 : 64;
    static constexpr int BIAS = RED <= 32 ? kept_shift(RED) : 0;
    static constexpr int BBYTES = UNITS * KS * kBlock;
    static constexpr int STAGE = kEpiWarps * 2048;
    static constexpr int ROWS = rows_bytes(D);
    static constexpr int SMEM = BBYTES + SLOTS * kSlot + STAGE + ROWS + kTiles * (128 * 4 + 8 * ITEMS) + 8 * (2 * SLOTS + 5) + 16;
};

struct Args {
    double2 *psi;
    const uint4 *dig;
    const double2 *Ut;
    const double2 *vw;  // as in dense_f64.cu
    long long ntiles;
    unsigned long long cmask, diag, beside;
    int su, sh, check, reach, nfix;  // as in dense_f64.cu
    int fix[kMaxFix];   // ascending: targets, controls, group bits inside a tile
    long long amp[64];  // offset (in amplitudes) of amplitude a of a group
    long long grp[7];   // ... of group bit b of a tile
};

__device__ __forceinline__ void mma_f16(unsigned d, uint64_t adesc, uint64_t bdesc, unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tmem_ld4(unsigned addr, float (&v)[4]) {
    unsigned r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
#pragma unroll
    for (int i = 0; i < 4; i++) v[i] = __uint_as_float(r[i]);
}

// The marked groups of a tile, in FP64: a warp takes every eighth (with 4 targets every eighth pair) and stores a group
// when all of its outputs are computed.  A lane has rows lane and lane + 32 and loads those amplitudes; U's columns come in
// the plain kernels' order, the column's amplitude from its lane.
template <int MODE>
__device__ __noinline__ void plain_groups(const Args &a, double2 *base, uint64_t m0, uint64_t m1, int ew, int lane) {
    using C = Cfg<MODE>;
    constexpr int D = C::D, L = D < 32 ? D : 32, ROWS = D / L;  // lanes per group, rows per lane
    int n = (32 / L) * ew + lane / L, r = lane % L;  // the warp's next mark, counted over the tile
    for (int w = 0; w < C::ITEMS; w++) {
        const uint64_t m = w ? m1 : m0;
        const int left = __popcll(m);
        while (__any_sync(~0u, n < left)) {
            const bool mine = n < left;
            uint64_t k = m;
            for (int i = 0; i < n && mine; i++) k &= k - 1;  // the n-th set bit
            const int g = 64 * w + (mine ? __ffsll((long long)k) - 1 : 0);
            double2 *p = base, x[ROWS], y[ROWS];
            for (int b = 0; b < C::GB; b++)
                if ((g >> b) & 1) p += a.grp[b];
#pragma unroll
            for (int o = 0; o < ROWS; o++) {
                x[o] = mine ? p[a.amp[r + 32 * o]] : make_double2(0.0, 0.0);
                y[o] = make_double2(0.0, 0.0);
            }
#pragma unroll
            for (int h = 0; h < ROWS; h++)
#pragma unroll 4
                for (int c = 0; c < L; c++) {  // amplitude c + 32 h, from its lane
                    const double zx = __shfl_sync(~0u, x[h].x, c, L), zy = __shfl_sync(~0u, x[h].y, c, L);
#pragma unroll
                    for (int o = 0; o < ROWS; o++) {
                        const double2 *w = a.Ut + (c + 32 * h) * D + r + 32 * o;
                        const double2 u = MODE == R6 ? make_double2(__ldg(&w->x), 0.0) : __ldg(w);
                        y[o].x = fma(u.x, zx, y[o].x);
                        if (MODE != R6) y[o].x = fma(-u.y, zy, y[o].x);
                        y[o].y = fma(u.x, zy, y[o].y);
                        if (MODE != R6) y[o].y = fma(u.y, zx, y[o].y);
                    }
                }
            __syncwarp();
            if (mine)
#pragma unroll
                for (int o = 0; o < ROWS; o++) p[a.amp[r + 32 * o]] = y[o];
            if (mine) n += kEpiWarps * (32 / L);
        }
        n -= left;
    }
}

// Where a diagonal entry is left to FP64: the sum z of the rest plus its product with the value at p.
template <int MODE>
__device__ __noinline__ double2 scaled_row(const Args &a, int row, const double2 *p, double2 z) {
    const double2 w = __ldg(a.Ut + row * Cfg<MODE>::D + row), o = *p;
    const double rest = (a.beside >> row) & 1ull ? __ldg(a.vw + row).y : 0.0;
    z.x = fma(w.x, o.x, rest * z.x);
    z.y = fma(w.x, o.y, rest * z.y);
    if (MODE != R6) {
        z.x = fma(-w.y, o.y, z.x);
        z.y = fma(w.y, o.x, z.y);
    }
    return z;
}
// The amplitudes of 8 columns from the warp's stage to their places: lane (4 lowest amplitudes, 8 groups).  SPEC: some
// rows have a diagonal entry left to FP64, or some of the warp's groups (bits of skip) are not stored here.
template <int MODE, bool SPEC>
__device__ __forceinline__ void store_body(const Args &a, const unsigned char *st, double2 *at, int h, int s, int lane, unsigned skip) {
    using C = Cfg<MODE>;
    const int sa = lane & 3, sr = lane >> 2;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        double2 z, *p = at;
        int row;
        if (SPEC && ((skip >> (8 * (C::PARTS ? i & 1 : i) + sr)) & 1u)) continue;
        if (C::PARTS) {
            const int g = 8 * (i & 1) + sr, c = sa + 4 * (i >> 1);
            z = *reinterpret_cast<const double2 *>(st + g * 128 + ((c ^ (g & 7)) * 16));
            row = 32 * h + 8 * s + c;
            p += ((i & 1) ? a.grp[3] : 0) + a.amp[32 * h + 8 * s + 4 * (i >> 1)];
        } else {
            const int r = 8 * i + sr;
            z = *reinterpret_cast<const double2 *>(st + r * 64 + ((sa ^ ((r >> 1) & 3)) * 16));
            row = 16 * h + 4 * s + sa;
            p += ((i & 1) ? a.grp[3] : 0) + ((i & 2) ? a.grp[4] : 0) + a.amp[16 * h + 4 * s];
        }
        if (SPEC && ((a.diag >> row) & 1ull)) z = scaled_row<MODE>(a, row, p, z);
        __stcs(p, z);
    }
}
template <int MODE>
__device__ __noinline__ void store_spec(const Args &a, const unsigned char *st, double2 *at, int h, int s, int lane, unsigned skip) {
    store_body<MODE, true>(a, st, at, h, s, lane, skip);
}

// SPEC: gates with diagonal entries multiplied in FP64, or whose groups are tested (as instructions of the one kernel that
// others pass by, 23 qubits: 4, 5, 6 real, 6 targets 87 106 111 185 us, without them 84 102 102 181).
template <int MODE, bool SPEC>
__global__ void __launch_bounds__(kThreads, 1) dense_f64_tc_kernel(const __grid_constant__ Args a) {
    using C = Cfg<MODE>;
    constexpr int KS = C::KS, SLOTS = C::SLOTS, ITEMS = C::ITEMS, EPT = C::EPT, STEP = C::STEP, UNITS = C::UNITS;
    constexpr bool PARTS = C::PARTS;
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *ring = sm + C::BBYTES;
    unsigned char *stage = ring + SLOTS * kSlot;
    unsigned char *rows = stage + C::STAGE;                        // bytes and thresholds of U's rows
    int *exps = reinterpret_cast<int *>(rows + C::ROWS);           // [kTiles][128 rows]
    uint64_t *marks = reinterpret_cast<uint64_t *>(exps + kTiles * 128);  // [kTiles][ITEMS], a bit per group: in FP64
    uint64_t *full = marks + kTiles * ITEMS;
    uint64_t *empty = full + SLOTS, *accfull = empty + SLOTS, *accempty = accfull + 2, *drain = accempty + 2;
    unsigned *tslot = reinterpret_cast<unsigned *>(drain + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < C::BBYTES / 16 + (SPEC && a.check ? C::ROWS / 16 : 0); i += kThreads)
        reinterpret_cast<uint4 *>(i < C::BBYTES / 16 ? sm : rows - C::BBYTES)[i] = a.dig[i];
    if (tid == 0) {
        for (int i = 0; i < SLOTS; i++) {
            mbar_init(&full[i], kProdWarps);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&accfull[i], 1);
            mbar_init(&accempty[i], kEpiWarps);
        }
        mbar_init(drain, 1);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = *tslot;
    const long long first = blockIdx.x, stride = gridDim.x;
    const long long ntl = first < a.ntiles ? (a.ntiles - first + stride - 1) / stride : 0;
    bool failed = false;
    auto tile_base = [&](long long i) -> double2 * {
        return a.psi + (insert_zeros((unsigned long long)(first + i * stride), a.fix, a.nfix) | a.cmask);
    };

    if (warp < kProdWarps) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kProdRegs));
        // ------------------------------------------------------------------ loads and digits
        // Lane (r8, kc): row (group) 8 warp + r8 of every item, amplitudes kc + 4 e.  A load covers the 4 lowest
        // amplitudes of 8 neighbouring groups.  K position of a thread's reals in a K-step: 4 kc ..
        const int r8 = lane & 7, kc = lane >> 3;
        long long off = a.amp[kc];
#pragma unroll
        for (int b = 0; b < 3; b++)
            if ((r8 >> b) & 1) off += a.grp[b];
#pragma unroll
        for (int b = 0; b < 3; b++)
            if ((warp >> b) & 1) off += a.grp[3 + b];
        double2 x[ITEMS][EPT];
        {
            const double2 *p = tile_base(0) + off;
#pragma unroll
            for (int it = 0; it < ITEMS; it++)
#pragma unroll
                for (int e = 0; e < EPT; e++)
                    if (ntl > 0) x[it][e] = __ldcs(p + (it ? a.grp[6] : 0) + a.amp[4 * e]);
        }
        const unsigned col = (unsigned)((kc >> 1) * 128 + (kc & 1) * 8);
        for (long long t = 0; t < ntl && !failed; t++) {
            int Er[ITEMS], Ei[ITEMS];
            bool out[ITEMS] = {};  // the group is outside the fixed-point range, or its sums would lose too much
            if (SPEC && a.diag) {  // amplitudes with a diagonal entry of their own: scaled to what else is in their column, or 0
                const unsigned long long mine = a.diag >> kc;
#pragma unroll
                for (int it = 0; it < ITEMS; it++)
#pragma unroll
                    for (int e = 0; e < EPT; e++)
                        if ((mine >> (4 * e)) & 1ull) {
                            out[it] |= max(mag_bits(x[it][e].x), mag_bits(x[it][e].y)) >= 0x7ff00000u;
                            if ((a.beside >> (kc + 4 * e)) & 1ull) {
                                const double v = __ldg(a.vw + kc + 4 * e).x;
                                x[it][e] = make_double2(x[it][e].x * v, x[it][e].y * v);
                            } else {
                                x[it][e] = make_double2(0.0, 0.0);
                            }
                        }
            }
#pragma unroll
            for (int it = 0; it < ITEMS; it++) {
                unsigned mr = 0, mi = 0, low = 0;
#pragma unroll
                for (int e = 0; e < EPT; e++) {
                    mr = max(mr, mag_bits(x[it][e].x));
                    mi = max(mi, mag_bits(x[it][e].y));
                }
                const unsigned ml = max(mr, mi);
                if (MODE != R6) mr = mi = ml;  // one exponent for both parts where they mix
                mr = max(mr, __shfl_xor_sync(~0u, mr, 8));
                mr = max(mr, __shfl_xor_sync(~0u, mr, 16));
                if (MODE == R6) {
                    mi = max(mi, __shfl_xor_sync(~0u, mi, 8));
                    mi = max(mi, __shfl_xor_sync(~0u, mi, 16));
                } else {
                    mi = mr;
                }
                Er[it] = mr ? (int)(mr >> 20) : 1023;
                Ei[it] = mi ? (int)(mi >> 20) : 1023;
                if (mr == 0 || mi == 0)  // all zero, or denormals whose high words are 0
#pragma unroll
                    for (int e = 0; e < EPT; e++) {
                        if (!mag_bits(x[it][e].x)) low |= (unsigned)__double2loint(x[it][e].x);
                        if (!mag_bits(x[it][e].y)) low |= (unsigned)__double2loint(x[it][e].y);
                    }
                out[it] |= Er[it] < kMinExp || Er[it] > kMaxExp || Ei[it] < kMinExp || Ei[it] > kMaxExp || low;
                if (SPEC && a.check) {  // by the larger part of an amplitude
                    const int E = PARTS ? max(mr ? Er[it] : 0, mi ? Ei[it] : 0) : Er[it];
                    const bool zero = mr == 0 && mi == 0;
                    if (!__all_sync(~0u, (int)(ml >> 20) >= E - a.reach || zero)) {
                        unsigned m[EPT];
#pragma unroll
                        for (int e = 0; e < EPT; e++) m[e] = max(mag_bits(x[it][e].x), mag_bits(x[it][e].y));
                        out[it] |= !rows_fit_of<C::D, 8, 16>(m, E, zero, kc, a.diag, rows);
                    }
                }
            }
            unsigned char mark[ITEMS];  // of the warp's 8 groups
#pragma unroll
            for (int it = 0; it < ITEMS; it++) {
                unsigned m = __ballot_sync(~0u, out[it]);
                m |= m >> 16;
                mark[it] = (unsigned char)(m | m >> 8);
            }
            auto post = [&] {  // after the wait for the tile's first ring slot (see kTiles)
                int *ex = exps + (t % kTiles) * 128;
                if (kc == 0) {
#pragma unroll
                    for (int it = 0; it < ITEMS; it++) {
                        if (PARTS) {
                            ex[2 * (8 * warp + r8)] = Er[it];
                            ex[2 * (8 * warp + r8) + 1] = Ei[it];
                        } else {
                            ex[64 * it + 8 * warp + r8] = Er[it];
                        }
                    }
                }
                if (lane == 0)
#pragma unroll
                    for (int it = 0; it < ITEMS; it++)
                        reinterpret_cast<unsigned char *>(marks + (t % kTiles) * ITEMS + it)[warp] = mark[it];
            };
            const bool more = t + 1 < ntl;
            const double2 *np = tile_base(more ? t + 1 : t) + off;
#pragma unroll
            for (int s = 0; s < EPT / STEP; s++) {
                constexpr int PER = MODE == C6 ? 2 : 1;  // slots per step
                const long long q0 = (t * (EPT / STEP) + s) * PER;
                auto wait_slot = [&](long long q) {  // the warp gives up together
                    const bool ok = q < SLOTS || mbar_wait(&empty[q % SLOTS], (unsigned)((q / SLOTS - 1) & 1));
                    if (!__all_sync(~0u, ok)) failed = true;
                };
                wait_slot(q0);
                if (failed) break;
                if (s == 0) post();
                unsigned char *sl = ring + (q0 % SLOTS) * kSlot + col;
                unsigned re[2][kDigits], im[2][kDigits];
#pragma unroll
                for (int it = 0; it < ITEMS; it++) {
                    if constexpr (PARTS) {
                        const double2 *v = x[it] + STEP * s;
                        digit_pairs(fixed_bytes(v[0].x, Er[it]), fixed_bytes(v[1].x, Er[it]), re[0]);
                        digit_pairs(fixed_bytes(v[2].x, Er[it]), fixed_bytes(v[3].x, Er[it]), re[1]);
                        digit_pairs(fixed_bytes(v[0].y, Ei[it]), fixed_bytes(v[1].y, Ei[it]), im[0]);
                        digit_pairs(fixed_bytes(v[2].y, Ei[it]), fixed_bytes(v[3].y, Ei[it]), im[1]);
                        const int g = 8 * warp + r8;
                        // rows 2 g and 2 g + 1, the order alternating so that 16 lanes fill distinct banks
                        const int r0 = 2 * g + (r8 >> 2), r1 = r0 ^ 1;
                        const unsigned o0 = (r0 >> 3) * 256 + (r0 & 7) * 16, o1 = (r1 >> 3) * 256 + (r1 & 7) * 16;
#pragma unroll
                        for (int d = 0; d < kDigits; d++) {
                            const uint2 vr = make_uint2(re[0][d], re[1][d]), vi = make_uint2(im[0][d], im[1][d]);
                            *reinterpret_cast<uint2 *>(sl + d * 4096 + o0) = (r8 >> 2) ? vi : vr;
                            *reinterpret_cast<uint2 *>(sl + d * 4096 + o1) = (r8 >> 2) ? vr : vi;
                        }
                        if constexpr (MODE == C6) {
                            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&full[q0 % SLOTS]);
                            wait_slot(q0 + 1);
                            sl = ring + ((q0 + 1) % SLOTS) * kSlot + col;
#pragma unroll
                            for (int d = 0; d < kDigits; d++) {  // -im in the re row, re in the im row
                                const uint2 vr = make_uint2(im[0][d] ^ 0x80008000u, im[1][d] ^ 0x80008000u);
                                const uint2 vi = make_uint2(re[0][d], re[1][d]);
                                *reinterpret_cast<uint2 *>(sl + d * 4096 + o0) = (r8 >> 2) ? vi : vr;
                                *reinterpret_cast<uint2 *>(sl + d * 4096 + o1) = (r8 >> 2) ? vr : vi;
                            }
                        }
                    } else {
                        const double2 *v = x[it] + STEP * s;
                        digit_pairs(fixed_bytes(v[0].x, Er[it]), fixed_bytes(v[0].y, Er[it]), re[0]);
                        digit_pairs(fixed_bytes(v[1].x, Er[it]), fixed_bytes(v[1].y, Er[it]), re[1]);
                        const int row = 64 * it + 8 * warp + r8;
                        unsigned char *p = sl + (row >> 3) * 256 + (row & 7) * 16;
#pragma unroll
                        for (int d = 0; d < kDigits; d++)
                            *reinterpret_cast<uint2 *>(p + d * 4096) = make_uint2(re[0][d], re[1][d]);
                    }
                    if (more)
#pragma unroll
                        for (int e = STEP * s; e < STEP * s + STEP; e++)
                            x[it][e] = __ldcs(np + (it ? a.grp[6] : 0) + a.amp[4 * e]);
                }
                if (failed) break;
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[(q0 + PER - 1) % SLOTS]);
            }
        }
    } else if (warp < kMmaWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kEpiRegs));
        // ------------------------------------------------------------------ sums and stores
        const int ew = warp - kProdWarps, sub = ew & 3;  // TMEM lanes 32 sub .. (warp mod 4 == sub)
        const int m = 32 * sub + lane;                   // row
        unsigned char *st = stage + ew * 2048;
        // place in a store: 4 lowest amplitudes x 8 groups
        const int sa = lane & 3, sr = lane >> 2;
        long long off = a.amp[sa];
#pragma unroll
        for (int b = 0; b < 3; b++)
            if ((sr >> b) & 1) off += a.grp[b];
        off += (sub & 1) ? a.grp[PARTS ? 4 : 5] : 0;
        off += (sub & 2) ? a.grp[PARTS ? 5 : 6] : 0;
        for (long long u = 0; u < ntl * UNITS && !failed; u++) {
            const long long t = u / UNITS;
            const int h = (int)(u % UNITS), ab = (int)(u & 1);
            bool ok = mbar_wait(&accfull[ab], (unsigned)((u >> 1) & 1));
            ok = __all_sync(~0u, ok);
            if (!ok) {
                failed = true;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            double2 *base = tile_base(t);
            const int ex = exps[(t % kTiles) * 128 + m] - 1022 + a.su - 68 + a.sh;
            const uint64_t *mt = marks + (t % kTiles) * ITEMS;
            const uint64_t m0 = mt[0], m1 = ITEMS > 1 ? mt[ITEMS - 1] : 0;
            const unsigned skip = PARTS ? (unsigned)(m0 >> (16 * sub)) & 0xffffu : (unsigned)((sub < 2 ? m0 : m1) >> (32 * (sub & 1)));
            const unsigned acc = tmem + (unsigned)(ab * 256) + ((unsigned)(32 * sub) << 16);
            if (skip != (PARTS ? 0xffffu : ~0u)) {
#pragma unroll 1
                for (int s = 2 * (ew >> 2); s < 2 * (ew >> 2) + 2; s++) {  // columns 8 s .. 8 s + 7 of the unit
                    __syncwarp();  // the previous step's amplitudes have been read
#pragma unroll
                    for (int c4 = 0; c4 < 8; c4 += 4) {  // four columns at a time: 32 registers of sums
                        float v[kDigits][4];
#pragma unroll
                        for (int d = 0; d < kDigits; d++) tmem_ld4(acc + (unsigned)(32 * d + 8 * s + c4), v[d]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                        double y[4];
#pragma unroll
                        for (int c = 0; c < 4; c++) {
                            float w[kDigits];
#pragma unroll
                            for (int d = 0; d < kDigits; d++) w[d] = C::BIAS > 0 ? v[d][c] + kBiasF : v[d][c];
                            y[c] = join<C::BIAS>(w, a.sh, ex);
                        }
                        if (PARTS) {  // row (group, part): parts of 8 amplitudes
                            const int g = lane >> 1;
#pragma unroll
                            for (int c = 0; c < 4; c++)
                                *reinterpret_cast<double *>(st + g * 128 + (((c4 + c) ^ (g & 7)) * 16) + (lane & 1) * 8) = y[c];
                        } else {      // row: 4 amplitudes
#pragma unroll
                            for (int c = 0; c < 2; c++)
                                *reinterpret_cast<double2 *>(st + lane * 64 + (((c4 / 2 + c) ^ ((lane >> 1) & 3)) * 16)) =
                                    make_double2(y[2 * c], y[2 * c + 1]);
                        }
                    }
                    __syncwarp();
                    // a function of its own: with the FP64 products as a condition here the FP64 pipe was 69 % busy
                    if ((SPEC && a.diag) || skip) store_spec<MODE>(a, st, base + off, h, s, lane, skip);
                    else store_body<MODE, false>(a, st, base + off, h, s, lane, 0u);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&accempty[ab]);
            // behind the release, by another warp first for every tile: the FP64 pipe of one scheduler takes 9 us for a group
            // of 6 targets with a real U, and the other warps and the MMAs go on meanwhile
            if (h == UNITS - 1 && (m0 | m1) != 0) plain_groups<MODE>(a, base, m0, m1, (int)((ew - t) & (kEpiWarps - 1)), lane);
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kMmaRegs));
        if (warp == kMmaWarp && lane == 0) {
        // ------------------------------------------------------------------ MMAs
        const unsigned b0 = smem_u32(sm), a0 = smem_u32(ring);
        constexpr unsigned IDESC = (1u << 4) | ((unsigned)(128 >> 4) << 24);  // FP32 += FP16 x FP16, M = 128
        auto kstep = [&](int slot, int h, int ks, int ab) {
            const unsigned as = a0 + slot * kSlot, bs = b0 + (unsigned)((h * KS + ks) * kBlock);
            const uint64_t ad = make_desc(as, 128, 256), bd = make_desc(bs, 128, 256);
#pragma unroll
            for (int i = 0; i < kDigits; i++)
                mma_f16(tmem + (unsigned)(ab * 256 + 32 * i), ad + (uint64_t)(i * 4096 >> 4), bd,
                        IDESC | ((unsigned)(32 * (kDigits - i) >> 3) << 17), (ks == 0 && i == 0) ? 0u : 1u);
        };
        auto free_unit = [&](long long u) {  // the unit's accumulators have been read
            return u < 2 || mbar_wait(&accempty[u & 1], (unsigned)(((u >> 1) - 1) & 1));
        };
        for (long long t = 0; t < ntl && !failed; t++) {
            if constexpr (MODE == C6) {
                if (!free_unit(2 * t)) failed = true;
#pragma unroll 1
                for (int ks = 0; ks < KS && !failed; ks++) {
                    const long long q = t * KS + ks;
                    if (!mbar_wait(&full[q % SLOTS], (unsigned)((q / SLOTS) & 1))) {
                        failed = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    kstep((int)(q % SLOTS), 0, ks, 0);
                    if (ks == 0 && !free_unit(2 * t + 1)) {
                        failed = true;
                        break;
                    }
                    kstep((int)(q % SLOTS), 1, ks, 1);
                    commit_to(&empty[q % SLOTS]);
                }
                if (!failed) {
                    commit_to(&accfull[0]);
                    commit_to(&accfull[1]);
                }
            } else {
#pragma unroll 1
                for (int h = 0; h < UNITS && !failed; h++) {
                    const long long u = t * UNITS + h;
                    if (!free_unit(u)) failed = true;
#pragma unroll 1
                    for (int ks = 0; ks < KS && !failed; ks++) {
                        const long long q = t * KS + ks;
                        if (h == 0 && !mbar_wait(&full[q % SLOTS], (unsigned)((q / SLOTS) & 1))) {
                            failed = true;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        kstep((int)(q % SLOTS), h, ks, (int)(u & 1));
                        if (h == UNITS - 1) commit_to(&empty[q % SLOTS]);
                    }
                    if (!failed) commit_to(&accfull[u & 1]);
                }
            }
        }
        commit_to(drain);  // tensor memory is released only after every MMA has completed
        if (!mbar_wait(drain, 0u)) failed = true;
        }
    }
    if (failed) atomicOr(&g_f64_error, 1u);
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// U's digits: [unit][K-step][row / 8][K half][row mod 8][8], row = 32 digit + output of the unit
template <int MODE>
static void pack(const Op &op, unsigned char *out) {
    using C = Cfg<MODE>;
    const double scale = std::ldexp(1.0, 62 - op.f64_su);
    auto entry = [&](int r, int c) { return op.f64_left[(size_t)r * C::D + c]; };
    for (int h = 0; h < C::UNITS; h++)
        for (int ks = 0; ks < C::KS; ks++) {
            unsigned short *blk = reinterpret_cast<unsigned short *>(out + (size_t)(h * C::KS + ks) * kBlock);
            for (int n = 0; n < 32; n++)
                for (int p = 0; p < 16; p++) {
                    const int kc = p >> 2, r = p & 3;  // loading lane and its real in the K-step
                    double u;
                    if (C::PARTS) {
                        const int step = MODE == C6 ? ks >> 1 : ks;
                        const cd z = entry(32 * h + n, kc + 4 * (4 * step + r));
                        u = MODE == C6 && (ks & 1) ? z.imag() : z.real();
                    } else {
                        const cd z = entry(16 * h + (n >> 1), kc + 4 * (2 * ks + (r >> 1)));
                        if (n & 1) u = (r & 1) ? z.real() : z.imag();
                        else u = (r & 1) ? -z.imag() : z.real();
                    }
                    const unsigned long long dg = digit_bytes(u, scale);
                    for (int j = 0; j < kDigits; j++) {
                        const int row = 32 * j + n;
                        blk[(size_t)(row >> 3) * 128 + (p >> 3) * 64 + (row & 7) * 8 + (p & 7)] = half_digit(dg, j);
                    }
                }
        }
    std::memcpy(out + C::BBYTES, op.f64_rows.data(), C::ROWS);
    dense_f64_pack_scales(op, out + C::BBYTES + C::ROWS);
}

static int mode_of(const Op &op) {
    const int k = (int)op.targets.size();
    if (k == 6) return op.real_u ? R6 : C6;
    if (op.real_u) return -1;
    return k == 5 ? C5 : k == 4 ? C4 : -1;
}

template <int MODE, bool SPEC>
static void launch(const Args &a, int sms, cudaStream_t st) {
    using C = Cfg<MODE>;
    static bool attr = false;
    if (!attr) {
        const cudaError_t e =
            cudaFuncSetAttribute(dense_f64_tc_kernel<MODE, SPEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
        if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("dense_f64_tc_kernel attribute: ") + cudaGetErrorString(e));
        attr = true;
    }
    // one CTA per SM: it holds all 512 tensor-memory columns
    dense_f64_tc_kernel<MODE, SPEC><<<(int)std::min<long long>(a.ntiles, sms), kThreads, C::SMEM, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("dense_f64_tc_kernel: ") + cudaGetErrorString(e));
    note_launches(1, QSIM_KERNEL_DENSE_TC);
}

#define QSIM_F64TC_SWITCH(m, CALL)  \
    switch (m) {                    \
        case C4: CALL(C4); break;   \
        case C5: CALL(C5); break;   \
        case R6: CALL(R6); break;   \
        case C6: CALL(C6); break;   \
        default: break;             \
    }

}  // namespace f64tc

// From 2^7 tiles up every SM has one (19 qubits, 4 / 5 / 6 real / 6 targets: 10.7 / 14 / 14 / 20 us here); below, the
// warp-level kernels spread a state over more SMs (18 qubits: 7.2 / 15 / 14 / 30 us).
size_t dense_f64_tc_blob_bytes(const Op &op, int n) {
    using namespace f64tc;
    size_t bytes = 0;
    int gb = 0;
#define QSIM_BYTES(M) bytes = Cfg<M>::BBYTES + Cfg<M>::ROWS + 16 * Cfg<M>::D, gb = Cfg<M>::GB
    QSIM_F64TC_SWITCH(mode_of(op), QSIM_BYTES)
#undef QSIM_BYTES
    return n - (int)(op.targets.size() + op.controls.size()) >= gb + 7 ? bytes : 0;
}

void dense_f64_tc_pack(const Op &op, unsigned char *out) {
    using namespace f64tc;
#define QSIM_PACK(M) pack<M>(op, out)
    QSIM_F64TC_SWITCH(mode_of(op), QSIM_PACK)
#undef QSIM_PACK
}

bool launch_dense_f64_tc(void *state, int n, const Op &op, const void *dig, const void *Ut, int sms, cudaStream_t st) {
    using namespace f64tc;
    const int mode = mode_of(op);
    if (mode < 0) return false;
    int gb = 0, vw = 0;
#define QSIM_GB(M) gb = Cfg<M>::GB, vw = Cfg<M>::BBYTES + Cfg<M>::ROWS
    QSIM_F64TC_SWITCH(mode, QSIM_GB)
#undef QSIM_GB
    Args a;
    std::memset(&a, 0, sizeof(a));
    unsigned long long used = 0;
    for (int q : op.targets) used |= 1ull << q;
    for (int q : op.controls) used |= 1ull << q, a.cmask |= 1ull << q;
    std::vector<int> fr, fix(op.targets);
    for (int q = 0; q < n; q++)
        if (!((used >> q) & 1ull)) fr.push_back(q);
    if ((int)fr.size() < gb) return false;  // not one tile
    if ((int)(op.targets.size() + op.controls.size()) + gb > kMaxFix) return false;
    a.psi = static_cast<double2 *>(state);
    a.dig = static_cast<const uint4 *>(dig);
    a.Ut = static_cast<const double2 *>(Ut);
    a.vw = reinterpret_cast<const double2 *>(static_cast<const unsigned char *>(dig) + vw);
    a.ntiles = 1ll << ((int)fr.size() - gb);
    a.diag = op.f64_diag;
    a.beside = dense_f64_beside(op);
    a.su = op.f64_su;
    a.sh = op.f64_sh;
    a.check = op.f64_check ? 1 : 0;
    a.reach = op.f64_reach;
    const int k = (int)op.targets.size();
    for (int v = 0; v < (1 << k); v++)
        for (int b = 0; b < k; b++)
            if ((v >> b) & 1) a.amp[v] += 1ll << op.targets[b];
    for (int b = 0; b < gb; b++) a.grp[b] = 1ll << fr[b];
    fix.insert(fix.end(), op.controls.begin(), op.controls.end());
    fix.insert(fix.end(), fr.begin(), fr.begin() + gb);
    std::sort(fix.begin(), fix.end());
    a.nfix = (int)fix.size();
    for (int i = 0; i < a.nfix; i++) a.fix[i] = fix[i];
#define QSIM_LAUNCH(M) (a.diag || a.check) ? launch<M, true>(a, sms, st) : launch<M, false>(a, sms, st)
    QSIM_F64TC_SWITCH(mode, QSIM_LAUNCH)
#undef QSIM_LAUNCH
    return true;
}

unsigned dense_f64_read_error() {
    unsigned v = 0;
    const cudaError_t e = cudaMemcpyFromSymbol(&v, g_f64_error, sizeof(v));
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("reading device status: ") + cudaGetErrorString(e));
    return v;
}

void dense_f64_clear_error() {
    const unsigned z = 0;
    const cudaError_t e = cudaMemcpyToSymbol(g_f64_error, &z, sizeof(z));
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("clearing device status: ") + cudaGetErrorString(e));
}

}  // namespace qsim
