// Fourier and Walsh-Hadamard passes on complex128 amplitudes in 64-bit fixed point (sm_103a).
//
// What bounds the FP64 form (dft_kernel<double>): FP64 adds and multiplies run at 2 per clock and SM
// on this GPU, and a 10-qubit pass needs about 10 adds and 12 products per real, so it ran at a tenth
// of the HBM rate.  Integer adds run 64 times as fast and a 62 x 60-bit product costs a few 32-bit
// multiply-adds, so the transform works on integers:
//   - a thread loads its points, takes their largest exponent and writes them as integers relative to
//     it, of as many bits as the growth of the step's sums leaves (58 for 16 points);
//   - butterflies are 64-bit adds; twiddles are 60-bit integers in two 32-bit halves;
//   - between the steps each thread leaves its exponent beside its integers, and the reader aligns
//     the points of a column to the column's largest (block floating point), so that the next steps
//     again start from as many bits as they can;
//   - the outputs, with the twiddle and the structured phase, are rounded once to FP64.
// An error of a few units of 2^-56 of a column's largest value is left, below the FP64 form's.
// Tile, layout and thread mapping are dft_kernel's (see dft_impl.cuh).  A tile with a point that is
// not finite, or a thread's largest exponent far from 1, is transformed in FP64 (plain_tile).
//
// 10 qubits of a 25-qubit state, FP64 form -> this one: Walsh-Hadamard 2030 -> 350 us, Fourier 2800 -> 515 us, Fourier with
// twiddles 2823 -> 620 us (1 GiB moved: 160 us at the copy rate).  What bounds it: issue slots (integer multiply-adds and
// shifts).  9 and 10 qubits run in three steps of 16 x 8 x (4 or 8) points: two steps of 32 points took 1044 us, their
// code outgrew the instruction cache.
#pragma once
#include "dft_impl.cuh"

namespace qsim {
namespace dftk {
namespace fx {

constexpr int kMinExp = 200, kMaxExp = 1900;  // biased exponents of a thread's largest value
constexpr int kMinK = 5;                      // narrower fields stay in FP64

struct Z {
    long long x, y;
};

// 2^60 (c + i s) in halves: c = ch 2^32 + cl, s = sh 2^32 + sl, cl and sl signed
constexpr int hi_half(long long v) { return (int)((v + 0x80000000ll) >> 32); }
constexpr int lo_half(long long v) { return (int)(unsigned)v; }
// 2^60 cos(pi k / 16), k = 0..8, to the nearest integer
constexpr long long kCos60[9] = {1152921504606846976ll, 1130768441178740757ll, 1065160580698383124ll,
                                 958619196450722178ll, 815238614083298888ll, 640528868967736374ll,
                                 441203958630471860ll, 224923827593068887ll, 0ll};
struct TwFx {
    int4 e[32];
};
constexpr TwFx make_tw_fx() {
    TwFx t{};
    for (int i = 0; i < 32; i++) {  // exp(-2 pi i e / 32)
        const int q = i / 8, r = i % 8;
        long long c = kCos60[r], s = kCos60[8 - r];
        for (int k = 0; k < q; k++) {
            const long long n = -s;
            s = c;
            c = n;
        }
        t.e[i].x = hi_half(c);
        t.e[i].y = lo_half(c);
        t.e[i].z = hi_half(-s);
        t.e[i].w = lo_half(-s);
    }
    return t;
}
static __constant__ TwFx kTwFx = make_tw_fx();

__device__ __forceinline__ int low(long long v) { return (int)(unsigned)v; }
__device__ __forceinline__ int high(long long v) { return (int)(v >> 32) + (int)((unsigned)v >> 31); }

constexpr long long kHalf = 1ll << 27;  // rounds the cross products' sum to the result's unit

// v t / 2^60 without the product of the low halves (below 4 units)
__device__ __forceinline__ Z cmul(Z v, int4 t) {
    const int al = low(v.x), ah = high(v.x), bl = low(v.y), bh = high(v.y), nh = -t.z, nl = -t.w;
    const long long mr = kHalf + (long long)ah * t.y + (long long)al * t.x + (long long)bh * nl + (long long)bl * nh;
    const long long mi = kHalf + (long long)ah * t.w + (long long)al * t.z + (long long)bh * t.y + (long long)bl * t.x;
    const unsigned long long hr = (unsigned long long)((long long)ah * t.x + (long long)bh * nh);
    const unsigned long long hi = (unsigned long long)((long long)ah * t.z + (long long)bh * t.x);
    return Z{(long long)((hr << 4) + (unsigned long long)(mr >> 28)), (long long)((hi << 4) + (unsigned long long)(mi >> 28))};
}
// v c / 2^60, c real
__device__ __forceinline__ long long rmul(long long v, int ch, int cl) {
    const int l = low(v), h = high(v);
    const long long m = kHalf + (long long)h * cl + (long long)l * ch;
    return (long long)(((unsigned long long)((long long)h * ch) << 4) + (unsigned long long)(m >> 28));
}

// dft_regs on integers
template <int R, int SGN, bool WALSH>
__device__ __forceinline__ void dft_regs_fx(Z *x) {
#pragma unroll
    for (int span = R / 2; span >= 1; span >>= 1) {
#pragma unroll
        for (int b = 0; b < R; b += 2 * span) {
#pragma unroll
            for (int j = 0; j < span; j++) {
                const Z u = x[b + j], v = x[b + j + span];
                x[b + j] = Z{u.x + v.x, u.y + v.y};
                Z d{u.x - v.x, u.y - v.y};
                const int e = WALSH ? 0 : j * (R / (2 * span));
                if (4 * e == R) {  // s i
                    d = SGN > 0 ? Z{-d.y, d.x} : Z{d.y, -d.x};
                } else if (8 * e == R || 8 * e == 3 * R) {  // (+-1 + s i) / sqrt(2)
                    const int4 h = kTwFx.e[4];
                    const long long p = rmul(d.x + d.y, h.x, h.y), q = rmul(d.y - d.x, h.x, h.y);
                    if (8 * e == R) d = SGN > 0 ? Z{-q, p} : Z{p, q};
                    else d = SGN > 0 ? Z{-p, -q} : Z{q, -p};
                } else if (e != 0) {
                    int4 t = kTwFx.e[e * (32 / R)];
                    if (SGN > 0) {
                        t.z = -t.z;
                        t.w = -t.w;
                    }
                    d = cmul(d, t);
                }
                x[b + j + span] = d;
            }
        }
    }
}

// x as an integer of B bits relative to 2^(E + 1) (E: a biased exponent not below x's)
template <int B>
__device__ __forceinline__ long long to_fixed(double x, int E) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int s = E - (int)((hi >> 20) & 0x7ffu);
    constexpr unsigned one = 1u << (B - 33);  // the leading bit of a normal number
    const unsigned mh = (__funnelshift_l(lo, hi, B - 53) & (one - 1u)) | one;
    unsigned long long v = ((unsigned long long)mh << 32) | (lo << (B - 53));
    asm("shr.u64 %0, %0, %1;" : "+l"(v) : "r"(s));  // 0 from 64 on
    const long long sg = (long long)((int)hi >> 31);
    return (long long)((v ^ (unsigned long long)sg) - (unsigned long long)sg);
}
// a point left by an earlier step, in units 2^s as large, rounded
__device__ __forceinline__ Z aligned(int4 p, int s) {
    unsigned long long r = 1;
    asm("shl.b64 %0, %0, %1;" : "+l"(r) : "r"(s));
    r >>= 1;
    long long x = (long long)((((unsigned long long)(unsigned)p.y << 32) | (unsigned)p.x) + r);
    long long y = (long long)((((unsigned long long)(unsigned)p.w << 32) | (unsigned)p.z) + r);
    asm("shr.s64 %0, %0, %1;" : "+l"(x) : "r"(s));
    asm("shr.s64 %0, %0, %1;" : "+l"(y) : "r"(s));
    return Z{x, y};
}
__device__ __forceinline__ double to_double(long long v, int ex) {  // v 2^ex
    const double d = (double)v;
    const int hi = __double2hiint(d);
    return __hiloint2double(hi ? hi + (ex << 20) : 0, __double2loint(d));
}

// (cos, sin) of half the inversion angle of clock value kk (see hhl_invert_kernel)
__device__ __forceinline__ double2 inversion(const DftArgs &a, unsigned long long kk) {
    double s = 0, c = 1;
    if (kk) {
        const long long ks = (a.inv_twos && (kk >> (a.inv_nc - 1))) ? (long long)kk - (1ll << a.inv_nc) : (long long)kk;
        s = a.inv_Cs / (double)ks;
        if (s > 1.0) s = 1.0;
        if (s < -1.0) s = -1.0;
        const double as = s < 0 ? -s : s;
        c = sqrt((1.0 - as) * (1.0 + as));
    }
    return make_double2(c, s);
}

// One tile in FP64 (dft_kernel's two steps, the tables read from global memory), by the threads
// u < 2^(K/2); pad: dft_kernel's gaps in S.
template <int K, int SGN, int KIND>
__device__ __noinline__ void plain_tile(const DftArgs &a, unsigned long long base, unsigned w, unsigned long long kb,
                                        double2 *S, int pad, int l, int u) {
    constexpr bool WALSH = KIND == 1;
    constexpr int k1 = K / 2, k2 = K - k1, N1 = 1 << k1, N2 = 1 << k2, RR = N2 / N1;
    const int L = a.L;
    double2 *psi = reinterpret_cast<double2 *>(a.psi);
    const double2 *W = reinterpret_cast<const double2 *>(a.W), *Tlo = reinterpret_cast<const double2 *>(a.Tlo),
                  *Thi = reinterpret_cast<const double2 *>(a.Thi), *qlo = reinterpret_cast<const double2 *>(a.qlo),
                  *qhi = reinterpret_cast<const double2 *>(a.qhi);
    const unsigned long long qcm = (1ull << a.qm) - 1ull, qhm = (1ull << a.qh) - 1ull;
    double2 x[N2];
    if (u < N1) {
#pragma unroll
    for (int v = 0; v < N2; v++) x[v] = psi[base + ((unsigned long long)(u + N1 * v) << a.f0)];
    dft_regs<N2, SGN, WALSH>(x);
#pragma unroll
    for (int i = 0; i < N2; i++) {
        const int aa = WALSH ? i : bitrev(i, k2);
        double2 y = x[i];
        if (!WALSH && aa != 0) y = dftk::cmul(y, W[u * aa]);
        S[((aa * N1 + u) << L) + l + (aa / RR) * pad] = y;
    }
    }
    __syncthreads();
    if (u >= N1) return;
#pragma unroll
    for (int r = 0; r < RR; r++) {
        const int aa = u * RR + r;
#pragma unroll
        for (int uu = 0; uu < N1; uu++) x[uu] = S[((aa * N1 + uu) << L) + l + u * pad];
        dft_regs<N1, SGN, WALSH>(x);
#pragma unroll
        for (int i = 0; i < N1; i++) {
            const int y = WALSH ? i + N1 * aa : aa + N2 * bitrev(i, k1);
            double2 z = x[i];
            z.x *= a.scale;
            z.y *= a.scale;
            if (a.twmode == 2) {
                const unsigned q = w * (unsigned)y;
                z = dftk::cmul(z, dftk::cmul(Tlo[q & ((1u << a.hT) - 1u)], Thi[q >> a.hT]));
            }
            const unsigned long long oi = base + ((unsigned long long)y << a.f0);
            if (a.qmode == 2) {
                const unsigned long long c = (oi >> a.qnb) & qcm, d = oi & ((1ull << a.qnb) - 1ull);
                z = dftk::cmul(z, dftk::cmul(qlo[((c & qhm) << a.qnb) + d], qhi[((c >> a.qh) << a.qnb) + d]));
            }
            if (KIND == 2) {
                const double2 cs = inversion(a, kb | ((unsigned long long)y << a.inv_fdst));
                psi[oi + (1ull << a.inv_bit)] = make_double2(cs.y * z.x, cs.y * z.y);
                z = make_double2(cs.x * z.x, cs.x * z.y);
            }
            psi[oi] = z;
        }
    }
}

// KIND as in dft_kernel; twiddle and structured phase on the outputs only (twmode 0, 2; qmode 0, 2)
template <int K, int SGN, int KIND>
__global__ void __launch_bounds__(256, 1) dft_fx_kernel(const __grid_constant__ DftArgs a) {
    constexpr bool WALSH = KIND == 1, INV = KIND == 2;
    constexpr int k1 = K / 2, k2 = K - k1, N1 = 1 << k1, N2 = 1 << k2, RR = N2 / N1, KN = 1 << K;
    constexpr int B1 = 62 - k2, B2 = 62 - k1;  // a sum of 2^k points grows by at most k + 1/2 bits
    const int L = a.L, NL = 1 << L, nthr = N1 << L;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int4 *S = reinterpret_cast<int4 *>(smem_raw);           // tile, padded as in dft_kernel
    int4 *Ws = S + (KN << L) + N1 * NL;                     // inner twiddles
    int4 *Ts = Ws + (WALSH ? 0 : KN);                       // twiddle tables (tw_smem)
    const int ntlo = 1 << a.hT, nthi = 1 << (K + a.ns - a.hT);
    double2 *cs = reinterpret_cast<double2 *>(Ts + (a.tw_smem ? ntlo + nthi : 0));  // inversion, per field value
    int *ex = reinterpret_cast<int *>(cs + (INV && a.inv_shared ? KN : 0));         // exponents [u][lane]
    int *top = ex + N1 * NL;                                // column exponents [2][lane]
    const int tid = threadIdx.x, l = tid & (NL - 1), u = tid >> L;
    const int4 *Wg = reinterpret_cast<const int4 *>(a.Wfx);
    if (!WALSH)
        for (int i = tid; i < KN; i += nthr) Ws[i] = Wg[i];
    const int4 *Tlo = Wg + KN, *Thi = Tlo + ntlo;
    if (a.tw_smem) {
        for (int i = tid; i < ntlo + nthi; i += nthr) Ts[i] = Tlo[i];
        Tlo = Ts;
        Thi = Ts + ntlo;
    }
    for (int i = tid; i < 2 * NL; i += nthr) top[i] = 0;
    unsigned long long lane_off = 0;
    for (int b = 0; b < L; b++)
        if ((l >> b) & 1) lane_off |= 1ull << a.lpos[b];
    __syncthreads();
    const unsigned tmask = (1u << a.hT) - 1u;
    double2 *psi = reinterpret_cast<double2 *>(a.psi);
    const int4 *qlo = reinterpret_cast<const int4 *>(a.qfx), *qhi = qlo + (1ll << (a.qh + a.qnb));
    int par = 0;

    for (long long tix = blockIdx.x; tix < a.ntiles; tix += gridDim.x, par ^= 1) {
        const unsigned long long base = insert_zero_bits((unsigned long long)tix, a.fix, a.nfix) + lane_off;
        unsigned long long kb = 0;
        if (INV) {
            for (int sg = 0; sg < a.inv_nseg; sg++)
                kb |= ((base >> a.inv_src[sg]) & ((1ull << a.inv_w[sg]) - 1ull)) << a.inv_dst[sg];
            if (a.inv_shared)  // the lanes lie outside the clock register: one rotation per field value
                for (int i = tid; i < KN; i += nthr) cs[i] = inversion(a, kb | ((unsigned long long)i << a.inv_fdst));
        }
        unsigned w = 0;
        for (int j = 0; j < a.ns; j++) w |= (unsigned)((base >> a.spos[j]) & 1ull) << j;
        int E;
        bool bad = false;
        {
            double2 x[N2];
            const double2 *src = psi + base + ((unsigned long long)u << a.f0);
            const long long step = 1ll << (a.f0 + k1);
#pragma unroll
            for (int v = 0; v < N2; v++) x[v] = src[v * step];
            unsigned m = 0, lows = 0;
#pragma unroll
            for (int v = 0; v < N2; v++) {
                m = max(m, (unsigned)__double2hiint(x[v].x) & 0x7fffffffu);
                m = max(m, (unsigned)__double2hiint(x[v].y) & 0x7fffffffu);
            }
            E = (int)(m >> 20);
            if (m == 0)
#pragma unroll
                for (int v = 0; v < N2; v++) lows |= (unsigned)__double2loint(x[v].x) | (unsigned)__double2loint(x[v].y);
            bad = m ? E < kMinExp || E > kMaxExp : lows != 0;
            const int Es = m ? E : 64;  // zeros shift out
            Z z[N2];
#pragma unroll
            for (int v = 0; v < N2; v++) z[v] = Z{to_fixed<B1>(x[v].x, Es), to_fixed<B1>(x[v].y, Es)};
            dft_regs_fx<N2, SGN, WALSH>(z);
            if (a.pf) {  // a later tile's lines into L2 (see dft_kernel)
                const long long nt = tix + (long long)a.pf * gridDim.x;
                if (nt < a.ntiles) {
                    const unsigned long long nb = insert_zero_bits((unsigned long long)nt, a.fix, a.nfix);
                    for (int v = l; v < N2; v += NL)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(psi + nb + ((unsigned long long)(u + N1 * v) << a.f0)));
                }
            }
            unsigned mag = 0;
#pragma unroll
            for (int i = 0; i < N2; i++) {
                const int aa = WALSH ? i : bitrev(i, k2);
                Z y = z[i];
                if (!WALSH && aa != 0) y = cmul(y, Ws[u * aa]);
                const int hx = (int)(y.x >> 32), hy = (int)(y.y >> 32);
                mag |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
                S[((aa * N1 + u) << L) + l + (aa / RR) * NL] = make_int4(low(y.x), hx, low(y.y), hy);
            }
            ex[u * NL + l] = E;
            // the column's exponent: its largest value back to 57 bits
            if (m) atomicMax(&top[par * NL + l], E + max(0, 64 - B2 - __clz((int)mag)));
        }
        if (__syncthreads_or(bad)) {
            plain_tile<K, SGN, KIND>(a, base, w, kb, reinterpret_cast<double2 *>(S), NL, l, u);
            if (u == 0) top[(par ^ 1) * NL + l] = 0;
            __syncthreads();
            continue;
        }
        const int Ec = top[par * NL + l];
        if (u == 0) top[(par ^ 1) * NL + l] = 0;
        const int eo = Ec - 1022 - B1 - K / 2;
#pragma unroll
        for (int r = 0; r < RR; r++) {
            const int aa = u * RR + r;
            Z z[N1];
#pragma unroll
            for (int uu = 0; uu < N1; uu++) {
                z[uu] = aligned(S[((aa * N1 + uu) << L) + l + u * NL], Ec - ex[uu * NL + l]);
            }
            dft_regs_fx<N1, SGN, WALSH>(z);
#pragma unroll
            for (int i = 0; i < N1; i++) {
                const int y = WALSH ? i + N1 * aa : aa + N2 * bitrev(i, k1);
                Z v = z[i];
                if (K & 1) {  // 2^(-K/2) = 2^(-floor(K/2)) / sqrt(2)
                    const int4 h = kTwFx.e[4];
                    v = Z{rmul(v.x, h.x, h.y), rmul(v.y, h.x, h.y)};
                }
                if (!WALSH && a.twmode == 2) {
                    const unsigned q = w * (unsigned)y;
                    v = cmul(cmul(v, Tlo[q & tmask]), Thi[q >> a.hT]);
                }
                const unsigned long long oi = base + ((unsigned long long)y << a.f0);
                if (a.qmode == 2) {
                    const unsigned long long c = (oi >> a.qnb) & ((1ull << a.qm) - 1ull), d = oi & ((1ull << a.qnb) - 1ull);
                    v = cmul(v, __ldg(qlo + (((c & ((1ull << a.qh) - 1ull)) << a.qnb) + d)));
                    v = cmul(v, __ldg(qhi + (((c >> a.qh) << a.qnb) + d)));
                }
                double2 o = make_double2(to_double(v.x, eo), to_double(v.y, eo));
                if (INV) {
                    const double2 t = a.inv_shared ? cs[y] : inversion(a, kb | ((unsigned long long)y << a.inv_fdst));
                    psi[oi + (1ull << a.inv_bit)] = make_double2(t.y * o.x, t.y * o.y);
                    o = make_double2(t.x * o.x, t.x * o.y);
                }
                psi[oi] = o;
            }
        }
        __syncthreads();  // S, ex, cs and the next column exponents are rewritten by the next tile
    }
}

// Fields of 9 and 10 qubits in three steps of 16, 8 and 4 or 8 points: two steps of 32 points ran
// out of the instruction cache (14 % of the issue slots used) and left 8 warps per SM.  y = u + Nr v:
// step 1 transforms over v (output digit a), step 2 over the high part of u = u2 + N3 v2 (digit a2),
// step 3 over u2 (digit b2); y' = a + 16 (a2 + 8 b2).  The tile's element (a, u) sits in row a Nr + u.
// The points are aligned to the column's exponent when step 2 reads them.
// TILE (see tile_twiddles): the products of the two twiddle tables' entries are made once a tile, 2^K of them for
// 2^(K + L) points, while step 1's loads are in flight.
template <int K, int SGN, int KIND, bool TILE>
__global__ void __launch_bounds__(512, 1) dft_fx3_kernel(const __grid_constant__ DftArgs a) {
    constexpr bool WALSH = KIND == 1, INV = KIND == 2;
    constexpr int RA = 16, RB = 8, RC = 1 << (K - 7), NR = RB * RC, KN = 1 << K;
    constexpr int B1 = 62 - 4, B2 = 62 - (K - 4);  // growth as in dft_fx_kernel; steps 2 and 3 together
    const int L = a.L, NL = 1 << L, nthr = NR << L;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int4 *S = reinterpret_cast<int4 *>(smem_raw);
    int4 *Ws = S + (KN << L);
    int4 *TW = Ws + (WALSH ? 0 : KN);
    int4 *Ts = TW + (TILE ? KN : 0);
    const int ntlo = 1 << a.hT, nthi = 1 << (K + a.ns - a.hT);
    double2 *cs = reinterpret_cast<double2 *>(Ts + (a.tw_smem ? ntlo + nthi : 0));
    int *ex = reinterpret_cast<int *>(cs + (INV && a.inv_shared ? KN : 0));  // [u][lane]
    int *top = ex + NR * NL;                                                 // [2][lane]
    const int tid = threadIdx.x, l = tid & (NL - 1), u = tid >> L;
    const int4 *Wg = reinterpret_cast<const int4 *>(a.Wfx);
    if (!WALSH)
        for (int i = tid; i < KN; i += nthr) Ws[i] = Wg[i];
    const int4 *Tlo = Wg + KN, *Thi = Tlo + ntlo;
    if (a.tw_smem) {
        for (int i = tid; i < ntlo + nthi; i += nthr) Ts[i] = Tlo[i];
        Tlo = Ts;
        Thi = Ts + ntlo;
    }
    for (int i = tid; i < 2 * NL; i += nthr) top[i] = 0;
    unsigned long long lane_off = 0;
    for (int b = 0; b < L; b++)
        if ((l >> b) & 1) lane_off |= 1ull << a.lpos[b];
    __syncthreads();
    const unsigned tmask = (1u << a.hT) - 1u;
    double2 *psi = reinterpret_cast<double2 *>(a.psi);
    const int4 *qlo = reinterpret_cast<const int4 *>(a.qfx), *qhi = qlo + (1ll << (a.qh + a.qnb));
    int par = 0;

    for (long long tix = blockIdx.x; tix < a.ntiles; tix += gridDim.x, par ^= 1) {
        const unsigned long long base = insert_zero_bits((unsigned long long)tix, a.fix, a.nfix) + lane_off;
        unsigned long long kb = 0;
        if (INV) {
            for (int sg = 0; sg < a.inv_nseg; sg++)
                kb |= ((base >> a.inv_src[sg]) & ((1ull << a.inv_w[sg]) - 1ull)) << a.inv_dst[sg];
            if (a.inv_shared)
                for (int i = tid; i < KN; i += nthr) cs[i] = inversion(a, kb | ((unsigned long long)i << a.inv_fdst));
        }
        unsigned w = 0;
        for (int j = 0; j < a.ns; j++) w |= (unsigned)((base >> a.spos[j]) & 1ull) << j;
        bool bad = false;
        {
            double2 x[RA];
            const double2 *src = psi + base + ((unsigned long long)u << a.f0);
            const long long step = (long long)NR << a.f0;
#pragma unroll
            for (int v = 0; v < RA; v++) x[v] = src[v * step];
            if (TILE)  // w is the tile's: its twiddles once, not once a lane
#pragma unroll 1
                for (int i = tid; i < KN; i += nthr) {
                    const unsigned q = w * (unsigned)i;
                    const int4 t = Tlo[q & tmask];
                    const Z y = cmul(Z{((long long)t.x << 32) + t.y, ((long long)t.z << 32) + t.w}, Thi[q >> a.hT]);
                    TW[i] = make_int4(high(y.x), low(y.x), high(y.y), low(y.y));
                }
            unsigned m = 0, lows = 0;
#pragma unroll
            for (int v = 0; v < RA; v++) {
                m = max(m, (unsigned)__double2hiint(x[v].x) & 0x7fffffffu);
                m = max(m, (unsigned)__double2hiint(x[v].y) & 0x7fffffffu);
            }
            const int E = (int)(m >> 20);
            if (m == 0)
#pragma unroll
                for (int v = 0; v < RA; v++) lows |= (unsigned)__double2loint(x[v].x) | (unsigned)__double2loint(x[v].y);
            bad = m ? E < kMinExp || E > kMaxExp : lows != 0;
            const int Es = m ? E : 64;
            Z z[RA];
#pragma unroll
            for (int v = 0; v < RA; v++) z[v] = Z{to_fixed<B1>(x[v].x, Es), to_fixed<B1>(x[v].y, Es)};
            dft_regs_fx<RA, SGN, WALSH>(z);
            unsigned mag = 0;
#pragma unroll
            for (int i = 0; i < RA; i++) {
                const int aa = WALSH ? i : bitrev(i, 4);
                Z y = z[i];
                if (!WALSH && aa != 0) y = cmul(y, Ws[u * aa]);
                const int hx = (int)(y.x >> 32), hy = (int)(y.y >> 32);
                mag |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
                S[((aa * NR + u) << L) + l] = make_int4(low(y.x), hx, low(y.y), hy);
            }
            ex[u * NL + l] = E;
            if (m) atomicMax(&top[par * NL + l], E + max(0, 64 - B2 - __clz((int)mag)));
        }
        if (__syncthreads_or(bad)) {
            plain_tile<K, SGN, KIND>(a, base, w, kb, reinterpret_cast<double2 *>(S), 0, l, u);
            if (u == 0) top[(par ^ 1) * NL + l] = 0;
            __syncthreads();
            continue;
        }
        const int Ec = top[par * NL + l];
        if (u == 0) top[(par ^ 1) * NL + l] = 0;
        if (a.pf) {  // a later tile's lines into L2 (see dft_kernel)
            const long long nt = tix + (long long)a.pf * gridDim.x;
            if (nt < a.ntiles) {
                const unsigned long long nb = insert_zero_bits((unsigned long long)nt, a.fix, a.nfix);
                for (int v = l; v < RA; v += NL)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(psi + nb + ((unsigned long long)(u + NR * v) << a.f0)));
            }
        }
        // step 2: thread u takes the groups (a, u2) with a RC + u2 = u, u + NR
#pragma unroll 1
        for (int g = u; g < RA * RC; g += NR) {
            const int aa = g / RC, u2 = g % RC;
            int4 *p = S + ((aa * NR + u2) << L) + l;
            const int *e = ex + u2 * NL + l;
            Z z[RB];
#pragma unroll
            for (int v = 0; v < RB; v++) {
                z[v] = aligned(p[(v * RC) << L], Ec - e[v * RC * NL]);
            }
            dft_regs_fx<RB, SGN, WALSH>(z);
#pragma unroll
            for (int i = 0; i < RB; i++) {
                const int a2 = WALSH ? i : bitrev(i, 3);
                Z y = z[i];
                if (!WALSH && a2 != 0) y = cmul(y, Ws[RA * u2 * a2]);
                p[(a2 * RC) << L] = make_int4(low(y.x), (int)(y.x >> 32), low(y.y), (int)(y.y >> 32));
            }
        }
        __syncthreads();
        const int eo = Ec - 1022 - B1 - K / 2;
#pragma unroll 1
        for (int g = u; g < RA * RB; g += NR) {  // step 3: groups (a, a2)
            const int aa = g / RB, a2 = g % RB;
            const int4 *p = S + ((aa * NR + a2 * RC) << L) + l;
            Z z[RC];
#pragma unroll
            for (int v = 0; v < RC; v++) {
                const int4 q = p[v << L];
                z[v] = Z{(long long)(((unsigned long long)(unsigned)q.y << 32) | (unsigned)q.x),
                         (long long)(((unsigned long long)(unsigned)q.w << 32) | (unsigned)q.z)};
            }
            dft_regs_fx<RC, SGN, WALSH>(z);
#pragma unroll
            for (int i = 0; i < RC; i++) {
                // Walsh: every step's digit stays in its place
                const int y = WALSH ? i + RC * a2 + NR * aa : aa + RA * (a2 + RB * bitrev(i, K - 7));
                Z v = z[i];
                if (K & 1) {
                    const int4 h = kTwFx.e[4];
                    v = Z{rmul(v.x, h.x, h.y), rmul(v.y, h.x, h.y)};
                }
                if (TILE) {
                    v = cmul(v, TW[y]);
                } else if (!WALSH && a.twmode == 2) {
                    const unsigned q = w * (unsigned)y;
                    v = cmul(cmul(v, Tlo[q & tmask]), Thi[q >> a.hT]);
                }
                const unsigned long long oi = base + ((unsigned long long)y << a.f0);
                if (a.qmode == 2) {
                    const unsigned long long c = (oi >> a.qnb) & ((1ull << a.qm) - 1ull), d = oi & ((1ull << a.qnb) - 1ull);
                    v = cmul(v, __ldg(qlo + (((c & ((1ull << a.qh) - 1ull)) << a.qnb) + d)));
                    v = cmul(v, __ldg(qhi + (((c >> a.qh) << a.qnb) + d)));
                }
                double2 o = make_double2(to_double(v.x, eo), to_double(v.y, eo));
                if (INV) {
                    const double2 t = a.inv_shared ? cs[y] : inversion(a, kb | ((unsigned long long)y << a.inv_fdst));
                    psi[oi + (1ull << a.inv_bit)] = make_double2(t.y * o.x, t.y * o.y);
                    o = make_double2(t.x * o.x, t.x * o.y);
                }
                psi[oi] = o;
            }
        }
        __syncthreads();
    }
}

template <int K, int SGN, int KIND, bool TILE = false>
void launch(DftArgs a, cudaStream_t st) {
    constexpr bool THREE = K >= 9;
    const size_t KN = (size_t)1 << K, N1 = THREE ? KN / 16 : (size_t)1 << (K / 2), NL = (size_t)1 << a.L;
    const int threads = (int)(N1 * NL);
    size_t smem = 16 * ((KN << a.L) + (THREE ? 0 : N1 * NL) + (KIND == 1 ? 0 : KN)) + 4 * (N1 * NL + 2 * NL);
    if (KIND == 2 && a.inv_shared) smem += 16 * KN;
    if (TILE) smem += 16 * KN;
    const size_t tw = 16 * (((size_t)1 << a.hT) + ((size_t)1 << (K + a.ns - a.hT)));
    // the tables too, unless they would take a second CTA's room (read once per amplitude, or once a tile)
    a.tw_smem = a.ns > 0 && smem + tw <= (TILE && threads <= 256 ? 112 : 220) * 1024 ? 1 : 0;
    if (a.tw_smem) smem += tw;
    void (*kern)(const DftArgs) = nullptr;
    if constexpr (TILE) kern = dft_fx3_kernel<K, SGN, KIND, TILE>;
    else if constexpr (THREE) kern = dft_fx3_kernel<K, SGN, KIND, false>;
    else kern = dft_fx_kernel<K, SGN, KIND>;
    static bool attr = false;
    if (!attr) {
        DFT_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        attr = true;
    }
    const int per_sm = occupancy_cached(reinterpret_cast<const void *>(kern), threads, smem);
    QSIM_REQUIRE(per_sm > 0, "Fourier pass does not fit on an SM");
    const long long grid = std::min<long long>(a.ntiles, (long long)num_sms_dft() * per_sm);
    kern<<<(int)grid, threads, smem, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("dft_fx_kernel: ") + cudaGetErrorString(e));
    note_launches(1, QSIM_KERNEL_FOURIER);
}

// Twiddles as one table a tile (no lane qubit is a twiddle source): a point then shares the product of the two
// tables' entries with the other lanes.  25 qubits, 10-qubit field, 8 lanes: 637 -> 569 us; 4 lanes 830 -> 713 us (tables
// left in global memory, so that two CTAs fit); with 2 lanes half of the products are left and the table's
// traffic comes on top.  Forms of their own: as a branch of the one kernel they cost the passes without a table 2 %.
inline bool tile_twiddles(const DftArgs &a) {
    bool ok = a.twmode == 2 && a.ns > 0 && a.L >= 2;
    for (int i = 0; i < a.ns; i++)
        for (int j = 0; j < a.L; j++) ok = ok && a.spos[i] != a.lpos[j];
    return ok;
}

template <int K>
void launch_k(const DftArgs &a, int sign, int kind, cudaStream_t st) {
    if constexpr (K >= 9)
        if (kind != 1 && tile_twiddles(a)) {
            if (kind == 2) launch<K, -1, 2, true>(a, st);
            else if (sign > 0) launch<K, 1, 0, true>(a, st);
            else launch<K, -1, 0, true>(a, st);
            return;
        }
    if (kind == 2) launch<K, -1, 2>(a, st);
    else if (kind == 1) launch<K, 1, 1>(a, st);
    else if (sign > 0) launch<K, 1, 0>(a, st);
    else launch<K, -1, 0>(a, st);
}

}  // namespace fx
}  // namespace dftk
}  // namespace qsim
