// Fixed-point Fourier-transform passes for complex128 amplitudes: launch and tables (kernels in
// dft_fx.cuh).
#include "dft_fx.cuh"

namespace qsim {
namespace dftk {
namespace fx {

// Outputs y = 1 .. 2^K - 1 of a pass onto a field that is still |0>, times the structured phase: psi[y 2^w + l]
// = scale psi[l] exp(i lam t c).  In FP64 (expand_kernel) the two products by table entries took 8 FP64
// operations an amplitude, 4 clocks per SM against 0.75 for its 16 bytes (2^26 amplitudes: 971 us); here they
// are integer products, the one whose table index does not depend on y is done once per thread, and the
// FP64 pipe only converts the results.
struct ExpandArgs {
    double2 *psi;
    const double2 *qlo, *qhi;
    const int4 *flo, *fhi;  // the same tables as integers
    long long count;
    double scale;
    int w, K, run, qnb, qm, qh;
};

__global__ void __launch_bounds__(256) expand_fx_kernel(const __grid_constant__ ExpandArgs a) {
    const unsigned long long dmask = (1ull << a.qnb) - 1ull, cmask = (1ull << a.qm) - 1ull, hmask = (1ull << a.qh) - 1ull;
    const unsigned long long ymax = 1ull << a.K;
    const int at = a.w - a.qnb;  // lowest clock bit of the field
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < a.count; g += (long long)gridDim.x * blockDim.x) {
        const unsigned long long l = (unsigned long long)g & ((1ull << a.w) - 1ull), d = l & dmask;
        const unsigned long long y0 = 1ull + ((unsigned long long)g >> a.w) * (unsigned long long)a.run;
        const unsigned long long y1 = min(ymax, y0 + a.run);
        const double2 z = a.psi[l];
        const unsigned m = max((unsigned)__double2hiint(z.x) & 0x7fffffffu, (unsigned)__double2hiint(z.y) & 0x7fffffffu);
        const int E = (int)(m >> 20);
        if (E < kMinExp || E > kMaxExp) {  // zero, not finite, or far from 1: in FP64
            for (unsigned long long y = y0; y < y1; y++) {
                const unsigned long long c = (((y << a.w) | l) >> a.qnb) & cmask;
                const double2 p = dftk::cmul(a.qlo[((c & hmask) << a.qnb) + d], a.qhi[((c >> a.qh) << a.qnb) + d]);
                a.psi[(y << a.w) | l] = dftk::cmul(make_double2(z.x * a.scale, z.y * a.scale), p);
            }
            continue;
        }
        Z v{to_fixed<61>(z.x, E), to_fixed<61>(z.y, E)};
        if (a.K & 1) {
            const int4 h = kTwFx.e[4];
            v = Z{rmul(v.x, h.x, h.y), rmul(v.y, h.x, h.y)};
        }
        const int ex = E - 1022 - 61 - a.K / 2;
        const unsigned long long c0 = (l >> a.qnb) & cmask;
        const bool lo_fixed = at >= a.qh, hi_fixed = at + a.K <= a.qh;
        if (lo_fixed) v = cmul(v, a.flo[((c0 & hmask) << a.qnb) + d]);
        else if (hi_fixed) v = cmul(v, a.fhi[((c0 >> a.qh) << a.qnb) + d]);
#pragma unroll 4
        for (unsigned long long y = y0; y < y1; y++) {
            const unsigned long long c = (((y << a.w) | l) >> a.qnb) & cmask;
            Z o = v;
            if (!lo_fixed) o = cmul(o, __ldg(a.flo + (((c & hmask) << a.qnb) + d)));
            if (!hi_fixed) o = cmul(o, __ldg(a.fhi + (((c >> a.qh) << a.qnb) + d)));
            a.psi[(y << a.w) | l] = make_double2(to_double(o.x, ex), to_double(o.y, ex));
        }
    }
}

}  // namespace fx
}  // namespace dftk

void launch_expand_fx(void *state, int w, int K, double scale, const void *qlo, const void *qhi, int qnb, int qm, int qh,
                      cudaStream_t st) {
    dftk::fx::ExpandArgs a;
    a.psi = static_cast<double2 *>(state);
    a.qlo = static_cast<const double2 *>(qlo);
    a.qhi = static_cast<const double2 *>(qhi);
    a.flo = reinterpret_cast<const int4 *>(a.qhi + (1ll << (qnb + qm - qh)));
    a.fhi = a.flo + (1ll << (qnb + qh));
    a.scale = scale;
    a.w = w;
    a.K = K;
    a.qnb = qnb;
    a.qm = qm;
    a.qh = qh;
    a.run = std::min(32, (1 << K) - 1);
    a.count = (((1ll << K) - 1 + a.run - 1) / a.run) << w;
    const long long grid = std::min<long long>((a.count + 255) / 256, (long long)dftk::num_sms_dft() * 8);
    dftk::fx::expand_fx_kernel<<<(int)grid, 256, 0, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string("expand_fx_kernel: ") + cudaGetErrorString(e));
    note_launches(1, QSIM_KERNEL_EXPAND);
}

bool dft_launch_fx(const dftk::DftArgs &a, int K, int sign, int kind, cudaStream_t st) {
    using namespace dftk;
    if (a.twmode == 1 || a.qmode == 1) return false;  // twiddle or phase on the inputs: FP64 form
    switch (K) {
        case 5: fx::launch_k<5>(a, sign, kind, st); break;
        case 6: fx::launch_k<6>(a, sign, kind, st); break;
        case 7: fx::launch_k<7>(a, sign, kind, st); break;
        case 8: fx::launch_k<8>(a, sign, kind, st); break;
        case 9: fx::launch_k<9>(a, sign, kind, st); break;
        case 10: fx::launch_k<10>(a, sign, kind, st); break;
        default: return false;  // narrower fields have too few additions to gain
    }
    return true;
}

namespace {
struct Unit {  // 2^62 (c + i s)
    long long c, s;
};
Unit operator*(const Unit &a, const Unit &b) {
    const __int128 half = (__int128)1 << 61;
    return Unit{(long long)(((__int128)a.c * b.c - (__int128)a.s * b.s + half) >> 62),
                (long long)(((__int128)a.c * b.s + (__int128)a.s * b.c + half) >> 62)};
}
// exp(2 pi i / 2^b), b = 0..31
const Unit &root(int b) {
    struct Roots {
        Unit r[32];
        Roots() {
            for (int i = 0; i < 32; i++) {
                const long double w = 6.283185307179586476925286766559005768L / (long double)(1ll << i);
                r[i] = Unit{std::llroundl(std::ldexp(std::cos(w), 62)), std::llroundl(std::ldexp(std::sin(w), 62))};
            }
            r[0] = Unit{1ll << 62, 0};
            r[1] = Unit{-(1ll << 62), 0};
            r[2] = Unit{0, 1ll << 62};
        }
    };
    static const Roots roots;
    return roots.r[b];
}
void put(std::vector<int> &out, long long c, long long s) {  // 2^60 (c + i s)
    out.push_back(dftk::fx::hi_half(c));
    out.push_back(dftk::fx::lo_half(c));
    out.push_back(dftk::fx::hi_half(s));
    out.push_back(dftk::fx::lo_half(s));
}
// exp(sign 2 pi i j 2^shift / 2^bits), j < 2^count, as products over the bits of j
void put_units(std::vector<int> &out, int count, int shift, int bits, int sign) {
    std::vector<Unit> t((size_t)1 << count);
    t[0] = Unit{1ll << 62, 0};
    for (size_t j = 1; j < t.size(); j++) {
        int low = 0;
        while (!((j >> low) & 1)) low++;
        t[j] = (j & (j - 1)) ? t[j & (j - 1)] * root(bits - shift - low) : root(bits - shift - low);
    }
    for (const Unit &u : t) put(out, (u.c + 2) >> 2, sign * ((u.s + 2) >> 2));
}
}  // namespace

void dft_fixed_tables(const Op &op, std::vector<int> &out) {
    const int K = (int)op.targets.size(), ns = (int)op.controls.size(), hT = dft_table_split(K, ns);
    put_units(out, K, 0, K, op.sign);
    put_units(out, hT, 0, K + ns, op.sign);
    put_units(out, K + ns - hT, hT, K + ns, op.sign);
}

void phase_fixed_table(const std::vector<cd> &v, std::vector<int> &out) {
    out.reserve(out.size() + 4 * v.size());
    for (const cd &z : v) put(out, std::llrint(z.real() * 0x1p60), std::llrint(z.imag() * 0x1p60));
}
}  // namespace qsim
