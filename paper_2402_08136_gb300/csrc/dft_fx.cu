// Fixed-point Fourier-transform passes for complex128 amplitudes: launch and tables (kernels in
// dft_fx.cuh).
#include "dft_fx.cuh"

namespace qsim {
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
    for (const cd &z : v) put(out, std::llrint(z.real() * 0x1p60), std::llrint(z.imag() * 0x1p60));
}
}  // namespace qsim
