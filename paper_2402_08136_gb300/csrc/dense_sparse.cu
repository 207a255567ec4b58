// Dense-gate kernels for two shapes on which the tiled kernels wait instead of working (sm_103a):
// complex128 gates whose matrix is mostly zeros, and states of a few groups.
//
// Mostly zero gates (sparse_kernel; fused Hadamards and phases, controlled gates and permutations
// written as dense matrices): the dense form spends 4 2^k FP64 multiply-adds per amplitude on them, at 2
// per clock and SM.  Here row r holds its W nonzero entries, so an amplitude costs 4 W (2 W for a
// real U), in the dense form's order: the terms left out are exact zeros.  17 qubits, 4 targets, 2 entries
// a row: 40 us dense.  A tile with a value that is not finite runs over whole rows, so that
// infinities and NaN spread as in the dense form.
//
// Few groups (group_kernel; the eigenvector rotation that opens an HHL run acts on the data register
// alone, one group): the tiled kernels give one warp a chain of 16 rows times 2^k columns (7 targets
// complex64 21 us, 6 targets complex128 80 us).  Here a CTA takes one group and a thread one part of
// one row, its columns in the tiled kernels' order (the same bits).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.h"

namespace qsim {
namespace sparse {

constexpr int kThreads = 256;
constexpr int kMaxFix = 40;

template <typename R> struct C2;
template <> struct C2<float> { using T = float2; };
template <> struct C2<double> { using T = double2; };

struct Args {
    double2 *psi;
    const double2 *val;       // W entries per row, columns ascending
    const int *col;
    const double2 *Ut;        // the whole matrix, transposed
    long long ntiles;
    unsigned long long cmask;
    int T, L0, nh, K, W, real_u;
    int hpos[16];             // qubits of tile bits L0..T-1
    int nfix;
    int fix[kMaxFix];         // ascending: tile qubits above L0, controls
    int tloc[8];              // tile-local bit of target b
};

__global__ void __launch_bounds__(kThreads) sparse_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int T = a.T, D = 1 << a.K, amps = 1 << T;
    double2 *tile = reinterpret_cast<double2 *>(smem_raw);
    double2 *val = tile + amps;                                       // [D][W]
    long long *hoff = reinterpret_cast<long long *>(val + D * a.W);   // 2^nh
    int *off = reinterpret_cast<int *>(hoff + (1 << a.nh));           // tile-local offset of a row's entry
    int *toff = off + D * a.W;                                        // ... and of amplitude c
    const int tid = threadIdx.x, lomask = (1 << a.L0) - 1;
    for (int c = tid; c < D; c += kThreads) {
        int o = 0;
        for (int b = 0; b < a.K; b++)
            if ((c >> b) & 1) o |= 1 << a.tloc[b];
        toff[c] = o;
    }
    for (int h = tid; h < (1 << a.nh); h += kThreads) {
        long long o = 0;
        for (int i = 0; i < a.nh; i++)
            if ((h >> i) & 1) o |= 1ll << a.hpos[i];
        hoff[h] = o;
    }
    __syncthreads();
    for (int i = tid; i < D * a.W; i += kThreads) {
        val[i] = a.val[i];
        off[i] = toff[a.col[i]];
    }
    int tmask = 0;
    for (int b = 0; b < a.K; b++) tmask |= 1 << a.tloc[b];
    for (long long t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        unsigned long long base = (unsigned long long)t << a.L0;
        for (int i = 0; i < a.nfix; i++) {
            const int p = a.fix[i];
            base = ((base >> p) << (p + 1)) | (base & ((1ull << p) - 1ull));
        }
        base |= a.cmask;
        bool bad = false;
        for (int l = tid; l < amps; l += kThreads) {
            const double2 z = a.psi[base + hoff[l >> a.L0] + (l & lomask)];
            bad |= !isfinite(z.x) || !isfinite(z.y);
            tile[l] = z;
        }
        bad = __syncthreads_or(bad);
        for (int l = tid; l < amps; l += kThreads) {
            int r = 0;
            for (int b = 0; b < a.K; b++) r |= ((l >> a.tloc[b]) & 1) << b;
            const double2 *x = tile + (l & ~tmask);
            double2 s = make_double2(0.0, 0.0);
            const int cnt = bad ? D : a.W;
            for (int j = 0; j < cnt; j++) {
                const double2 u = bad ? a.Ut[j * D + r] : val[r * a.W + j];
                const double2 z = x[bad ? toff[j] : off[r * a.W + j]];
                s.x = fma(u.x, z.x, s.x);
                if (!a.real_u) s.x = fma(-u.y, z.y, s.x);
                s.y = fma(u.x, z.y, s.y);
                if (!a.real_u) s.y = fma(u.y, z.x, s.y);
            }
            a.psi[base + hoff[l >> a.L0] + (l & lomask)] = s;
        }
        __syncthreads();
    }
}

// One group per CTA: thread (row, re or im).
struct GroupArgs {
    void *psi;
    const void *Ut;
    unsigned long long cmask;
    int K, real_u, nfix;
    int fix[kMaxFix];
    int targets[8];
};

template <typename R>
__global__ void __launch_bounds__(256) group_kernel(const __grid_constant__ GroupArgs a) {
    using V = typename C2<R>::T;
    __shared__ V x[128];
    const int D = 1 << a.K, tid = threadIdx.x, r = tid >> 1;
    unsigned long long base = blockIdx.x;
    for (int i = 0; i < a.nfix; i++) {
        const int p = a.fix[i];
        base = ((base >> p) << (p + 1)) | (base & ((1ull << p) - 1ull));
    }
    base |= a.cmask;
    for (int b = 0; b < a.K; b++)
        if ((r >> b) & 1) base |= 1ull << a.targets[b];
    V *psi = static_cast<V *>(a.psi) + base;
    if (!(tid & 1)) x[r] = *psi;
    __syncthreads();
    const V *u = static_cast<const V *>(a.Ut) + r;
    R s = 0;
    if (a.real_u) {
#pragma unroll 16
        for (int c = 0; c < D; c++) s = fma(u[c * D].x, (tid & 1) ? x[c].y : x[c].x, s);
    } else {
#pragma unroll 16
        for (int c = 0; c < D; c++) {
            const V w = u[c * D], z = x[c];
            s = fma(w.x, (tid & 1) ? z.y : z.x, s);
            s = fma((tid & 1) ? w.y : -w.y, (tid & 1) ? z.x : z.y, s);
        }
    }
    reinterpret_cast<R *>(psi)[tid & 1] = s;
}

}  // namespace sparse

static void cuda_check(const char *what) {
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw Error(QSIM_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Largest number of nonzero entries in a row, when that is at most half of the row (0: not sparse).
int sparse_width(const Op &op) {
    const int k = (int)op.targets.size(), D = 1 << k;
    if (op.kind != OP_DENSE || k > 7) return 0;
    int W = 0;
    for (int r = 0; r < D; r++) {
        int nz = 0;
        for (int c = 0; c < D; c++) nz += op.U[(size_t)r * D + c] != cd(0.0, 0.0);
        W = std::max(W, nz);
    }
    return W >= 1 && 2 * W <= D && D * W <= 1024 ? W : 0;
}

// W entries per row (values, then columns); rows with fewer end in zeros on the row's own column
void sparse_pack(const Op &op, std::vector<unsigned char> &blob) {
    const int D = 1 << (int)op.targets.size(), W = op.sparse_w;
    std::vector<double> val;
    std::vector<int> col;
    for (int r = 0; r < D; r++) {
        int n = 0;
        for (int c = 0; c < D; c++) {
            const cd u = op.U[(size_t)r * D + c];
            if (u == cd(0.0, 0.0)) continue;
            val.push_back(u.real());
            val.push_back(u.imag());
            col.push_back(c);
            n++;
        }
        for (; n < W; n++) {
            val.insert(val.end(), {0.0, 0.0});
            col.push_back(r);
        }
    }
    const unsigned char *p = reinterpret_cast<const unsigned char *>(val.data());
    blob.insert(blob.end(), p, p + val.size() * sizeof(double));
    p = reinterpret_cast<const unsigned char *>(col.data());
    blob.insert(blob.end(), p, p + col.size() * sizeof(int));
}

// False (nothing launched): a real U with half of a row nonzero on 2^20 amplitudes or more.  The row form is bound by the
// reads of its entries there, as long for a real U as for a complex one, and the tiled kernels' real form is ahead: 25
// qubits, 1..5 targets 428, 650, 1081, 1945, 3715 us here and 270, 517, 1027, 1785, 3520 there (20 qubits: 29.5, 38.5, 54, 87,
// 151 and 27, 36, 54, 84, 148; 18 qubits: 19, 22, 26, 34, 51 and 20, 22, 27, 36, 54).  With fewer entries, or a complex U, the
// row form is never behind.
bool launch_sparse(void *state, int n, const Op &op, const void *ell, const void *Ut, int sms, cudaStream_t st) {
    sparse::Args a;
    std::memset(&a, 0, sizeof(a));
    const int K = (int)op.targets.size(), D = 1 << K, avail = n - (int)op.controls.size();
    if (op.real_u && 2 * op.sparse_w == D && avail >= 20) return false;
    a.psi = static_cast<double2 *>(state);
    a.W = op.sparse_w;
    a.K = K;
    a.val = static_cast<const double2 *>(ell);
    a.col = reinterpret_cast<const int *>(a.val + (size_t)D * a.W);
    a.Ut = static_cast<const double2 *>(Ut);
    a.real_u = op.real_u ? 1 : 0;
    unsigned long long cm = 0, tm = 0;
    for (int q : op.controls) cm |= 1ull << q;
    for (int q : op.targets) tm |= 1ull << q;
    a.cmask = cm;
    // tiles of 2^11 amplitudes (32 KB), smaller on states with too few of them for the chip
    a.T = std::min(avail, std::max(K + 3, std::min(11, avail - 9)));
    std::vector<int> ts(op.targets.begin(), op.targets.end());
    for (int q = 0; q < n && (int)ts.size() < a.T; q++)
        if (!(((cm | tm) >> q) & 1ull)) ts.push_back(q);
    std::sort(ts.begin(), ts.end());
    while (a.L0 < a.T && ts[a.L0] == a.L0) a.L0++;
    a.nh = a.T - a.L0;
    std::vector<int> fix(ts.begin() + a.L0, ts.end());
    for (int i = 0; i < a.nh; i++) a.hpos[i] = ts[a.L0 + i];
    fix.insert(fix.end(), op.controls.begin(), op.controls.end());
    std::sort(fix.begin(), fix.end());
    QSIM_REQUIRE((int)fix.size() <= sparse::kMaxFix && a.nh <= 16, "tile layout");
    a.nfix = (int)fix.size();
    for (int i = 0; i < a.nfix; i++) a.fix[i] = fix[i];
    for (int b = 0; b < K; b++) a.tloc[b] = (int)(std::find(ts.begin(), ts.end(), op.targets[b]) - ts.begin());
    a.ntiles = 1ll << (avail - a.T);
    const size_t smem = ((size_t)16 << a.T) + (size_t)D * a.W * 20 + (8ull << a.nh) + 4 * D;
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(sparse::sparse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        cuda_check("sparse_kernel attribute");
        attr = true;
    }
    const int per_sm = occupancy_cached(reinterpret_cast<const void *>(sparse::sparse_kernel), sparse::kThreads, smem);
    QSIM_REQUIRE(per_sm > 0, "sparse_kernel does not fit on an SM");
    const long long grid = std::min<long long>(a.ntiles, (long long)sms * per_sm);
    sparse::sparse_kernel<<<(int)grid, sparse::kThreads, smem, st>>>(a);
    cuda_check("sparse_kernel");
    note_launches(1, QSIM_KERNEL_DENSE_SIMT);
    return true;
}

// At most 8 groups (a CTA each): larger states fill the tiled kernels' warps.
bool launch_group(void *state, int n, int dtype, const Op &op, const void *Ut, cudaStream_t st) {
    const int K = (int)op.targets.size(), free_bits = n - K - (int)op.controls.size();
    if (K < 3 || free_bits < 0 || free_bits > 3) return false;
    sparse::GroupArgs a;
    std::memset(&a, 0, sizeof(a));
    a.psi = state;
    a.Ut = Ut;
    a.K = K;
    a.real_u = op.real_u ? 1 : 0;
    std::vector<int> fix(op.targets.begin(), op.targets.end());
    for (int q : op.controls) {
        fix.push_back(q);
        a.cmask |= 1ull << q;
    }
    std::sort(fix.begin(), fix.end());
    QSIM_REQUIRE((int)fix.size() <= sparse::kMaxFix, "too many fixed qubits");
    a.nfix = (int)fix.size();
    for (int i = 0; i < a.nfix; i++) a.fix[i] = fix[i];
    for (int b = 0; b < K; b++) a.targets[b] = op.targets[b];
    if (dtype == QSIM_C128) sparse::group_kernel<double><<<1 << free_bits, 2 << K, 0, st>>>(a);
    else sparse::group_kernel<float><<<1 << free_bits, 2 << K, 0, st>>>(a);
    cuda_check("group_kernel");
    note_launches(1, QSIM_KERNEL_DENSE_SIMT);
    return true;
}

}  // namespace qsim
