// Navier-Stokes projection step on the periodic square (Section 4.1), the
// velocity the stress step is coupled to.  One step t_n -> t_{n+1}, BDF2 with
// the extrapolation E(f) = 2 f^n - f^{n-1} (eq. BDF_and_extrapolation),
// nu = beta/Re, sigma the polymer stress whose divergence drives the momentum
// equation (eq. Navier_Stokes):
//   Xi = (b1 u^n + b2 u^{n-1})/dt + E(nu curl curl u + (u.grad)u - div sigma)
//        (eq. time_discretization_NS; curl curl u = grad div u - Lap u, eq. velocity_correction)
//   Lap p = -div Xi, mean(p) = 0                                   (eq. NS_Poisson)
//   (b0/dt) u^{n+1} - nu Lap u^{n+1} = -grad p - (b1 u^n + b2 u^{n-1})/dt
//        + E(-(u.grad)u + div sigma)                               (eq. NS_Helmholtz)
// On the periodic grid every operator is diagonal in Fourier space: d/dx_a
// multiplies mode k by i k_a (zero at the Nyquist wavenumber of the axis), the
// Laplacian is the square of that, so Poisson and Helmholtz are divisions per
// mode and the result is divergence-free to rounding.  Products are formed on
// the grid.  The transforms are this file's own: a Stockham autosort FFT of
// each row in shared memory (the formulation of Govindaraju et al.,
// "High performance discrete Fourier transforms on graphics processors",
// SC 2008) in radix 4, FP64 complex; spectral arrays are kept transposed, [kx][ky].
//
// Bound: the FP64 pipe (2 operations per clock and SM); a row pass over 1024^2 points is
// 33.5 M FP64 operations, 57 us of it.  So the step is arranged to transform
// and to compute as little as possible:
//   - real fields go two to a complex transform (f + i g forward, split by the
//     Hermitian symmetry of real spectra; A + i B inverse);
//   - of the stress only xx - yy and xy are transformed: an isotropic part adds
//     a gradient to the explicit terms, which the projection removes, so a step
//     takes 5 two-dimensional transforms (convection 1, stress 1, velocity 1, gradient 2);
//   - one kernel per mode goes from the two forward transforms to the three
//     inverse ones (splitting, divergence, Helmholtz update, gradient, packing);
//   - products, packing and rounding happen where the row passes load and store,
//     and a pass whose rows become columns next writes them transposed.
// Six launches per step.  Measured per step (FP32 exchange, CUDA events): 1024^2 1.40 -> 0.92 ms (a row
// pass 73 - 86 us, was 83 and its transposes, packing and splitting apart; the kernel per mode 150 us, was
// 153 and 125 in four others), 128^2 49 us.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/tfs.h"
#include "tfs_internal.h"

namespace tfs {
namespace {

constexpr int kMaxLen = 1024;          // longest row transform (two rows of complex doubles in 32 KB)
constexpr int kNsThreads = 256;

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
// conjugate, on the integer pipe
__device__ __forceinline__ double2 conj_of(double2 a) {
    return make_double2(a.x, __longlong_as_double(__double_as_longlong(a.y) ^ (long long)0x8000000000000000ull));
}
// i d a for a real d (the first-derivative multiplier)
__device__ __forceinline__ double2 cimul(double d, double2 a) { return make_double2(-d * a.y, d * a.x); }

// What a row pass reads: complex rows, two real fields as f + i g (g absent: 0),
// the stress as (xx - yy) + i xy, or the convective term of the grid fields
// u [2][N] and kap [4][N], (u.grad)u_x + i (u.grad)u_y.
enum { kLoadComplex, kLoadPair, kLoadStress, kLoadConvection };
// What it writes: complex rows, complex rows transposed (out[c][r]), or the real
// and imaginary parts as real fields (FP64 and the caller's type, each when given).
enum { kStoreRows, kStoreTransposed, kStoreFields };

template <typename T>
struct RowPass {
    const double2* in[3];      // one per blockIdx.y
    double2* out[3];
    const T *f, *g;            // kLoadPair, kLoadStress (f: packed xx, xy, yy)
    const double *u, *kap;     // kLoadConvection
    double *da[3], *db[3];     // kStoreFields
    T *ta[3], *tb[3];
    int n, rows, per_block;    // row length, rows, rows per block
    const double2* tw;
    int inverse;
    long long N;
};

// Points a block transforms at most (measured at 1024^2: 925 us per step against 974 with 2048, whose
// 512 blocks of a pass leave an SM's last wave nearly empty), and blocks a pass should have at
// least: shorter rows go one to a block on small grids.
constexpr int kRowElems = 1024;
constexpr int kRowBlocks = 152;

// DFT of each row of length n (a power of two, 2 .. kMaxLen) with
// exp(-+ 2 pi i j k / n) (forward / inverse), unscaled; a block takes per_block
// rows.  tw[t] = exp(-2 pi i t / n), t < n (computed once on the host
// in FP64).  Stockham autosort, radix 4: stage Ns = 1, 4, 16, ... takes the
// four operands j + r n/4 (r = 0..3) of butterfly j, turns operand r by
// exp(-+ 2 pi i r k / (4 Ns)) = tw[r k n / (4 Ns)], k = j mod Ns, applies the
// 4-point DFT and writes output r to (j / Ns) 4 Ns + k + r Ns; a length that is
// not a power of four ends with one radix-2 stage (Ns = n/2).  A stage holds its butterflies in
// registers between reading and writing the one shared buffer, whose
// rows are n + 1 apart (the transposed store then reads different banks).
// Several blocks per SM and more than one wave of them, so that the loads and
// stores of some run beside the arithmetic of others.
template <typename T, int LOAD, int STORE>
__global__ void __launch_bounds__(kNsThreads, 5) fft_pass_kernel(const RowPass<T> A) {
    extern __shared__ double2 fft_buf[];
    const int n = A.n, R = A.per_block, ld = n + 1;
    const int which = blockIdx.y;
    const int r0 = blockIdx.x * R;
    const int tid = threadIdx.x;
    const int count = R * n;
    const int lg = 31 - __clz(n);
    for (int e = tid; e < count; e += kNsThreads) {
        const int r = e >> lg, c = e & (n - 1);
        const long long q = ((long long)(r0 + r) << lg) + c;
        double2 v;
        if (LOAD == kLoadComplex) v = A.in[which][q];
        else if (LOAD == kLoadPair) v = make_double2((double)A.f[q], A.g ? (double)A.g[q] : 0.0);
        else if (LOAD == kLoadStress) v = make_double2((double)A.f[q] - (double)A.f[2 * A.N + q], (double)A.f[A.N + q]);
        else {
            const double ux = A.u[q], uy = A.u[A.N + q];
            v = make_double2(ux * A.kap[q] + uy * A.kap[A.N + q], ux * A.kap[2 * A.N + q] + uy * A.kap[3 * A.N + q]);
        }
        fft_buf[r * ld + c] = v;
    }
    __syncthreads();
    const int quarter = n >> 2;
    const bool inverse = A.inverse != 0;
    constexpr int kMine = kRowElems / 4 / kNsThreads;   // butterflies of a thread, held in registers
    int ns = 1;
    for (; 4 * ns <= n; ns <<= 2) {
        const int step = n / (4 * ns), lq = lg - 2;
        double2 o[kMine][4];
#pragma unroll
        for (int i = 0; i < kMine; ++i) {
            const int b = tid + i * kNsThreads;
            if (b >= R * quarter) continue;
            const int j = b & (quarter - 1), k = j & (ns - 1);
            const double2* x = fft_buf + (b >> lq) * ld;
            const double2 v0 = x[j];
            double2 v1 = x[j + quarter], v2 = x[j + 2 * quarter], v3 = x[j + 3 * quarter];
            if (ns > 1) {   // the first stage's twiddles are all 1
                double2 t1 = __ldg(A.tw + k * step), t2 = __ldg(A.tw + 2 * k * step), t3 = __ldg(A.tw + 3 * k * step);
                if (inverse) {
                    t1 = conj_of(t1);
                    t2 = conj_of(t2);
                    t3 = conj_of(t3);
                }
                v1 = cmul(v1, t1);
                v2 = cmul(v2, t2);
                v3 = cmul(v3, t3);
            }
            const double2 a0 = cadd(v0, v2), a1 = csub(v0, v2), a2 = cadd(v1, v3), d = csub(v1, v3);
            // (v1 - v3) times -i (forward) or +i (inverse) joins a1
            const double2 p = make_double2(a1.x - d.y, a1.y + d.x), m = make_double2(a1.x + d.y, a1.y - d.x);
            o[i][0] = cadd(a0, a2);
            o[i][2] = csub(a0, a2);
            o[i][1] = inverse ? p : m;
            o[i][3] = inverse ? m : p;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kMine; ++i) {
            const int b = tid + i * kNsThreads;
            if (b >= R * quarter) continue;
            const int j = b & (quarter - 1), k = j & (ns - 1);
            double2* y = fft_buf + (b >> lq) * ld + ((j - k) << 2) + k;
            y[0] = o[i][0];
            y[ns] = o[i][1];
            y[2 * ns] = o[i][2];
            y[3 * ns] = o[i][3];
        }
        __syncthreads();
    }
    if (ns < n) {   // radix-2 stage, Ns = n/2: reads and writes the same two places
        const int half = n >> 1, lh = lg - 1;
        for (int b = tid; b < R * half; b += kNsThreads) {
            const int j = b & (half - 1);
            double2* x = fft_buf + (b >> lh) * ld;
            double2 t = __ldg(A.tw + j);
            if (inverse) t = conj_of(t);
            const double2 a = x[j], v = cmul(x[j + half], t);
            x[j] = cadd(a, v);
            x[j + half] = csub(a, v);
        }
        __syncthreads();
    }
    if (STORE == kStoreTransposed) {
        const int lr = 31 - __clz(R);
        for (int e = tid; e < count; e += kNsThreads) {
            const int r = e & (R - 1), c = e >> lr;
            A.out[which][(long long)c * A.rows + r0 + r] = fft_buf[r * ld + c];
        }
    } else {
        for (int e = tid; e < count; e += kNsThreads) {
            const int r = e >> lg, c = e & (n - 1);
            const long long q = ((long long)(r0 + r) << lg) + c;
            const double2 v = fft_buf[r * ld + c];
            if (STORE == kStoreRows) {
                A.out[which][q] = v;
            } else {
                if (A.da[which]) A.da[which][q] = v.x;
                if (A.ta[which]) A.ta[which][q] = (T)v.x;
                if (A.db[which]) A.db[which][q] = v.y;
                if (A.tb[which]) A.tb[which][q] = (T)v.y;
            }
        }
    }
}

// Spectra of the two real fields of Z = DFT(f + i g) ([kx][ky], row kx of n1
// entries): with W = conj(Z(-k)), F = (Z + W)/2 and G = (Z - W)/(2i), the
// Hermitian and anti-Hermitian parts (G not written when absent).
__global__ void unpack_pair_kernel(const double2* Z, double2* F, double2* G, int n0, int n1) {
    const long long n = (long long)n0 * n1;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(q / n1), j = (int)(q - (long long)i * n1);
        const long long qm = (long long)(i == 0 ? 0 : n0 - i) * n1 + (j == 0 ? 0 : n1 - j);
        const double2 z = Z[q], zm = Z[qm];
        F[q] = make_double2(0.5 * (z.x + zm.x), 0.5 * (z.y - zm.y));
        if (G) G[q] = make_double2(0.5 * (z.y + zm.y), -0.5 * (z.x - zm.x));
    }
}

// First-derivative multipliers d_x, d_y of spectral entry idx of the
// transposed layout [kx][ky] (row kx of n1 entries): wavenumber times 2 pi / L,
// zero at the Nyquist index of each axis.
__device__ __forceinline__ void wavenumbers(long long idx, int n0, int n1, double sx, double sy, double& dx,
                                            double& dy) {
    const int qi = (int)idx;   // n0 n1 <= kMaxLen^2
    const int i = qi / n1, j = qi - i * n1;
    dx = i == n0 / 2 ? 0.0 : (double)(i < n0 / 2 ? i : i - n0) * sx;
    dy = j == n1 / 2 ? 0.0 : (double)(j < n1 / 2 ? j : j - n1) * sy;
}

#define NS_LOOP(i, n) for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (n); \
                           i += (long long)gridDim.x * blockDim.x)

// divergence-free part of (ux, uy) in place: u -= grad phi, Lap phi = div u (mode 0 kept)
__global__ void ns_project_kernel(double2* ux, double2* uy, int n0, int n1, double sx, double sy) {
    NS_LOOP(q, (long long)n0 * n1) {
        double dx, dy;
        wavenumbers(q, n0, n1, sx, sy, dx, dy);
        const double k2 = dx * dx + dy * dy;
        if (k2 <= 0.0) continue;
        const double2 div = cadd(cimul(dx, ux[q]), cimul(dy, uy[q]));
        const double2 phi = cscale(div, -1.0 / k2);
        ux[q] = csub(ux[q], cimul(dx, phi));
        uy[q] = csub(uy[q], cimul(dy, phi));
    }
}

// Inputs of the three inverse transforms of the velocity (ux, uy) at mode (dx, dy),
// times scale: ux + i uy, and per component d_x u + i d_y u = (-dy + i dx) u
// (the gradient entries 0, 1 and 2, 3 of kappa as real and imaginary parts).
__device__ __forceinline__ void pack_velocity(double2 ux, double2 uy, double dx, double dy, double scale, double2* zu,
                                              double2* z0, double2* z1) {
    const double2 a = cscale(ux, scale), b = cscale(uy, scale);
    *zu = make_double2(a.x - b.y, a.y + b.x);
    *z0 = make_double2(-dy * a.x - dx * a.y, dx * a.x - dy * a.y);
    *z1 = make_double2(-dy * b.x - dx * b.y, dx * b.x - dy * b.y);
}

__global__ void ns_pack_kernel(const double2* ux, const double2* uy, double2* zu, double2* z0, double2* z1, int n0,
                               int n1, double sx, double sy, double scale) {
    NS_LOOP(q, (long long)n0 * n1) {
        double dx, dy;
        wavenumbers(q, n0, n1, sx, sy, dx, dy);
        pack_velocity(ux[q], uy[q], dx, dy, scale, zu + q, z0 + q, z1 + q);
    }
}

// One step per Fourier mode.  With the explicit terms f = (u.grad)u - div sigma
// (div sigma up to a gradient: of (xx - yy) and xy alone), h = (b1 u^n + b2 u^{n-1})/dt
// and w = h + E(f): Xi = h + E(nu curl curl u + f), p = i k.Xi / k^2 (Lap p =
// -div Xi), (b0/dt + nu k^2) u^{n+1} = -i k p - w.  In Fourier space
// k.(curl curl u) = k.(k^2 u - k (k.u)) = 0 for every k, so k.Xi = k.w and
//   u^{n+1} = -(w - k (k.w)/k^2) / (b0/dt + nu k^2),
// the projection of -w onto divergence-free fields, which the kernel forms
// directly (the rotational term changes the pressure of the scheme only on a
// bounded domain).  Mode 0: u^{n+1} = -w dt/b0.
// Zc, Zs: the forward transforms of the convective term and of the stress
// (nullptr: none), split by Hermitian symmetry; f1: twice f at level n-1 (nullptr: the
// empty past, f^{n-1} = f^n); f2 receives twice f^n; u^{n+1} goes over u^{n-1}.
struct NsModes {
    const double2 *Zc, *Zs;
    const double2 *ax, *ay;       // u^n
    double2 *bx, *by;             // u^{n-1} in, u^{n+1} out
    const double2 *f1x, *f1y;
    double2 *f2x, *f2y;
    double2 *zu, *z0, *z1;        // packed for the inverse transforms
};

// 2 f at entry q (mode (i, j)) from the two transforms
__device__ __forceinline__ void explicit_terms(const double2* Zc, const double2* Zs, long long q, long long qm,
                                               double dx, double dy, double2& fx, double2& fy) {
    const double2 z = Zc[q], zm = Zc[qm];
    fx = make_double2(z.x + zm.x, z.y - zm.y);
    fy = make_double2(z.y + zm.y, zm.x - z.x);
    if (!Zs) return;
    const double2 s = Zs[q], sm = Zs[qm];
    const double2 D = make_double2(s.x + sm.x, s.y - sm.y), S = make_double2(s.y + sm.y, sm.x - s.x);
    // minus i (dx D + dy S, dx S)
    fx.x += dx * D.y + dy * S.y;
    fx.y -= dx * D.x + dy * S.x;
    fy.x += dx * S.y;
    fy.y -= dx * S.x;
}

__device__ __forceinline__ long long mirrored(long long q, int n0, int n1) {
    const int i = (int)q / n1, j = (int)q - i * n1;
    return (long long)(i == 0 ? 0 : n0 - i) * n1 + (j == 0 ? 0 : n1 - j);
}

__global__ void __launch_bounds__(kNsThreads) ns_update_kernel(const NsModes M, int n0, int n1, double sx, double sy,
                                                               double nu, double b0dt, double b1dt, double b2dt,
                                                               double inv0, double scale) {
    NS_LOOP(q, (long long)n0 * n1) {
        double dx, dy;
        wavenumbers(q, n0, n1, sx, sy, dx, dy);
        double2 fx, fy;
        explicit_terms(M.Zc, M.Zs, q, mirrored(q, n0, n1), dx, dy, fx, fy);
        // w = h + 2 f^n - f^{n-1}; without a past f^{n-1} = f^n
        const double2 gx = M.f1x ? M.f1x[q] : fx, gy = M.f1y ? M.f1y[q] : fy;
        M.f2x[q] = fx;
        M.f2y[q] = fy;
        const double2 ax = M.ax[q], ay = M.ay[q], bx = M.bx[q], by = M.by[q];
        auto w1 = [&](double a, double b, double f, double g) { return fma(-0.5, g, f + fma(b1dt, a, b2dt * b)); };
        double2 wx = make_double2(w1(ax.x, bx.x, fx.x, gx.x), w1(ax.y, bx.y, fx.y, gx.y));
        double2 wy = make_double2(w1(ay.x, by.x, fy.x, gy.x), w1(ay.y, by.y, fy.y, gy.y));
        const double k2 = dx * dx + dy * dy;
        double inv = inv0;
        if (k2 > 0.0) {
            // one division gives both 1/k^2 and 1/(b0/dt + nu k^2)
            const double den = b0dt + nu * k2;
            const double r = 1.0 / (k2 * den), ik2 = den * r;
            const double2 s = make_double2((dx * wx.x + dy * wy.x) * ik2, (dx * wx.y + dy * wy.y) * ik2);   // (k.w)/k^2
            wx = make_double2(fma(-dx, s.x, wx.x), fma(-dx, s.y, wx.y));
            wy = make_double2(fma(-dy, s.x, wy.x), fma(-dy, s.y, wy.y));
            inv = k2 * r;
        }
        const double2 ux = cscale(wx, -inv), uy = cscale(wy, -inv);
        M.bx[q] = ux;
        M.by[q] = uy;
        pack_velocity(ux, uy, dx, dy, scale, M.zu + q, M.z0 + q, M.z1 + q);
    }
}

// twice f (no stress) of a level from the transform of its convective term
__global__ void ns_terms_kernel(const double2* Zc, double2* fx, double2* fy, int n0, int n1) {
    NS_LOOP(q, (long long)n0 * n1) explicit_terms(Zc, nullptr, q, mirrored(q, n0, n1), 0.0, 0.0, fx[q], fy[q]);
}

}  // namespace
}  // namespace tfs

using namespace tfs;

struct tfs_ns_ctx {
    int n0 = 0, n1 = 0;
    long long N = 0;
    double sx = 0, sy = 0;        // 2 pi / L per axis
    double nu = 0, dt = 0;
    int precision = TFS_FP64;
    char* ws = nullptr;
    size_t ws_bytes = 0;
    // spectral (complex, [kx][ky]): velocity levels and twice the explicit terms
    // of levels n and n-1 ([level slot][component]); the transforms' inputs and outputs
    double2* uh[2][2] = {};
    double2* fh[2][2] = {};
    double2* za[3] = {};
    double2* zb[3] = {};
    // grid fields (FP64): u^n [2][N], kappa^n [4][N]
    double* u = nullptr;
    double* kap = nullptr;
    double2* tw0 = nullptr;       // exp(-2 pi i t / n0), t < n0; and for n1
    double2* tw1 = nullptr;
    std::vector<double2> tw_host; // both tables, uploaded by tfs_ns_set_state
    int cur = 0;                  // slot of level n (n-1 in the other)
    bool have_prev_terms = false; // f^{n-1} exists (else the empty past: f^{n-1} = f^n)
    bool state_set = false;
    long long step = 0;
};

namespace {

constexpr size_t kNsAlign = 256;
size_t ns_up(size_t v) { return (v + kNsAlign - 1) / kNsAlign * kNsAlign; }

size_t ns_bytes(const tfs_ns_ctx* h) {
    const size_t cplx = ns_up(sizeof(double2) * (size_t)h->N), real = ns_up(sizeof(double) * (size_t)h->N);
    return 14 * cplx + 6 * real + ns_up(sizeof(double2) * (size_t)(h->n0 + h->n1));
}

void ns_layout(tfs_ns_ctx* h) {
    const size_t cplx = ns_up(sizeof(double2) * (size_t)h->N), real = ns_up(sizeof(double) * (size_t)h->N);
    char* p = h->ws;
    auto take_c = [&]() { double2* r = (double2*)p; p += cplx; return r; };
    for (int l = 0; l < 2; ++l)
        for (int a = 0; a < 2; ++a) h->uh[l][a] = take_c();
    for (int l = 0; l < 2; ++l)
        for (int a = 0; a < 2; ++a) h->fh[l][a] = take_c();
    for (int c = 0; c < 3; ++c) h->za[c] = take_c();
    for (int c = 0; c < 3; ++c) h->zb[c] = take_c();
    h->u = (double*)p;
    p += 2 * real;
    h->kap = (double*)p;
    p += 4 * real;
    h->tw0 = (double2*)p;
    h->tw1 = h->tw0 + h->n0;
}

unsigned ns_grid(long long n) {
    long long b = (n + kNsThreads - 1) / kNsThreads;
    return (unsigned)(b > 4096 ? 4096 : (b < 1 ? 1 : b));
}

// one pass over the rows of `arrays` arrays: axis 0 rows of n0, axis 1 rows of n1
template <typename T, int LOAD, int STORE>
cudaError_t row_pass(const tfs_ns_ctx* h, RowPass<T>& A, int axis, int arrays, bool inverse, cudaStream_t s) {
    A.n = axis == 0 ? h->n0 : h->n1;
    A.rows = axis == 0 ? h->n1 : h->n0;
    A.per_block = kRowElems / A.n < A.rows ? kRowElems / A.n : A.rows;
    while (A.per_block > 1 && A.rows / A.per_block < kRowBlocks) A.per_block /= 2;
    A.tw = axis == 0 ? h->tw0 : h->tw1;
    A.inverse = inverse ? 1 : 0;
    A.N = h->N;
    const size_t smem = (size_t)A.per_block * (A.n + 1) * sizeof(double2);
    fft_pass_kernel<T, LOAD, STORE><<<dim3(A.rows / A.per_block, arrays), kNsThreads, smem, s>>>(A);
    return cudaGetLastError();
}

// Z [kx][ky] = DFT of what the first pass loads
template <typename T, int LOAD>
cudaError_t forward(const tfs_ns_ctx* h, RowPass<T> A, double2* Z, cudaStream_t s) {
    A.out[0] = Z;
    return row_pass<T, LOAD, kStoreTransposed>(h, A, 0, 1, false, s);
}
template <typename T>
cudaError_t forward_second(const tfs_ns_ctx* h, double2* Z0, double2* Z1, cudaStream_t s) {
    RowPass<T> A{};
    A.in[0] = A.out[0] = Z0;
    A.in[1] = A.out[1] = Z1;
    return row_pass<T, kLoadComplex, kStoreRows>(h, A, 1, Z1 ? 2 : 1, false, s);
}

// spectra of two real fields by one transform of f + i g
template <typename T>
cudaError_t fft2_pair(tfs_ns_ctx* h, const T* f, const T* g, double2* F, double2* G, cudaStream_t s) {
    RowPass<T> A{};
    A.f = f;
    A.g = g;
    cudaError_t e = forward<T, kLoadPair>(h, A, h->za[0], s);
    if (e == cudaSuccess) e = forward_second<T>(h, h->za[0], nullptr, s);
    if (e == cudaSuccess) {
        unpack_pair_kernel<<<ns_grid(h->N), kNsThreads, 0, s>>>(h->za[0], F, G, h->n0, h->n1);
        e = cudaGetLastError();
    }
    return e;
}

// grid velocity and gradient of the packed spectra in za (zu, z0, z1): into the FP64
// fields u, kap and, when given, the caller's fields uo [2][N], ko [4][N]
template <typename T>
cudaError_t grid_fields(tfs_ns_ctx* h, T* uo, T* ko, cudaStream_t s) {
    const long long N = h->N;
    RowPass<T> A{};
    for (int c = 0; c < 3; ++c) {
        A.in[c] = h->za[c];
        A.out[c] = h->zb[c];
    }
    cudaError_t e = row_pass<T, kLoadComplex, kStoreTransposed>(h, A, 1, 3, true, s);
    if (e != cudaSuccess) return e;
    for (int c = 0; c < 3; ++c) {
        double* d = c == 0 ? h->u : h->kap + (c == 1 ? 0 : 2) * N;
        T* t = c == 0 ? uo : (ko ? ko + (c == 1 ? 0 : 2) * N : nullptr);
        A.in[c] = h->zb[c];
        A.da[c] = d;
        A.db[c] = d + N;
        A.ta[c] = t;
        A.tb[c] = t ? t + N : nullptr;
    }
    return row_pass<T, kLoadComplex, kStoreFields>(h, A, 0, 3, true, s);
}

template <typename T>
cudaError_t fields_of_level(tfs_ns_ctx* h, const double2* ux, const double2* uy, cudaStream_t s) {
    ns_pack_kernel<<<ns_grid(h->N), kNsThreads, 0, s>>>(ux, uy, h->za[0], h->za[1], h->za[2], h->n0, h->n1, h->sx,
                                                        h->sy, 1.0 / (double)h->N);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? grid_fields<T>(h, nullptr, nullptr, s) : e;
}

template <typename T>
int ns_set_state(tfs_ns_ctx* h, const T* u0, const T* uprev, cudaStream_t s) {
    const long long N = h->N;
    const int c = h->cur, o = 1 - c;
    cudaError_t e = cudaMemcpyAsync(h->tw0, h->tw_host.data(), sizeof(double2) * h->tw_host.size(),
                                    cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = fft2_pair<T>(h, u0, u0 + N, h->uh[c][0], h->uh[c][1], s);
    if (e == cudaSuccess) {
        ns_project_kernel<<<ns_grid(N), kNsThreads, 0, s>>>(h->uh[c][0], h->uh[c][1], h->n0, h->n1, h->sx, h->sy);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && uprev) {
        // the given level n-1 and its explicit terms (no stress)
        e = fft2_pair<T>(h, uprev, uprev + N, h->uh[o][0], h->uh[o][1], s);
        if (e == cudaSuccess) {
            ns_project_kernel<<<ns_grid(N), kNsThreads, 0, s>>>(h->uh[o][0], h->uh[o][1], h->n0, h->n1, h->sx, h->sy);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = fields_of_level<T>(h, h->uh[o][0], h->uh[o][1], s);
        RowPass<T> A{};
        A.u = h->u;
        A.kap = h->kap;
        if (e == cudaSuccess) e = forward<T, kLoadConvection>(h, A, h->za[0], s);
        if (e == cudaSuccess) e = forward_second<T>(h, h->za[0], nullptr, s);
        if (e == cudaSuccess) {
            ns_terms_kernel<<<ns_grid(N), kNsThreads, 0, s>>>(h->za[0], h->fh[o][0], h->fh[o][1], h->n0, h->n1);
            e = cudaGetLastError();
        }
    } else if (e == cudaSuccess) {
        for (int a = 0; a < 2 && e == cudaSuccess; ++a)
            e = cudaMemcpyAsync(h->uh[o][a], h->uh[c][a], sizeof(double2) * (size_t)N, cudaMemcpyDeviceToDevice, s);
    }
    if (e == cudaSuccess) e = fields_of_level<T>(h, h->uh[c][0], h->uh[c][1], s);
    if (e != cudaSuccess) return TFS_ERR_CUDA;
    h->have_prev_terms = uprev != nullptr;
    h->state_set = true;
    h->step = 0;
    return TFS_OK;
}

template <typename T>
int ns_step(tfs_ns_ctx* h, const T* sigma, T* u_out, T* kap_out, cudaStream_t s) {
    const int c = h->cur, o = 1 - c;
    // transforms of the convective term (from the stored grid fields) and of the stress
    RowPass<T> A{};
    A.u = h->u;
    A.kap = h->kap;
    A.f = sigma;
    cudaError_t e = forward<T, kLoadConvection>(h, A, h->zb[0], s);
    if (e == cudaSuccess && sigma) e = forward<T, kLoadStress>(h, A, h->zb[1], s);
    if (e == cudaSuccess) e = forward_second<T>(h, h->zb[0], sigma ? h->zb[1] : nullptr, s);
    if (e != cudaSuccess) return TFS_ERR_CUDA;
    // u^{n+1} is written over u^{n-1}: each mode reads its own entries before writing them
    const bool past = h->have_prev_terms;
    const NsModes M{h->zb[0], sigma ? h->zb[1] : nullptr, h->uh[c][0], h->uh[c][1], h->uh[o][0], h->uh[o][1],
                    past ? h->fh[o][0] : nullptr, past ? h->fh[o][1] : nullptr, h->fh[c][0], h->fh[c][1],
                    h->za[0], h->za[1], h->za[2]};
    ns_update_kernel<<<ns_grid(h->N), kNsThreads, 0, s>>>(M, h->n0, h->n1, h->sx, h->sy, h->nu, kB0 / h->dt,
                                                          kB1 / h->dt, kB2 / h->dt, h->dt / kB0, 1.0 / (double)h->N);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = grid_fields<T>(h, u_out, kap_out, s);
    if (e != cudaSuccess) return TFS_ERR_CUDA;
    h->cur = o;
    h->have_prev_terms = true;
    h->step += 1;
    return TFS_OK;
}

bool pow2(int n) { return n >= 2 && (n & (n - 1)) == 0; }

}  // namespace

extern "C" {

int tfs_ns_create(tfs_ns_handle* out, int n0, int n1, double L0, double L1, double beta, double Re, double dt,
                  int precision) {
    if (!out) return TFS_ERR_ARG;
    *out = nullptr;
    if (!pow2(n0) || !pow2(n1) || n0 > kMaxLen || n1 > kMaxLen) return TFS_ERR_ARG;
    if (!(L0 > 0.0) || !(L1 > 0.0) || !std::isfinite(L0) || !std::isfinite(L1)) return TFS_ERR_ARG;
    if (!(beta > 0.0 && beta <= 1.0) || !(Re > 0.0) || !std::isfinite(Re) || !(dt > 0.0) || !std::isfinite(dt))
        return TFS_ERR_ARG;
    if (precision != TFS_FP64 && precision != TFS_FP32 && precision != TFS_FP32_PLAIN) return TFS_ERR_ARG;
    tfs_ns_ctx* h = new (std::nothrow) tfs_ns_ctx();
    if (!h) return TFS_ERR_ARG;
    h->n0 = n0;
    h->n1 = n1;
    h->N = (long long)n0 * n1;
    h->sx = 2.0 * 3.14159265358979323846 / L0;
    h->sy = 2.0 * 3.14159265358979323846 / L1;
    h->nu = beta / Re;
    h->dt = dt;
    h->precision = precision;
    // twiddle tables exp(-2 pi i t / n), t < n, of both axes (FP64, host)
    for (int n : {n0, n1})
        for (int t = 0; t < n; ++t) {
            const double a = -2.0 * 3.14159265358979323846 * (double)t / (double)n;
            h->tw_host.push_back(make_double2(std::cos(a), std::sin(a)));
        }
    *out = h;
    return TFS_OK;
}

size_t tfs_ns_workspace_bytes(tfs_ns_handle h) { return h ? ns_bytes(h) : 0; }

int tfs_ns_bind_workspace(tfs_ns_handle h, void* dev_ptr, size_t bytes) {
    if (!h || !dev_ptr || ((uintptr_t)dev_ptr % kNsAlign) != 0) return TFS_ERR_ARG;
    if (bytes < ns_bytes(h)) return TFS_ERR_NOWORKSPACE;
    h->ws = (char*)dev_ptr;
    h->ws_bytes = bytes;
    ns_layout(h);
    h->state_set = false;
    return TFS_OK;
}

int tfs_ns_set_state(tfs_ns_handle h, const void* u0, const void* u_prev, void* stream) {
    if (!h || !u0) return TFS_ERR_ARG;
    if (!h->ws) return TFS_ERR_NOWORKSPACE;
    return h->precision == TFS_FP64
               ? ns_set_state<double>(h, (const double*)u0, (const double*)u_prev, (cudaStream_t)stream)
               : ns_set_state<float>(h, (const float*)u0, (const float*)u_prev, (cudaStream_t)stream);
}

int tfs_ns_step(tfs_ns_handle h, const void* sigma, void* u_out, void* grad_u_out, void* stream) {
    if (!h) return TFS_ERR_ARG;
    if (!h->ws) return TFS_ERR_NOWORKSPACE;
    if (!h->state_set) return TFS_ERR_STATE;
    return h->precision == TFS_FP64
               ? ns_step<double>(h, (const double*)sigma, (double*)u_out, (double*)grad_u_out, (cudaStream_t)stream)
               : ns_step<float>(h, (const float*)sigma, (float*)u_out, (float*)grad_u_out, (cudaStream_t)stream);
}

int tfs_ns_destroy(tfs_ns_handle h) {
    delete h;
    return TFS_OK;
}

}  // extern "C"
