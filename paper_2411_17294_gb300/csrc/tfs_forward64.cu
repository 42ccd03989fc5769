// Forward stress step in FP64 storage: one launch advances every grid point
// from t_n to t_{n+1} (the same step as tfs_forward.cu, which serves FP32
// storage), all arithmetic in FP64.
//
// Bound.  FP64 runs at about 2 operations per clock and SM on this GPU
// (0.5 - 0.6 T/s), so the step is bound by the number of FP64 instructions, not
// by its bytes: 4 per (mode, component) here and about 160 (3D) or 66 (2D) per
// point for the rest (an FP64 elimination alone takes 250 in 3D).  Hence
//   - Q'_j = x - y/4 instead of Q_j = b1 x + b2 y = -2 Q'_j, with the power of two
//     in the constants (-2 eta_j, 2 c_j): one FMA for Q', one for the history
//     sum, two for the push-forward, and bitwise the same values (5 before);
//   - the transport stencil inside the step: its coefficients are formed once
//     per point, each component then takes 3 taps per axis (the tap that the
//     upwinding leaves out is not loaded), no separate launch, no term
//     written and read back;
//   - no staging of whole tiles: a warp owns one component of 32 points and
//     loads both levels of its modes straight into registers, eight modes ahead;
//     only Q' stays in shared memory (m nc 256 bytes, read back by the thread
//     that wrote it).  Two to eight tiles fit an SM where the staged form held one
//     (3D, m = 48) to four, so one tile's memory latency hides behind the others;
//   - the point systems by FP32 LU and refinement with FP64 residuals: a thread
//     owns one component of one point throughout, the warps of a tile factor its
//     32 matrices in FP32 (each for itself, the FP32 pipe is idle), and each
//     thread forms its component's residual, so a solve costs about 20 FP64
//     operations per component and none of it waits for one warp.  FP64 Gaussian
//     elimination with partial pivoting serves the points whose refinement does
//     not contract, or whose numbers leave the FP32 range;
//   - grids of few tiles split a tile's modes over several warps.
// Measured per step (CUDA events, back to back) against the staged form this replaces: 3D 160^3,
// m = 48: 26.7 -> 11.1 ms; 3D 192^3, m = 32 with transport: 22.9 -> 14.5 ms; 2D 1024^2, m = 32:
// 1.18 -> 0.87 ms, with transport 1.45 -> 1.00 ms; 2D 64^2, m = 16 with transport: 27.3 -> 10.3 us.
// The FP64 pipe is 83% (3D) and 87% (2D) busy with 927 FP64 instructions per 32-point tile at 3D,
// m = 32.  Error against 64-bit references no larger than before (3.2e-16 against 4.8e-16 normwise
// at 3D 160^3, 7.3e-16 against 8.9e-16 at 2D 1024^2).
#include <cuda_runtime.h>

#include <cmath>

#include "tfs_device.cuh"
#include "tfs_internal.h"
#include "tfs_solve64.cuh"

namespace tfs {
namespace {

constexpr int kAhead = 8;    // modes whose two levels a thread loads before using them

// where the transport term comes from
enum { kNoTransport = 0, kInStep = 1, kFromPrepass = 2 };

template <int DIM>
struct Shape64 {
    static constexpr int NC = Packed<DIM>::NC;
    static constexpr int kSplit = 12 / NC;    // mode groups of a tile on small grids
    static constexpr int kCoef = 3 * DIM + 1; // stencil coefficients of a point
};

template <int DIM>
__host__ __device__ constexpr size_t smem64_bytes(int m, int groups) {
    constexpr int NC = Packed<DIM>::NC;
    return (size_t)kT64 * sizeof(double) *
               ((size_t)m * NC + (size_t)groups * NC + 3 * NC + DIM * DIM + Shape64<DIM>::kCoef) +
           (size_t)kT64 * sizeof(float) * DIM * DIM;
}

// Products of the step's scalars, formed once on the host.
struct Step64 {
    // what kappa* is scaled by: dt, in the paper's variable dt xi with xi's power of two apart (xi = frac 2^kexp,
    // frac in [1, 2), so that xi = 0, a table without weight, divides nothing; then kexp is far out of range)
    double scale;
    double src;        // dt G g / scale
    double inv_frac;   // 1 / frac
    double pow2;       // 2^kexp, or 0
    int kexp;
    double g6[3];      // dt / (6 h_a)
    double lap[3];     // eps dt / h_a^2
    float inv_h[3];
    float a;
};

// v >= 0 (-0 included)
__device__ __forceinline__ bool not_negative(double v) { return __double2hiint(v) >= 0 || zero64(v); }

// Stencil coefficients of point p (times dt): per axis the taps at -1, +1 and at
// the far upwind point, then the centre, into cf[k * 32].  Returns sum_a |u_a| / h_a.
template <int DIM>
__device__ __forceinline__ float stencil_coefs(const FwdArgs<double>& A, const Step64& B, int stencil, const double u[DIM],
                                               double* cf) {
    double c0 = 0.0;
    float cr = 0.0f;
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
        const double g = u[ax] * B.g6[ax];
        double lo, hi, far;
        if (stencil == 1) {
            lo = -3.0 * g;
            hi = 3.0 * g;
            far = 0.0;
        } else {
            const bool pos = not_negative(u[ax]);
            lo = g * (pos ? -6.0 : -2.0);
            hi = g * (pos ? 2.0 : 6.0);
            far = pos ? g : -g;
            c0 = fma(g, pos ? 3.0 : -3.0, c0);
        }
        if (A.eps != 0.0) {
            lo -= B.lap[ax];
            hi -= B.lap[ax];
            c0 = fma(2.0, B.lap[ax], c0);
        }
        cf[(3 * ax + 0) * kT64] = lo;
        cf[(3 * ax + 1) * kT64] = hi;
        cf[(3 * ax + 2) * kT64] = far;
        cr += fabsf((float)u[ax]) * B.inv_h[ax];
    }
    cf[3 * DIM * kT64] = c0;
    return cr;
}

// The transport term of component c at point p from the coefficients in cf.
template <int DIM>
__device__ __forceinline__ double stencil_term(const FwdArgs<double>& A, int stencil, int c, long long p,
                                               const double* cf) {
    constexpr int NC = Packed<DIM>::NC;
    const unsigned pu = (unsigned)p;
    const int nn[3] = {A.n0, A.n1, A.n2};
    const unsigned r1 = pu / (unsigned)A.n0;
    const int co[3] = {(int)(pu % (unsigned)A.n0), (int)(DIM == 3 ? r1 % (unsigned)A.n1 : r1),
                       (int)(DIM == 3 ? r1 / (unsigned)A.n1 : 0)};
    const long long stride[3] = {1, A.n0, (long long)A.n0 * A.n1};
    const double* sn = A.sig_n + (long long)c * A.N;
    const double* sm = A.sig_nm1 + (long long)c * A.N;
    // E = 2 sigma^n - sigma^{n-1} at offset off along axis ax: periodic wrap, or on a slab
    // the slowest axis beyond the grid from the halo planes
    auto at = [&](int ax, int off) -> double {
        int v = co[ax] + off;
        if ((v < 0 || v >= nn[ax]) && ax == DIM - 1 && A.halo_lo) {
            const long long pl = stride[DIM - 1];
            const double* hb = v < 0 ? A.halo_lo : A.halo_hi;
            const int k = v < 0 ? v + A.halo_r : v - nn[ax];
            const long long q = ((long long)c * A.halo_r + k) * pl + (p - (long long)co[ax] * pl);
            return fma(2.0, __ldg(hb + q), -__ldg(hb + (long long)NC * A.halo_r * pl + q));
        }
        if (v < 0) v += nn[ax];
        if (v < 0) v += nn[ax];
        if (v >= nn[ax]) v -= nn[ax];
        if (v >= nn[ax]) v -= nn[ax];
        const long long q = p + (long long)(v - co[ax]) * stride[ax];
        return fma(2.0, __ldg(sn + q), -__ldg(sm + q));
    };
    double acc = cf[3 * DIM * kT64] * fma(2.0, __ldg(sn + p), -__ldg(sm + p));
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
        const double lo = at(ax, -1), hi = at(ax, 1);
        acc = fma(cf[(3 * ax + 0) * kT64], lo, acc);
        acc = fma(cf[(3 * ax + 1) * kT64], hi, acc);
        if (stencil == 0) {
            // the sign of the coefficient is that of u (far = g or -g: u >= 0 takes the tap at -2)
            const double fc = cf[(3 * ax + 2) * kT64];
            const double ua = __ldg(A.u + (long long)ax * A.N + p);
            acc = fma(fc, at(ax, not_negative(ua) ? -2 : 2), acc);
        }
    }
    return acc;
}

// One tile of 32 points per block; warp (c, g) takes component c and the modes
// j = g mod G, and with g = 0 the component's part of the point systems.
template <int DIM, int TR, bool PAPER, int G>
__global__ void __launch_bounds__(kT64* Packed<DIM>::NC* G, G > 1 ? 1 : (DIM == 2 ? 8 : 3))
    fwd64_kernel(const FwdArgs<double> A, const Step64 B, const int classic, const int stencil) {
    constexpr int NC = Packed<DIM>::NC;
    constexpr int DD = DIM * DIM;
    extern __shared__ __align__(16) double sm64[];
    const int lane = threadIdx.x;
    const int w = threadIdx.y;
    const int c = w % NC, grp = w / NC;
    const int m = classic ? 0 : A.m;
    double* sQ = sm64;                          // Q'_j [m][NC][32]
    double* sH = sQ + (size_t)m * NC * kT64;    // partial history sums [G][NC][32]
    double* sR = sH + G * NC * kT64;            // right-hand side, then two buffers of residuals [3][NC][32]
    double* sK = sR + 3 * NC * kT64;            // dt kappa* (the paper's variable: dt frac kappa*) [DD][32]
    double* sC = sK + DD * kT64;                // stencil coefficients
    // dt kappa* in FP32 (the paper's variable: dt xi kappa*, the operator's)
    float* sKf = reinterpret_cast<float*>(sC + Shape64<DIM>::kCoef * kT64);
    const long long t0 = (long long)blockIdx.x * kT64;
    const long long p = t0 + lane;
    const bool active = p < A.N;
    const long long pc = active ? p : A.N - 1;  // a point to read where the tile ends past the grid
    const bool has_s0 = A.sigma0 != nullptr;

    // ---- velocity gradient entries and stencil coefficients, spread over the warps
    for (int k = w; k < DD; k += NC * G) {
        const long long q = (long long)k * A.N + pc;
        const double v = B.scale * fma(2.0, A.kap_n[q], -A.kap_nm1[q]);
        sK[k * kT64 + lane] = v;
        sKf[k * kT64 + lane] = PAPER ? (float)v * (float)B.pow2 : (float)v;
    }
    if (TR == kInStep && w == NC * G - 1) {
        double u[DIM];
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) u[ax] = __ldg(A.u + (long long)ax * A.N + pc);
        const float cr = stencil_coefs<DIM>(A, B, stencil, u, sC + lane);
        const float ccoef = (float)A.courant_coef;
        const bool over = active && ccoef > 0.0f && ccoef * cr > (float)A.courant_limit;
        if (__any_sync(0xffffffffu, over) && lane == 0) atomicOr(A.flags, 4u);
    }

    // ---- history sum over this warp's modes (constants: -2 eta_j in mc.eta): one partial
    //      sum per residue of j mod kSplit, added in the order of the residues, whether
    //      one warp holds them all or each has its own (a slab of a domain may be split
    //      where the domain is not, and gives the same bits)
    constexpr int kSums = Shape64<DIM>::kSplit / G;
    double part[kSums];
#pragma unroll
    for (int k = 0; k < kSums; ++k) part[k] = 0.0;
    if (classic) {
        if (grp == 0) {
            const long long q = (long long)c * A.N + pc;
            part[0] = kB1 * A.sig_n[q] + kB2 * A.sig_nm1[q] + (has_s0 ? kB0 * A.sigma0[q] : 0.0);
        }
    } else {
        constexpr long long row = (long long)NC * kT64;
        const long long base = mode_index(t0, c, m * NC) + lane;
        const double* xs = A.modes_n + base;
        const double* ys = A.modes_nm1 + base;
        double* q = sQ + c * kT64 + lane;
#pragma unroll 1
        for (int jb = grp; jb < m; jb += G * kAhead) {
            double x[kAhead], y[kAhead];
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                const int j = jb + k * G;
                if (j < m) {
                    x[k] = __ldcs(xs + j * row);
                    y[k] = __ldcs(ys + j * row);
                }
            }
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                const int j = jb + k * G;
                if (j < m) {
                    const double qp = fma(-0.25, y[k], x[k]);
                    part[k % kSums] = fma(A.mc.eta[j], qp, part[k % kSums]);
                    q[j * row] = qp;
                }
            }
        }
    }
    double H = part[0];
#pragma unroll
    for (int k = 1; k < kSums; ++k) H += part[k];
    if (G > 1 || PAPER) sH[(grp * NC + c) * kT64 + lane] = H;
    __syncthreads();

    // ---- right-hand side of this thread's component
    double x = 0.0, r = 0.0, s0 = 0.0;
    const int ci = Packed<DIM>::I(c), cj = Packed<DIM>::J(c);
    if (grp == 0) {
#pragma unroll
        for (int g = 1; g < G; ++g) H += sH[(g * NC + c) * kT64 + lane];
        const long long q = (long long)c * A.N + pc;
        const double ks = sK[(ci * DIM + cj) * kT64 + lane] + sK[(cj * DIM + ci) * kT64 + lane];
        if constexpr (PAPER) {
            // -b1 Phi^n - b2 Phi^{n-1} + dt (L(kappa*) h - h/Wi) + dt G (kappa* + kappa*^T) Psi0 [- A]
            // against (b0 + dt xi/Wi) Phi - dt xi L(kappa*) Phi; h_ab of the other components
            // from shared memory (their partial sums, added in the same order)
            auto hat = [&](int a, int b) {
                const int k = PackedIndex<DIM>::at(a, b);
                double v = sH[k * kT64 + lane];
#pragma unroll
                for (int g = 1; g < G; ++g) v += sH[(g * NC + k) * kT64 + lane];
                return v;
            };
            double lh = 0.0;
#pragma unroll
            for (int l = 0; l < DIM; ++l)
                lh = fma(sK[(ci * DIM + l) * kT64 + lane], hat(l, cj),
                         fma(hat(ci, l), sK[(cj * DIM + l) * kT64 + lane], lh));
            r = fma(2.0, A.sig_n[q], -0.5 * A.sig_nm1[q]) - A.dt * A.inv_wi * H + fma(B.src, ks, B.inv_frac * lh);
            if (TR == kFromPrepass) r -= A.trans[q];
        } else {
            s0 = has_s0 ? A.sigma0[q] : 0.0;
            r = fma(B.src, ks, fma(A.eta, s0, -H));
            if (TR == kInStep) r -= stencil_term<DIM>(A, stencil, c, pc, sC + lane);
        }
        sR[c * kT64 + lane] = r;
    }
    __syncthreads();
    if (grp == 0) {
        unsigned fl = 0u;
        if (!refine_solve64<DIM, false, PAPER>(sK + lane, sKf + lane, sR + lane, A.a, B.a, c, r, &x, B.pow2, B.kexp) &&
            active)
            fl |= 2u;
        const long long q = (long long)c * A.N + p;
        bool finite = finite64(x);
        if (active) {
            A.sig_np1[q] = x;
            if constexpr (PAPER) {
                const double psi = fma(A.xi, x, H);
                finite = finite && finite64(psi);
                A.psi[q] = psi;
                if (A.sig_copy) A.sig_copy[q] = psi;
            } else {
                if (A.sig_copy) A.sig_copy[q] = x;
            }
            if (!finite) fl |= 1u;
            if (fl) atomicOr(A.flags, fl);
        }
        x -= s0;
        if (G > 1) sH[c * kT64 + lane] = x;
    }
    if (G > 1) {
        __syncthreads();
        x = sH[c * kT64 + lane];
    }

    // ---- push-forward over the oldest level (constants: 2 c_j in mc.c)
    if (!classic && active) {
        constexpr long long row = (long long)NC * kT64;
        const double* q = sQ + c * kT64 + lane;
        double* out = A.modes_nm1 + mode_index(p, c, m * NC);
#pragma unroll 4
        for (int j = grp; j < m; j += G) __stcs(out + j * row, fma(A.mc.rho[j], x, A.mc.c[j] * q[j * row]));
    }
}

// Raises a kernel's dynamic shared-memory limit once per device.
template <int DIM, int TR, bool PAPER, int G>
cudaError_t smem_ready() {
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(fwd64_kernel<DIM, TR, PAPER, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem64_bytes<DIM>(kMaxModes, G));
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

template <int DIM, int TR, bool PAPER, int G>
cudaError_t launch64(const FwdArgs<double>& a, const LaunchCfg& cfg, long long tiles, cudaStream_t s) {
    cudaError_t e = smem_ready<DIM, TR, PAPER, G>();
    if (e != cudaSuccess) return e;
    const size_t dyn = smem64_bytes<DIM>(cfg.classic ? 0 : a.m, G);
    Step64 b;
    const bool has = !PAPER || (a.xi > 0.0 && std::isfinite(a.xi));
    const int kexp = PAPER && has ? std::ilogb(a.xi) : 0;
    const double frac = PAPER && has ? std::ldexp(a.xi, -kexp) : 1.0;
    b.scale = a.dt * frac;
    b.src = a.G * a.g / frac;
    b.inv_frac = 1.0 / frac;
    b.pow2 = has ? std::ldexp(1.0, kexp) : 0.0;
    b.kexp = has ? kexp : -10000;
    for (int i = 0; i < 3; ++i) {
        b.g6[i] = a.dt * a.inv_h[i] / 6.0;
        b.lap[i] = a.eps * a.dt * a.inv_h[i] * a.inv_h[i];
        b.inv_h[i] = (float)a.inv_h[i];
    }
    b.a = (float)a.a;
    fwd64_kernel<DIM, TR, PAPER, G><<<(unsigned)tiles, dim3(kT64, Packed<DIM>::NC * G), dyn, s>>>(
        a, b, cfg.classic ? 1 : 0, cfg.stencil);
    return cudaGetLastError();
}

// Tiles up to which a tile's modes are split over several warps: one block per SM.  Measured, split
// against not: 128 tiles (2D 64^2, m = 16, with transport) 10.3 us against 12.2; beyond it 288 tiles
// 14.2 against 12.4, 480 (m = 24) 20.5 against 16.4, 512 (m = 32) 26.6 against 23.1; 3D, 183 tiles
// (m = 24) 24.2 against 18.5.
constexpr long long kSplitTiles = 152;

template <int DIM, int TR, bool PAPER>
cudaError_t launch_split(const FwdArgs<double>& a, const LaunchCfg& cfg, cudaStream_t s) {
    const long long tiles = (a.N + kT64 - 1) / kT64;
    if (tiles <= kSplitTiles) return launch64<DIM, TR, PAPER, Shape64<DIM>::kSplit>(a, cfg, tiles, s);
    return launch64<DIM, TR, PAPER, 1>(a, cfg, tiles, s);
}

template <int DIM>
cudaError_t launch_dim(const FwdArgs<double>& a, const LaunchCfg& cfg, cudaStream_t s) {
    if (cfg.paper) {
        if (cfg.transport) return launch_split<DIM, kFromPrepass, true>(a, cfg, s);
        return launch_split<DIM, kNoTransport, true>(a, cfg, s);
    }
    if (cfg.transport) return launch_split<DIM, kInStep, false>(a, cfg, s);
    return launch_split<DIM, kNoTransport, false>(a, cfg, s);
}

}  // namespace

cudaError_t launch_forward_f64(const FwdArgs<double>& args, const LaunchCfg& cfg, cudaStream_t s) {
    if (cfg.paper && (cfg.classic || !args.psi)) return cudaErrorInvalidValue;
    if (cfg.paper && cfg.transport) {
        // Psi^{n+1} is written over Psi^{n-1}, which its neighbours' stencils
        // still need: this variable keeps the pre-pass
        if (!args.psi_n || !args.psi_nm1 || !args.trans) return cudaErrorInvalidValue;
        FwdArgs<double> ta = args;
        ta.sig_n = args.psi_n;
        ta.sig_nm1 = args.psi_nm1;
        const cudaError_t e = launch_prepass_f64(ta, cfg, s);
        if (e != cudaSuccess) return e;
    }
    FwdArgs<double> a = args;
    for (int j = 0; j < a.m; ++j) {   // Q = -2 Q'
        a.mc.c[j] *= 2.0;
        a.mc.eta[j] *= -2.0;
    }
    if (cfg.ev_before) {
        const cudaError_t e = cudaEventRecord(cfg.ev_before, s);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cfg.dim == 2 ? launch_dim<2>(a, cfg, s) : launch_dim<3>(a, cfg, s);
    if (e == cudaSuccess && cfg.ev_after) e = cudaEventRecord(cfg.ev_after, s);
    return e;
}

}  // namespace tfs
