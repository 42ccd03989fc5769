// Adjoint of one forward stress step in FP64 storage (the formulas are those at
// the head of tfs_adjoint.cu, which serves FP32 storage), laid out like the
// FP64 forward step (tfs_forward64.cu) and for the same reason: the FP64 pipe's
// instruction rate bounds it.  A warp owns one component of a tile's 32 points: its two
// adjoint mode levels go straight to registers, z_j = b1 lamQ'_j + b2 lamQ''_j =
// -2 q_j with q_j = x - y/4 costs one FMA, the sum another, the new level two; the
// transposed point system is solved by FP32 factors with FP64 residuals; the
// gradient accumulations are spread over the component warps.  Measured per reverse step, 2D
// 250 x 198, m = 32: 86 -> 63 us against the staged form with one solving warp.
#include <cuda_runtime.h>

#include "tfs_internal.h"
#include "tfs_solve64.cuh"

namespace tfs {
namespace {

constexpr int kAhead = 8;    // modes whose two levels a thread loads before using them

template <int DIM>
__host__ __device__ constexpr size_t adj64_smem(int m) {
    constexpr int NC = Packed<DIM>::NC;
    return (size_t)kT64 * sizeof(double) * ((size_t)m * NC + 6 * NC + DIM * DIM) +
           (size_t)kT64 * sizeof(float) * DIM * DIM;
}

template <int DIM>
__global__ void __launch_bounds__(kT64* Packed<DIM>::NC, DIM == 2 ? 8 : 3)
    adj64_kernel(const AdjArgs<double> A, const int classic, const float af) {
    constexpr int NC = Packed<DIM>::NC;
    constexpr int DD = DIM * DIM;
    extern __shared__ __align__(16) double sm[];
    const int lane = threadIdx.x, c = threadIdx.y;
    const int m = classic ? 0 : A.m;
    double* sQ = sm;                         // q_j [m][NC][32]
    double* sR = sQ + (size_t)m * NC * kT64; // right-hand side and two residual buffers [3][NC][32]
    double* sL = sR + 3 * NC * kT64;         // lamR
    double* sG = sL + NC * kT64;             // sigma^{n+1}
    double* sW = sG + NC * kT64;             // lamR (kappa + kappa^T), per component
    double* sK = sW + NC * kT64;             // dt kappa* [DD][32]
    float* sKf = reinterpret_cast<float*>(sK + DD * kT64);
    const long long t0 = (long long)blockIdx.x * kT64, p = t0 + lane, N = A.N;
    const bool active = p < N;
    const long long pc = active ? p : N - 1;
    const long long qc = (long long)c * N + pc;

    for (int k = c; k < DD; k += NC) {
        const long long q = (long long)k * N + pc;
        const double v = A.dt * fma(2.0, A.kap_n[q], -A.kap_nm1[q]);
        sK[k * kT64 + lane] = v;
        sKf[k * kT64 + lane] = (float)v;
    }
    // ---- S = sum_j rho_j z_j over this component's modes (constants: -2 rho_j in mc.rho)
    constexpr long long row = (long long)NC * kT64;
    const long long base = mode_index(t0, c, m * NC) + lane;
    double* qs = sQ + c * kT64 + lane;
    double S0 = 0.0, S1 = 0.0;
    if (!classic) {
        const double* xs = A.ell_prev + base;
        const double* ys = A.ell_prev2 + base;
#pragma unroll 1
        for (int jb = 0; jb < m; jb += kAhead) {
            double x[kAhead], y[kAhead];
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                x[k] = y[k] = 0.0;
                if (jb + k < m && !A.first) {
                    x[k] = __ldcs(xs + (jb + k) * row);
                    y[k] = __ldcs(ys + (jb + k) * row);
                }
            }
#pragma unroll
            for (int k = 0; k < kAhead; ++k)
                if (jb + k < m) {
                    const double q = fma(-0.25, y[k], x[k]);
                    if (k & 1) S1 = fma(A.mc.rho[jb + k], q, S1);
                    else S0 = fma(A.mc.rho[jb + k], q, S0);
                    qs[(jb + k) * row] = q;
                }
        }
    }
    const double S = S0 + S1;
    const double v = A.s1[qc] + S;
    const double sig = A.sig_np1[qc];
    sR[c * kT64 + lane] = v;
    sG[c * kT64 + lane] = sig;
    __syncthreads();
    // ---- M(kappa*)^T lamR = s1 + S
    double lam = 0.0;
    if (!refine_solve64<DIM, true>(sK + lane, sKf + lane, sR + lane, A.a, af, c, v, &lam) && active)
        atomicOr(A.flags, 2u);
    sL[c * kT64 + lane] = lam;
    {
        const int i = Packed<DIM>::I(c), j = Packed<DIM>::J(c);
        // times dt (sK carries it); taken out of the block's sum
        sW[c * kT64 + lane] = lam * (sK[(i * DIM + j) * kT64 + lane] + sK[(j * DIM + i) * kT64 + lane]);
    }
    __syncthreads();
    if (active) {
        A.lamR[qc] = lam;
        double gs = fma(A.eta, lam, -S), s1o = A.s0[qc], s0o = 0.0;
        if (classic) {
            s1o = fma(-kB1, lam, s1o);
            s0o = -kB2 * lam;
            gs = fma(-kB0, lam, gs);
        }
        A.g_sigma0[qc] += gs;
        A.s1_out[qc] = s1o;
        A.s0_out[qc] = s0o;
        // dJ/dkappa_ab += dt sum_s Lam_as sigma_bs + dt G g Lam_ab, Lam symmetric with doubled diagonal
        const double src = A.G * A.g;
#pragma unroll
        for (int e = c; e < DD; e += NC) {
            const int a = e / DIM, b = e % DIM;
            auto Lam = [&](int i, int j) {
                const double l = sL[PackedIndex<DIM>::at(i, j) * kT64 + lane];
                return i == j ? 2.0 * l : l;
            };
            double g = src * Lam(a, b);
#pragma unroll
            for (int s = 0; s < DIM; ++s) g = fma(Lam(a, s), sG[PackedIndex<DIM>::at(b, s) * kT64 + lane], g);
            const long long q = (long long)e * N + p;
            A.g_kap[q] = fma(A.dt, g, A.g_kap[q]);
        }
        // ---- lamQ_j = -c_j z_j - eta_j lamR over the oldest slot (constants: 2 c_j in mc.c)
        if (!classic) {
            double* out = A.ell_prev2 + base;
#pragma unroll 4
            for (int j = 0; j < m; ++j) __stcs(out + j * row, fma(-A.mc.eta[j], lam, A.mc.c[j] * qs[j * row]));
        }
    }
    // ---- the tile's sums of the two scalar derivatives (one warp, which rotates)
    if (c == (int)(blockIdx.x % (unsigned)NC)) {
        double sig_dot = 0.0, sym_dot = 0.0;   // sym_dot times dt
        if (active) {
#pragma unroll
            for (int r = 0; r < NC; ++r) {
                sig_dot = fma(sL[r * kT64 + lane], sG[r * kT64 + lane], sig_dot);
                sym_dot += sW[r * kT64 + lane];
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            sig_dot += __shfl_xor_sync(0xffffffffu, sig_dot, off);
            sym_dot += __shfl_xor_sync(0xffffffffu, sym_dot, off);
        }
        if (lane == 0) {
            const double lam_G = A.g * sym_dot;
            A.partials[2 * (long long)blockIdx.x + 0] += A.dt / (A.Wi * A.Wi) * sig_dot - A.G / A.Wi * lam_G;
            A.partials[2 * (long long)blockIdx.x + 1] += -lam_G / (A.Wi * A.Re);
        }
    }
}

template <int DIM>
cudaError_t launch(const AdjArgs<double>& args, bool classic, cudaStream_t s) {
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !done[dev]) {
        e = cudaFuncSetAttribute(adj64_kernel<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)adj64_smem<DIM>(kMaxModes));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) done[dev] = true;
    }
    AdjArgs<double> a = args;
    for (int j = 0; j < a.m; ++j) {   // z = -2 q
        a.mc.c[j] *= 2.0;
        a.mc.rho[j] *= -2.0;
    }
    const unsigned tiles = (unsigned)((a.N + kT64 - 1) / kT64);
    adj64_kernel<DIM><<<tiles, dim3(kT64, Packed<DIM>::NC), adj64_smem<DIM>(classic ? 0 : a.m), s>>>(
        a, classic ? 1 : 0, (float)a.a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adjoint_f64(const AdjArgs<double>& a, const LaunchCfg& cfg, cudaStream_t s) {
    return cfg.dim == 2 ? launch<2>(a, cfg.classic, s) : launch<3>(a, cfg.classic, s);
}

}  // namespace tfs
