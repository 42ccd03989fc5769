// Many steps of the pointwise law in one launch (tfs_run, tfs_backward,
// tfs_backward_run): FP32 storage, the stress form, alpha < 1, BDF2 start, frozen
// velocity gradient.
//
// Without transport a point depends on no other, so a run need not return its
// modes to memory between steps: thread (point, component) keeps both levels of
// its m modes in registers (64 at m = 32) and takes step after step with the
// arithmetic of the single step (tfs_forward.cu) and of its adjoint
// (tfs_adjoint.cu), operation for operation, so that every stress, adjoint mode and
// adjoint of a right-hand side is bitwise the one that stepping gives.  The gradients are
// their sums over the steps, which stepping adds up in FP64 and a run in three floats
// (no less accurate; the FP64 additions took 4.8 us per reverse step at 2D 512^2, these
// 1.5 us more than two floats).  Per step a tile of 32
// points exchanges only its right-hand sides and solutions through shared
// memory; the point matrix is factored once.
//
// Bound: instruction issue.  8 (forward) and 7 (reverse) FP32 operations per mode
// value and step, most of them one dependent chain per thread (the compensated
// sum runs over the modes in order), plus the 32 point solves on one warp of the
// tile, which rotates with the tile so that the solves spread over the SM's
// schedulers.  Nothing but one stress row per step and, per launch, the mode levels moves:
// a single step is bound by 3 words per (mode, component) from HBM.  Measured at 2D
// 512^2, m = 32, 100 steps: 15.7 us per step against 49 for tfs_step, 14.6 us per
// reverse step against 77; a training pass (forward and gradients) 19.2 -> 3.5 ms, of which
// 4.9 ms are the segments' recomputation that stored stresses make unnecessary.
// Tried and not kept: one mode sweep per block of eight steps with the steps' own drives convolved
// by scalar weights (4.5 ms; smaller rounding errors, but not the values that stepping gives).
#include <cuda_runtime.h>

#include "tfs_device.cuh"
#include "tfs_resident.h"

namespace tfs {
namespace {

constexpr int kT = 32;

// f(j, integral constant) for the modes j < m, eight at a time without a test each.
template <int MM, class F>
__device__ __forceinline__ void for_modes(int m, F&& f) {
    static_for<0, MM / 8>([&](auto gg) {
        constexpr int g = decltype(gg)::value;
        if (8 * g + 8 <= m) {
            static_for<0, 8>([&](auto ii) { f(std::integral_constant<int, 8 * g + decltype(ii)::value>{}); });
        } else {
            static_for<0, 8>([&](auto ii) {
                constexpr int j = 8 * g + decltype(ii)::value;
                if (j < m) f(std::integral_constant<int, j>{});
            });
        }
    });
}

// Factors of a tile's matrices in shared memory, lane = point.
template <int NC>
struct SharedLU {
    float a[NC][NC][kT];
    unsigned swaps[kT];
    __device__ __forceinline__ void put(const LU32<NC>& F, int lane) {
        unsigned s = 0u;
        int bit = 0;
#pragma unroll
        for (int k = 0; k < NC; ++k)
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                a[k][i][lane] = F.a[k][i];
                if (i > k) s |= (F.sw[k][i] ? 1u : 0u) << bit++;
            }
        swaps[lane] = s;
    }
    __device__ __forceinline__ void get(LU32<NC>& F, int lane) const {
        const unsigned s = swaps[lane];
        int bit = 0;
#pragma unroll
        for (int k = 0; k < NC; ++k)
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                F.a[k][i] = a[k][i][lane];
                if (i > k) F.sw[k][i] = (s >> bit++) & 1u;
            }
    }
};

template <int DIM, int MM, bool COMP>
__global__ void __launch_bounds__(kT* Packed<DIM>::NC) resident_run_kernel(const ResidentRun A) {
    constexpr int NC = Packed<DIM>::NC;
    __shared__ f2 sR[NC][kT];
    __shared__ float sD[NC][kT];
    __shared__ float sK[DIM * DIM][kT];
    __shared__ float sS0[NC][kT];
    __shared__ SharedLU<NC> sF;
    const int lane = threadIdx.x, c = threadIdx.y;
    const int ws = (int)(blockIdx.x % (unsigned)NC);   // the solving warp
    const long long t0 = (long long)blockIdx.x * kT, p = t0 + lane, N = A.N;
    const bool active = p < N;
    const long long pc = active ? p : N - 1;
    const int m = A.m;
    constexpr int row = NC * kT;
    const long long base = mode_index(t0, c, m * NC) + lane;
    float x[MM], y[MM];
    for_modes<MM>(m, [&](auto jj) {
        constexpr int j = decltype(jj)::value;
        x[j] = __ldcs(A.modes_n + base + j * row);
        y[j] = __ldcs(A.modes_nm1 + base + j * row);
    });
    const int ci = Packed<DIM>::I(c), cj = Packed<DIM>::J(c);
    const float s0 = A.sigma0 ? __ldg(A.sigma0 + (long long)c * N + pc) : 0.0f;
    sS0[c][lane] = s0;
    // kappa* = 2 kappa - kappa as the step forms it: kappa exactly, and a NaN from an infinite one
    auto star = [&](int e) {
        const float v = __ldg(A.kap + (long long)e * N + pc);
        return two_sum_f2(2.0f * v, -v);
    };
    const f2 ks = f2_add(star(ci * DIM + cj), star(cj * DIM + ci));
    const f2 es0 = f2_mul_f(f2{A.eta.hi, A.eta.lo}, s0);
    unsigned fl = 0u;
    if (c == ws) {
        f2 K[3][3];
#pragma unroll
        for (int i = 0; i < DIM; ++i)
#pragma unroll
            for (int j = 0; j < DIM; ++j) {
                K[i][j] = star(i * DIM + j);
                sK[i * DIM + j][lane] = K[i][j].hi;
            }
        LU32<NC> F;
        if (!factor_point_f32<DIM>(K, A.a, A.dt, F)) fl |= 2u;
        sF.put(F, lane);
    }
#pragma unroll 1
    for (int k = 0; k < A.steps; ++k) {
        // history sum (Q_j = -2 q: the power of two goes into the constants, the bits stay)
        float hs = 0.0f, comp = 0.0f;
        for_modes<MM>(m, [&](auto jj) {
            constexpr int j = decltype(jj)::value;
            const float q = __fmaf_rn(-0.25f, y[j], x[j]);
            if constexpr (COMP) {
                const float yv = __fmaf_rn(A.mc.eta_hi[j], q, __fmaf_rn(A.mc.eta_lo[j], q, -comp));
                const float t = __fadd_rn(hs, yv);
                comp = __fsub_rn(__fsub_rn(t, hs), yv);
                hs = t;
            } else {
                hs = __fmaf_rn(A.mc.eta_hi[j], q, hs);
            }
            y[j] = x[j];
            x[j] = A.mc.c[j] * q;      // the push-forward's part without the new stress
        });
        const f2 H = COMP ? fast_two_sum(hs, -comp) : f2_from(hs);
        const f2 R = f2_add(f2_add(es0, f2_neg(H)), f2_mul(f2{A.src[k].hi, A.src[k].lo}, ks));
        sR[c][lane] = R;
        __syncthreads();
        if (c == ws) {
            f2 K[3][3], Rv[NC], xv[NC];
            LU32<NC> F;
            sF.get(F, lane);
#pragma unroll
            for (int i = 0; i < DIM; ++i)
#pragma unroll
                for (int j = 0; j < DIM; ++j) K[i][j] = f2{sK[i * DIM + j][lane], 0.0f};
#pragma unroll
            for (int r = 0; r < NC; ++r) Rv[r] = sR[r][lane];
            refine_point_f32<DIM>(K, A.a, A.dt, F, Rv, xv);
            float* out = A.rows + (long long)k * A.stride;
#pragma unroll
            for (int r = 0; r < NC; ++r) {
                const float v = xv[r].hi + xv[r].lo;
                if (!isfinite(v)) fl |= 1u;
                if (active) out[(long long)r * N + p] = v;
                sD[r][lane] = __fsub_rn(v, sS0[r][lane]);
            }
        }
        __syncthreads();
        const float d = sD[c][lane];
        for_modes<MM>(m, [&](auto jj) {
            constexpr int j = decltype(jj)::value;
            x[j] = __fmaf_rn(A.mc.rho[j], d, x[j]);
        });
    }
    if (active) {
        if (fl) atomicOr(A.flags, fl);
        for_modes<MM>(m, [&](auto jj) {
            constexpr int j = decltype(jj)::value;
            __stcs(A.modes_n + base + j * row, x[j]);
            __stcs(A.modes_nm1 + base + j * row, y[j]);
        });
    }
}

template <int DIM, int MM>
__global__ void __launch_bounds__(kT* Packed<DIM>::NC) resident_back_kernel(const ResidentBack A) {
    constexpr int NC = Packed<DIM>::NC;
    constexpr int DD = DIM * DIM;
    constexpr int kPer = (DD + NC - 1) / NC;           // entries of dJ/dkappa a thread accumulates
    __shared__ float sS[NC][kT];                       // S = sum_j rho_j z_j, rounded once
    __shared__ float sL[NC][kT];                       // lamR
    __shared__ float sSig[2][NC][kT];                  // sigma^{n+1} (by step parity)
    __shared__ float sK[DD][kT];
    __shared__ SharedLU<NC> sF;
    const int lane = threadIdx.x, c = threadIdx.y;
    const int ws = (int)(blockIdx.x % (unsigned)NC);
    const long long t0 = (long long)blockIdx.x * kT, p = t0 + lane, N = A.N;
    const bool active = p < N;
    const long long pc = active ? p : N - 1;
    const int m = A.m;
    constexpr int row = NC * kT;
    const long long base = mode_index(t0, c, m * NC) + lane;
    float x[MM], y[MM];
    for_modes<MM>(m, [&](auto jj) {
        constexpr int j = decltype(jj)::value;
        x[j] = __ldcs(A.ell_prev + base + j * row);
        y[j] = __ldcs(A.ell_prev2 + base + j * row);
    });
    unsigned fl = 0u;
    if (c == ws) {
        float K[3][3];
#pragma unroll
        for (int i = 0; i < DIM; ++i)
#pragma unroll
            for (int j = 0; j < DIM; ++j) {
                const float v = __ldg(A.kap + (long long)(i * DIM + j) * N + pc);
                K[i][j] = __fmaf_rn(2.0f, v, -v);   // kappa* (a NaN from an infinite kappa)
                sK[i * DIM + j][lane] = K[i][j];
            }
        LU32<NC> F;
        static_for<0, NC>([&](auto rr) {
            constexpr int r = decltype(rr)::value;
            static_for<0, NC>([&](auto kk) {
                // transpose: entry (r, k) of M^T is entry (k, r) of M
                constexpr int k = decltype(kk)::value;
                const float v = uc_entry<DIM, float>(K, k, r);
                F.a[r][k] = (r == k) ? __fmaf_rn(-A.dt, v, A.a) : -A.dt * v;
            });
        });
        if (!lu32_factor<NC>(F, 1e-30f)) fl |= 2u;
        sF.put(F, lane);
    }
    f3 l_sum{0.0f, 0.0f, 0.0f}, s_sum{0.0f, 0.0f, 0.0f}, gk[kPer];   // of lamR, S, dJ/dkappa
    double sig_sum = 0.0, sym_sum = 0.0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) gk[e] = f3{0.0f, 0.0f, 0.0f};
    // to the FP64 fields: the sum of eta lamR - S, and of dJ/dkappa's entries
    auto flush = [&] {
        double lh, ll, sh, sl;
        l_sum.value(lh, ll);
        s_sum.value(sh, sl);
        if (active) A.g_sigma0[(long long)c * N + p] += fma(A.eta, lh, -sh) + fma(A.eta, ll, -sl);
        l_sum = s_sum = f3{0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            if (c + e * NC < DD && active) A.g_kap[(long long)(c + e * NC) * N + p] += gk[e].value();
            gk[e] = f3{0.0f, 0.0f, 0.0f};
        }
    };
#pragma unroll 1
    for (int k = 0; k < A.steps; ++k) {
        const int n = A.steps - 1 - k;
        const float sig = __ldg(A.rows + (long long)n * A.stride + (long long)c * N + pc);
        float ss = 0.0f, comp = 0.0f;
        for_modes<MM>(m, [&](auto jj) {
            constexpr int j = decltype(jj)::value;
            const float q = __fmaf_rn(-0.25f, y[j], x[j]);   // z = -2 q
            const float yv = __fmaf_rn(A.mc.rho[j], q, -comp);
            const float t = __fadd_rn(ss, yv);
            comp = __fsub_rn(__fsub_rn(t, ss), yv);
            ss = t;
            y[j] = x[j];
            x[j] = A.mc.c[j] * q;
        });
        const float S = __fsub_rn(ss, comp);
        const bool last = k == 0 && A.dJ;
        // with dJ these are the first reverse steps: the adjoint modes, and S, are zero
        sS[c][lane] = last ? __ldg(A.dJ + (long long)c * N + pc) : S;
        sSig[k & 1][c][lane] = sig;
        __syncthreads();
        if (c == ws) {
            LU32<NC> F;
            sF.get(F, lane);
            float lam[NC];
#pragma unroll
            for (int r = 0; r < NC; ++r) lam[r] = sS[r][lane];
            lu32_solve<NC>(F, lam);
            float sym_dot = 0.0f, sig_dot = 0.0f;
#pragma unroll
            for (int r = 0; r < NC; ++r) {
                const int i = Packed<DIM>::I(r), j = Packed<DIM>::J(r);
                sym_dot = __fmaf_rn(lam[r], sK[i * DIM + j][lane] + sK[j * DIM + i][lane], sym_dot);
                sig_dot = __fmaf_rn(lam[r], sSig[k & 1][r][lane], sig_dot);
                sL[r][lane] = lam[r];
            }
            sig_sum += (double)sig_dot;
            sym_sum = fma(A.dtg[k], (double)sym_dot, sym_sum);
        }
        __syncthreads();
        const float l = sL[c][lane];
        for_modes<MM>(m, [&](auto jj) {
            constexpr int j = decltype(jj)::value;
            x[j] = __fmaf_rn(-A.mc.eta_hi[j], l, x[j]);
        });
        l_sum.add(l);
        if (!last) {
            s_sum.add(ss);
            s_sum.add_small(-comp);
        }
        bool large = l_sum.large() | s_sum.large();
        // dJ/dkappa_ab += dt sum_s Lam_as sigma_bs + dt G g Lam_ab, Lam symmetric with doubled diagonal
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const int q = c + e * NC;
            if (q < DD) {
                const int a = q / DIM, b = q % DIM;
                auto at = [&](int i, int j) { return i == j ? (DIM == 2 ? 2 * i : i) : (DIM == 2 ? 1 : 6 - i - j); };
                // (dt lamR before sigma: their product may leave the float range where dt times it does not)
                const float lab = sL[at(a, b)][lane];
                float g = A.src[k] * (a == b ? 2.0f * lab : lab);
#pragma unroll
                for (int s = 0; s < DIM; ++s) {
                    const float la = A.dt * sL[at(a, s)][lane];
                    g = __fmaf_rn(a == s ? 2.0f * la : la, sSig[k & 1][at(b, s)][lane], g);
                }
                gk[e].add(g);
                large |= gk[e].large();
            }
        }
        if (large) flush();
    }
    if (active) {
        if (fl) atomicOr(A.flags, fl);
        for_modes<MM>(m, [&](auto jj) {
            constexpr int j = decltype(jj)::value;
            __stcs(A.ell_prev + base + j * row, x[j]);
            __stcs(A.ell_prev2 + base + j * row, y[j]);
        });
        flush();
    }
    if (c == ws) {
        const double sd = active ? sig_sum : 0.0, sy = active ? sym_sum : 0.0;
        double wi = A.dt_wi2 * sd - A.g_wi * sy, be = -A.inv_wire * sy;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            wi += __shfl_xor_sync(0xffffffffu, wi, off);
            be += __shfl_xor_sync(0xffffffffu, be, off);
        }
        if (lane == 0) {
            A.partials[2 * (long long)blockIdx.x + 0] += wi;
            A.partials[2 * (long long)blockIdx.x + 1] += be;
        }
    }
}

template <int DIM, int MM>
cudaError_t run_m(const ResidentRun& a, bool compensated, cudaStream_t s) {
    const unsigned tiles = (unsigned)((a.N + kT - 1) / kT);
    const dim3 block(kT, Packed<DIM>::NC);
    if (compensated) resident_run_kernel<DIM, MM, true><<<tiles, block, 0, s>>>(a);
    else resident_run_kernel<DIM, MM, false><<<tiles, block, 0, s>>>(a);
    return cudaGetLastError();
}

template <int DIM>
cudaError_t run_dim(const ResidentRun& a, bool compensated, cudaStream_t s) {
    if (a.m <= 16) return run_m<DIM, 16>(a, compensated, s);
    if (a.m <= 32) return run_m<DIM, 32>(a, compensated, s);
    if (a.m <= 48) return run_m<DIM, 48>(a, compensated, s);
    return run_m<DIM, 64>(a, compensated, s);
}

template <int DIM, int MM>
cudaError_t back_m(const ResidentBack& a, cudaStream_t s) {
    const unsigned tiles = (unsigned)((a.N + kT - 1) / kT);
    resident_back_kernel<DIM, MM><<<tiles, dim3(kT, Packed<DIM>::NC), 0, s>>>(a);
    return cudaGetLastError();
}

template <int DIM>
cudaError_t back_dim(const ResidentBack& a, cudaStream_t s) {
    if (a.m <= 16) return back_m<DIM, 16>(a, s);
    if (a.m <= 32) return back_m<DIM, 32>(a, s);
    if (a.m <= 48) return back_m<DIM, 48>(a, s);
    return back_m<DIM, 64>(a, s);
}

}  // namespace

cudaError_t launch_resident_run(const ResidentRun& args, int dim, bool compensated, cudaStream_t s) {
    ResidentRun a = args;
    for (int j = 0; j < a.m; ++j) {   // Q = -2 q
        a.mc.c[j] *= 2.0f;
        a.mc.eta_hi[j] *= -2.0f;
        a.mc.eta_lo[j] *= -2.0f;
    }
    return dim == 2 ? run_dim<2>(a, compensated, s) : run_dim<3>(a, compensated, s);
}

cudaError_t launch_resident_back(const ResidentBack& args, int dim, cudaStream_t s) {
    ResidentBack a = args;
    for (int j = 0; j < a.m; ++j) {   // z = -2 q
        a.mc.c[j] *= 2.0f;
        a.mc.rho[j] *= -2.0f;
    }
    return dim == 2 ? back_dim<2>(a, s) : back_dim<3>(a, s);
}

}  // namespace tfs
