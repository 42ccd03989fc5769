// Point systems of a 32-point tile in FP64 by FP32 factors and refinement, one
// thread per (point, component): the FP64 step and its adjoint
// (tfs_forward64.cu, tfs_adjoint64.cu).
#pragma once

#include "tfs_device.cuh"

namespace tfs {

constexpr int kT64 = 32;     // points per tile

// Tests that keep off the FP64 pipe.
__device__ __forceinline__ bool finite64(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool zero64(double v) {
    return ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) == 0;
}

// ---- FP32 images of FP64 numbers by integer operations (a conversion costs what
// an FP64 operation does).  A vector is scaled by the power of two that brings
// its largest component to [1, 2); smaller components lose the bits below that
// of the float format, which the refinement recovers.
__device__ __forceinline__ int biased_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

__device__ __forceinline__ float scaled_float(double v, int emax) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int be = (hi >> 20) & 0x7ff, e = be - emax + 127;
    const unsigned bits = ((unsigned)hi & 0x80000000u) | ((unsigned)e << 23) | (((unsigned)hi & 0xfffffu) << 3) |
                          ((unsigned)lo >> 29);
    return be > 0 && e > 0 ? __uint_as_float(bits) : 0.0f;
}

// f 2^(emax - 1023), exactly, for a finite f whose scaled exponent is in range (0 below it).
__device__ __forceinline__ double unscaled_double(float f, int emax) {
    const unsigned b = __float_as_uint(f);
    const int e = (int)((b >> 23) & 0xffu) - 127 + emax;
    const int hi = (int)((b & 0x80000000u) | ((unsigned)e << 20) | ((b & 0x7fffffu) >> 3));
    return ((b >> 23) & 0xffu) != 0u && e > 0 ? __hiloint2double(hi, (int)(b << 29)) : 0.0;
}

// Barrier of the first N threads of a block.
template <int N>
__device__ __forceinline__ void named_sync() {
    asm volatile("bar.sync 1, %0;\n" ::"n"(N) : "memory");
}

// Packed component of the symmetric entry (a, b).
template <int DIM>
struct PackedIndex {
    __host__ __device__ static constexpr int at(int a, int b) {
        return a == b ? (DIM == 2 ? 2 * a : a) : (DIM == 2 ? 1 : 6 - a - b);
    }
};

// The point system M = a I - scale L(K) (scale 1 where none is given: a further argument spills in the 3D
// step) by FP64 Gaussian elimination: component c of M^-1 R.  Returns false when a pivot vanishes.
template <int DIM, bool TRANSPOSED, typename... Scale>
__device__ __noinline__ bool solve_by_elimination(const double* sK, const double* sR, double a, int c, double* out,
                                                   Scale... given) {
    constexpr int NC = Packed<DIM>::NC;
    const double scale = (1.0 * ... * given);
    double K[3][3], x[NC], M[NC][NC];
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int j = 0; j < DIM; ++j) K[i][j] = sK[(i * DIM + j) * kT64];
#pragma unroll
    for (int r = 0; r < NC; ++r) x[r] = sR[r * kT64];
    assemble_M<DIM>(K, a, scale, M);
    if (TRANSPOSED) {
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int j = i + 1; j < NC; ++j) {
                const double t = M[i][j];
                M[i][j] = M[j][i];
                M[j][i] = t;
            }
    }
    const bool ok = gauss_pp<NC>(M, x, 1e-300);
    *out = x[0];
#pragma unroll
    for (int r = 1; r < NC; ++r)
        if (c == r) *out = x[r];
    return ok;
}

// Component c of M^-1 R (TRANSPOSED: M^-T R), M = a I - scale L(K), for this lane's point; every
// lane of the NC warps of the tile calls it.  sK: K in FP64 [d*d][32]; sKf: scale K in FP32
// (SCALED false: scale is 1; else a power of two 2^kexp, or 0 with kexp far below the
// exponents' range); sR: R [NC][32] followed by two buffers of that size for the residuals (all
// at this lane); r: this thread's entry of R.  Returns false when a pivot vanishes.
//
// The warps factor the tile's 32 matrices in FP32, each for itself (the FP32 pipe is idle),
// and x = y0 + y1 + ..., each y the FP32 solution for the residual so far, each thread
// forming its component's FP64 residual.  With contraction q per pass the error after
// y2 is |y2| q: q < 2^-18 leaves it below the last bit, and then |y2| is below 2^-36 |x|;
// otherwise further passes follow.  FP64 elimination with partial pivoting takes over where
// the refinement does not contract, where a right-hand side or solution is outside the FP32
// images' range, where the matrix is (its entries' sum, or its dominant diagonal's, from 2^64 up:
// what a y below the FP32 normal numbers contributes to a residual is then not negligible any
// more, and from 2^128 the factors are not finite), and for a component whose own residual is so far below the point's
// others (2^-126) that its image or its y vanishes.
template <int DIM, bool TRANSPOSED, bool SCALED = false>
__device__ __forceinline__ bool refine_solve64(const double* sK, const float* sKf, double* sR, double a, float af,
                                               int c, double r, double* out, double scale = 1.0, int kexp = 0) {
    constexpr int NC = Packed<DIM>::NC;
    LU32<NC> F;
    static_for<0, NC>([&](auto rr) {
        constexpr int ro = decltype(rr)::value;
        static_for<0, NC>([&](auto kk) {
            constexpr int k = decltype(kk)::value;
            constexpr int e1 = TRANSPOSED ? k : ro, e2 = TRANSPOSED ? ro : k;   // entry (e1, e2) of M
            constexpr int i1 = Packed<DIM>::I(e1), j1 = Packed<DIM>::J(e1);
            constexpr int i = Packed<DIM>::I(e2), j = Packed<DIM>::J(e2);
            float v = ro == k ? af : 0.0f;
            if (j1 == j) v -= sKf[(i1 * DIM + i) * kT64];
            if (i != j && j1 == i) v -= sKf[(i1 * DIM + j) * kT64];
            if (i1 == i) v -= sKf[(j1 * DIM + j) * kT64];
            if (i != j && i1 == j) v -= sKf[(j1 * DIM + i) * kT64];
            F.a[ro][k] = v;
        });
    });
    // the entries' magnitude: of a dominant matrix the diagonal bounds all
    const bool dominant = row_dominant<NC>(F);
    float entries = 0.0f;
    static_for<0, NC>([&](auto rr) {
        constexpr int ro = decltype(rr)::value;
        entries += fabsf(F.a[ro][ro]);
    });
    bool good;
    if (dominant) {
        good = lu32_factor_nopivot<NC>(F, 1e-30f);
    } else {
        static_for<0, NC>([&](auto rr) {
            constexpr int ro = decltype(rr)::value;
            static_for<0, NC>([&](auto kk) {
                constexpr int k = decltype(kk)::value;
                if (k != ro) entries += fabsf(F.a[ro][k]);
            });
        });
        good = lu32_factor<NC>(F, 1e-30f);
    }
    good = good && entries < 18446744073709551616.0f;   // 2^64; false for a NaN
    int e0 = 0;
    constexpr int kMaxPass = 8;
    bool done = false;
    double x = 0.0;
    for (int pass = 0; pass < kMaxPass; ++pass) {
        const double* rb = pass == 0 ? sR : sR + (1 + (pass & 1)) * NC * kT64;
        double rv[NC];
        int emax = 0;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            rv[k] = rb[k * kT64];
            emax = max(emax, biased_exp(rv[k]));
        }
        // a residual of zeros (or below the range of a scaled float) is solved
        bool zero = true;
        float y[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            zero = zero && zero64(rv[k]);
            y[k] = scaled_float(rv[k], emax);
        }
        if (pass == 0) good = good && emax < 0x7ff && (emax > 200 || zero);
        lu32_solve<NC>(F, y);
        unsigned ymax = 0u;
#pragma unroll
        for (int k = 0; k < NC; ++k) ymax = max(ymax, __float_as_uint(y[k]) & 0x7fffffffu);
        const int ey = (int)(ymax >> 23) + emax;       // exponent of the correction (biased by 127 + 1023)
        if (pass == 0) {
            good = good && ymax < 0x7f800000u && ey - 127 + (SCALED ? max(kexp, 0) : 0) < 0x7ff;
            e0 = ey;
        }
        const bool small = ymax != 0u && ey <= e0 - 36;
        static_for<0, NC>([&](auto kk) {
            constexpr int k = decltype(kk)::value;
            // a point's passes are its own, whatever the other points of its tile still need
            if (c == k && !done) {
                x += unscaled_double(y[k], emax);
                // lost in scaling: marked for elimination (nothing else makes x a NaN from finite numbers)
                if (!zero64(r) && (biased_exp(r) <= emax - 127 || (__float_as_uint(y[k]) & 0x7fffffffu) < 0x00800000u))
                    x = __hiloint2double(0x7ff80000, 0);
            }
        });
        done = done || zero || (pass >= 2 && small);
        // the same data in every warp of the tile: they leave together
        if (__all_sync(0xffffffffu, done || !good)) break;
        static_for<0, NC>([&](auto kk) {
            constexpr int k = decltype(kk)::value;
            if (c == k) {
                constexpr int i = Packed<DIM>::I(k), j = Packed<DIM>::J(k);
                r = fma(-a, unscaled_double(y[k], emax), r);
                const int ek = SCALED ? emax + kexp : emax;   // y scale
                static_for<0, DIM>([&](auto ll) {
                    constexpr int l = decltype(ll)::value;
                    constexpr int lj = PackedIndex<DIM>::at(l, j), li = PackedIndex<DIM>::at(l, i);
                    if constexpr (!TRANSPOSED) {
                        r = fma(sK[(i * DIM + l) * kT64], unscaled_double(y[lj], ek), r);
                        r = fma(sK[(j * DIM + l) * kT64], unscaled_double(y[li], ek), r);
                    } else {
                        // (L^T y)_ij = sum_l K_li Y_lj + K_lj Y_li (once for i = j), Y symmetric
                        // with the diagonal doubled
                        r = fma(sK[(l * DIM + i) * kT64], unscaled_double(l == j ? 2.0f * y[lj] : y[lj], ek), r);
                        if constexpr (i != j)
                            r = fma(sK[(l * DIM + j) * kT64], unscaled_double(l == i ? 2.0f * y[li] : y[li], ek), r);
                    }
                });
            }
        });
        sR[(1 + ((pass + 1) & 1)) * NC * kT64 + c * kT64] = r;
        named_sync<NC * 32>();
    }
    bool ok = true;
    if (!good || !done || !finite64(x)) {
        if constexpr (SCALED) ok = solve_by_elimination<DIM, TRANSPOSED>(sK, sR, a, c, &x, scale);
        else ok = solve_by_elimination<DIM, TRANSPOSED>(sK, sR, a, c, &x);
    }
    *out = x;
    return ok;
}

}  // namespace tfs
