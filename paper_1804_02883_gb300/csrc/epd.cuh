// epd.cuh -- arguments and pointwise parts shared by the EPD operator passes
// (epd.cu: radix-8 kernels of the MIXED power-of-two grids; epd_line.cu: every
// other grid and FP64).
#pragma once

#include "common.cuh"
#include "engine.h"

namespace epdlb {

enum RowMode { ROW_GRAD = 0, ROW_LAP = 1, ROW_FWD_S = 2, ROW_INV_FORCE = 3, ROW_DIVX = 4 };
enum ColMode { COL_CONVECT = 0, COL_DIFFUSE = 1, COL_FORCE = 2, COL_DIVY = 3 };

struct EpdK {
    GroupGeom g;
    const double *omega, *omega_t, *phi, *phi_t;
    double *omega_dst;
    double *phi_dst;  // convected densities (ROW_DIVX / COL_DIVY)
    void *cz;  // [run][4][n] complex of the transform type
    const void *vel;
    void *force;
    int bulk_double;
    const void *twx, *twy;  // twiddles of the transform type
    const float2 *tab8x, *tab8y;  // pass tables of each axis' best radix plan (FP32 radix-8/16 kernels)
    const float2 *tab16y, *tab8y_r8;  // column tables of the radix-16 and radix-8 plans (tile-dependent)
    double kunit_x, kunit_y;  // 2 pi / (n dx) per axis
    double mu_c[3][3], mu_0[3];  // mu_I minus its homogeneous value = sum_J mu_c[I][J] Phi_J - mu_0[I] - omega_I
    double phibar[3];         // the homogeneous composition
    double inv_dp, inv_ds;    // 1 / D_P, 1 / D_S
};

// signed wavenumber of bin m; odd operators drop the Nyquist bin
template <typename TT> __device__ __forceinline__ TT kvec(int m, int n, TT unit) { return unit * (TT)signed_bin(m, n); }
template <typename TT> __device__ __forceinline__ TT kvec_odd(int m, int n, TT unit) { return (2 * m == n) ? (TT)0 : kvec<TT>(m, n, unit); }

// Chemical potential of Eq. (1), mu_I = sum_{J != I} chi_IJ Phi_J + kappa_H (sum Phi - 1) - omega_I,
// minus its homogeneous value, in FP64: three FMAs per field on the merged
// coefficients (an FP64 instruction is 1/64 of the FP32 rate here)
__device__ __forceinline__ double mu_one(const EpdK &k, int i, double pa, double pb, double ps, double om)
{
    return fma(k.mu_c[i][0], pa, fma(k.mu_c[i][1], pb, fma(k.mu_c[i][2], ps, -(om + k.mu_0[i]))));
}

// The same in FP32 from the FP64 deviations dPhi_J = Phi_J - Phi-bar_J:
// mu_I - mu_I(Phi-bar, 0) = sum_{J != I} chi_IJ dPhi_J + kappa_H sum_J dPhi_J - omega_I
// (linear in Phi), so FP32 rounding scales with the fluctuations.
__device__ __forceinline__ float2 mu_pair_f(const EpdK &k, const double *phi, const double *om, long long n, long long i, int pair)
{
    const GroupGeom &g = k.g;
    const float da = (float)(phi[i] - k.phibar[0]), db = (float)(phi[n + i] - k.phibar[1]),
                dsv = (float)(phi[2 * n + i] - k.phibar[2]);
    const float inc = (float)g.kappa_h * (da + db + dsv);
    if (pair == 0)
        return make_float2((float)g.chi_ab * db + (float)g.chi_as * dsv + inc - (float)om[i],
                           (float)g.chi_ab * da + (float)g.chi_bs * dsv + inc - (float)om[n + i]);
    return make_float2((float)g.chi_as * da + (float)g.chi_bs * db + inc - (float)om[2 * n + i], 0.f);
}

__device__ __forceinline__ double2 vel_at(const EpdK &k, size_t idx)
{
    if (k.bulk_double) return reinterpret_cast<const double2 *>(k.vel)[idx];
    const float2 v = reinterpret_cast<const float2 *>(k.vel)[idx];
    return make_double2((double)v.x, (double)v.y);
}

// Row and column passes on any grid (epd_line.cu): the operators of EpdK's
// mode in FP64 (fp64) or FP32 transforms, over every run of the group.
cudaError_t epd_line_row(const EpdK &k, int mode, bool fp64, cudaStream_t s);
cudaError_t epd_line_col(const EpdK &k, int mode, bool fp64, cudaStream_t s);

} // namespace epdlb
