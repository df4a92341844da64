// epd.cu -- EPD part of the hybrid LB/EPD step of arXiv:1804.02883 on sm_103a:
//   auxiliary convection of omega (App. C, item 1),
//   diffusion step omega <- omega~ - dt D_I Lap mu_I (Sec. 2, Eq. (5); App. C),
//   force reconstruction from the composition change (Sec. 2, Eqs. (19)-(20)),
//   convection of the composition fields Phi~ = Phi - dt div(v Phi) (the
//   convective part of Eq. (2); the exact step of App. C).
//
// Spatial derivatives are spectral with continuum wavenumbers; first
// derivatives drop the Nyquist bin, the Laplacian keeps it.  d/dx and d2/dx2
// act on rows only and d/dy, d2/dy2 on columns only, so each operator is one
// row pass plus one column pass; two real fields travel as one complex field.
//
// The fields (omega, Phi) are FP64.  The transforms run in the type TT: FP64
// in PLAIN_FP64, FP32 in MIXED_FP32.  In FP32 the transformed quantities are
// small differences: mu_I minus its homogeneous value (the constant drops
// out of every derivative, and FP32 rounding then scales with the
// fluctuations rather than with mu itself), omega (zero-mean noise), and
// dPhi^D.  Pointwise combinations with the fields are done in FP64.
#include <cmath>
#include <cstdlib>

#include "common.cuh"
#include "engine.h"
#include "epd.cuh"
#include "fft8.cuh"

namespace epdlb {

// ---------------------------------------------------------------------------
// FP32 radix-8 row and column passes (MIXED_FP32, grids with 64..2048 points
// per axis): the operators and data flow of epd_line.cu, transforms and tiles
// (RowTile, ColTile) from fft8.cuh.
// ---------------------------------------------------------------------------

// i k / n (first derivative, Nyquist bin dropped) and -k^2 / n along one axis
struct OpGrad {
    int n;
    float unit, inv_n;
    __device__ __forceinline__ float2 operator()(int, int bin, float2 v) const
    {
        const float kk = (2 * bin == n ? 0.f : unit * (float)signed_bin(bin, n)) * inv_n;
        return f2(-kk * v.y, kk * v.x);
    }
};
struct OpLap {
    int n;
    float unit, inv_n;
    __device__ __forceinline__ float2 operator()(int, int bin, float2 v) const
    {
        const float kk = unit * (float)signed_bin(bin, n), f = -kk * kk * inv_n;
        return f2(v.x * f, v.y * f);
    }
};
// force of Eq. (20) on a column of the row spectrum: c (i kx - ky) / |k|^2
struct OpForce {
    int nx, ny, x0;
    float ux, uy, cforce;
    __device__ __forceinline__ float2 operator()(int c, int my, float2 v) const
    {
        const int mx = x0 + c;
        const float kx = ux * (float)signed_bin(mx, nx), ky = uy * (float)signed_bin(my, ny);
        const float k2 = kx * kx + ky * ky;
        if (k2 == 0.f) return f2(0.f, 0.f);
        const float cc = cforce / k2;
        const float kxo = 2 * mx == nx ? 0.f : kx, kyo = 2 * my == ny ? 0.f : ky;
        return fmul(v, f2(-cc * kyo, cc * kxo));
    }
};

template <int LOGX, int MODE>
__global__ void __launch_bounds__(RowTile<LOGX>::T) epd_row8(EpdK k)
{
    using RT = RowTile<LOGX>;
    using RL = RowLayout<LOGX>;
    constexpr int NX = RT::NX, P = RT::P, T = RT::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *buf = reinterpret_cast<float2 *>(smem_raw);
    float2 *tab = buf + RT::ROWS * RL::PITCH;
    const GroupGeom &g = k.g;
    const int run = blockIdx.y, pair = blockIdx.z, tid = threadIdx.x;
    const long long n = g.n;
    const long long base = (long long)blockIdx.x * P;
    float2 *cz = reinterpret_cast<float2 *>(k.cz);
    copy_tables(tab, k.tab8x, RT::TAB, tid, T);
    // the inputs of this thread in batches, each batch's loads before its
    // stores (the scratch planes written below could alias the fields as far
    // as the compiler knows, so interleaving would serialise the loads
    // behind the stores)
    constexpr int UB = P / T < 8 ? P / T : 8;  // inputs per batch
#pragma unroll
    for (int u0 = 0; u0 < P / T; u0 += UB) {
        float2 vin[UB];
#pragma unroll
        for (int u = u0; u < u0 + UB; ++u) {
            const int i = tid + u * T;
            const long long s = base + i;
            float2 v;
            if (MODE == ROW_GRAD) {
                const double *om = k.omega + (size_t)run * 3 * n;
                v = pair == 0 ? f2((float)om[s], (float)om[n + s]) : f2((float)om[2 * n + s], 0.f);
            } else if (MODE == ROW_LAP) {
                v = mu_pair_f(k, k.phi_t + (size_t)run * 3 * n, k.omega_t + (size_t)run * 3 * n, n, s, pair);
            } else if (MODE == ROW_FWD_S) {
                // S = sum_I dPhi_I^D / D_I from the FP64 differences, in FP32
                const double *p1 = k.phi + (size_t)run * 3 * n, *p0 = k.phi_t + (size_t)run * 3 * n;
                const float da = (float)(p1[s] - p0[s]), db = (float)(p1[n + s] - p0[n + s]), dsv = (float)(p1[2 * n + s] - p0[2 * n + s]);
                v = f2((da + db) * (float)(1.0 / g.d_p) + dsv * (float)(1.0 / g.d_s), 0.f);
            } else {
                v = cz[((size_t)run * 4 + 2) * n + s];
            }
            vin[u - u0] = v;
        }
#pragma unroll
        for (int u = u0; u < u0 + UB; ++u) {
            const int i = tid + u * T;
            // the column pass of the same operator reads this FP32 input from the
            // free scratch planes 2, 3 instead of forming it again from FP64 fields
            if (MODE == ROW_GRAD || MODE == ROW_LAP) cz[((size_t)run * 4 + 2 + pair) * n + base + i] = vin[u - u0];
            buf[RL::at(i / NX, i % NX)] = vin[u - u0];
        }
    }
    __syncthreads();
    if (MODE == ROW_FWD_S) {
        forward<LOGX, T, RL, P, RT::MR>(buf, tab, tid);
#pragma unroll
        for (int u = 0; u < P / T; ++u) {
            const int i = tid + u * T;
            cz[((size_t)run * 4 + 2) * n + base + i] = buf[RL::at(i / NX, i % NX)];
        }
        return;
    }
    const float unit = (float)k.kunit_x, inv_n = 1.f / (float)NX;
    if (MODE == ROW_GRAD)
        transform_pair<LOGX, T, RL, P, OpGrad, RT::MR>(buf, tab, OpGrad{NX, unit, inv_n}, tid);
    else if (MODE == ROW_LAP)
        transform_pair<LOGX, T, RL, P, OpLap, RT::MR>(buf, tab, OpLap{NX, unit, inv_n}, tid);
    else
        inverse_open<LOGX, T, RL, P, RT::MR>(buf, tab, tid);
    constexpr int RLOG_L = inv_rlog(LOGX, npasses(LOGX, RT::MR) - 1, RT::MR), RR = 1 << RLOG_L, PER_L = NX / RR, NB_L = P / RR / T;
    float2 h[NB_L][RR];
    int bb[NB_L], tt[NB_L];
    last_inverse<LOGX, NB_L, T, RL, RT::MR>(buf, h, bb, tt, tid);
#pragma unroll
    for (int j = 0; j < NB_L; ++j)
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            const long long s = base + (long long)bb[j] * NX + tt[j] + r * PER_L;
            if (MODE == ROW_INV_FORCE) {
                const float2 f = f2(h[j][r].x * inv_n, h[j][r].y * inv_n);
                if (k.bulk_double) reinterpret_cast<double2 *>(k.force)[(size_t)run * n + s] = make_double2((double)f.x, (double)f.y);
                else reinterpret_cast<float2 *>(k.force)[(size_t)run * n + s] = f;
            } else {
                cz[((size_t)run * 4 + pair) * n + s] = h[j][r];
            }
        }
}

template <int LOGY, int MODE, int CW>
__global__ void __launch_bounds__(ColTile<LOGY, CW>::T) epd_col8(EpdK k)
{
    using CT = ColTile<LOGY, CW>;
    using CL = ColLayout<LOGY, CT::C>;
    constexpr int NY = CT::NY, C = CT::C, P = CT::P, T = CT::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *buf = reinterpret_cast<float2 *>(smem_raw);
    float2 *tab = buf + P;
    const GroupGeom &g = k.g;
    const int nx = g.nx, run = blockIdx.y, pair = blockIdx.z, x0 = blockIdx.x * C, tid = threadIdx.x;
    const long long n = g.n;
    float2 *cz = reinterpret_cast<float2 *>(k.cz);
    copy_tables(tab, CT::MR == 4 ? k.tab16y : k.tab8y_r8, CT::TAB, tid, T);
#pragma unroll
    for (int u = 0; u < P / T; ++u) {
        const int i = tid + u * T;
        const long long s = (long long)(i / C) * nx + x0 + (i % C);
        float2 v;
        if (MODE == COL_CONVECT || MODE == COL_DIFFUSE) {
            v = cz[((size_t)run * 4 + 2 + pair) * n + s];  // stored by the row pass (omega, mu in FP32)
        } else {
            v = cz[((size_t)run * 4 + 2) * n + s];
        }
        buf[i] = v;  // CL::at(i % C, i / C)
    }
    __syncthreads();
    const float uy = (float)k.kunit_y, inv_n = 1.f / (float)NY;
    if (MODE == COL_CONVECT)
        transform_pair<LOGY, T, CL, P, OpGrad, CT::MR>(buf, tab, OpGrad{NY, uy, inv_n}, tid);
    else if (MODE == COL_DIFFUSE)
        transform_pair<LOGY, T, CL, P, OpLap, CT::MR>(buf, tab, OpLap{NY, uy, inv_n}, tid);
    else
        transform_pair<LOGY, T, CL, P, OpForce, CT::MR>(
            buf, tab, OpForce{nx, NY, x0, (float)k.kunit_x, uy, (float)(g.inv_beta_v * g.fstar / (g.dt * (double)NY))}, tid);
    constexpr int RLOG_L = inv_rlog(LOGY, npasses(LOGY, CT::MR) - 1, CT::MR), RR = 1 << RLOG_L, PER_L = NY / RR, NB_L = P / RR / T;
    float2 h[NB_L][RR];
    int bb[NB_L], tt[NB_L];
    last_inverse<LOGY, NB_L, T, CL, CT::MR>(buf, h, bb, tt, tid);
    // in batches of SB points: every load first, then the stores (the output
    // field could alias the inputs as far as the compiler knows, which would
    // serialise each load behind the previous stores)
    constexpr int SB = RR < 4 ? RR : 4;
#pragma unroll
    for (int j = 0; j < NB_L; ++j)
#pragma unroll
        for (int r0 = 0; r0 < RR; r0 += SB) {
            long long sj[SB];
#pragma unroll
            for (int b = 0; b < SB; ++b) sj[b] = (long long)(tt[j] + (r0 + b) * PER_L) * nx + x0 + bb[j];
            if (MODE == COL_FORCE) {
#pragma unroll
                for (int b = 0; b < SB; ++b) cz[((size_t)run * 4 + 2) * n + sj[b]] = h[j][r0 + b];
            } else if (MODE == COL_CONVECT) {
                // omega~ = omega - dt v . grad omega, v = u_lat dx/dt (increment in FP32)
                const double *om = k.omega + (size_t)run * 3 * n;
                double *ot = k.omega_dst + (size_t)run * 3 * n;
                const float cv = (float)(g.vscale * g.dt);
                float2 dxf[SB], u[SB];
                double o0[SB], o1[SB];
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    const long long s = sj[b];
                    dxf[b] = cz[((size_t)run * 4 + pair) * n + s];
                    u[b] = reinterpret_cast<const float2 *>(k.vel)[(size_t)run * n + s];  // FP32 bulk
                    o0[b] = pair == 0 ? om[s] : om[2 * n + s];
                    o1[b] = pair == 0 ? om[n + s] : 0.0;
                }
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    const long long s = sj[b];
                    const float2 dyf = h[j][r0 + b];
                    const float vx = u[b].x * cv, vy = u[b].y * cv;
                    if (pair == 0) {
                        ot[s] = o0[b] - (double)(vx * dxf[b].x + vy * dyf.x);
                        ot[n + s] = o1[b] - (double)(vx * dxf[b].y + vy * dyf.y);
                    } else {
                        ot[2 * n + s] = o0[b] - (double)(vx * dxf[b].x + vy * dyf.x);
                    }
                }
            } else {
                // omega(t+dt) = omega~ - dt D_I Lap mu_I (increment in FP32)
                const double *ot = k.omega_t + (size_t)run * 3 * n;
                double *om = k.omega_dst + (size_t)run * 3 * n;
                float2 lxf[SB];
                double o0[SB], o1[SB];
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    const long long s = sj[b];
                    lxf[b] = cz[((size_t)run * 4 + pair) * n + s];
                    o0[b] = pair == 0 ? ot[s] : ot[2 * n + s];
                    o1[b] = pair == 0 ? ot[n + s] : 0.0;
                }
#pragma unroll
                for (int b = 0; b < SB; ++b) {
                    const long long s = sj[b];
                    const float2 dyf = h[j][r0 + b];
                    if (pair == 0) {
                        const float c = (float)(g.dt * g.d_p);
                        om[s] = o0[b] - (double)(c * (lxf[b].x + dyf.x));
                        om[n + s] = o1[b] - (double)(c * (lxf[b].y + dyf.y));
                    } else {
                        om[2 * n + s] = o0[b] - (double)((float)(g.dt * g.d_s) * (lxf[b].x + dyf.x));
                    }
                }
            }
        }
}

// Launch of the radix-8 row / column pass for the group's grid, or false
// when the grid has no radix-8 instantiation.
template <int MODE, int L>
static bool row8_at(int logx, const EpdK &k, dim3 grid_yz, cudaStream_t s)
{
    if constexpr (L > 11) {
        return false;
    } else {
        if (logx != L) return row8_at<MODE, L + 1>(logx, k, grid_yz, s);
        using RT = RowTile<L>;
        static PerDevice conf;
        if (conf.once([] { return cudaFuncSetAttribute(epd_row8<L, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RT::SMEM); }))
            return false;
        const int blocks = (int)(k.g.n / RT::P);
        epd_row8<L, MODE><<<dim3(blocks, grid_yz.y, grid_yz.z), RT::T, RT::SMEM, s>>>(k);
        return true;
    }
}
template <int MODE, int L, int CW>
static bool col8_launch(const EpdK &k, dim3 grid_yz, cudaStream_t s)
{
    using CT = ColTile<L, CW>;
    if (k.g.nx % CT::C) return false;
    static PerDevice conf;
    if (conf.once([] { return cudaFuncSetAttribute(epd_col8<L, MODE, CW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CT::SMEM); }))
        return false;
    epd_col8<L, MODE, CW><<<dim3(k.g.nx / CT::C, grid_yz.y, grid_yz.z), CT::T, CT::SMEM, s>>>(k);
    return true;
}
// colw: column tile width (4, 8, 16; 0 = default)
template <int MODE, int L>
static bool col8_at(int logy, const EpdK &k, dim3 grid_yz, cudaStream_t s, int colw)
{
    if constexpr (L > 11) {
        return false;
    } else {
        if (logy != L) return col8_at<MODE, L + 1>(logy, k, grid_yz, s, colw);
        switch (colw) {
        case 4: return col8_launch<MODE, L, 4>(k, grid_yz, s);
        case 8: return col8_launch<MODE, L, 8>(k, grid_yz, s);
        case 16: return col8_launch<MODE, L, 16>(k, grid_yz, s);
        default: return col8_launch<MODE, L, ColTile<L>::C>(k, grid_yz, s);
        }
    }
}
// radix-8 passes apply to MIXED_FP32 groups with 64 <= nx, ny <= 2048 and at
// least 2048 sites
static bool use_r8(const Group &G)
{
    return G.prec == EPD_LB_MIXED_FP32 && G.tab8x && G.tab8y && G.g.logx >= 6 && G.g.logy >= 6 && G.g.logx <= 11 &&
           G.g.logy <= 11 && G.g.n >= 2048;
}

static EpdK make_k(Group &G)
{
    EpdK k;
    k.g = G.g;
    k.omega = G.omega;
    k.omega_t = G.omega_t;
    k.phi = G.phi;
    k.phi_t = G.phi_t;
    k.omega_dst = nullptr;
    k.phi_dst = nullptr;
    k.cz = G.cz;
    k.vel = G.vel;
    k.force = G.force;
    k.bulk_double = G.prec == EPD_LB_PLAIN_FP64;
    // FP32 transforms use the bulk (FP32) twiddle tables, FP64 ones the FP64 tables
    k.twx = k.bulk_double ? (const void *)G.twx_d : G.twx;
    k.twy = k.bulk_double ? (const void *)G.twy_d : G.twy;
    // tables of each axis' radix plan (RowTile / ColTile pick best_mr)
    k.tab8x = best_mr(G.g.logx) == 4 ? G.tab16x : G.tab8x;
    k.tab8y = best_mr(G.g.logy) == 4 ? G.tab16y : G.tab8y;
    k.tab16y = G.tab16y;
    k.tab8y_r8 = G.tab8y;
    const double pi = 3.14159265358979323846;
    k.kunit_x = 2.0 * pi / ((double)G.g.nx * G.g.dx);
    k.kunit_y = 2.0 * pi / ((double)G.g.ny * G.g.dx);
    // homogeneous composition: Phi_A = phi_p N_A/N_s, Phi_B = phi_p (1 - N_A/N_s), Phi_S = 1 - phi_p
    const double fa = (double)G.g.na / (double)G.g.ns;
    const double pa = G.g.phi_p * fa, pb = G.g.phi_p * (1.0 - fa), ps = 1.0 - G.g.phi_p;
    const double inc = G.g.kappa_h * (pa + pb + ps - 1.0);
    const double mu_ref[3] = {G.g.chi_ab * pb + G.g.chi_as * ps + inc, G.g.chi_ab * pa + G.g.chi_bs * ps + inc,
                              G.g.chi_as * pa + G.g.chi_bs * pb + inc};
    const double chi[3][3] = {{0.0, G.g.chi_ab, G.g.chi_as}, {G.g.chi_ab, 0.0, G.g.chi_bs}, {G.g.chi_as, G.g.chi_bs, 0.0}};
    for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j) k.mu_c[i][j] = chi[i][j] + G.g.kappa_h;
        k.mu_0[i] = G.g.kappa_h + mu_ref[i];
    }
    k.inv_dp = 1.0 / G.g.d_p;
    k.inv_ds = 1.0 / G.g.d_s;
    k.phibar[0] = pa;
    k.phibar[1] = pb;
    k.phibar[2] = ps;
    return k;
}

cudaError_t launch_aux_convection(Group &G, cudaStream_t s)
{
    EpdK k = make_k(G);
    k.omega_dst = G.omega_t;
    if (use_r8(G)) {
        const dim3 gz(1, G.g.nruns, 2);
        if (row8_at<ROW_GRAD, 6>(G.g.logx, k, gz, s) && col8_at<COL_CONVECT, 6>(G.g.logy, k, gz, s, G.colw)) return cudaGetLastError();
        return cudaErrorInvalidConfiguration;
    }
    const bool d = G.prec == EPD_LB_PLAIN_FP64;
    const cudaError_t e = epd_line_row(k, ROW_GRAD, d, s);
    return e ? e : epd_line_col(k, COL_CONVECT, d, s);
}

cudaError_t launch_diffusion(Group &G, cudaStream_t s)
{
    EpdK k = make_k(G);
    k.omega_dst = G.omega;
    if (use_r8(G)) {
        const dim3 gz(1, G.g.nruns, 2);
        if (row8_at<ROW_LAP, 6>(G.g.logx, k, gz, s) && col8_at<COL_DIFFUSE, 6>(G.g.logy, k, gz, s, G.colw)) return cudaGetLastError();
        return cudaErrorInvalidConfiguration;
    }
    const bool d = G.prec == EPD_LB_PLAIN_FP64;
    const cudaError_t e = epd_line_row(k, ROW_LAP, d, s);
    return e ? e : epd_line_col(k, COL_DIFFUSE, d, s);
}

cudaError_t launch_force(Group &G, cudaStream_t s)
{
    EpdK k = make_k(G);
    if (use_r8(G)) {
        const dim3 gz(1, G.g.nruns, 1);
        if (row8_at<ROW_FWD_S, 6>(G.g.logx, k, gz, s) && col8_at<COL_FORCE, 6>(G.g.logy, k, gz, s, G.colw) &&
            row8_at<ROW_INV_FORCE, 6>(G.g.logx, k, gz, s))
            return cudaGetLastError();
        return cudaErrorInvalidConfiguration;
    }
    const bool d = G.prec == EPD_LB_PLAIN_FP64;
    cudaError_t e = epd_line_row(k, ROW_FWD_S, d, s);
    if (!e) e = epd_line_col(k, COL_FORCE, d, s);
    return e ? e : epd_line_row(k, ROW_INV_FORCE, d, s);
}

// Column tile autotuner (radix-8 EPD column passes and streaming propagator
// column passes): each candidate width runs the diffusion column pass a few
// times on the group's state, writing only scratch (omega~, the EPD scratch);
// the fastest width is kept in G.colw.  Every width computes the same
// per-column transforms, so the results do not depend on the choice.
// EPD_LB_COLUMN_TILE=4|8|16 in the environment forces a width.
cudaError_t tune_column_tiles(Group &G, cudaStream_t s)
{
    if (!use_r8(G)) return cudaSuccess;
    if (const char *env = std::getenv("EPD_LB_COLUMN_TILE")) {
        const int w = std::atoi(env);
        if (w == 4 || w == 8 || w == 16) {
            G.colw = w;
            return cudaSuccess;
        }
    }
    EpdK k = make_k(G);
    k.omega_t = G.omega;      // read the current state ...
    k.phi_t = G.phi;
    k.omega_dst = G.omega_t;  // ... write only scratch (rewritten by the next step)
    const dim3 gz(1, G.g.nruns, 2);
    cudaEvent_t a, b;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) return cudaGetLastError();
    float best = 1e30f;
    int best_w = 0;
    for (int w : kColWidths) {
        if (G.g.nx % w) continue;
        if (!col8_at<COL_DIFFUSE, 6>(G.g.logy, k, gz, s, w)) {
            cudaGetLastError();
            continue;
        }
        float t = 1e30f;
        for (int rep = 0; rep < 4; ++rep) {
            cudaEventRecord(a, s);
            col8_at<COL_DIFFUSE, 6>(G.g.logy, k, gz, s, w);
            cudaEventRecord(b, s);
            cudaEventSynchronize(b);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, a, b);
            if (rep > 0 && ms < t) t = ms;  // the first launch is a warm-up
        }
        if (t < best) {
            best = t;
            best_w = w;
        }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    G.colw = best_w;
    return cudaGetLastError();
}

// Convection of the composition fields, always with FP64 transforms (the
// FP64 twiddles exist in both precisions; the FP64 scratch planes fit the
// EPD scratch): the densities of every run of the group.
cudaError_t launch_convect_phi(Group &G, const double *phi, double *phi_dst, cudaStream_t s)
{
    EpdK k = make_k(G);
    k.phi = phi;
    k.phi_dst = phi_dst;
    k.twx = G.twx_d;
    k.twy = G.twy_d;
    const cudaError_t e = epd_line_row(k, ROW_DIVX, true, s);
    return e ? e : epd_line_col(k, COL_DIVY, true, s);
}

} // namespace epdlb
