// epd_line.cu -- row and column passes of the EPD operators on any grid (App.
// C item 1; Eqs. (2), (5), (19)-(20) of arXiv:1804.02883): FP64 transforms in
// PLAIN_FP64 and for the convection of Phi, FP32 in MIXED_FP32 where a grid
// has no radix-8 passes (epd.cu).  The fields are FP64, two real fields travel
// as one complex one, pointwise combinations with the fields are in FP64.
//
// Each operator is one row and one column pass, once per time step; the tiles
// are small (line_logb) so that a 64 x 64 grid has 64-128 CTAs instead of 2,
// and what a row pass forms from FP64 fields (mu, omega) it leaves in the
// transform's type for the column pass.  The x spectrum of the force travels
// in the plan's digit-reversed order.  The FP64 unit bounds the FP64 passes (4 x
// 256 x 512: 180 us a column pass), latency the FP32 ones: the seven passes of
// a 64 x 150 x 150 step 0.48 -> 0.42 ms as kernel time (cold, serialised).
#include "common.cuh"
#include "engine.h"
#include "epd.cuh"
#include "fftg.cuh"

namespace epdlb {

// Spectral multiplier of a bin, by mode (one type, so that the passes are
// compiled once per precision).
enum EpdOpMode { OP_ONE = 0, OP_GRAD = 1, OP_LAP = 2, OP_FORCE = 3 };
template <typename T> struct EpdOp {
    int mode, n;
    T unit, inv_n;
    // OP_FORCE: the column's x bin from its place in the row spectrum
    int nx, x0;
    LinePlan px;
    T ux, cforce;
    using Pre = V2<T>;
    __device__ __forceinline__ V2<T> pre(int b, int bin) const
    {
        if (mode == OP_GRAD) return mk<T>((T)0, kvec_odd<T>(bin, n, unit) * inv_n);  // i k / n
        if (mode == OP_LAP) {                                                        // -k^2 / n
            const T kk = kvec<T>(bin, n, unit);
            return mk<T>(-kk * kk * inv_n, (T)0);
        }
        if (mode == OP_ONE || x0 + b >= nx) return mk<T>((T)1, (T)0);
        // f(k) = (1/(beta v)) S(k) / dt * i k / |k|^2, Eq. (20), in lattice units;
        // f_x + i f_y is real + i real, so one transform carries both:
        // multiply by c (i kx - ky) / |k|^2 and invert.
        const int mx = line_bin(px, nx, x0 + b);
        const T kx = kvec<T>(mx, nx, ux), ky = kvec<T>(bin, n, unit), k2 = kx * kx + ky * ky;
        if (k2 == (T)0) return mk<T>((T)0, (T)0);
        const T c = cforce / k2;
        return mk<T>(-c * kvec_odd<T>(bin, n, unit), c * kvec_odd<T>(mx, nx, ux));
    }
    __device__ __forceinline__ V2<T> operator()(V2<T> f, V2<T> v) const
    {
        if (mode == OP_GRAD) return mk<T>(-f.y * v.y, f.y * v.x);
        if (mode == OP_LAP) return mk<T>(f.x * v.x, f.x * v.y);
        return mode == OP_ONE ? v : cmul(v, f);
    }
};

template <typename TT, int MODE>
__global__ void __launch_bounds__(256) epd_row(EpdK k, int logb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V2<TT> *buf = reinterpret_cast<V2<TT> *>(smem_raw);
    const GroupGeom &g = k.g;
    const int nx = g.nx, run = blockIdx.y, pair = blockIdx.z, y0 = blockIdx.x << logb, limit = (g.ny - y0) * nx;
    const long long n = g.n, base = (long long)y0 * nx;
    V2<TT> *cz = reinterpret_cast<V2<TT> *>(k.cz) + (size_t)run * 4 * n + base;
    const LineTile tl(true, nx, logb, g.px);
    const V2<TT> *tw = reinterpret_cast<const V2<TT> *>(k.twx);
    line_batches<4, V2<TT>>(
        tl,
        [&](int b, int p, V2<TT> &v) {
            const int i = b * nx + p;
            v = mk<TT>((TT)0, (TT)0);
            if (i >= limit) return;
            const long long s = base + i;
            if (MODE == ROW_GRAD) {
                const double *om = k.omega + (size_t)run * 3 * n;
                v = pair == 0 ? mk<TT>((TT)om[s], (TT)om[n + s]) : mk<TT>((TT)om[2 * n + s], (TT)0);
            } else if (MODE == ROW_LAP) {
                const double *ph = k.phi_t + (size_t)run * 3 * n, *om = k.omega_t + (size_t)run * 3 * n;
                const double pa = ph[s], pb = ph[n + s], ps = ph[2 * n + s];
                v = pair == 0 ? mk<TT>((TT)mu_one(k, 0, pa, pb, ps, om[s]), (TT)mu_one(k, 1, pa, pb, ps, om[n + s]))
                              : mk<TT>((TT)mu_one(k, 2, pa, pb, ps, om[2 * n + s]), (TT)0);
            } else if (MODE == ROW_FWD_S) {
                // S = sum_I dPhi_I^D / D_I, dPhi^D = Phi(t+dt) - Phi~ (Eq. (19))
                const double *p1 = k.phi + (size_t)run * 3 * n, *p0 = k.phi_t + (size_t)run * 3 * n;
                const double sa = (p1[s] - p0[s]) + (p1[n + s] - p0[n + s]);
                v = mk<TT>((TT)(sa * k.inv_dp + (p1[2 * n + s] - p0[2 * n + s]) * k.inv_ds), (TT)0);
            } else if (MODE == ROW_DIVX) {
                // x flux v_x Phi_I, v = u_lat dx/dt
                const double *ph = k.phi + (size_t)run * 3 * n;
                const double vx = vel_at(k, (size_t)run * n + s).x * g.vscale;
                v = pair == 0 ? mk<TT>((TT)(vx * ph[s]), (TT)(vx * ph[n + s])) : mk<TT>((TT)(vx * ph[2 * n + s]), (TT)0);
            } else {
                v = cz[2 * n + i];
            }
        },
        [&](int b, int p, int at, V2<TT> v) {
            buf[at] = v;
            // omega and mu in the transform's type, for the column pass
            if ((MODE == ROW_GRAD || MODE == ROW_LAP) && b * nx + p < limit) cz[(2 + pair) * n + b * nx + p] = v;
        });
    __syncthreads();
    EpdOp<TT> op;
    op.mode = MODE == ROW_GRAD || MODE == ROW_DIVX ? OP_GRAD : (MODE == ROW_LAP ? OP_LAP : OP_ONE);
    op.n = nx;
    op.unit = (TT)k.kunit_x;
    op.inv_n = (TT)(1.0 / (double)nx);
    line_operator<TT, MODE != ROW_INV_FORCE, MODE != ROW_FWD_S>(buf, tl, g.px, tw, op);
    for (LineIter it(tl); it.in(); it.next()) {
        const int i = it.b * nx + it.p;
        if (i >= limit) continue;
        const V2<TT> v = buf[it.at()];
        if (MODE == ROW_INV_FORCE) {
            const V2<TT> f = cscale(v, op.inv_n);
            const size_t s = (size_t)run * n + base + i;
            if (k.bulk_double) reinterpret_cast<double2 *>(k.force)[s] = make_double2((double)f.x, (double)f.y);
            else reinterpret_cast<float2 *>(k.force)[s] = make_float2((float)f.x, (float)f.y);
        } else {
            cz[(MODE == ROW_FWD_S ? 2 : pair) * n + i] = v;
        }
    }
}

template <typename TT, int MODE>
__global__ void __launch_bounds__(256) epd_col(EpdK k, int logb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V2<TT> *buf = reinterpret_cast<V2<TT> *>(smem_raw);
    const GroupGeom &g = k.g;
    const int nx = g.nx, ny = g.ny, run = blockIdx.y, pair = blockIdx.z, x0 = blockIdx.x << logb;
    const long long n = g.n;
    V2<TT> *cz = reinterpret_cast<V2<TT> *>(k.cz) + (size_t)run * 4 * n + x0;
    const LineTile tl(false, ny, logb, g.py);
    const V2<TT> *tw = reinterpret_cast<const V2<TT> *>(k.twy);
    line_batches<4, V2<TT>>(
        tl,
        [&](int b, int p, V2<TT> &v) {
            v = mk<TT>((TT)0, (TT)0);
            if (x0 + b >= nx) return;
            const int i = p * nx + b;
            if (MODE == COL_DIVY) {
                // y flux v_y Phi_I
                const long long s = x0 + i;
                const double *ph = k.phi + (size_t)run * 3 * n;
                const double vy = vel_at(k, (size_t)run * n + s).y * g.vscale;
                v = pair == 0 ? mk<TT>((TT)(vy * ph[s]), (TT)(vy * ph[n + s])) : mk<TT>((TT)(vy * ph[2 * n + s]), (TT)0);
            } else {
                v = cz[(2 + (MODE == COL_FORCE ? 0 : pair)) * n + i];
            }
        },
        [&](int, int, int at, V2<TT> v) { buf[at] = v; });
    __syncthreads();
    EpdOp<TT> op;
    op.mode = MODE == COL_CONVECT || MODE == COL_DIVY ? OP_GRAD : (MODE == COL_DIFFUSE ? OP_LAP : OP_FORCE);
    op.n = ny;
    op.unit = (TT)k.kunit_y;
    op.inv_n = (TT)(1.0 / (double)ny);
    op.nx = nx;
    op.x0 = x0;
    op.px = g.px;
    op.ux = (TT)k.kunit_x;
    op.cforce = (TT)(g.inv_beta_v * g.fstar / (g.dt * (double)ny));
    line_operator<TT, true, true>(buf, tl, g.py, tw, op);
    if (MODE == COL_FORCE) {
        for (LineIter it(tl); it.in(); it.next())
            if (x0 + it.b < nx) cz[2 * n + it.p * nx + it.b] = buf[it.at()];
        return;
    }
    // the row pass's part, the field(s) and the velocity of a batch, then the
    // new field(s): dst = src - c . (row part + column part)
    struct In {
        V2<TT> d;
        double2 u;
        double f0, f1;
    };
    const double *src = (MODE == COL_CONVECT ? k.omega : (MODE == COL_DIFFUSE ? k.omega_t : k.phi)) + (size_t)run * 3 * n + x0;
    double *dst = (MODE == COL_DIVY ? k.phi_dst : k.omega_dst) + (size_t)run * 3 * n + x0;
    const double cv = g.dt * g.vscale, cd = g.dt * (pair == 0 ? g.d_p : g.d_s);
    line_batches<2, In>(
        tl,
        [&](int b, int p, In &v) {
            if (x0 + b >= nx) return;
            const int i = p * nx + b;
            v.d = cz[pair * n + i];
            v.f0 = pair == 0 ? src[i] : src[2 * n + i];
            v.f1 = pair == 0 ? src[n + i] : 0.0;
            if (MODE == COL_CONVECT) v.u = vel_at(k, (size_t)run * n + x0 + i);
        },
        [&](int b, int p, int at, const In &v) {
            if (x0 + b >= nx) return;
            const int i = p * nx + b;
            const V2<TT> y = buf[at];
            double r0, r1 = 0.0;
            if (MODE == COL_CONVECT) {
                // omega~ = omega - dt v . grad omega, v = u_lat dx/dt
                const double vx = v.u.x * cv, vy = v.u.y * cv;
                r0 = v.f0 - (vx * (double)v.d.x + vy * (double)y.x);
                if (pair == 0) r1 = v.f1 - (vx * (double)v.d.y + vy * (double)y.y);
            } else if (MODE == COL_DIFFUSE) {
                // omega(t+dt) = omega~ - dt D_I Lap mu_I
                r0 = v.f0 - cd * ((double)v.d.x + (double)y.x);
                if (pair == 0) r1 = v.f1 - cd * ((double)v.d.y + (double)y.y);
            } else {
                // Phi~ = Phi - dt (d/dx (v_x Phi) + d/dy (v_y Phi))
                r0 = v.f0 - g.dt * ((double)v.d.x + (double)y.x);
                if (pair == 0) r1 = v.f1 - g.dt * ((double)v.d.y + (double)y.y);
            }
            if (pair == 0) {
                dst[i] = r0;
                dst[n + i] = r1;
            } else {
                dst[2 * n + i] = r0;
            }
        });
}

template <typename TT> static cudaError_t row_t(const EpdK &k, int mode, cudaStream_t s)
{
    const int n = k.g.nx, pairs = mode == ROW_FWD_S || mode == ROW_INV_FORCE ? 1 : 2;
    const int l = line_logb(true, n, k.g.px, k.g.ny, k.g.nruns * pairs, sizeof(V2<TT>), 3, 0, 1LL << 30);
    const dim3 grid((k.g.ny + (1 << l) - 1) >> l, k.g.nruns, pairs);
    const size_t sm = LineTile(true, n, l, k.g.px).points() * sizeof(V2<TT>);
    const int th = line_threads(n, k.g.px.r(0), l);
    switch (mode) {
    case ROW_GRAD: epd_row<TT, ROW_GRAD><<<grid, th, sm, s>>>(k, l); break;
    case ROW_LAP: epd_row<TT, ROW_LAP><<<grid, th, sm, s>>>(k, l); break;
    case ROW_FWD_S: epd_row<TT, ROW_FWD_S><<<grid, th, sm, s>>>(k, l); break;
    case ROW_INV_FORCE: epd_row<TT, ROW_INV_FORCE><<<grid, th, sm, s>>>(k, l); break;
    default:
        if constexpr (sizeof(TT) == 8) epd_row<TT, ROW_DIVX><<<grid, th, sm, s>>>(k, l);
        else return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}
template <typename TT> static cudaError_t col_t(const EpdK &k, int mode, cudaStream_t s)
{
    const int n = k.g.ny, pairs = mode == COL_FORCE ? 1 : 2;
    const int l = line_logb(false, n, k.g.py, k.g.nx, k.g.nruns * pairs, sizeof(V2<TT>), sizeof(TT) == 4 ? 3 : 2,
                            sizeof(TT) == 4 ? 1 : 0, 1LL << 30);
    const dim3 grid((k.g.nx + (1 << l) - 1) >> l, k.g.nruns, pairs);
    const size_t sm = LineTile(false, n, l, k.g.py).points() * sizeof(V2<TT>);
    const int th = line_threads(n, k.g.py.r(0), l);
    switch (mode) {
    case COL_CONVECT: epd_col<TT, COL_CONVECT><<<grid, th, sm, s>>>(k, l); break;
    case COL_DIFFUSE: epd_col<TT, COL_DIFFUSE><<<grid, th, sm, s>>>(k, l); break;
    case COL_FORCE: epd_col<TT, COL_FORCE><<<grid, th, sm, s>>>(k, l); break;
    default:
        if constexpr (sizeof(TT) == 8) epd_col<TT, COL_DIVY><<<grid, th, sm, s>>>(k, l);
        else return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t epd_line_row(const EpdK &k, int mode, bool fp64, cudaStream_t s) { return fp64 ? row_t<double>(k, mode, s) : row_t<float>(k, mode, s); }
cudaError_t epd_line_col(const EpdK &k, int mode, bool fp64, cudaStream_t s) { return fp64 ? col_t<double>(k, mode, s) : col_t<float>(k, mode, s); }

} // namespace epdlb
