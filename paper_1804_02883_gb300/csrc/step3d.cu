// step3d.cu -- the coupled hybrid LB/EPD step on a 3D box (the extension the
// paper names in Sec. 2 and Sec. 5), FP64 spectral operators on sm_103a:
//   omega~ = omega - dt v . grad omega            (App. C, item 1)
//   Phi~ = solve3d(omega~)                        (Eqs. (6)-(11))
//   omega(t+dt) = omega~ - dt D_I Lap mu_I(Phi~)  (Eq. (5))
//   Phi(t+dt) = solve3d(omega(t+dt))
//   f = (1/(beta v)) sum_I dPhi_I/(D_I dt) i k/|k|^2 (Eqs. (19)-(20)) + f_P(y) x^
//   one D3Q19 collide-stream.
// A derivative along one axis needs the transforms of that axis only, and two
// real fields travel as one complex one, so the gradient and the Laplacian are
// three fused line passes each per pair of fields (fftg.cuh: fill from the
// fields, forward, factor, inverse, combine with the fields): 24 one-way
// sweeps of the box for both, where full 3D transforms of each field take 54
// and an elementwise pass per derivative.  The force is one 3D transform
// forward, in the plans' digit-reversed order, and two back: f_x + i f_y as one
// complex field, f_z as another.  FP64 instructions bound all of it (2 lanes
// per SM and cycle).  64 x 128 x 128 (ns = 16): these operators 5.2 -> 2.4 ms
// of kernel time (cold, serialised).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "engine.h"
#include "fftg.cuh"

namespace epdlb {
namespace {

using C2 = V2<double>;

// Lines along one axis of the box: point p of line i = j lines + c (c < lines,
// planes j) at j PS + c LS + p S.
struct Lines {
    int n, row;       // length; 1: contiguous points (x), 0: contiguous lines
    long long S, LS, PS;
    long long lines;  // lines per plane
    int planes;
    LinePlan plan;
    const C2 *tw;
    double unit;      // 2 pi / (n dx)
};

enum Op3 { D3_ONE = 0, D3_GRAD = 1, D3_LAP = 2, D3_FORCE_XY = 3, D3_FORCE_Z = 4 };

// Spectral multiplier along the pass's axis; the force's at the (x, y) bins of
// the pillar as well.
struct Op3D {
    int mode, n;
    double unit, inv_n;
    int nx, ny;
    long long c0;  // first pillar of the tile
    LinePlan px, py;
    double ux, uy, c;  // c: the force's constant over the number of sites
    using Pre = C2;
    __device__ __forceinline__ C2 pre(int b, int bin) const
    {
        const double k = unit * signed_bin(bin, n), ko = 2 * bin == n ? 0.0 : k;  // odd operators drop the Nyquist bin
        if (mode == D3_GRAD) return mk<double>(0.0, ko * inv_n);
        if (mode == D3_LAP) return mk<double>(-k * k * inv_n, 0.0);
        if (mode == D3_ONE) return mk<double>(1.0, 0.0);
        const long long cb = c0 + b;
        if (cb >= (long long)nx * ny) return mk<double>(0.0, 0.0);
        const int yi = (int)(cb / nx), bx = line_bin(px, nx, (int)(cb - (long long)yi * nx)), by = line_bin(py, ny, yi);
        const double kx = ux * signed_bin(bx, nx), ky = uy * signed_bin(by, ny), k2 = kx * kx + ky * ky + k * k;
        if (k2 == 0.0) return mk<double>(0.0, 0.0);
        const double m = c / k2;
        if (mode == D3_FORCE_Z) return mk<double>(0.0, m * ko);
        const double kxo = 2 * bx == nx ? 0.0 : kx, kyo = 2 * by == ny ? 0.0 : ky;
        return mk<double>(-m * kyo, m * kxo);  // i kx + i (i ky): f_x + i f_y
    }
    __device__ __forceinline__ C2 operator()(C2 f, C2 v) const
    {
        if (mode == D3_GRAD || mode == D3_FORCE_Z) return mk<double>(-f.y * v.y, f.y * v.x);
        if (mode == D3_LAP) return mk<double>(f.x * v.x, f.x * v.y);
        return mode == D3_ONE ? v : cmul(v, f);
    }
};

// What a pass reads and writes.
enum Pass3 { P3_CONVECT, P3_DIFFUSE, P3_FWD, P3_BOTH, P3_INV, P3_INV_OUT };
struct Args3 {
    long long n;
    int first;                 // first axis of a sum of derivatives: dst = src - .., else dst -= ..
    const double *omega, *wt_c, *phi, *phi0, *vel;  // vel: the axis' component
    double *dst, *mu;
    C2 *in, *out;
    double mu_c[3][3], mu_0[3];
    double ca, cb;             // CONVECT: ca; DIFFUSE: ca (A, B), cb (S); FWD: 1/D_P, 1/D_S
    double *force, *ftot;      // INV_OUT: component(s)
    int comp, nx, ny;
    double f0, scale;
};

template <int MODE>
__global__ void __launch_bounds__(256) line3(Lines L, Op3D op, Args3 a, int logb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *buf = reinterpret_cast<C2 *>(smem_raw);
    const LineTile tl(L.row, L.n, logb, L.plan);
    const long long c0 = (long long)blockIdx.x << logb, base = (long long)blockIdx.y * L.PS + c0 * L.LS;
    const int pair = blockIdx.z;  // fields (A, B) or (S)
    const long long n = a.n, f0 = pair == 0 ? 0 : 2 * n;
    auto site = [&](int b, int p) { return base + b * L.LS + p * L.S; };
    auto in = [&](int b) { return c0 + b < L.lines; };
    op.c0 = c0;
    line_batches<4, C2>(
        tl,
        [&](int b, int p, C2 &v) {
            v = mk<double>(0.0, 0.0);
            if (!in(b)) return;
            const long long s = site(b, p);
            if (MODE == P3_CONVECT) {
                v = mk<double>(a.omega[f0 + s], pair == 0 ? a.omega[n + s] : 0.0);
            } else if (MODE == P3_DIFFUSE) {
                if (a.first) {  // mu of Eq. (1) from the fields, kept for the other axes
                    const double pa = a.phi[s], pb = a.phi[n + s], ps = a.phi[2 * n + s];
                    auto mu = [&](int i, double om) {
                        return fma(a.mu_c[i][0], pa, fma(a.mu_c[i][1], pb, fma(a.mu_c[i][2], ps, -(om + a.mu_0[i]))));
                    };
                    v = pair == 0 ? mk<double>(mu(0, a.wt_c[s]), mu(1, a.wt_c[n + s])) : mk<double>(mu(2, a.wt_c[2 * n + s]), 0.0);
                } else {
                    v = mk<double>(a.mu[f0 + s], pair == 0 ? a.mu[n + s] : 0.0);
                }
            } else if (MODE == P3_FWD && a.phi) {
                // S = sum_I dPhi_I / D_I
                const double sa = (a.phi[s] - a.phi0[s]) + (a.phi[n + s] - a.phi0[n + s]);
                v = mk<double>(sa * a.ca + (a.phi[2 * n + s] - a.phi0[2 * n + s]) * a.cb, 0.0);
            } else {
                v = a.in[s];
            }
        },
        [&](int b, int p, int at, C2 v) {
            buf[at] = v;
            if (MODE == P3_DIFFUSE && a.first && in(b)) {
                const long long s = site(b, p);
                a.mu[f0 + s] = v.x;
                if (pair == 0) a.mu[n + s] = v.y;
            }
        });
    __syncthreads();
    constexpr bool FWD = MODE != P3_INV && MODE != P3_INV_OUT, BWD = MODE != P3_FWD;
    line_operator<double, FWD, BWD>(buf, tl, L.plan, L.tw, op);
    if (MODE == P3_CONVECT || MODE == P3_DIFFUSE) {
        struct In {
            double s0, s1, v;
        };
        const double *src = a.first ? (MODE == P3_CONVECT ? a.omega : a.wt_c) : a.dst;
        const double c = MODE == P3_DIFFUSE && pair ? a.cb : a.ca;
        line_batches<4, In>(
            tl,
            [&](int b, int p, In &v) {
                if (!in(b)) return;
                const long long s = site(b, p);
                v.s0 = src[f0 + s];
                v.s1 = pair == 0 ? src[n + s] : 0.0;
                v.v = MODE == P3_CONVECT ? c * a.vel[s] : c;
            },
            [&](int b, int p, int at, const In &v) {
                if (!in(b)) return;
                const long long s = site(b, p);
                const C2 d = buf[at];
                a.dst[f0 + s] = v.s0 - v.v * d.x;
                if (pair == 0) a.dst[n + s] = v.s1 - v.v * d.y;
            });
        return;
    }
    for (LineIter it(tl); it.in(); it.next()) {
        if (!in(it.b)) continue;
        const long long s = site(it.b, it.p);
        const C2 v = buf[it.at()];
        if (MODE == P3_INV_OUT) {
            // force component(s); the total adds the body force of Eq. (23)
            // along x, -f0 for y < ny/2 and +f0 above
            const double f = a.scale * v.x;
            a.force[(size_t)a.comp * n + s] = f;
            double fb = 0.0;
            if (a.comp == 0) {
                fb = (int)((s / a.nx) % a.ny) < a.ny / 2 ? -a.f0 : a.f0;
                const double fy = a.scale * v.y;
                a.force[n + s] = fy;
                a.ftot[n + s] = fy;
            }
            a.ftot[(size_t)a.comp * n + s] = f + fb;
        } else {
            a.out[s] = v;
        }
    }
}

template <int MODE> cudaError_t run3(const Lines &L, const Op3D &op, const Args3 &a, cudaStream_t s)
{
    const int fields = MODE == P3_CONVECT || MODE == P3_DIFFUSE ? 2 : 1;
    const int l = line_logb(L.row, L.n, L.plan, L.lines, L.planes * fields, sizeof(C2), L.row ? 3 : 2, 0, 1LL << 30);
    const size_t sm = LineTile(L.row, L.n, l, L.plan).points() * sizeof(C2);
    const dim3 grid((unsigned)((L.lines + (1 << l) - 1) >> l), L.planes, fields);
    line3<MODE><<<grid, line_threads(L.n, L.plan.r(0), l), sm, s>>>(L, op, a, l);
    return cudaGetLastError();
}

} // namespace

cudaError_t launch_step3d(const Step3 &T, double *omega, double *pop, double *vel, double *phi, double *q, double *force,
                          cudaStream_t s)
{
    const GroupGeom &g = T.S.vx;
    const int nx = T.nx, ny = T.ny, nz = T.nz;
    const long long n = g.n, nxy = (long long)nx * ny;
    const double pi = 3.14159265358979323846;
    auto unit = [&](int m) { return 2.0 * pi / ((double)m * g.dx); };
    const Lines L[3] = {
        {nx, 1, 1, nx, 0, (long long)ny * nz, 1, T.S.vx.px, T.twx, unit(nx)},
        {ny, 0, nx, 1, nxy, nx, nz, T.S.vy.py, T.twy, unit(ny)},
        {nz, 0, nxy, 1, 0, nxy, 1, T.S.vz.py, T.twz, unit(nz)},
    };
    auto op_of = [&](int axis, int mode) {
        Op3D o = {};
        o.mode = mode;
        o.n = L[axis].n;
        o.unit = L[axis].unit;
        o.inv_n = 1.0 / (double)L[axis].n;
        o.nx = nx;
        o.ny = ny;
        o.px = L[0].plan;
        o.py = L[1].plan;
        o.ux = L[0].unit;
        o.uy = L[1].unit;
        o.c = g.inv_beta_v / (g.dt * (double)n);
        return o;
    };
    Args3 a = {};
    a.n = n;
    a.nx = nx;
    a.ny = ny;
    cudaError_t e;
    // (1) omega~ = omega - dt v . grad omega, v = u_lat dx/dt
    a.omega = omega;
    a.dst = T.wt;
    a.ca = g.dt * g.vscale;
    for (int ax = 0; ax < 3; ++ax) {
        a.first = ax == 0;
        a.vel = vel + (size_t)ax * n;
        if ((e = run3<P3_CONVECT>(L[ax], op_of(ax, D3_GRAD), a, s))) return e;
    }
    // (2) Phi~
    if ((e = launch_solve3d(T.S, T.wt, T.pt, T.qt, s))) return e;
    // (3) mu and the diffusion step
    const double chi[3][3] = {{0.0, g.chi_ab, g.chi_as}, {g.chi_ab, 0.0, g.chi_bs}, {g.chi_as, g.chi_bs, 0.0}};
    for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j) a.mu_c[i][j] = chi[i][j] + g.kappa_h;
        a.mu_0[i] = g.kappa_h;
    }
    a.phi = T.pt;
    a.wt_c = T.wt;
    a.mu = T.mu;
    a.dst = omega;
    a.ca = g.dt * g.d_p;
    a.cb = g.dt * g.d_s;
    for (int ax = 0; ax < 3; ++ax) {
        a.first = ax == 0;
        if ((e = run3<P3_DIFFUSE>(L[ax], op_of(ax, D3_LAP), a, s))) return e;
    }
    // (4) Phi(t + dt)
    if ((e = launch_solve3d(T.S, omega, phi, q, s))) return e;
    // (5) the force from S = sum_I dPhi_I / D_I: x and y forward, z with the
    // factor of (f_x, f_y) into b1 and of f_z in place, y and x back
    a.phi = phi;
    a.phi0 = T.pt;
    a.ca = 1.0 / g.d_p;
    a.cb = 1.0 / g.d_s;
    a.out = T.b0;
    if ((e = run3<P3_FWD>(L[0], op_of(0, D3_ONE), a, s))) return e;
    a.phi = nullptr;
    a.in = T.b0;
    if ((e = run3<P3_FWD>(L[1], op_of(1, D3_ONE), a, s))) return e;
    a.out = T.b1;
    if ((e = run3<P3_BOTH>(L[2], op_of(2, D3_FORCE_XY), a, s))) return e;
    a.out = T.b0;
    if ((e = run3<P3_BOTH>(L[2], op_of(2, D3_FORCE_Z), a, s))) return e;
    a.force = force;
    a.ftot = T.ftot;
    a.f0 = T.f0_lat;
    a.scale = g.fstar;
    for (int c = 0; c < 2; ++c) {
        a.in = a.out = c == 0 ? T.b1 : T.b0;
        a.comp = c == 0 ? 0 : 2;
        if ((e = run3<P3_INV>(L[1], op_of(1, D3_ONE), a, s))) return e;
        if ((e = run3<P3_INV_OUT>(L[0], op_of(0, D3_ONE), a, s))) return e;
    }
    // (6) D3Q19 with the total force
    if ((e = launch_lb3d_step(nx, ny, nz, g.gamma_s, g.gamma_b, g.gamma_g, pop, T.ftot, T.pop2, vel, s))) return e;
    return cudaMemcpyAsync(pop, T.pop2, 19 * n * sizeof(double), cudaMemcpyDeviceToDevice, s);
}

} // namespace epdlb
