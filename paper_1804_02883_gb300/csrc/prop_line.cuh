// prop_line.cuh -- the streaming propagator passes that run on every grid
// (Sec. 2, Eqs. (6)-(10) of arXiv:1804.02883): one contour step is a column
// pass and a row pass over the packed chain z = g + i g', each a forward
// transform, the axis' Fourier factor and an inverse transform of every line
// (fftg.cuh).  Included by one translation unit per precision.
//
// What bounds them.  FP32: L2 traffic and, on small grids, the latency of a
// pass; FP64: the FP64 unit (2 lanes per SM and cycle), so what counts there
// is FP64 instructions per point and an even load of the SMs.  A CTA holds few
// lines (line_logb) so that every grid gives each SM several tiles.
// Per launch (cold, serialised), 64 x 150 x 150 in FP32, 32 runs as Stockham
// passes -> 64 runs now: column 24.3 -> 14.6 us, row 37.7 -> 24.4 us (1.9 TB/s
// of the chain, factors and history; no instruction to issue for a third of the
// stalls).  FP64, 4 x 256 x 512, N_s = 64: 53 and 73 us, a step 20.4 -> 15.0 ms.
#pragma once

#include "common.cuh"
#include "engine.h"
#include "fftg.cuh"

namespace epdlb {

template <typename T> struct PropK {
    GroupGeom g;
    V2<T> *chain;
    V2<T> *hist;          // [run][hnodes][n]: nodes 0..half_lo, or all N_s + 1 (reference of a differential solve)
    V2<T> *hd;            // differential solve: (dg, dg') at every node, [run][N_s + 1][n]
    const float2 *rho;    // differential solve: (rho_A, rho_B), [run][n]
    int hnodes;
    const V2<T> *efac;
    double *ia, *ib, *part;
    const V2<T> *twx, *twy;
    const T *kx, *ky;
    bool stateless;  // launches as programmatic dependents (see line_dependents), every twiddle read
};

// Boltzmann factor (E_A, E_B) of the half-step at node j of chain g (fac_g)
// or g' (fac_gp), arriving or departing (half_step_block)
template <typename T> __device__ __forceinline__ T fac_g(V2<T> e, const GroupGeom &g, int j, bool arriving)
{
    return half_step_block(g.jr, 0, j, g.ns, g.na, arriving) ? e.y : e.x;
}
template <typename T> __device__ __forceinline__ T fac_gp(V2<T> e, const GroupGeom &g, int j, bool arriving)
{
    return half_step_block(g.jr, 1, j, g.ns, g.na, arriving) ? e.y : e.x;
}

// Trapezoid weights on [0, s_{N_A}] (block A) and [s_{N_A}, 1] (block B).
__host__ __device__ inline double weight_a(int j, int na, double ds)
{
    if (na == 0 || j > na) return 0.0;
    return (j == 0 || j == na) ? 0.5 * ds : ds;
}
__host__ __device__ inline double weight_b(int j, int na, int ns, double ds)
{
    if (na == ns || j < na) return 0.0;
    return (j == na || j == ns) ? 0.5 * ds : ds;
}

// The launches of a stateless solve are programmatic dependents of the one
// before: the next one's CTAs are placed while its last CTAs finish (128 x 128,
// N_s = 64: 1.03 -> 0.75 ms; 48 x 90 x 96 box 0.95 -> 0.80 ms).  Inside a
// handle's captured step they are not: there the graph already launches
// back to back (alone 14.4 against 14.1 ms on 64 x 150 x 150, 17.0 against 17.7
// in FP64 on 4 x 256 x 512), and with several handles on one GPU the waiting
// CTAs hold the other graphs' launches up (three 64 x 64 FP64 handles: 5.2 ms
// a pass without, 8.4 with).
__device__ __forceinline__ void line_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename T> struct LineScale {  // the Fourier factor of Eq. (8)
    const T *__restrict__ kf;
    using Pre = T;
    __device__ __forceinline__ T pre(int, int bin) const { return __ldg(&kf[bin]); }
    __device__ __forceinline__ V2<T> operator()(T f, V2<T> v) const { return cscale(v, f); }
};

// Column pass: Ty = IFFT_y Ky FFT_y on the tile's adjacent columns.
template <typename T, int R0, class Tile, class Plan>
__device__ __forceinline__ void col_tile(const PropK<T> &k, const Tile &tl, const Plan &pl)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V2<T> *buf = reinterpret_cast<V2<T> *>(smem_raw);
    const int nx = k.g.nx, x0 = blockIdx.x << tl.logb;
    V2<T> *data = k.chain + (size_t)blockIdx.y * k.g.n + x0;
    line_dependents();
    line_pair<T, R0>(
        buf, tl, pl, k.twy,
        [&](int b, int t, int q, V2<T>(&x)[R0]) {
            const bool in = Tile::fixed || x0 + b < nx;  // whole tiles on power-of-two grids
            const int i0 = t * nx + b, di = q * nx;
#pragma unroll
            for (int u = 0; u < R0; ++u) x[u] = in ? data[i0 + u * di] : mk<T>((T)0, (T)0);
        },
        LineScale<T>{k.ky},
        [&](int b, int t, int q, V2<T>(&x)[R0]) {
            if (!Tile::fixed && x0 + b >= nx) return;
            const int i0 = t * nx + b, di = q * nx;
#pragma unroll
            for (int u = 0; u < R0; ++u) data[i0 + u * di] = x[u];
        });
}

// What a row pass adds to the contour sums: the trapezoid weights of node m
// (block A, B) and of its mirror N_s - m.
struct RowWeights {
    double a1, b1, a2, b2;
    bool a, b;  // whether a block has a weight there at all (compared on the host: FP64 comparisons were 9% of an FP32 row pass)
};
inline RowWeights row_weights(const GroupGeom &g, int m)
{
    const int ns = g.ns, na = g.na, s2 = ns - m;
    RowWeights w = {weight_a(m, na, g.ds), weight_b(m, na, ns, g.ds), s2 == m ? 0.0 : weight_a(s2, na, g.ds),
                    s2 == m ? 0.0 : weight_b(s2, na, ns, g.ds), false, false};
    w.a = w.a1 != 0.0 || w.a2 != 0.0;
    w.b = w.b1 != 0.0 || w.b2 != 0.0;
    return w;
}

// Row pass producing contour node m (1 <= m <= ns): Tx, node factors, history
// store / contour accumulation, Q_P partial sums at m = ns, next half step.
// Differential solve (DIFF): the chain carries the change d a of the state
// E_d g; with U = T(d a_{m-1}) and the reference node g~_m from the history,
//   dg_m = E'_a U + rho_a g~_m,   d a_m = E'_d dg_m + E_d rho_d g~_m
// (E' = E (1 + rho)), the exact differences of g_m = E'_a T(a_{m-1}) and
// a_m = E'_d g_m from the reference solve's g~_m = E_a T(a~_{m-1}) and
// a~_m = E_d g~_m; dg_m is stored at every node, dQ_P partials at m = ns.
// With the full history (hnodes = N_s + 1) the contour sums are a pass of
// their own (prop_contour_stream); otherwise node m >= N_s / 2 meets its
// mirror from the half history here.
template <typename T, int R0, bool DIFF, class Tile, class Plan>
__device__ __forceinline__ void row_tile(const PropK<T> &k, const Tile &tl, const Plan &pl, int m, const RowWeights &w)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[32];
    V2<T> *buf = reinterpret_cast<V2<T> *>(smem_raw);
    const int nx = Tile::fixed ? tl.n : k.g.nx, ny = k.g.ny, run = blockIdx.y, y0 = blockIdx.x << tl.logb;
    const int ns = k.g.ns, na = k.g.na, jr = k.g.jr, hlo = k.g.half_lo, hhi = k.g.half_hi, s2 = ns - m;
    const long long n = k.g.n, base = (long long)y0 * nx;
    V2<T> *data = k.chain + (size_t)run * n + base;
    const V2<T> *efac = k.efac + (size_t)run * n + base;
    V2<T> *hist = k.hist + (size_t)run * k.hnodes * n + base;
    // blocks of the arriving and departing half-steps of both chains
    const bool bag = half_step_block(jr, 0, m, ns, na, true), bap = half_step_block(jr, 1, m, ns, na, true);
    const bool bdg = half_step_block(jr, 0, m, ns, na, false), bdp = half_step_block(jr, 1, m, ns, na, false);
    double qsum = 0.0;
    // points whose loads are issued together, ahead of the stores
    constexpr int CH = R0 % 4 == 0 ? 4 : (R0 % 5 == 0 ? 5 : (R0 % 3 == 0 ? 3 : 2));
    line_dependents();
    line_pair<T, R0>(
        buf, tl, pl, k.twx,
        [&](int b, int t, int q, V2<T>(&x)[R0]) {
            const bool in = Tile::fixed || y0 + b < ny;
            const int i0 = b * nx + t;
#pragma unroll
            for (int u = 0; u < R0; ++u) x[u] = in ? data[i0 + u * q] : mk<T>((T)0, (T)0);
        },
        LineScale<T>{k.kx},
        [&](int b, int t, int q, V2<T>(&x)[R0]) {
            if (!Tile::fixed && y0 + b >= ny) return;
            const int i0 = b * nx + t;
            if constexpr (DIFF) {
                const float2 *rho = k.rho + (size_t)run * n + base;
                V2<T> *hd = k.hd + ((size_t)run * (ns + 1) + m) * n + base;
                const V2<T> *gref = hist + (size_t)m * n;
                // eight points' operands in flight where the tile is known at compile time
                // (1024 x 2048: 21.4 -> 19.3 us a launch)
                constexpr int CD = Tile::fixed && R0 % 8 == 0 ? 8 : CH;
#pragma unroll
                for (int u0 = 0; u0 < R0; u0 += CD) {
                    V2<T> eb[CD], grb[CD];
                    float2 qb[CD];
#pragma unroll
                    for (int c = 0; c < CD; ++c) {
                        const int i = i0 + (u0 + c) * q;
                        eb[c] = efac[i];
                        grb[c] = gref[i];
                        qb[c] = rho[i];
                    }
#pragma unroll
                    for (int c = 0; c < CD; ++c) {
                        const int i = i0 + (u0 + c) * q;
                        const V2<T> e = eb[c], gr = grb[c], h = x[u0 + c];
                        const float2 r = qb[c];
                        const T ea = bag ? e.y : e.x, eap = bap ? e.y : e.x, qa = bag ? r.y : r.x, qap = bap ? r.y : r.x;
                        const V2<T> dg = mk<T>(ea * ((T)1 + qa) * h.x + qa * gr.x, eap * ((T)1 + qap) * h.y + qap * gr.y);
                        hd[i] = dg;
                        if (m == ns) {
                            qsum += (double)dg.x;
                        } else {
                            const T ed = bdg ? e.y : e.x, edp = bdp ? e.y : e.x, qd = bdg ? r.y : r.x, qdp = bdp ? r.y : r.x;
                            data[i] = mk<T>(ed * ((T)1 + qd) * dg.x + ed * qd * gr.x,
                                            edp * ((T)1 + qdp) * dg.y + edp * qdp * gr.y);
                        }
                    }
                }
            } else {
                const bool store_all = k.hnodes == ns + 1, acc = !store_all && m >= hhi;
                // only the block(s) with a weight at this node or its mirror
                const bool use_a = acc && (m == hhi || w.a);
                const bool use_b = acc && (m == hhi || w.b);
                double *ia = k.ia + (size_t)run * n + base, *ib = k.ib + (size_t)run * n + base;
                if constexpr (Tile::fixed) {
                    if (store_all) {  // no sums: the factors of all the thread's points at once (1024 x 2048, 2 steps: 16.1 -> 15.3 ms)
                        V2<T> eb[R0];
#pragma unroll
                        for (int u = 0; u < R0; ++u) eb[u] = efac[i0 + u * q];
#pragma unroll
                        for (int u = 0; u < R0; ++u) {
                            const int i = i0 + u * q;
                            const V2<T> e = eb[u], h = x[u];
                            const V2<T> z = mk<T>((bag ? e.y : e.x) * h.x, (bap ? e.y : e.x) * h.y);
                            hist[(size_t)m * n + i] = z;
                            if (m == ns) qsum += (double)z.x;
                            else data[i] = mk<T>((bdg ? e.y : e.x) * z.x, (bdp ? e.y : e.x) * z.y);
                        }
                        return;
                    }
                }
#pragma unroll
                for (int u0 = 0; u0 < R0; u0 += CH) {
                    V2<T> eb[CH], hvb[CH];
                    double iab[CH], ibb[CH];
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const int i = i0 + (u0 + c) * q;
                        eb[c] = efac[i];
                        iab[c] = ibb[c] = 0.0;
                        if (acc && s2 != m) hvb[c] = hist[(size_t)s2 * n + i];
                        if (use_a && m > hhi) iab[c] = ia[i];
                        if (use_b && m > hhi) ibb[c] = ib[i];
                    }
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const int i = i0 + (u0 + c) * q;
                        const V2<T> e = eb[c], h = x[u0 + c];
                        // z = (g_m, g'_m): the arriving half-step's factor; the
                        // chain goes on with the departing one
                        const V2<T> z = mk<T>((bag ? e.y : e.x) * h.x, (bap ? e.y : e.x) * h.y);
                        if (m <= hlo || store_all) hist[(size_t)m * n + i] = z;
                        if (acc) {
                            const V2<T> hv = (s2 == m) ? z : hvb[c];
                            const double t1 = (double)z.x * (double)hv.y;                  // g(s_m) g'(1 - s_m)
                            const double t2 = s2 == m ? 0.0 : (double)hv.x * (double)z.y;  // g(s_{ns-m}) g'(s_m)
                            if (use_a) ia[i] = iab[c] + (w.a1 * t1 + w.a2 * t2);
                            if (use_b) ib[i] = ibb[c] + (w.b1 * t1 + w.b2 * t2);
                        }
                        if (m == ns) qsum += (double)z.x;
                        else data[i] = mk<T>((bdg ? e.y : e.x) * z.x, (bdp ? e.y : e.x) * z.y);
                    }
                }
            }
        });
    if (m == ns) {
        const double s = block_sum(qsum, red);
        if (threadIdx.x == 0) k.part[(size_t)run * kMaxPart + blockIdx.x] = s;
    }
}

template <typename T, int R0>
__global__ void __launch_bounds__(256) prop_col(PropK<T> k, int logb)
{
    col_tile<T, R0>(k, LineTile(false, k.g.ny, logb, k.g.py), k.g.py);
}
template <typename T, int R0, bool DIFF>
__global__ void __launch_bounds__(256, 2) prop_row(PropK<T> k, int m, int logb, RowWeights w)
{
    row_tile<T, R0, DIFF>(k, LineTile(true, k.g.nx, logb, k.g.px), k.g.px, m, w);
}

constexpr size_t kMaxTile = 200 * 1024;  // shared memory of a tile at most

template <typename K, typename... A>
cudaError_t launch_line(bool dependent, K kernel, dim3 grid, int threads, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = dependent ? 1 : 0;
    // Tiles past the default limit: wide column tiles on long axes, and the
    // row tiles of 3D boxes that fill the Q partials.  The limit belongs to the
    // function on the current device and every host thread sees it, so each
    // such launch sets the same value, on whichever device is current.
    if (smem > kMaxTile) return cudaErrorInvalidConfiguration;
    if (smem > 48 * 1024)
        if (cudaError_t e = cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxTile)) return e;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename T> cudaError_t line_col_t(const PropK<T> &k, cudaStream_t s)
{
    const int n = k.g.ny, nx = k.g.nx, r0 = k.g.py.r(0);
    const int maxlog = sizeof(T) == 4 ? 3 : 2;  // 64-byte row segments
    const int l = line_logb(false, n, k.g.py, nx, k.g.nruns, sizeof(V2<T>), maxlog, sizeof(T) == 4 ? 1 : 0, 1LL << 30);
    const dim3 grid((nx + (1 << l) - 1) >> l, k.g.nruns);
    const size_t sm = LineTile(false, n, l, k.g.py).points() * sizeof(V2<T>);
    const int th = line_threads(n, r0, l);
    switch (r0) {
    case 2: return launch_line(k.stateless, prop_col<T, 2>, grid, th, sm, s, k, l);
    case 4: return launch_line(k.stateless, prop_col<T, 4>, grid, th, sm, s, k, l);
    case 6: return launch_line(k.stateless, prop_col<T, 6>, grid, th, sm, s, k, l);
    case 8: return launch_line(k.stateless, prop_col<T, 8>, grid, th, sm, s, k, l);
    case 10: return launch_line(k.stateless, prop_col<T, 10>, grid, th, sm, s, k, l);
    default: return launch_line(k.stateless, prop_col<T, 12>, grid, th, sm, s, k, l);
    }
}

template <typename T, bool DIFF> cudaError_t line_row_t(const PropK<T> &k, int m, int *blocks, cudaStream_t s)
{
    const int n = k.g.nx, ny = k.g.ny, r0 = k.g.px.r(0);
    // The tiles of the last pass set the order of the Q_P sum, so they follow the
    // grid alone and a run's results do not depend on the batch it is in: four
    // rows, near enough to both ends of the rule (64 x 150 x 150 a step: 1.60 ms
    // with the tile of one run in its last passes, 1.56 with four rows).
    const bool last = m == k.g.ns;
    const int l = line_logb(true, n, k.g.px, ny, last ? 1 << 20 : k.g.nruns, sizeof(V2<T>), last ? 2 : 3, 0, kMaxPart / 2);
    const dim3 grid((ny + (1 << l) - 1) >> l, k.g.nruns);
    *blocks = (int)grid.x;
    const size_t sm = LineTile(true, n, l, k.g.px).points() * sizeof(V2<T>);
    const int th = line_threads(n, r0, l);
    const RowWeights w = row_weights(k.g, m);
    switch (r0) {
    case 2: return launch_line(k.stateless, prop_row<T, 2, DIFF>, grid, th, sm, s, k, m, l, w);
    case 4: return launch_line(k.stateless, prop_row<T, 4, DIFF>, grid, th, sm, s, k, m, l, w);
    case 6: return launch_line(k.stateless, prop_row<T, 6, DIFF>, grid, th, sm, s, k, m, l, w);
    case 8: return launch_line(k.stateless, prop_row<T, 8, DIFF>, grid, th, sm, s, k, m, l, w);
    case 10: return launch_line(k.stateless, prop_row<T, 10, DIFF>, grid, th, sm, s, k, m, l, w);
    default: return launch_line(k.stateless, prop_row<T, 12, DIFF>, grid, th, sm, s, k, m, l, w);
    }
}

// One column pass; one row pass producing node m (blocks: its Q partials per
// run); instantiated in prop_line_f32.cu and prop_line_f64.cu.
cudaError_t line_col(const PropK<float> &k, cudaStream_t s);
cudaError_t line_col(const PropK<double> &k, cudaStream_t s);
cudaError_t line_row(const PropK<float> &k, int m, bool diff, int *blocks, cudaStream_t s);
cudaError_t line_row(const PropK<double> &k, int m, bool diff, int *blocks, cudaStream_t s);
// The same on power-of-two grids of 64..2048 points per axis in FP32, on
// compile-time tiles (prop_stream.cu); colw: columns per tile (4, 8, 16; 0: by
// the rule of line_logb).
cudaError_t stream_col(const PropK<float> &k, int colw, cudaStream_t s);
cudaError_t stream_row(const PropK<float> &k, int m, bool diff, int *blocks, cudaStream_t s);
bool stream_col_fits(int ny, int colw);  // whether a tile of colw columns fits an SM

} // namespace epdlb
