// prop.cu -- single-chain solve of the hybrid LB/EPD step (Sec. 2, Eqs. (6)-(11)
// of arXiv:1804.02883) on sm_103a.
//
// Both propagators advance together: the forward propagator g (from the A end,
// Eq. (6)) and the backward propagator g' (from the B end, Eq. (7)) are real, so
// they travel as the real and imaginary parts of one complex field z = g + i g'.
// The Fourier factor exp(-R_G^2 |k|^2 ds) of the split step, Eq. (8), is
// separable, exp(-R_G^2 kx^2 ds) exp(-R_G^2 ky^2 ds), and maps real fields to
// real fields, so one contour step is
//   column pass : z <- IFFT_y[ Ky * FFT_y[ z ] ]              (all columns)
//   row pass    : h <- IFFT_x[ Kx * FFT_x[ z ] ]              (all rows)
//                 z_{j+1} = E(s_{j+1}) h  (g and g' each with its own node field),
//                 store or consume the contour history,
//                 z <- E(s_{j+1}) z_{j+1} (first half of the next step)
// with E = exp(-N w ds / 2).  The history holds nodes 0..floor(N_s/2): while
// the chains run through the second half, node m of g meets node N_s - m of g'
// from the history (and vice versa), and the trapezoid sums of Eqs. (9)-(10)
// are accumulated in FP64 on the fly.  A MIXED_FP32 handle stores every node:
// the full history is the reference of the differential second solve, and the
// contour sums are a separate pass over the stored nodes (prop_contour_stream).
// The column and row passes are in prop_line.cuh (every grid, both precisions)
// and prop_stream.cu (FP32 on power-of-two grids); this file holds the pointwise
// and contour passes and the solves' host side.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "common.cuh"
#include "engine.h"
#include "fft8.cuh"
#include "prop_line.cuh"

namespace epdlb {

template <typename T> __device__ __forceinline__ T exp_t(T v);
template <> __device__ __forceinline__ float exp_t<float>(float v) { return expf(v); }
template <> __device__ __forceinline__ double exp_t<double>(double v) { return exp(v); }

// Place of site i in the packed-row layout of the cluster solve, in floats
// (site (y, x) -> packed row y / 2, component y & 1; power-of-two grids).
__device__ __forceinline__ size_t packed_site(const GroupGeom &g, long long i)
{
    const long long y = i >> g.logx, x = i & (g.nx - 1);
    return (size_t)((y >> 1) * g.nx + x) * 2 + (y & 1);
}

// Boltzmann factors E_{A,B} = exp(-N w_{A,B} ds / 2) and exp(-w_S) in the bulk
// precision; exp(-w_S) into the S slot of phi_out and its block sums for Q_S
// in FP64.
template <typename T>
__global__ void __launch_bounds__(kThreads) prop_prep(GroupGeom g, const double *omega, V2<T> *efac, T *fac, double *phi_out, double *part)
{
    __shared__ double red[32];
    const int run = blockIdx.y;
    const long long n = g.n;
    const double *wa = omega + (size_t)run * 3 * n, *wb = wa + n, *ws = wb + n;
    double *es = phi_out + (size_t)run * 3 * n + 2 * n;
    const T c = (T)(-0.5 * g.nseg * g.ds);
    double acc = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const T ea = exp_t<T>(c * (T)wa[i]), eb = exp_t<T>(c * (T)wb[i]);
        efac[(size_t)run * n + i] = mk<T>(ea, eb);
        if (fac) {  // node factors of the cluster solve
            const size_t o = packed_site(g, i), hn = (size_t)n;
            T *f = fac + (size_t)run * 3 * hn;
            f[o] = ea * ea;
            f[hn + o] = eb * eb;
            f[2 * hn + o] = ea * eb;
        }
        // exp(-w_S) in the bulk precision (FP32 in MIXED_FP32), kept in FP64
        const double e = (double)exp_t<T>(-(T)ws[i]);
        es[i] = e;
        acc += e;
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) part[(size_t)run * kMaxPart + kMaxPart / 2 + blockIdx.x] = s;
}

// Node 0: g = g' = 1 stored; chain <- E(s_0) z_0.  Differential solve: the
// change of node 0 is 0, the chain starts from d a_0 = E' - E = E rho of the
// departing half-step.
template <typename T, bool DIFF>
__global__ void __launch_bounds__(kThreads) prop_start(PropK<T> k)
{
    const int run = blockIdx.y;
    const long long n = k.g.n;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const V2<T> e = k.efac[(size_t)run * n + i];
        if constexpr (!DIFF) {
            k.hist[(size_t)run * k.hnodes * n + i] = mk<T>((T)1, (T)1);
            k.chain[(size_t)run * n + i] = mk<T>(fac_g<T>(e, k.g, 0, false), fac_gp<T>(e, k.g, 0, false));
        } else {
            const float2 q = k.rho[(size_t)run * n + i];
            k.hd[(size_t)run * (k.g.ns + 1) * n + i] = mk<T>((T)0, (T)0);
            k.chain[(size_t)run * n + i] = mk<T>(fac_g<T>(e, k.g, 0, false) * fac_g<float>(q, k.g, 0, false),
                                                 fac_gp<T>(e, k.g, 0, false) * fac_gp<float>(q, k.g, 0, false));
        }
    }
}

// Normalisation, Eqs. (9)-(11) with Q as spatial means.
__global__ void __launch_bounds__(kThreads) prop_finalize(GroupGeom g, int nrow_blocks, int nprep_blocks, const double *ia,
                                                      const double *ib, const double *part, double *phi, double *q,
                                                      int *err)
{
    __shared__ double bc, fac[2];
    const int run = blockIdx.y;
    const long long n = g.n;
    const double *pr = part + (size_t)run * kMaxPart;
    const double sp = sum_partials(pr, nrow_blocks, 1, &bc), ss = sum_partials(pr + kMaxPart / 2, nprep_blocks, 1, &bc);
    // the FP64 divisions once per block: a division is tens of FP64
    // instructions, at 2 lanes per SM and cycle
    if (threadIdx.x == 0) {
        const double qp = sp / (double)n, qs = ss / (double)n;
        fac[0] = g.phi_p / qp;
        fac[1] = (1.0 - g.phi_p) / qs;
        if (blockIdx.x == 0) {
            q[2 * run] = qp;
            q[2 * run + 1] = qs;
            if (!(qp > 0.0) || !(qs > 0.0) || !isfinite(qp) || !isfinite(qs)) atomicOr(err, 1);
        }
    }
    __syncthreads();
    const double cp = fac[0], cs = fac[1];
    double *pa = phi + (size_t)run * 3 * n, *pb = pa + n, *ps = pb + n;
    const double *ja = ia + (size_t)run * n, *jb = ib + (size_t)run * n;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        pa[i] = cp * ja[i];
        pb[i] = cp * jb[i];
        ps[i] = cs * ps[i];
    }
}

// Differential second solve (MIXED_FP32, cluster solve).  The step's second
// solve differs from its first only by the diffusion update d omega = omega -
// omega~ (Eq. (5)), small next to omega.  Its node factors are E~ (1 + rho),
// rho = expm1(-N d omega ds / 2), and its solvent factor e~ (1 + expm1(
// -d omega_S)), so the changes follow from the FP64 difference with the
// rounding of FP32 relative to the change itself.  The solvent change de goes
// to the S slot of phi, its block sums to the S partials.
__global__ void __launch_bounds__(kThreads) prop_prep_delta(GroupGeom g, const double *omega, const double *omega_t,
                                                            float2 *rho, float *cdiff, const float2 *efac, float *fac,
                                                            double *phi_out, double *part)
{
    __shared__ double red[32];
    const int run = blockIdx.y;
    const long long n = g.n;
    const double *wa = omega + (size_t)run * 3 * n, *wb = wa + n, *ws = wb + n;
    const double *ta = omega_t + (size_t)run * 3 * n, *tb = ta + n, *ts = tb + n;
    double *ds_out = phi_out + (size_t)run * 3 * n + 2 * n;
    const float c = (float)(-0.5 * g.nseg * g.ds);
    double acc = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float da = (float)(wa[i] - ta[i]), db = (float)(wb[i] - tb[i]);
        const float qa = expm1f(c * da), qb = expm1f(c * db);
        rho[(size_t)run * n + i] = make_float2(qa, qb);
        if (cdiff) {
            // (1 + rho_d)(1 + rho_a) - 1 and the node factors E'_d E'_a for the
            // block pairs (A, A), (B, B), (A, B) of a node's departing and
            // arriving half-steps, in the packed-row layout
            const size_t o = packed_site(g, i), hn = (size_t)n;
            float *cd = cdiff + (size_t)run * 3 * hn, *f = fac + (size_t)run * 3 * hn;
            cd[o] = qa * (2.f + qa);
            cd[hn + o] = qb * (2.f + qb);
            cd[2 * hn + o] = qa + qb + qa * qb;
            const float2 e = efac[(size_t)run * n + i];
            const float pa = 1.f + qa, pb = 1.f + qb;
            f[o] = e.x * e.x * (pa * pa);
            f[hn + o] = e.y * e.y * (pb * pb);
            f[2 * hn + o] = e.x * e.y * (pa * pb);
        }
        // e~_S exactly as the first solve formed it
        const float es = expf(-(float)ts[i]);
        const double de = (double)(es * expm1f(-(float)(ws[i] - ts[i])));
        ds_out[i] = de;
        acc += de;
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) part[(size_t)run * kMaxPart + kMaxPart / 2 + blockIdx.x] = s;
}

// Contour sums and normalisation over the full history (Eqs. (9)-(11)).  Plain
// solve: exact products and exact additions in pairs of FP32 values, so that a
// sum is good to ~2^-44 (N_s terms of 2^-47) and the densities of every grid
// have the error of FP64 sums to four digits against a 64-bit solve, at a
// fraction of the FP64 unit's time (64 x 150 x 150, N_s = 17, a step: 1.60 ms,
// 1.78 with FP64 sums; 1024 x 2048, N_s = 128: 8.5 and 10.6; plain compensated
// sums, which keep ~2^-24 of each term, 1.62 and 8.6).  The solvent slot of phi
// holds exp(-omega_S) from prop_prep.
// Differential solve (DIFF): the sums of the product's change
// g~ dg' + dg g~' + dg dg' (reference history hist, changes hd), the
// partials hold dQ_P and the solvent factor's change, and
// Phi = Phi~ + (phi_p ds dI - Phi~ dQ) / (Q~ + dQ) per species.
template <bool DIFF>
__global__ void __launch_bounds__(kThreads) prop_contour_stream(GroupGeom g, const float2 *hist, const float2 *hd,
                                                                int nrow_blocks, int nprep_blocks, const double *part,
                                                                double *phi, double *q, const double *phi_ref,
                                                                const double *q_ref, int *err)
{
    __shared__ double bc, fac[4];
    const int run = blockIdx.y, ns = g.ns, na = g.na;
    const long long n = g.n;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < n;
    const float2 *hz = hist + (size_t)run * (ns + 1) * n + i;
    const float2 *dz = DIFF ? hd + (size_t)run * (ns + 1) * n + i : nullptr;
    // Nodes m and N_s - m are read together: z_m = (g_m, g'_m) and z_{N_s-m}
    // give the terms g_m g'_{N_s-m} (node m) and g_{N_s-m} g'_m (node N_s - m).
    // Sums s + c per block; the trapezoid weights 1 and 1/2 scale terms exactly.
    // Changes (DIFF): compensated (Kahan).  Plain: two-sum (Knuth), the exact
    // rounding error of each addition and product into c.
    float sa = 0.f, ca = 0.f, sb = 0.f, cb = 0.f;
    auto kadd = [](float &s_, float &c_, float t) {
        const float y = t + c_, u = s_ + y;
        c_ = y - (u - s_);
        s_ = u;
    };
    auto two_add = [](float &s_, float &c_, float t, float e) {
        const float u = s_ + t, v = u - s_;
        c_ += ((s_ - (u - v)) + (t - v)) + e;
        s_ = u;
    };
    auto add = [&](int j, float t) {
        const float wa = (na == 0 || j > na) ? 0.f : ((j == 0 || j == na) ? 0.5f : 1.f);
        const float wb = (na == ns || j < na) ? 0.f : ((j == na || j == ns) ? 0.5f : 1.f);
        if (wa != 0.f) kadd(sa, ca, wa * t);
        if (wb != 0.f) kadd(sb, cb, wb * t);
    };
    auto add_exact = [&](int j, float x, float y) {
        const float wa = (na == 0 || j > na) ? 0.f : ((j == 0 || j == na) ? 0.5f : 1.f);
        const float wb = (na == ns || j < na) ? 0.f : ((j == na || j == ns) ? 0.5f : 1.f);
        const float t = x * y, e = fmaf(x, y, -t);
        if (wa != 0.f) two_add(sa, ca, wa * t, wa * e);
        if (wb != 0.f) two_add(sb, cb, wb * t, wb * e);
    };
    const int half = ns / 2;
    constexpr int U = DIFF ? 4 : 8;
    for (int m0 = 0; m0 <= (valid ? half : -1); m0 += U) {
        float2 zl[U], zr[U], dl[U], dr[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int m = m0 + u;
            if (m <= half) {
                zl[u] = hz[(size_t)m * n];
                zr[u] = hz[(size_t)(ns - m) * n];
                if (DIFF) {
                    dl[u] = dz[(size_t)m * n];
                    dr[u] = dz[(size_t)(ns - m) * n];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int m = m0 + u;
            if (m > half) break;
            if (!DIFF) {
                add_exact(m, zl[u].x, zr[u].y);
                if (ns - m != m) add_exact(ns - m, zr[u].x, zl[u].y);
            } else {
                // node m: g_m g'_{ns-m}; node ns - m: g_{ns-m} g'_m
                add(m, zl[u].x * dr[u].y + dl[u].x * zr[u].y + dl[u].x * dr[u].y);
                if (ns - m != m) add(ns - m, zr[u].x * dl[u].y + dr[u].x * zl[u].y + dr[u].x * dl[u].y);
            }
        }
    }
    // Q from the partials (after the streaming loop, so that its latency
    // overlaps other blocks' loads; every thread of the block takes part).
    // The FP64 divisions once per block, by one thread.
    const double *pr = part + (size_t)run * kMaxPart;
    const double tp = sum_partials(pr, nrow_blocks, 1, &bc), ts = sum_partials(pr + kMaxPart / 2, nprep_blocks, 1, &bc);
    if (threadIdx.x == 0) {
        const double sq = tp / (double)n, ss = ts / (double)n;
        const double qp = DIFF ? q_ref[2 * run] + sq : sq, qs = DIFF ? q_ref[2 * run + 1] + ss : ss;
        fac[0] = g.phi_p * g.ds / qp;
        fac[1] = (1.0 - g.phi_p) / qs;
        fac[2] = sq / qp;
        fac[3] = ss / qs;
        if (blockIdx.x == 0) {
            q[2 * run] = qp;
            q[2 * run + 1] = qs;
            if (!(qp > 0.0) || !(qs > 0.0) || !isfinite(qp) || !isfinite(qs)) atomicOr(err, 1);
        }
    }
    __syncthreads();
    if (!valid) return;
    const double ia = (double)sa + (double)ca, ib = (double)sb + (double)cb;
    const double cp = fac[0], cs = fac[1];
    double *ph = phi + (size_t)run * 3 * n;
    if (!DIFF) {
        ph[i] = cp * ia;
        ph[n + i] = cp * ib;
        ph[2 * n + i] *= cs;
    } else {
        const double *pt = phi_ref + (size_t)run * 3 * n;
        const double rp = fac[2], rs = fac[3], pa = pt[i], pb = pt[n + i], ps = pt[2 * n + i];
        ph[i] = pa + (cp * ia - pa * rp);
        ph[n + i] = pb + (cp * ib - pb * rp);
        ph[2 * n + i] = ps + (cs * ph[2 * n + i] - ps * rs);
    }
}

template <typename T> static PropK<T> prop_args(const Group &G)
{
    PropK<T> k;
    k.g = G.g;
    k.chain = reinterpret_cast<V2<T> *>(G.chain);
    k.hist = reinterpret_cast<V2<T> *>(G.hist);
    k.hd = reinterpret_cast<V2<T> *>(G.hd);
    k.rho = reinterpret_cast<const float2 *>(G.rho);
    k.hnodes = G.hnodes;
    k.efac = reinterpret_cast<const V2<T> *>(G.efac);
    k.ia = G.ia;
    k.ib = G.ib;
    k.part = G.part;
    k.twx = reinterpret_cast<const V2<T> *>(G.twx);
    k.twy = reinterpret_cast<const V2<T> *>(G.twy);
    k.kx = reinterpret_cast<const T *>(G.kx);
    k.ky = reinterpret_cast<const T *>(G.ky);
    k.stateless = G.stateless;
    return k;
}

// Column tile autotuner of the power-of-two streaming column pass (see
// tune_column_tiles): times it at each width on the group's chain buffer
// (scratch until the next solve starts it) and keeps the fastest.
cudaError_t tune_stream_tiles(Group &G, cudaStream_t s)
{
    if (!(G.prec == EPD_LB_MIXED_FP32 && G.hist_full)) return cudaSuccess;
    if (const char *env = std::getenv("EPD_LB_COLUMN_TILE")) {
        const int w = std::atoi(env);
        if ((w == 4 || w == 8 || w == 16) && stream_col_fits(G.g.ny, w)) {
            G.colw_prop = w;
            return cudaSuccess;
        }
    }
    const PropK<float> k = prop_args<float>(G);
    cudaError_t e = cudaMemsetAsync(G.chain, 0, (size_t)G.g.nruns * G.g.n * sizeof(float2), s);
    if (e != cudaSuccess) return e;
    cudaEvent_t a, b;
    if ((e = cudaEventCreate(&a)) != cudaSuccess) return e;
    if ((e = cudaEventCreate(&b)) != cudaSuccess) {
        cudaEventDestroy(a);
        return e;
    }
    float best = 1e30f;
    for (int w : kColWidths) {
        if (!stream_col_fits(G.g.ny, w)) continue;
        for (int rep = 0; rep < 4 && !e; ++rep) {
            cudaEventRecord(a, s);
            e = stream_col(k, w, s);
            cudaEventRecord(b, s);
            cudaEventSynchronize(b);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, a, b);
            if (!e && rep > 0 && ms < best) {
                best = ms;
                G.colw_prop = w;
            }
        }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return e ? e : cudaGetLastError();
}

bool stream8_eligible(int prec, int logx, int logy)
{
    return prec == EPD_LB_MIXED_FP32 && !cluster_shape_exists(logx, logy) && logx >= 6 && logy >= 6 && logx <= 11 &&
           logy <= 11 && logx + logy >= 11;
}

// Blocks of the pointwise passes: four sites per thread (the FP64 block sums
// of the solvent factor cost ten FP64 additions per thread), at most 1024.
// Depends on one run's grid only: so does the order of the sums.
static int grid_for(long long n)
{
    const long long b = (n + 4 * kThreads - 1) / (4 * kThreads);
    return (int)(b > 1024 ? 1024 : b);
}

// One pass of either axis: compile-time tiles on the FP32 grids that have them
// (powers of two, 64..2048 points per axis), the general passes otherwise.
static bool has_stream_tiles(const GroupGeom &g) { return g.pow2 && g.logx >= 6 && g.logx <= 11 && g.logy >= 6 && g.logy <= 11; }
static cudaError_t col_pass(const PropK<float> &k, const Group &G, cudaStream_t s)
{
    return has_stream_tiles(k.g) ? stream_col(k, G.colw_prop, s) : line_col(k, s);
}
static cudaError_t col_pass(const PropK<double> &k, const Group &, cudaStream_t s) { return line_col(k, s); }
static cudaError_t row_pass(const PropK<float> &k, const Group &, int m, bool diff, int *blocks, cudaStream_t s)
{
    return has_stream_tiles(k.g) ? stream_row(k, m, diff, blocks, s) : line_row(k, m, diff, blocks, s);
}
static cudaError_t row_pass(const PropK<double> &k, const Group &, int m, bool diff, int *blocks, cudaStream_t s)
{
    return line_row(k, m, diff, blocks, s);
}

// The contour loop of the streaming solves (column pass, row pass per node);
// blocks: the Q partials of the last row pass per run.
template <typename T>
static cudaError_t generic_loop(const Group &G, const PropK<T> &k, bool diff, int *blocks, cudaStream_t s, const SolveProbe *probe)
{
    cudaError_t e = cudaSuccess;
    for (int m = 1; m <= k.g.ns && !e; ++m) {
        const bool pa = probe && m == probe->m_acc, ps = probe && m == probe->m_store;
        if (pa) cudaEventRecordWithFlags(probe->ev[2], s, cudaEventRecordExternal);
        e = col_pass(k, G, s);
        if (pa) cudaEventRecordWithFlags(probe->ev[3], s, cudaEventRecordExternal);
        if (ps) cudaEventRecordWithFlags(probe->ev[0], s, cudaEventRecordExternal);
        if (!e) e = row_pass(k, G, m, diff, blocks, s);
        if (ps) cudaEventRecordWithFlags(probe->ev[1], s, cudaEventRecordExternal);
        if (pa) cudaEventRecordWithFlags(probe->ev[4], s, cudaEventRecordExternal);
    }
    return e;
}

template <typename T>
static cudaError_t solve_t(Group &G, const double *omega, double *phi, double *q, cudaStream_t s, const SolveProbe *probe)
{
    const GroupGeom &g = G.g;
    PropK<T> k = prop_args<T>(G);

    const int pg = grid_for(g.n);
    prop_prep<T><<<dim3(pg, g.nruns), kThreads, 0, s>>>(g, omega, reinterpret_cast<V2<T> *>(G.efac), reinterpret_cast<T *>(G.facp), phi, G.part);
    if (sizeof(T) == sizeof(float) && G.hc && G.tab8x && cluster_solve_supported(G)) {
        // whole contour in one cluster-resident launch, then the contour sums
        return launch_cluster_solve(G, s, false, pg, phi, q, probe);
    }
    prop_start<T, false><<<dim3(pg, g.nruns), kThreads, 0, s>>>(k);
    int blocks = 0;
    if (cudaError_t e = generic_loop<T>(G, k, false, &blocks, s, probe)) return e;
    if (sizeof(T) == sizeof(float) && k.hnodes == g.ns + 1)  // full history: the sums are one pass over it
        prop_contour_stream<false><<<dim3((unsigned)((g.n + kThreads - 1) / kThreads), g.nruns), kThreads, 0, s>>>(
            g, reinterpret_cast<const float2 *>(G.hist), nullptr, blocks, pg, G.part, phi, q, nullptr, nullptr, G.err);
    else
        prop_finalize<<<dim3(pg, g.nruns), kThreads, 0, s>>>(g, blocks, pg, G.ia, G.ib, G.part, phi, q, G.err);
    return cudaGetLastError();
}

// Streaming differential solve (MIXED_FP32 grids without the cluster
// solve): the changes against the reference history of the last plain
// solve, then the contour pass of the changes.
static cudaError_t stream_delta(Group &G, int pg, double *phi, double *q, const double *phi_ref, const double *q_ref,
                                cudaStream_t s, const SolveProbe *probe)
{
    const GroupGeom &g = G.g;
    const dim3 gcon((unsigned)((g.n + kThreads - 1) / kThreads), g.nruns);
    PropK<float> k = prop_args<float>(G);
    prop_start<float, true><<<dim3(pg, g.nruns), kThreads, 0, s>>>(k);
    int blocks = 0;
    if (cudaError_t e = generic_loop<float>(G, k, true, &blocks, s, probe)) return e;
    prop_contour_stream<true><<<gcon, kThreads, 0, s>>>(g, reinterpret_cast<const float2 *>(G.hist),
                                                       reinterpret_cast<const float2 *>(G.hd), blocks, pg, G.part, phi,
                                                       q, phi_ref, q_ref, G.err);
    return cudaGetLastError();
}

cudaError_t launch_solve(Group &G, const double *omega, double *phi, double *q, cudaStream_t s, const SolveProbe *probe)
{
    if (G.prec == EPD_LB_MIXED_FP32) return solve_t<float>(G, omega, phi, q, s, probe);
    return solve_t<double>(G, omega, phi, q, s, probe);
}

cudaError_t launch_solve_delta_at(Group &G, const double *omega, const double *omega_ref, const double *phi_ref,
                                  const double *q_ref, double *phi, double *q, cudaStream_t s, const SolveProbe *probe)
{
    if (!G.diff || !G.hd) return cudaErrorInvalidValue;
    const GroupGeom &g = G.g;
    const int pg = grid_for(g.n);
    prop_prep_delta<<<dim3(pg, g.nruns), kThreads, 0, s>>>(g, omega, omega_ref, reinterpret_cast<float2 *>(G.rho),
                                                          reinterpret_cast<float *>(G.cdiff), reinterpret_cast<const float2 *>(G.efac),
                                                          reinterpret_cast<float *>(G.facd), phi, G.part);
    if (!G.hc) return stream_delta(G, pg, phi, q, phi_ref, q_ref, s, probe);
    return launch_cluster_solve(G, s, true, pg, phi, q, probe, phi_ref, q_ref);
}

cudaError_t launch_solve_delta(Group &G, cudaStream_t s, const SolveProbe *probe)
{
    return launch_solve_delta_at(G, G.omega, G.omega_t, G.phi_t, G.q_t, G.phi, G.q, s, probe);
}

// Single-chain solve on a 3D box: per contour step the z-column, y-column and
// x-row passes (the Fourier factor exp(-R_G^2 |k|^2 ds) is the product of the
// three axes' factors, each applied inside its own axis transform), the row
// pass carrying the node factors, history and contour sums as in 2D.
template <typename T>
static cudaError_t solve3d_t(const Solve3 &S, const double *omega, double *phi, double *q, cudaStream_t s)
{
    auto view = [&](const GroupGeom &g, const void *tw_row, const void *tw_col, const void *k_row, const void *k_col) {
        PropK<T> k;
        k.g = g;
        k.chain = reinterpret_cast<V2<T> *>(S.chain);
        k.hist = reinterpret_cast<V2<T> *>(S.hist);
        k.hd = nullptr;
        k.rho = nullptr;
        k.hnodes = g.half_lo + 1;
        k.efac = reinterpret_cast<const V2<T> *>(S.efac);
        k.ia = S.ia;
        k.ib = S.ib;
        k.part = S.part;
        k.twx = reinterpret_cast<const V2<T> *>(tw_row);
        k.twy = reinterpret_cast<const V2<T> *>(tw_col);
        k.kx = reinterpret_cast<const T *>(k_row);
        k.ky = reinterpret_cast<const T *>(k_col);
        k.stateless = true;
        return k;
    };
    const PropK<T> kx = view(S.vx, S.twx, S.twy, S.kx, S.ky);
    const PropK<T> ky = view(S.vy, S.twx, S.twy, S.kx, S.ky);
    const PropK<T> kz = view(S.vz, S.twx, S.twz, S.kx, S.kz);
    const GroupGeom &g = S.vx;
    const int pg = grid_for(g.n);
    prop_prep<T><<<dim3(pg, 1), kThreads, 0, s>>>(g, omega, reinterpret_cast<V2<T> *>(S.efac), (T *)nullptr, phi, S.part);
    prop_start<T, false><<<dim3(pg, 1), kThreads, 0, s>>>(kx);
    int blocks = 0;
    cudaError_t e = cudaSuccess;
    for (int m = 1; m <= g.ns && !e; ++m) {
        e = line_col(kz, s);
        if (!e) e = line_col(ky, s);
        if (!e) e = line_row(kx, m, false, &blocks, s);
    }
    if (e) return e;
    prop_finalize<<<dim3(pg, 1), kThreads, 0, s>>>(g, blocks, pg, S.ia, S.ib, S.part, phi, q, S.err);
    return cudaGetLastError();
}

cudaError_t launch_solve3d(const Solve3 &S, const double *omega, double *phi, double *q, cudaStream_t s)
{
    return S.prec == EPD_LB_MIXED_FP32 ? solve3d_t<float>(S, omega, phi, q, s) : solve3d_t<double>(S, omega, phi, q, s);
}

} // namespace epdlb
