// fftg.cuh -- in-place transforms of any length 2^a 3^b 5^c in shared memory
// (FP32 and FP64), for the passes that run on every grid.
//
// A sequence of N points is transformed with decimation in frequency over the
// radices r_0, r_1, .., r_last of its plan: the butterfly of pass i reads and
// writes the same R points, M_i = N / (r_0 .. r_i) apart, so a pass needs one
// buffer and one barrier, and the spectrum ends in digit-reversed order.  A
// spectral operator acts on it there, by the natural bin of each position
// (line_bin), and the inverse runs the passes backwards (decimation in time),
// so the order never has to be restored.  The last forward pass, the operator
// and the first inverse pass are one: a length up to 256 is two radices, three
// trips through shared memory for a whole transform pair.
//
// Radices up to 16: a pass costs the tile one trip through shared memory and
// one twiddle per point whatever its radix, so few large ones win (150 = 10 x
// 15).  Butterflies of coprime factors (6, 10, 12, 15) are prime-factor
// transforms (Good 1958, Thomas 1963) without inner twiddles.
//
// The first forward pass takes its points from global memory and the last
// inverse pass hands its points to the caller's epilogue, both templated on
// the plan's first radix; the passes between are called by radix.
#pragma once

#include "common.cuh"
#include "engine.h"

namespace epdlb {

// (x, y) -> i (x, y) times the direction's sign: forward -i, inverse +i
template <bool INV, typename V> __device__ __forceinline__ V mul_i(V a)
{
    V r;
    r.x = INV ? -a.y : a.y;
    r.y = INV ? a.x : -a.x;
    return r;
}

// a conj(b)
template <typename V> __device__ __forceinline__ V cmul_conj(V a, V b)
{
    V r;
    r.x = a.x * b.x + a.y * b.y;
    r.y = a.y * b.x - a.x * b.y;
    return r;
}

// 2^e 2^-(bits of the fraction) of 2^e <= |v| < 2^(e + 1)
__host__ __device__ inline float ulp(float v)
{
    unsigned b;
    memcpy(&b, &v, sizeof b);
    b &= 0x7f800000u;
    memcpy(&v, &b, sizeof b);
    return v * 1.1920928955078125e-7f;
}
__host__ __device__ inline double ulp(double v)
{
    unsigned long long b;
    memcpy(&b, &v, sizeof b);
    b &= 0x7ff0000000000000ull;
    memcpy(&v, &b, sizeof b);
    return v * 2.220446049250313e-16;
}

// a b rounded, never fused with what follows (by the compiler of either side)
template <typename T> __host__ __device__ inline T mul_rounded(T a, T b)
{
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(T) == 4) return __fmul_rn(a, b);
    else return __dmul_rn(a, b);
#else
    volatile T p = a * b;
    return p;
#endif
}

// The pair next to (c, s) = (cos, -sin) in T's numbers that is nearest to the
// unit circle.  A forward and an inverse pass multiply by w and conj(w), so over a
// contour every step adds the same |w|^2 - 1 at the same points; of the rounded
// pair and its neighbours (an ulp away at most) this takes the one where that is
// least, with a small weight on the distance, which turns the phase only.  RMS
// error of MIXED solves: 270 x 384 1.07e-7 -> 0.99e-7, 90 x 96 1.58e-7 -> 1.37e-7, 512 x
// 512 1.25e-7 -> 1.14e-7; of 14 general grids 1.02 -> 0.96 times
// that of radix-2 to radix-5 passes (geometric mean, 0.76 to 1.08).
template <typename T> __host__ __device__ inline V2<T> unit_pair(double c, double s)
{
    const T c0 = (T)c, s0 = (T)s;
    V2<T> best;
    best.x = c0;
    best.y = s0;
    if (c0 == (T)0 || s0 == (T)0) return best;
    // c0^2 + s0^2 - 1, the products exact by FMA, the larger minus one first (exact)
    const T p = mul_rounded(c0, c0), q = mul_rounded(s0, s0), low = fma(c0, c0, -p) + fma(s0, s0, -q);
    const T m0 = (p > q ? (p - (T)1) + q : (q - (T)1) + p) + low;
    const T uc = ulp(c0), us = ulp(s0);
    const T ec = (T)((double)c0 - c), es = (T)((double)s0 - s);
    T least = (T)1;
    for (int i = -1; i <= 1; ++i)
        for (int j = -1; j <= 1; ++j) {
            const T dc = (T)i * uc, ds = (T)j * us;
            T m = m0 + (T)2 * (c0 * dc + s0 * ds), d = ec + dc, e = es + ds;
            m = m < (T)0 ? -m : m;
            d = d < (T)0 ? -d : d;
            e = e < (T)0 ? -e : e;
            const T cost = m + (T)0.05 * (d + e);
            if (cost < least) {
                least = cost;
                best.x = c0 + dc;
                best.y = s0 + ds;
            }
        }
    return best;
}

// DFT of R points in registers, natural order in and out.
template <typename T, int R, bool INV> struct DftN;

template <typename T, bool INV> struct DftN<T, 1, INV> {
    static __device__ __forceinline__ void run(V2<T> *) {}
};
template <typename T, bool INV> struct DftN<T, 2, INV> {
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        const V2<T> a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = csub(a, b);
    }
};
template <typename T, bool INV> struct DftN<T, 3, INV> {
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        const T h = (T)0.86602540378443864676;  // sin(2 pi / 3)
        const V2<T> s = cadd(x[1], x[2]), d = mul_i<INV>(csub(x[1], x[2]));
        const V2<T> m = mk<T>(x[0].x - (T)0.5 * s.x, x[0].y - (T)0.5 * s.y);
        x[0] = cadd(x[0], s);
        x[1] = mk<T>(m.x + h * d.x, m.y + h * d.y);
        x[2] = mk<T>(m.x - h * d.x, m.y - h * d.y);
    }
};
template <typename T, bool INV> struct DftN<T, 4, INV> {
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        const V2<T> s02 = cadd(x[0], x[2]), d02 = csub(x[0], x[2]);
        const V2<T> s13 = cadd(x[1], x[3]), d13 = mul_i<INV>(csub(x[1], x[3]));
        x[0] = cadd(s02, s13);
        x[2] = csub(s02, s13);
        x[1] = cadd(d02, d13);
        x[3] = csub(d02, d13);
    }
};
template <typename T, bool INV> struct DftN<T, 5, INV> {
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        const T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;  // cos(2 pi / 5), cos(4 pi / 5)
        const T s1 = (T)0.95105651629515357212, s2 = (T)0.58778525229247312917;   // sin(2 pi / 5), sin(4 pi / 5)
        const V2<T> a1 = cadd(x[1], x[4]), a2 = cadd(x[2], x[3]);
        const V2<T> b1 = mul_i<INV>(csub(x[1], x[4])), b2 = mul_i<INV>(csub(x[2], x[3]));
        const V2<T> m1 = mk<T>(x[0].x + c1 * a1.x + c2 * a2.x, x[0].y + c1 * a1.y + c2 * a2.y);
        const V2<T> m2 = mk<T>(x[0].x + c2 * a1.x + c1 * a2.x, x[0].y + c2 * a1.y + c1 * a2.y);
        const V2<T> n1 = mk<T>(s1 * b1.x + s2 * b2.x, s1 * b1.y + s2 * b2.y);
        const V2<T> n2 = mk<T>(s2 * b1.x - s1 * b2.x, s2 * b1.y - s1 * b2.y);
        x[0] = cadd(x[0], cadd(a1, a2));
        x[1] = cadd(m1, n1);
        x[4] = csub(m1, n1);
        x[2] = cadd(m2, n2);
        x[3] = csub(m2, n2);
    }
};
template <typename T, bool INV> struct DftN<T, 8, INV> {
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        V2<T> e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
        DftN<T, 4, INV>::run(e);
        DftN<T, 4, INV>::run(o);
        const T h = (T)0.70710678118654752440;
        // W8 o_1 = h (o_1 + (-+i) o_1), W8^3 o_3 = h ((-+i) o_3 - o_3): the
        // factor h goes into the sums
        const V2<T> o1 = cadd(o[1], mul_i<INV>(o[1])), o2 = mul_i<INV>(o[2]), o3 = csub(mul_i<INV>(o[3]), o[3]);
        x[0] = cadd(e[0], o[0]);
        x[4] = csub(e[0], o[0]);
        x[1] = mk<T>(e[1].x + h * o1.x, e[1].y + h * o1.y);
        x[5] = mk<T>(e[1].x - h * o1.x, e[1].y - h * o1.y);
        x[2] = cadd(e[2], o2);
        x[6] = csub(e[2], o2);
        x[3] = mk<T>(e[3].x + h * o3.x, e[3].y + h * o3.y);
        x[7] = mk<T>(e[3].x - h * o3.x, e[3].y - h * o3.y);
    }
};
// x times exp(-+2 pi i / n) given its cosine and sine
template <typename T, bool INV> __device__ __forceinline__ V2<T> rot(V2<T> v, T c, T s)
{
    if (!INV) s = -s;
    return mk<T>(v.x * c - v.y * s, v.x * s + v.y * c);
}
// 9 = 3 x 3 and 16 = 4 x 4: X[k1 + P k2] = DFT over n2 of W^(n2 k1) DFT over n1 of x[P n1 + n2]
template <typename T, bool INV> struct DftN<T, 9, INV> {
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        const T c1 = (T)0.76604444311897803520, s1 = (T)0.64278760968653932632;   // 2 pi / 9
        const T c2 = (T)0.17364817766693034885, s2 = (T)0.98480775301220805937;   // 4 pi / 9
        const T c4 = (T)-0.93969262078590838405, s4 = (T)0.34202014332566873304;  // 8 pi / 9
        V2<T> y[3][3];
#pragma unroll
        for (int n2 = 0; n2 < 3; ++n2) {
            y[n2][0] = x[n2];
            y[n2][1] = x[3 + n2];
            y[n2][2] = x[6 + n2];
            DftN<T, 3, INV>::run(y[n2]);
        }
        y[1][1] = rot<T, INV>(y[1][1], c1, s1);
        y[1][2] = rot<T, INV>(y[1][2], c2, s2);
        y[2][1] = rot<T, INV>(y[2][1], c2, s2);
        y[2][2] = rot<T, INV>(y[2][2], c4, s4);
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            V2<T> v[3] = {y[0][k1], y[1][k1], y[2][k1]};
            DftN<T, 3, INV>::run(v);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) x[k1 + 3 * k2] = v[k2];
        }
    }
};
template <typename T, bool INV> struct DftN<T, 16, INV> {
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        const T c = (T)0.92387953251128675613, s = (T)0.38268343236508977173, h = (T)0.70710678118654752440;
        V2<T> y[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            y[n2][0] = x[n2];
            y[n2][1] = x[4 + n2];
            y[n2][2] = x[8 + n2];
            y[n2][3] = x[12 + n2];
            DftN<T, 4, INV>::run(y[n2]);
        }
        auto w2 = [&](V2<T> v) { return cscale(cadd(v, mul_i<INV>(v)), h); };   // exp(-+2 pi i 2 / 16)
        auto w6 = [&](V2<T> v) { return cscale(csub(mul_i<INV>(v), v), h); };   // exp(-+2 pi i 6 / 16)
        y[1][1] = rot<T, INV>(y[1][1], c, s);
        y[1][2] = w2(y[1][2]);
        y[1][3] = rot<T, INV>(y[1][3], s, c);
        y[2][1] = w2(y[2][1]);
        y[2][2] = mul_i<INV>(y[2][2]);
        y[2][3] = w6(y[2][3]);
        y[3][1] = rot<T, INV>(y[3][1], s, c);
        y[3][2] = w6(y[3][2]);
        y[3][3] = rot<T, INV>(y[3][3], -c, -s);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            V2<T> v[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
            DftN<T, 4, INV>::run(v);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) x[k1 + 4 * k2] = v[k2];
        }
    }
};
// Prime-factor transform of A B points, gcd(A, B) = 1: input n = B n1 + A n2
// (mod AB), output the k with k = k1 (mod A), k = k2 (mod B).
template <typename T, int A, int B, bool INV> struct DftPf {
    static constexpr int out(int k1, int k2)
    {
        for (int k = 0; k < A * B; ++k)
            if (k % A == k1 && k % B == k2) return k;
        return 0;
    }
    static __device__ __forceinline__ void run(V2<T> *x)
    {
        V2<T> y[B][A];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) y[n2][n1] = x[(B * n1 + A * n2) % (A * B)];
            DftN<T, A, INV>::run(y[n2]);
        }
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            V2<T> v[B];
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) v[n2] = y[n2][k1];
            DftN<T, B, INV>::run(v);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) x[out(k1, k2)] = v[k2];
        }
    }
};
template <typename T, bool INV> struct DftN<T, 6, INV> : DftPf<T, 2, 3, INV> {};
template <typename T, bool INV> struct DftN<T, 10, INV> : DftPf<T, 2, 5, INV> {};
template <typename T, bool INV> struct DftN<T, 12, INV> : DftPf<T, 3, 4, INV> {};
template <typename T, bool INV> struct DftN<T, 15, INV> : DftPf<T, 3, 5, INV> {};

// Tile of B = 2^logb sequences of n points: point p of sequence b at
// (p + pad (p / rl)) bp + b, rl the plan's last radix, pad = 1 where it is
// even.  Every pass but the middle one has legs a multiple of rl apart, so
// the pad only changes their constant distance, and the middle one's blocks
// start an odd number of points apart.  Columns: bp = B, consecutive threads
// on consecutive sequences; rows: bp odd, and consecutive threads on
// consecutive points (the global order) where the legs are far enough apart.
// No access then meets the same bank more than twice.
struct LineTile {
    static constexpr bool fixed = false, products = false;
    int n, logb, bp, rl, pad;
    bool row;
    __host__ __device__ LineTile(bool row_, int n_, int logb_, LinePlan pl)
        : n(n_), logb(logb_), bp(row_ ? (1 << logb_) | 1 : 1 << logb_), rl(pl.r(pl.nf - 1)), pad(rl % 2 ? 0 : 1), row(row_)
    {
    }
    __host__ __device__ size_t points() const { return (size_t)(n + pad * (n / rl)) * bp; }
    // distance of points M apart (M a multiple of rl)
    __device__ int leg(int M) const { return (M + pad * (M / rl)) * bp; }
};
// The same with everything known at compile time, for the power-of-two axes
// of the streaming solves: offsets become immediates, indices shifts, loops
// straight code (a third fewer instructions per point than above).
// NT: threads of the block; READ: every twiddle is read (LineTw).
constexpr int ct_radix(int logn, int i)
{
    // 64 = 8.8, 128 = 16.8, 256 = 16.16, 512 = 8.8.8, 1024 = 16.8.8, 2048 = 16.8.16
    constexpr int plan[6][4] = {{2, 8, 8, 0}, {2, 16, 8, 0}, {2, 16, 16, 0}, {3, 8, 8, 8}, {3, 16, 8, 8}, {3, 16, 8, 16}};
    return plan[logn - 6][i + 1];
}
template <int LOGN> struct LinePlanCT {
    static constexpr int nf = ct_radix(LOGN, -1);
    static __host__ __device__ constexpr int r(int i) { return ct_radix(LOGN, i); }
};
template <int LOGN, int LOGB, bool ROW, int NT, bool READ> struct LineTileCT {
    static constexpr bool fixed = true, products = !READ;
    static constexpr int n = 1 << LOGN, logb = LOGB, bp = ROW ? (1 << LOGB) | 1 : 1 << LOGB;
    static constexpr int rl = LinePlanCT<LOGN>::r(LinePlanCT<LOGN>::nf - 1), pad = 1, nt = NT;
    static constexpr bool row = ROW;
    static constexpr int POINTS = (n + n / rl) * bp;
    static __device__ constexpr int leg(int M) { return (M + M / rl) * bp; }
};
// a / d of a tile: shifts where d is known, FastDiv otherwise
template <class Tile> struct TileDiv {
    FastDiv f;
    __device__ __forceinline__ explicit TileDiv(int d) : f(d) {}
    __device__ __forceinline__ int div(int a) const { return f.div(a); }
    __device__ __forceinline__ int d() const { return f.d; }
};
template <int LOGN, int LOGB, bool ROW, int NT, bool READ> struct TileDiv<LineTileCT<LOGN, LOGB, ROW, NT, READ>> {
    int v;
    __device__ __forceinline__ explicit TileDiv(int d) : v(d) {}
    __device__ __forceinline__ int div(int a) const { return (int)((unsigned)a / (unsigned)v); }  // a shift once inlined
    __device__ __forceinline__ int d() const { return v; }
};
// f(bf) for the thread's butterflies bf < total
template <class Tile, class F> __device__ __forceinline__ void line_for(const Tile &, int total, F f)
{
    if constexpr (Tile::fixed) {
#pragma unroll
        for (int i = 0; i < total / Tile::nt; ++i) f((int)threadIdx.x + i * Tile::nt);  // one butterfly of the largest radix per thread: whole rounds
    } else {
        for (int bf = threadIdx.x; bf < total; bf += blockDim.x) f(bf);
    }
}
// sequence b and butterfly t of butterfly number bf (dq.d per sequence)
template <class Tile>
__device__ __forceinline__ void line_split(const Tile &tl, bool bfast, const TileDiv<Tile> &dq, int bf, int &b, int &t)
{
    if (bfast) {
        b = bf & ((1 << tl.logb) - 1);
        t = bf >> tl.logb;
    } else {
        b = dq.div(bf);
        t = bf - b * dq.d();
    }
}

// Natural bin of position p of a spectrum in the plan's digit-reversed order.
__device__ __forceinline__ int line_bin(LinePlan pl, int n, int p)
{
    int m = n, s = 1, k = 0;
    for (int i = 0; i < pl.nf; ++i) {
        m /= pl.r(i);
        const int v = p / m;
        p -= v * m;
        k += s * v;
        s *= pl.r(i);
    }
    return k;
}

// Twiddles of a butterfly, tw[u j] (tw[i] = exp(-2 pi i i / n)), read before
// its points: with few warps per SM the reads' latency is exposed, and taken
// one by one next to their uses it is exposed at every butterfly.  PROD: the powers
// of two are read, the others are products, w_u = w_(u mod 8) w_(u - u mod 8)
// (power-of-two axes in FP32: a gather at stride u j touches a line per lane,
// and fewer factors stay in registers).
template <int R, bool PROD, typename V> struct LineTw {
    V w[R];
    __device__ __forceinline__ LineTw(const V *__restrict__ tw, int j)
    {
#pragma unroll
        for (int u = 1; u < R; ++u) w[u] = __ldg(&tw[u * j]);
    }
    __device__ __forceinline__ V get(int u) const { return w[u]; }
};
template <int R, typename V> struct LineTw<R, true, V> {
    static constexpr int NA = R < 8 ? R : 8, NB = (R + 7) / 8;
    V a[NA], b[NB];
    __device__ __forceinline__ LineTw(const V *__restrict__ tw, int j)
    {
        a[1] = __ldg(&tw[j]);
        if constexpr (R > 2) a[2] = __ldg(&tw[2 * j]);
        if constexpr (R > 4) a[4] = __ldg(&tw[4 * j]);
        if constexpr (R > 8) b[1] = __ldg(&tw[8 * j]);
        if constexpr (R > 3) a[3] = cmul(a[1], a[2]);
        if constexpr (R > 5) a[5] = cmul(a[1], a[4]);
        if constexpr (R > 6) a[6] = cmul(a[2], a[4]);
        if constexpr (R > 7) a[7] = cmul(a[3], a[4]);
    }
    __device__ __forceinline__ V get(int u) const
    {
        if (u < 8) return a[u];
        return u % 8 ? cmul(b[u / 8], a[u % 8]) : b[u / 8];
    }
};

// One pass: radix R, M = points between the legs of a butterfly, S = product
// of the radices before it; tw[i] = exp(-2 pi i i / n).
template <typename T, int R, bool INV, class Tile>
__device__ __forceinline__ void line_pass(V2<T> *buf, Tile tl, int M, int S, const V2<T> *__restrict__ tw)
{
    const int q = tl.n / R, total = q << tl.logb, leg = tl.leg(M);
    const TileDiv<Tile> dq(q), dm(M), dl(tl.rl);
    line_for(tl, total, [&](int bf) {
        int b, t;
        line_split(tl, !tl.row || M < 8, dq, bf, b, t);
        const int blk = dm.div(t), j = t - blk * M;
        V2<T> *p = buf + (j + (tl.pad ? dl.div(j) : 0)) * tl.bp + blk * R * leg + b;
        V2<T> x[R];
        const LineTw<R, Tile::products && sizeof(T) == 4, V2<T>> w(tw, j * S);
#pragma unroll
        for (int u = 0; u < R; ++u) x[u] = p[u * leg];
        if (INV) {
#pragma unroll
            for (int u = 1; u < R; ++u) x[u] = cmul_conj(x[u], w.get(u));
            DftN<T, R, true>::run(x);
        } else {
            DftN<T, R, false>::run(x);
#pragma unroll
            for (int u = 1; u < R; ++u) x[u] = cmul(x[u], w.get(u));
        }
#pragma unroll
        for (int u = 0; u < R; ++u) p[u * leg] = x[u];
    });
    __syncthreads();
}

// Last forward pass, operator, first inverse pass (adjacent points).
// op(op.pre(b, bin), v): the operator applied to natural bin `bin` of
// sequence b (pre: what it reads from memory, ahead of the points).
// FWD, BWD: which halves run.
template <typename T, int R, bool FWD, bool BWD, class Op, class Tile, class Plan>
__device__ __forceinline__ void line_middle(V2<T> *buf, Tile tl, Plan pl, const Op &op)
{
    const int q = tl.n / R, total = q << tl.logb;
    line_for(tl, total, [&](int bf) {
        const int b = bf & ((1 << tl.logb) - 1), t = bf >> tl.logb;
        int bin = t;  // digits of the block, reversed (one radix before the last: the digit itself)
        if (pl.nf > 2) {
            int m = q, p = t, s = 1;
            bin = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                if (i + 1 >= pl.nf) break;
                m /= pl.r(i);
                const int v = p / m;
                p -= v * m;
                bin += s * v;
                s *= pl.r(i);
            }
        }
        V2<T> *p = buf + t * (R + tl.pad) * tl.bp + b;
        V2<T> x[R];
        typename Op::Pre f[R];
#pragma unroll
        for (int u = 0; u < R; ++u) f[u] = op.pre(b, bin + u * q);
#pragma unroll
        for (int u = 0; u < R; ++u) x[u] = p[u * tl.bp];
        if (FWD) DftN<T, R, false>::run(x);
#pragma unroll
        for (int u = 0; u < R; ++u) x[u] = op(f[u], x[u]);
        if (BWD) DftN<T, R, true>::run(x);
#pragma unroll
        for (int u = 0; u < R; ++u) p[u * tl.bp] = x[u];
    });
    __syncthreads();
}

template <typename T, bool INV, class Tile>
__device__ __forceinline__ void line_pass_any(int R, V2<T> *buf, Tile tl, int M, int S, const V2<T> *tw)
{
    switch (R) {
    case 3: line_pass<T, 3, INV>(buf, tl, M, S, tw); break;
    case 4: line_pass<T, 4, INV>(buf, tl, M, S, tw); break;
    case 5: line_pass<T, 5, INV>(buf, tl, M, S, tw); break;
    case 8: line_pass<T, 8, INV>(buf, tl, M, S, tw); break;
    default: line_pass<T, 9, INV>(buf, tl, M, S, tw); break;
    }
}
template <typename T, bool FWD, bool BWD, class Op, class Tile, class Plan>
__device__ __forceinline__ void line_middle_any(V2<T> *buf, Tile tl, Plan pl, const Op &op)
{
    if constexpr (Tile::fixed) {
        line_middle<T, Plan::r(Plan::nf - 1), FWD, BWD>(buf, tl, pl, op);
        return;
    }
    switch (pl.r(pl.nf - 1)) {
    case 1: line_middle<T, 1, FWD, BWD>(buf, tl, pl, op); break;
    case 2: line_middle<T, 2, FWD, BWD>(buf, tl, pl, op); break;
    case 3: line_middle<T, 3, FWD, BWD>(buf, tl, pl, op); break;
    case 4: line_middle<T, 4, FWD, BWD>(buf, tl, pl, op); break;
    case 5: line_middle<T, 5, FWD, BWD>(buf, tl, pl, op); break;
    case 8: line_middle<T, 8, FWD, BWD>(buf, tl, pl, op); break;
    case 9: line_middle<T, 9, FWD, BWD>(buf, tl, pl, op); break;
    case 10: line_middle<T, 10, FWD, BWD>(buf, tl, pl, op); break;
    case 15: line_middle<T, 15, FWD, BWD>(buf, tl, pl, op); break;
    default: line_middle<T, 16, FWD, BWD>(buf, tl, pl, op); break;
    }
}
// The passes between the first and the middle one, forward or back.
template <typename T, bool INV, class Tile, class Plan>
__device__ __forceinline__ void line_inner(V2<T> *buf, Tile tl, Plan pl, const V2<T> *tw)
{
    if constexpr (Tile::fixed) {
        static_assert(Plan::nf <= 3, "at most one pass between");
        if constexpr (Plan::nf == 3) line_pass<T, Plan::r(1), INV>(buf, tl, Plan::r(2), Plan::r(0), tw);
        return;
    }
    if (!INV) {
        int S = pl.r(0);
        for (int i = 1; i + 1 < pl.nf; ++i) {
            const int r = pl.r(i);
            line_pass_any<T, false>(r, buf, tl, tl.n / (S * r), S, tw);
            S *= r;
        }
    } else {
        int S = tl.n / pl.r(pl.nf - 1);
        for (int i = pl.nf - 2; i >= 1; --i) {
            const int r = pl.r(i);
            S /= r;
            line_pass_any<T, true>(r, buf, tl, tl.n / (S * r), S, tw);
        }
    }
}
// First pass of a forward transform (R0 = the plan's first radix):
// src(b, t, q, x) gives the points t + u q, u < R0, of sequence b.
template <typename T, int R0, class Src, class Tile>
__device__ __forceinline__ void line_open(V2<T> *buf, Tile tl, const V2<T> *__restrict__ tw, const Src &src)
{
    const int q = tl.n / R0, total = q << tl.logb, leg = tl.leg(q);
    const TileDiv<Tile> dq(q), dl(tl.rl);
    line_for(tl, total, [&](int bf) {
        int b, t;
        line_split(tl, !tl.row, dq, bf, b, t);
        V2<T> x[R0];
        src(b, t, q, x);
        const LineTw<R0, Tile::products && sizeof(T) == 4, V2<T>> w(tw, t);
        DftN<T, R0, false>::run(x);
        V2<T> *p = buf + (t + (tl.pad ? dl.div(t) : 0)) * tl.bp + b;
        p[0] = x[0];
#pragma unroll
        for (int u = 1; u < R0; ++u) p[u * leg] = cmul(x[u], w.get(u));
    });
    __syncthreads();
}
// Last pass of an inverse transform: sink(b, t, q, x) takes the points t + u q.
template <typename T, int R0, class Sink, class Tile>
__device__ __forceinline__ void line_close(const V2<T> *buf, Tile tl, const V2<T> *__restrict__ tw, const Sink &sink)
{
    const int q = tl.n / R0, total = q << tl.logb, leg = tl.leg(q);
    const TileDiv<Tile> dq(q), dl(tl.rl);
    line_for(tl, total, [&](int bf) {
        int b, t;
        line_split(tl, !tl.row, dq, bf, b, t);
        const V2<T> *p = buf + (t + (tl.pad ? dl.div(t) : 0)) * tl.bp + b;
        V2<T> x[R0];
        const LineTw<R0, Tile::products && sizeof(T) == 4, V2<T>> w(tw, t);
        x[0] = p[0];
#pragma unroll
        for (int u = 1; u < R0; ++u) x[u] = cmul_conj(p[u * leg], w.get(u));
        DftN<T, R0, true>::run(x);
        sink(b, t, q, x);
    });
}
// Forward transform, operator, inverse transform of the tile's sequences.
template <typename T, int R0, class Src, class Op, class Sink, class Tile, class Plan>
__device__ __forceinline__ void line_pair(V2<T> *buf, Tile tl, Plan pl, const V2<T> *tw, const Src &src, const Op &op,
                                          const Sink &sink)
{
    line_open<T, R0>(buf, tl, tw, src);
    line_inner<T, false>(buf, tl, pl, tw);
    line_middle_any<T, true, true>(buf, tl, pl, op);
    line_inner<T, true>(buf, tl, pl, tw);
    line_close<T, R0>(buf, tl, tw, sink);
}

// ---------------------------------------------------------------------------
// The same transforms on a tile filled and emptied by the caller, every pass
// called by its radix: less code per kernel, for the operators that run once
// per time step.
// ---------------------------------------------------------------------------

template <typename T, int R, bool INV>
__device__ __noinline__ void line_pass_call(V2<T> *buf, LineTile tl, int M, int S, const V2<T> *tw)
{
    line_pass<T, R, INV>(buf, tl, M, S, tw);
}
template <typename T, int R, bool FWD, bool BWD, class Op>
__device__ __noinline__ void line_middle_call(V2<T> *buf, LineTile tl, LinePlan pl, Op op)
{
    line_middle<T, R, FWD, BWD>(buf, tl, pl, op);
}
template <typename T, bool INV> __device__ __forceinline__ void line_pass_by(int R, V2<T> *buf, LineTile tl, int M, int S, const V2<T> *tw)
{
    switch (R) {
    case 2: line_pass_call<T, 2, INV>(buf, tl, M, S, tw); break;
    case 3: line_pass_call<T, 3, INV>(buf, tl, M, S, tw); break;
    case 4: line_pass_call<T, 4, INV>(buf, tl, M, S, tw); break;
    case 5: line_pass_call<T, 5, INV>(buf, tl, M, S, tw); break;
    case 6: line_pass_call<T, 6, INV>(buf, tl, M, S, tw); break;
    case 8: line_pass_call<T, 8, INV>(buf, tl, M, S, tw); break;
    case 9: line_pass_call<T, 9, INV>(buf, tl, M, S, tw); break;
    case 10: line_pass_call<T, 10, INV>(buf, tl, M, S, tw); break;
    default: line_pass_call<T, 12, INV>(buf, tl, M, S, tw); break;
    }
}
// FWD: forward transform; then op in digit-reversed order; BWD: inverse.
template <typename T, bool FWD, bool BWD, class Op>
__device__ __forceinline__ void line_operator(V2<T> *buf, LineTile tl, LinePlan pl, const V2<T> *tw, Op op)
{
    if (FWD) {
        int S = 1;
        for (int i = 0; i + 1 < pl.nf; ++i) {
            const int r = pl.r(i);
            line_pass_by<T, false>(r, buf, tl, tl.n / (S * r), S, tw);
            S *= r;
        }
    }
    switch (pl.r(pl.nf - 1)) {
    case 1: line_middle_call<T, 1, FWD, BWD>(buf, tl, pl, op); break;
    case 2: line_middle_call<T, 2, FWD, BWD>(buf, tl, pl, op); break;
    case 3: line_middle_call<T, 3, FWD, BWD>(buf, tl, pl, op); break;
    case 4: line_middle_call<T, 4, FWD, BWD>(buf, tl, pl, op); break;
    case 5: line_middle_call<T, 5, FWD, BWD>(buf, tl, pl, op); break;
    case 8: line_middle_call<T, 8, FWD, BWD>(buf, tl, pl, op); break;
    case 9: line_middle_call<T, 9, FWD, BWD>(buf, tl, pl, op); break;
    case 10: line_middle_call<T, 10, FWD, BWD>(buf, tl, pl, op); break;
    case 15: line_middle_call<T, 15, FWD, BWD>(buf, tl, pl, op); break;
    default: line_middle_call<T, 16, FWD, BWD>(buf, tl, pl, op); break;
    }
    if (BWD) {
        int S = tl.n / pl.r(pl.nf - 1);
        for (int i = pl.nf - 2; i >= 0; --i) {
            const int r = pl.r(i);
            S /= r;
            line_pass_by<T, true>(r, buf, tl, tl.n / (S * r), S, tw);
        }
    }
}

// The tile elements of one thread in the global order: columns with
// consecutive threads on consecutive sequences, rows on consecutive points.
// (b, p) is the current element, at() its place in the tile; next() moves on.
struct LineIter {
    LineTile tl;
    FastDiv dl;
    int b, p, db, dp;
    __device__ __forceinline__ explicit LineIter(const LineTile &t) : tl(t), dl(t.rl)
    {
        const int tid = threadIdx.x, nt = blockDim.x;
        if (tl.row) {
            b = tid / tl.n;
            p = tid - b * tl.n;
            db = nt / tl.n;
            dp = nt - db * tl.n;
        } else {
            b = tid & ((1 << tl.logb) - 1);
            p = tid >> tl.logb;
            db = 0;
            dp = nt >> tl.logb;  // at least 1: a block has 32 threads or more, a tile at most 16 columns
        }
    }
    __device__ __forceinline__ void next()
    {
        b += db;
        p += dp;
        if (tl.row && p >= tl.n) {
            p -= tl.n;
            ++b;
        }
    }
    __device__ __forceinline__ bool in() const { return tl.row ? b < (1 << tl.logb) : p < tl.n; }
    __device__ __forceinline__ int at() const { return (p + (tl.pad ? dl.div(p) : 0)) * tl.bp + b; }
};

// f(b, p, at) for every tile element of the thread in batches of U: load
// reads into v, use consumes (loads of a batch before its stores).
template <int U, typename V, class Load, class Use> __device__ __forceinline__ void line_batches(const LineTile &tl, Load load, Use use)
{
    LineIter it(tl);
    while (it.in()) {
        V v[U];
        int b[U], p[U], at[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            b[u] = -1;
            if (it.in()) {
                b[u] = it.b;
                p[u] = it.p;
                at[u] = it.at();
                load(it.b, it.p, v[u]);
            }
            it.next();
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (b[u] >= 0) use(b[u], p[u], at[u], v[u]);
    }
}

// Host: log2 of the lines per CTA: at most 2^maxlog, halved down to 2^minlog
// while the launch has fewer than four CTAs per SM (152 SMs) or a tile more
// than 40 KB; then doubled while the launch has more than maxblocks CTAs per
// run.  batch: launches of nseq lines side by side (runs, fields).
inline int line_logb(bool row, int n, LinePlan pl, long long nseq, int batch, size_t elem, int maxlog, int minlog, long long maxblocks)
{
    auto tiles = [&](int l) { return (nseq + (1 << l) - 1) >> l; };
    int l = maxlog;
    while (l > 0 && LineTile(row, n, l, pl).points() * elem > 40 * 1024) --l;
    while (l > minlog && tiles(l) * batch < 4 * 152) --l;
    while (tiles(l) > maxblocks) ++l;
    return l;
}
// Host: threads of a tile, one butterfly of the first pass each, in whole warps
inline int line_threads(int n, int r0, int logb)
{
    const int t = (((n / r0) << logb) + 31) / 32 * 32;
    return t > 256 ? 256 : t;
}

} // namespace epdlb
