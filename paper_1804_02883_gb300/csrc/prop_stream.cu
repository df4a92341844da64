// prop_stream.cu -- the streaming propagator passes on power-of-two grids of
// 64..2048 points per axis in FP32 (grids without a cluster shape, such as 1024
// x 2048, and stateless solves): the passes of prop_line.cuh on tiles known at compile
// time.
//
// Bound: instruction issue, then the L2 traffic of the chain.  With the axis,
// the tile and the radices fixed, offsets are immediates, and a transform pair
// of 1024 points is eight accesses of shared memory per point and five
// barriers (ten and nine as load, Stockham passes and store).  Radix 32 would
// save two more of each but holds 168-250 registers: 512 x 512 (9 runs, N_s =
// 24) 2.27 ms a step with 32.16, 2.14 with 8.8.8.  1024 x 2048, N_s = 128:
// 8.8 -> 7.6 ms a step; per launch (cold, serialised) column 19.9 -> 15.6 us
// (2.2 TB/s), differential row 23.5 -> 19.4 us (5.2 TB/s), plain row 17.9 -> 20.6 us
// (in digit-reversed order both transforms of a pair read twiddles; the pair of
// passes is what gains).
//
// READ: stateless solves read every twiddle, a handle's form most as products
// of the powers of two (one or two roundings more each).  512 x 512, N_s = 32:
// 0.80 ms and an RMS error of 1.25e-7 read, 0.75 ms and 1.86e-7 as products;
// 1024 x 2048: 1.84 and 1.71 ms.
#include "prop_line.cuh"

namespace epdlb {
namespace {

template <int LOGN, int LOGB> constexpr int tile_threads()
{
    return ((1 << LOGN) / LinePlanCT<LOGN>::r(0)) << LOGB;
}
template <int LOGN, int LOGB, bool ROW, bool READ = false> using TileOf = LineTileCT<LOGN, LOGB, ROW, tile_threads<LOGN, LOGB>(), READ>;

template <int LOGY, int LOGB, bool READ>
__global__ void __launch_bounds__(tile_threads<LOGY, LOGB>()) stream_col_k(PropK<float> k)
{
    col_tile<float, LinePlanCT<LOGY>::r(0)>(k, TileOf<LOGY, LOGB, false, READ>(), LinePlanCT<LOGY>());
}
template <int LOGX, int LOGB, bool DIFF, bool READ>
__global__ void __launch_bounds__(tile_threads<LOGX, LOGB>()) stream_row_k(PropK<float> k, int m, RowWeights w)
{
    row_tile<float, LinePlanCT<LOGX>::r(0), DIFF>(k, TileOf<LOGX, LOGB, true, READ>(), LinePlanCT<LOGX>(), m, w);
}

template <int LOGY, int LOGB> cudaError_t col_at(const PropK<float> &k, cudaStream_t s)
{
    constexpr size_t sm = (size_t)TileOf<LOGY, LOGB, false>::POINTS * sizeof(float2);
    if constexpr (sm > kMaxTile || tile_threads<LOGY, LOGB>() > 512) {
        return cudaErrorInvalidConfiguration;
    } else {
        constexpr int th = tile_threads<LOGY, LOGB>();
        const dim3 grid(k.g.nx >> LOGB, k.g.nruns);
        return k.stateless ? launch_line(true, stream_col_k<LOGY, LOGB, true>, grid, th, sm, s, k)
                           : launch_line(false, stream_col_k<LOGY, LOGB, false>, grid, th, sm, s, k);
    }
}
template <int LOGX, int LOGB> cudaError_t row_at(const PropK<float> &k, int m, bool diff, const RowWeights &w, cudaStream_t s)
{
    constexpr size_t sm = (size_t)TileOf<LOGX, LOGB, true>::POINTS * sizeof(float2);
    const dim3 grid(k.g.ny >> LOGB, k.g.nruns);
    constexpr int th = tile_threads<LOGX, LOGB>();
    if (k.stateless) return launch_line(true, stream_row_k<LOGX, LOGB, false, true>, grid, th, sm, s, k, m, w);
    return diff ? launch_line(false, stream_row_k<LOGX, LOGB, true, false>, grid, th, sm, s, k, m, w)
                : launch_line(false, stream_row_k<LOGX, LOGB, false, false>, grid, th, sm, s, k, m, w);
}

template <int LOGY> cudaError_t col_by(const PropK<float> &k, int colw, cudaStream_t s)
{
    if (!colw) {  // the widest that fits, narrower while the launch has fewer than four tiles per SM
        colw = LOGY >= 10 ? 8 : 16;
        while (colw > 4 && (!stream_col_fits(1 << LOGY, colw) || (long long)(k.g.nx / colw) * k.g.nruns < 4 * 152)) colw /= 2;
    }
    switch (colw) {
    case 4: return col_at<LOGY, 2>(k, s);
    case 16: return col_at<LOGY, 4>(k, s);
    default: return col_at<LOGY, 3>(k, s);
    }
}
// rows per tile: 64 to 256 threads; 16 to 64 while the launch has fewer than two
// tiles per SM, but for the last pass, whose tiles set the order of the Q_P sum
// and follow the grid alone
template <int LOGX> cudaError_t row_by(const PropK<float> &k, int m, bool diff, int *blocks, const RowWeights &w, cudaStream_t s)
{
    constexpr int big = LOGX == 11 ? 0 : (LOGX == 10 ? 1 : (LOGX == 9 ? 2 : 3)), small = LOGX <= 7 ? 2 : (LOGX == 8 ? 1 : 0);
    if (big == small || m == k.g.ns || (long long)(k.g.ny >> big) * k.g.nruns >= 2 * 152) {
        *blocks = k.g.ny >> big;
        return row_at<LOGX, big>(k, m, diff, w, s);
    }
    *blocks = k.g.ny >> small;
    return row_at<LOGX, small>(k, m, diff, w, s);
}

} // namespace

bool stream_col_fits(int ny, int colw)
{
    const int log = ilog2(ny), r0 = ct_radix(log, 0);
    return (size_t)(ny + ny / ct_radix(log, ct_radix(log, -1) - 1)) * colw * sizeof(float2) <= kMaxTile && ny / r0 * colw <= 512;
}

cudaError_t stream_col(const PropK<float> &k, int colw, cudaStream_t s)
{
    switch (k.g.logy) {
    case 6: return col_by<6>(k, colw, s);
    case 7: return col_by<7>(k, colw, s);
    case 8: return col_by<8>(k, colw, s);
    case 9: return col_by<9>(k, colw, s);
    case 10: return col_by<10>(k, colw, s);
    case 11: return col_by<11>(k, colw, s);
    default: return cudaErrorInvalidConfiguration;
    }
}

cudaError_t stream_row(const PropK<float> &k, int m, bool diff, int *blocks, cudaStream_t s)
{
    const RowWeights w = row_weights(k.g, m);
    switch (k.g.logx) {
    case 6: return row_by<6>(k, m, diff, blocks, w, s);
    case 7: return row_by<7>(k, m, diff, blocks, w, s);
    case 8: return row_by<8>(k, m, diff, blocks, w, s);
    case 9: return row_by<9>(k, m, diff, blocks, w, s);
    case 10: return row_by<10>(k, m, diff, blocks, w, s);
    case 11: return row_by<11>(k, m, diff, blocks, w, s);
    default: return cudaErrorInvalidConfiguration;
    }
}

} // namespace epdlb
