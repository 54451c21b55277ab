// Tile shapes of the FP64-mode product-sum and the launches that cover a
// result with them (the kernel is in prodsum_f64w_kernel.cuh).
#include <cstdlib>
#include <cstring>

#include "launchers.cuh"

namespace emu {

constexpr int kTileRows = 128;

// Tile shape of the FP64 product-sum.  Every shape forms the same exact sums
// and adds them with the same roundings, so C does not depend on the choice.
// The table below holds per-SM rates relative to 256 x 256 tiles on CTA pairs.
// Measured at 4096^3 with 21 products, every SM busy (256 x 256: 1446 TFLOP/s), they
// are 0.82 for 256 x 128 on pairs, 0.85, 0.68 and 0.39; a narrower tile moves more
// operand bytes through shared memory per FLOP.  A single wave of 256 x 128 tiles takes
// a little more than the rate says (kRateHalf), and the two narrowest are 0.66 and
// 0.38 in the table, which leaves near ties to the wider tile.
// - The shape with the least waves x columns / rate is taken.  Pairs need two
//   128-row tile rows.
// - 128 x 128 tiles are taken only where 256 x 128 pairs would leave half of the
//   SMs idle or more, and 64-column tiles where 128 x 128 ones would leave more
//   than 60 % idle: with so few CTAs the time is that of one CTA's chain of
//   products, which is shorter for half the columns (256^3, 21 products: 40
//   against 54 us; 3001 x 203 x 2999: 283 against 378 us).
// - When 256 x 256 tiles leave the last wave partly empty, the full waves run
//   as such and a second launch takes the remaining tiles as 256 x 128 halves,
//   if that is estimated faster (4096^3, 21 products: 1996 us in four waves,
//   1901 us as three and one of halves).
// EMU_F64_TILE=128x64 / 128x128 / 256x128 / 128x256 / 256x256 forces one shape
// for every result (and no mixed last wave).
constexpr double kRateHalf = 0.75;
static int f64_tile_forced()
{
    static const int forced = [] {
        const char *e = std::getenv("EMU_F64_TILE");
        if (!e) return 0;
        if (std::strcmp(e, "256x256") == 0) return 1;
        if (std::strcmp(e, "128x256") == 0) return 2;
        if (std::strcmp(e, "256x128") == 0) return 3;
        if (std::strcmp(e, "128x128") == 0) return 4;
        if (std::strcmp(e, "128x64") == 0) return 5;
        return 0;
    }();
    return forced;
}

static int device_sms()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 2)
        sms = 152;
    return sms;
}

F64Plan f64_plan(int64_t M, int64_t N)
{
    F64Plan p;
    if (M < 1 || N < 1) return p;
    const int forced = f64_tile_forced();
    const int sms = device_sms();
    const int64_t tiles_m = (M + kTileRows - 1) / kTileRows;
    struct Shape { int rows, cols; double rate; };
    static const Shape shapes[5] = {
        {256, 256, 1.0}, {128, 256, 0.85}, {256, 128, kRateHalf}, {128, 128, 0.66}, {128, 64, 0.38}};
    const bool few = tiles_m * ((N + 127) / 128) * 10 < (int64_t)sms * 4;
    // 128-column tiles of 128 rows only where pairs would leave half of the SMs idle
    const bool few_pairs = ((tiles_m + 1) / 2) * ((N + 127) / 128) * 4 <= (int64_t)sms || tiles_m < 2;
    p.launches = 1;
    double best = 0.0;
    for (int i = 0; i < 5; ++i) {
        const Shape &h = shapes[i];
        if (forced ? forced != i + 1 : (h.cols == 256 && (h.rows == 256) != (tiles_m >= 2)) ||
                         (h.rows == 256 && tiles_m < 2) || (h.cols == 128 && (h.rows == 256) == few_pairs) || (h.cols == 64 && !few))
            continue;
        const int64_t tiles = ((M + h.rows - 1) / h.rows) * ((N + h.cols - 1) / h.cols);
        const int64_t slots = sms / (h.rows / kTileRows);
        const double t = (double)((tiles + slots - 1) / slots) * h.cols / h.rate;
        if (best == 0.0 || t < 0.98 * best) {          // the wider tile on near ties
            best = t;
            p.rows = h.rows;
            p.cols = h.cols;
            p.tiles = tiles;
        }
    }
    if (!forced && p.rows == 256 && p.cols == 256) {
        const int64_t slots = sms / 2, full = (p.tiles / slots) * slots, rem = p.tiles - full;
        const double t_mixed =
            (double)(full / slots) * 256.0 + (double)((2 * rem + slots - 1) / slots) * 128.0 / kRateHalf;
        if (full > 0 && rem > 0 && t_mixed < 0.97 * best) {
            p.tiles = full;
            p.rest = 2 * rem;
            p.launches = 2;
        }
    }
    return p;
}

int f64_tile_columns(int64_t M, int64_t N)
{
    return f64_plan(M, N).cols;
}

cudaError_t launch_prodsum_f64(int64_t M, int64_t N, int64_t K, const uint16_t *Ap, const uint16_t *Bp,
                               int64_t ldcomp, const int32_t *vA, const int32_t *vB, int nprod, double *C,
                               int64_t ldc, double *acc, uint32_t *flags, cudaStream_t st, int64_t a_plane,
                               bool rowcol, const float *T, int64_t ldt)
{
    const F64Plan p = f64_plan(M, N);
    // 128-row tiles on at most half of the SMs: two CTAs per tile, each with half of the
    // first ten products (any K that diag_exact lets through)
    const bool duo = p.cols < 256 && p.rows == 128 && !rowcol && !T && vA && 2 * p.tiles <= device_sms() && K <= 8097;
    if (p.cols < 256)
        return launch_prodsum_f64_narrow(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane,
                                         rowcol, T, ldt, p.cols, p.rows == 256, p.tiles, -1, duo);
    cudaError_t e = launch_prodsum_f64_wide(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane,
                                            rowcol, T, ldt, p.rows == 256, p.tiles);
    if (e != cudaSuccess || p.rest == 0) return e;
    return launch_prodsum_f64_narrow(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane, rowcol, T,
                                     ldt, 128, true, p.rest, (int)p.tiles, false);
}

}  // namespace emu
