// FP64 fixed six-slice simplified Ozaki split, Eq. (fp64split), with one set
// of level exponents per matrix, writing BF16 component planes row-major or
// transposed (K-major for the B operand).
//
// The FP64 split reads a 64 x 64 tile of X with coalesced vector loads,
// splits it in registers, stages it in shared memory and writes 16-byte
// chunks of whole plane rows, so transposed B planes are written as
// coalesced as row-major A planes.
//
// FP64 level exponents need a whole-matrix max per level (v^(r) of
// Eq. (fp64split)), i.e. six dependent grid-wide reductions.  The split does
// them speculatively in one pass: after the exact max of level 0, the fused
// pass assumes v^(r) = v^(0) - 8r (a residual always shrinks by at least 2^-8
// per level, and on full-size dense data by exactly that), writes the planes
// (all six, or only the d a product-sum of d diagonals reads) and records the
// true per-level maxima.  One cooperative launch then checks the assumption
// level by level and, only if it fails, recomputes the remaining levels
// literally.  The result is identical to the literal definition in every
// case.
#include "split_common.cuh"

namespace emu {

namespace {


// Row-major planes: thread = 4 consecutive entries of a row (two 16-byte
// loads, one 8-byte store per plane), rows advancing by the grid's y size.
// Block (bx, by) of a grid with gy rows of blocks; red: 5 * kThreads / 32
// words of shared memory.
template <int NLEV>
__device__ __forceinline__ void f64_spec_rows_body(const double *__restrict__ X, int64_t rows, int64_t cols,
                                                   int64_t ldx, uint16_t *__restrict__ comps, int64_t ldcomp,
                                                   int64_t plane, WsHeader *ws, int slot, int64_t bx, int64_t by,
                                                   int64_t gy, uint32_t *red)
{
    const int v0 = spec_v0(ws, slot);
    const bool fast = v0 >= -78;
    float P[3] = {};
    if (fast) spec_units(v0 - 50, P);
    const bool vin = ((ldx & 1) == 0) && ((reinterpret_cast<uintptr_t>(X) & 15u) == 0);
    const bool vout = ((ldcomp & 3) == 0) && ((plane & 3) == 0) && ((reinterpret_cast<uintptr_t>(comps) & 7u) == 0);
    const int64_t j0 = (bx * kThreads + threadIdx.x) * 4;
    SpecState st;
    if (j0 < cols) {
        const bool full = j0 + 4 <= cols;
        for (int64_t i = by; i < rows; i += gy) {
            const double *src = X + i * ldx + j0;
            double x[4];
            if (vin && full) {
                const double2 a = reinterpret_cast<const double2 *>(src)[0], c = reinterpret_cast<const double2 *>(src)[1];
                x[0] = a.x; x[1] = a.y; x[2] = c.x; x[3] = c.y;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = (j0 + e < cols) ? src[e] : 0.0;
            }
            uint32_t w[NLEV][2];
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                uint32_t sa[6], sb[6];
                spec_element<NLEV>(x[e], v0, fast, P, sa, st);
                spec_element<NLEV>(x[e + 1], v0, fast, P, sb, st);
#pragma unroll
                for (int r = 0; r < NLEV; ++r) w[r][e >> 1] = pack2(sa[r], sb[r]);
            }
            uint16_t *dst = comps + i * ldcomp + j0;
#pragma unroll
            for (int r = 0; r < NLEV; ++r) {
                if (vout && full) {
                    *reinterpret_cast<uint2 *>(dst + r * plane) = make_uint2(w[r][0], w[r][1]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (j0 + e < cols) dst[r * plane + e] = (uint16_t)(w[r][e >> 1] >> (16 * (e & 1)));
                }
            }
        }
    }
    spec_publish(st, v0, ws, slot, red);
}

template <int NLEV>
__global__ void __launch_bounds__(kThreads)
f64_spec_rows_kernel(const double *__restrict__ X, int64_t rows, int64_t cols, int64_t ldx,
                     uint16_t *__restrict__ comps, int64_t ldcomp, int64_t plane, WsHeader *ws, int slot)
{
    __shared__ uint32_t red[5 * (kThreads / 32)];
    f64_spec_rows_body<NLEV>(X, rows, cols, ldx, comps, ldcomp, plane, ws, slot, blockIdx.x, blockIdx.y, gridDim.y, red);
}

// Transposed (K-major) planes: a 64 x 64 tile; lane p of warp q takes rows
// 2rp and 2rp+1 (rp = 4q + p / 8) and columns 16j + 2(p % 8) + {0, 1},
// j = 0..3, so eight lanes read 128 contiguous bytes of a row.  Each plane
// word packs the two entries adjacent in the transposed row; it is staged
// with each transposed row's 16-byte K-chunks permuted by an XOR with the
// column (a warp's stores hit 32 different banks) and written as 16-byte
// chunks of whole transposed rows.  Shared memory: [6][64][32] words.
// Block bid of nblk (tiles with a stride of nblk); smw: [6][kTile][kTile / 2]
// words, red: 5 * kThreads / 32 words of shared memory.
template <int NLEV>
__device__ __forceinline__ void f64_spec_transpose_body(const double *__restrict__ X, int64_t rows, int64_t cols,
                                                        int64_t ldx, uint16_t *__restrict__ comps, int64_t ldcomp,
                                                        int64_t plane, WsHeader *ws, int slot, int64_t bid,
                                                        int64_t nblk, uint32_t *smw, uint32_t *red)
{
    const int v0 = spec_v0(ws, slot);
    const bool fast = v0 >= -78;
    float P[3] = {};
    if (fast) spec_units(v0 - 50, P);
    const bool vin = ((ldx & 1) == 0) && ((reinterpret_cast<uintptr_t>(X) & 15u) == 0);
    const bool vout = ((ldcomp & 7) == 0) && ((plane & 7) == 0) && ((reinterpret_cast<uintptr_t>(comps) & 15u) == 0);
    const int q = threadIdx.x >> 5, p = lane_id();
    const int rp = 4 * q + (p >> 3), cg = p & 7;       // rows 2rp, 2rp + 1; columns 16j + 2cg + {0, 1}
    const int64_t tiles_r = (rows + kTile - 1) / kTile, tiles_c = (cols + kTile - 1) / kTile;
    SpecState st;
    // this thread's two entries in step j of tile t: eight lanes read 128
    // contiguous bytes of one row
    auto load = [&](int64_t t, int j, double (&x)[2][2]) {
        const int64_t r0 = (t / tiles_c) * kTile, gj = (t % tiles_c) * kTile + 16 * j + 2 * cg;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t gi = r0 + 2 * rp + h;
            const double *src = X + gi * ldx + gj;
            if (gi < rows && vin && gj + 2 <= cols) {
                const double2 a = *reinterpret_cast<const double2 *>(src);
                x[h][0] = a.x; x[h][1] = a.y;
            } else {
#pragma unroll
                for (int e = 0; e < 2; ++e) x[h][e] = (gi < rows && gj + e < cols) ? src[e] : 0.0;
            }
        }
    };
    double xn[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    if (bid < tiles_r * tiles_c) load(bid, 0, xn);
    for (int64_t t = bid; t < tiles_r * tiles_c; t += nblk) {
        const int64_t r0 = (t / tiles_c) * kTile, c0 = (t % tiles_c) * kTile;
        // two adjacent columns per step (one 16-byte load per row), so that
        // the element body appears four times in the loop, not sixteen; the
        // next step's entries are loaded before this step is split
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
            double x[2][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) { x[h][0] = xn[h][0]; x[h][1] = xn[h][1]; }
            if (j + 1 < 4) load(t, j + 1, xn);
            else if (t + nblk < tiles_r * tiles_c) load(t + nblk, 0, xn);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                uint32_t s0[6], s1[6];
                spec_element<NLEV>(x[0][e], v0, fast, P, s0, st);
                spec_element<NLEV>(x[1][e], v0, fast, P, s1, st);
                // transposed row col, K-chunk rp / 4 stored at chunk (rp / 4) ^ cg: conflict-free
                const int col = 16 * j + 2 * cg + e;
#pragma unroll
                for (int r = 0; r < NLEV; ++r)
                    smw[(r * kTile + col) * (kTile / 2) + (((q ^ cg) << 2) | (p >> 3))] = pack2(s0[r], s1[r]);
            }
        }
        __syncthreads();
        // NLEV planes x 64 transposed rows x 8 chunks (two iterations per plane)
#pragma unroll 4
        for (int it = 0; it < NLEV * kTile * 8 / kThreads; ++it) {
            const int c = threadIdx.x + it * kThreads;
            const int r = c >> 9, orow = (c >> 3) & 63, ch = c & 7;
            const int64_t go = c0 + orow, gk = r0 + 8 * ch;
            if (go < cols && gk < rows) {
                const uint4 v = *reinterpret_cast<const uint4 *>(&smw[(r * kTile + orow) * (kTile / 2) + 4 * (ch ^ ((orow >> 1) & 7))]);
                uint16_t *dst = comps + r * plane + go * ldcomp + gk;
                if (vout && gk + 8 <= rows) {
                    *reinterpret_cast<uint4 *>(dst) = v;
                } else {
                    const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (gk + e < rows) dst[e] = (uint16_t)(wv[e >> 1] >> (16 * (e & 1)));
                }
            }
        }
        __syncthreads();
    }
    spec_publish(st, v0, ws, slot, red);
}

template <int NLEV>
__global__ void __launch_bounds__(kThreads)
f64_spec_transpose_kernel(const double *__restrict__ X, int64_t rows, int64_t cols, int64_t ldx,
                          uint16_t *__restrict__ comps, int64_t ldcomp, int64_t plane, WsHeader *ws, int slot)
{
    extern __shared__ __align__(16) uint32_t smw[];                  // [6][kTile][kTile / 2]
    __shared__ uint32_t red[5 * (kThreads / 32)];
    f64_spec_transpose_body<NLEV>(X, rows, cols, ldx, comps, ldcomp, plane, ws, slot, blockIdx.x, gridDim.x, smw, red);
}

// Row-major planes of an operand too small for the row pass to fill its blocks:
// a 64 x 64 tile per step, 16 threads to a row of it (four entries each).
// Block bid of nblk; red: 5 * kThreads / 32 words of shared memory.
template <int NLEV>
__device__ __forceinline__ void f64_spec_tile_body(const double *__restrict__ X, int64_t rows, int64_t cols, int64_t ldx,
                                                   uint16_t *__restrict__ comps, int64_t ldcomp, int64_t plane,
                                                   WsHeader *ws, int slot, int64_t bid, int64_t nblk, uint32_t *red)
{
    const int v0 = spec_v0(ws, slot);
    const bool fast = v0 >= -78;
    float P[3] = {};
    if (fast) spec_units(v0 - 50, P);
    const bool vin = ((ldx & 1) == 0) && ((reinterpret_cast<uintptr_t>(X) & 15u) == 0);
    const bool vout = ((ldcomp & 3) == 0) && ((plane & 3) == 0) && ((reinterpret_cast<uintptr_t>(comps) & 7u) == 0);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t tiles_r = (rows + kTile - 1) / kTile, tiles_c = (cols + kTile - 1) / kTile;
    SpecState st;
    for (int64_t t = bid; t < tiles_r * tiles_c; t += nblk) {
        const int64_t j0 = (t % tiles_c) * kTile + 4 * tx;
        const bool full = j0 + 4 <= cols;
#pragma unroll 1
        for (int p = 0; p < 4; ++p) {
            const int64_t i = (t / tiles_c) * kTile + ty + 16 * p;
            if (i >= rows || j0 >= cols) continue;
            const double *src = X + i * ldx + j0;
            double x[4];
            if (vin && full) {
                const double2 a = reinterpret_cast<const double2 *>(src)[0], c = reinterpret_cast<const double2 *>(src)[1];
                x[0] = a.x; x[1] = a.y; x[2] = c.x; x[3] = c.y;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = (j0 + e < cols) ? src[e] : 0.0;
            }
            uint32_t w[NLEV][2];
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                uint32_t sa[6], sb[6];
                spec_element<NLEV>(x[e], v0, fast, P, sa, st);
                spec_element<NLEV>(x[e + 1], v0, fast, P, sb, st);
#pragma unroll
                for (int r = 0; r < NLEV; ++r) w[r][e >> 1] = pack2(sa[r], sb[r]);
            }
            uint16_t *dst = comps + i * ldcomp + j0;
#pragma unroll
            for (int r = 0; r < NLEV; ++r) {
                if (vout && full) {
                    *reinterpret_cast<uint2 *>(dst + r * plane) = make_uint2(w[r][0], w[r][1]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (j0 + e < cols) dst[r * plane + e] = (uint16_t)(w[r][e >> 1] >> (16 * (e & 1)));
                }
            }
        }
    }
    spec_publish(st, v0, ws, slot, red);
}

// One operand of a split of two: X as stored, its planes, whether they are
// written transposed, and where its levels go.
struct SplitOperand {
    const double *X;
    int64_t rows, cols, ldx;
    uint16_t *comps;
    int64_t plane;
    int32_t *v_out;
    bool transpose;
};

// The literal passes of one operand whose speculative levels failed from level
// ff on, as f64_fix_kernel runs them (every block of a cooperative launch).
__device__ __noinline__ void fix_operand(const SplitOperand &o, int64_t ldcomp, WsHeader *ws, int slot, int ff,
                                         const int (&v)[6], int nlev, unsigned long long *red, uint16_t *smdyn)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int r = 0; r < 6; ++r) ws->v[slot][r] = v[r];
        ws->fix_from[slot] = ff;
    }
    grid_sync(ws, slot);
    f64_max_pass<1>(o.X, o.rows, o.cols, o.ldx, ws, slot, blockIdx.x, gridDim.x, red);
    grid_sync(ws, slot);
    f64_max_pass<2>(o.X, o.rows, o.cols, o.ldx, ws, slot, blockIdx.x, gridDim.x, red);
    grid_sync(ws, slot);
    f64_max_pass<3>(o.X, o.rows, o.cols, o.ldx, ws, slot, blockIdx.x, gridDim.x, red);
    grid_sync(ws, slot);
    f64_max_pass<4>(o.X, o.rows, o.cols, o.ldx, ws, slot, blockIdx.x, gridDim.x, red);
    grid_sync(ws, slot);
    f64_max_pass<5>(o.X, o.rows, o.cols, o.ldx, ws, slot, blockIdx.x, gridDim.x, red);
    grid_sync(ws, slot);
    if (o.transpose)
        split_tile_pass<double, 2, true>(o.X, o.rows, o.cols, o.ldx, o.comps, ldcomp, o.plane, ws, slot, nullptr,
                                         nullptr, blockIdx.x, gridDim.x, smdyn);
    else
        split_tile_pass<double, 2, false>(o.X, o.rows, o.cols, o.ldx, o.comps, ldcomp, o.plane, ws, slot, nullptr,
                                          nullptr, blockIdx.x, gridDim.x, smdyn);
    grid_sync(ws, slot);
    if (blockIdx.x == 0 && threadIdx.x == 0) f64_finalize(ws, slot, o.v_out, nlev);
}

// After the speculative passes of both operands: every block checks both; the
// usual case publishes the levels and ends, no block waiting on another.
__device__ __forceinline__ void verify_and_fix(const SplitOperand &a, const SplitOperand &b, int64_t ldcomp, WsHeader *ws,
                                               int nlev, unsigned long long *red, uint16_t *smdyn)
{
    auto one = [&](const SplitOperand &o, int slot) {
        int v[6];
        const int ff = f64_verify_levels(ws, slot, v, nlev);
        if (ff == 6) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                for (int r = 0; r < 6; ++r) ws->v[slot][r] = v[r];
                ws->fix_from[slot] = 6;
                f64_finalize(ws, slot, o.v_out, nlev);
            }
        } else {
            fix_operand(o, ldcomp, ws, slot, ff, v, nlev, red, smdyn);
        }
    };
    one(a, 0);
    one(b, 1);
}

// The verifier of both operands as one cooperative launch.  It does not let its
// dependent, the product-sum, start early: blocks of a grid smaller than the GPU
// then land wherever an SM falls free first, both SMs of a TPC before others'
// first, and the long product-sums that follow ran 1.5 % slower (2048 x 2048 x
// 65536, 128 CTAs: 4640 against 4566 us a call).
__global__ void __launch_bounds__(kThreads)
f64_fix_pair_kernel(const __grid_constant__ SplitOperand a, const __grid_constant__ SplitOperand b, int64_t ldcomp,
                    WsHeader *ws, int nlev)
{
    extern __shared__ __align__(16) uint16_t smdyn[];
    __shared__ unsigned long long red[kThreads / 32];
    verify_and_fix(a, b, ldcomp, ws, nlev, red, smdyn);
}

// The whole split of two small operands in one cooperative launch: level-0
// maxima, grid barrier, speculative pass by tiles, grid barrier, verifier.  Five
// launches and their gaps took 28 us for operands of 256 x 256, whose entries
// are read and written in well under one.
template <int NLEV>
__global__ void __launch_bounds__(kThreads)
f64_split_small_kernel(const __grid_constant__ SplitOperand a, const __grid_constant__ SplitOperand b, int64_t ldcomp,
                       WsHeader *ws)
{
    extern __shared__ __align__(16) uint32_t smw[];
    __shared__ unsigned long long red[5 * (kThreads / 32)];
    uint32_t *red32 = reinterpret_cast<uint32_t *>(red);
    griddep_launch_dependents();
    f64_max_pass<0>(a.X, a.rows, a.cols, a.ldx, ws, 0, blockIdx.x, gridDim.x, red);
    f64_max_pass<0>(b.X, b.rows, b.cols, b.ldx, ws, 1, blockIdx.x, gridDim.x, red);
    grid_sync(ws, 0);
    // B's tiles go on where A's end, so that a block has tiles of one operand only while
    // there are blocks enough
    const int64_t ta = ((a.rows + kTile - 1) / kTile) * ((a.cols + kTile - 1) / kTile);
    const int64_t bid_b = (blockIdx.x + gridDim.x - ta % gridDim.x) % gridDim.x;
    auto spec = [&](const SplitOperand &o, int slot, int64_t bid) {
        if (o.transpose)
            f64_spec_transpose_body<NLEV>(o.X, o.rows, o.cols, o.ldx, o.comps, ldcomp, o.plane, ws, slot, bid, gridDim.x,
                                          smw, red32);
        else
            f64_spec_tile_body<NLEV>(o.X, o.rows, o.cols, o.ldx, o.comps, ldcomp, o.plane, ws, slot, bid, gridDim.x, red32);
        __syncthreads();                                  // red is reused
    };
    spec(a, 0, blockIdx.x);
    spec(b, 1, bid_b);
    grid_sync(ws, 1);
    verify_and_fix(a, b, ldcomp, ws, NLEV, red, reinterpret_cast<uint16_t *>(smw));
}

// Block b of a launch that holds nA blocks of one kind and nB of another:
// the first 2 min(nA, nB) blocks alternate between the kinds (blocks are
// dispatched roughly in index order, so both kinds run side by side), the
// rest belong to the larger kind.  Returns the block's index within its kind.
__device__ __forceinline__ int64_t pair_block(int64_t b, int64_t nA, int64_t nB, bool &is_a)
{
    const int64_t m = nA < nB ? nA : nB;
    if (b < 2 * m) { is_a = (b & 1) == 0; return b >> 1; }
    is_a = nA > nB;
    return m + (b - 2 * m);
}

// The level-0 maxima of both operands of an FP64 GEMM in one launch: nA
// blocks on A (header slot 0) and nB on B (slot 1), interleaved.
__global__ void __launch_bounds__(kThreads)
f64_max_gemm_kernel(const double *__restrict__ A, int64_t rows_a, int64_t cols_a, int64_t lda,
                    const double *__restrict__ B, int64_t rows_b, int64_t cols_b, int64_t ldb, WsHeader *ws, int64_t nA,
                    int64_t nB)
{
    __shared__ unsigned long long red[kThreads / 32];
    bool is_a;
    const int64_t i = pair_block(blockIdx.x, nA, nB, is_a);
    if (is_a) f64_max_pass<0>(A, rows_a, cols_a, lda, ws, 0, i, nA, red);
    else f64_max_pass<0>(B, rows_b, cols_b, ldb, ws, 1, i, nB, red);
}

// The fused speculative pass for slices 0 .. NLEV-1.
template <int NLEV>
cudaError_t launch_spec(const double *X, int64_t rows, int64_t cols, int64_t ldx, bool transpose, uint16_t *comps,
                        int64_t ldcomp, int64_t plane, WsHeader *ws, int slot, int gt, cudaStream_t st)
{
    if (transpose) {
        cudaError_t e = cudaFuncSetAttribute(f64_spec_transpose_kernel<NLEV>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpecTransposeSmem);
        if (e != cudaSuccess) return e;
        f64_spec_transpose_kernel<NLEV><<<gt, kThreads, kSpecTransposeSmem, st>>>(X, rows, cols, ldx, comps, ldcomp,
                                                                                  plane, ws, slot);
    } else {
        // about eight blocks per SM, each over several rows
        const int64_t bx = (cols + 4 * kThreads - 1) / (4 * kThreads);
        const int64_t want = (152 * 8 + bx - 1) / bx;
        const int64_t by = rows < want ? rows : (want < 65535 ? want : 65535);
        f64_spec_rows_kernel<NLEV><<<dim3((unsigned)bx, (unsigned)by), kThreads, 0, st>>>(X, rows, cols, ldx, comps,
                                                                                          ldcomp, plane, ws, slot);
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_split_f64(const double *X, int64_t rows, int64_t cols, int64_t ldx, bool transpose,
                             uint16_t *comps, int64_t ldcomp, int32_t *v_out, WsHeader *ws, int slot,
                             cudaStream_t st, int nlev)
{
    if (nlev < 3 || nlev > 6) return cudaErrorInvalidValue;
    const int64_t plane = (transpose ? cols : rows) * ldcomp;
    if (rows > 0 && cols > 0) {
        const int64_t segs = rows * ((cols + 4 * kThreads - 1) / (4 * kThreads));
        const int gmax = grid_for(segs, 152 * 8);
        const int64_t tiles = ((rows + kTile - 1) / kTile) * ((cols + kTile - 1) / kTile);
        const int gt = grid_for(tiles, 152 * 8);
        cudaError_t e = cudaSuccess;
        f64_max_kernel<0><<<gmax, kThreads, 0, st>>>(X, rows, cols, ldx, ws, slot);
        switch (nlev) {
        case 3: e = launch_spec<3>(X, rows, cols, ldx, transpose, comps, ldcomp, plane, ws, slot, gt, st); break;
        case 4: e = launch_spec<4>(X, rows, cols, ldx, transpose, comps, ldcomp, plane, ws, slot, gt, st); break;
        case 5: e = launch_spec<5>(X, rows, cols, ldx, transpose, comps, ldcomp, plane, ws, slot, gt, st); break;
        default: e = launch_spec<6>(X, rows, cols, ldx, transpose, comps, ldcomp, plane, ws, slot, gt, st); break;
        }
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess)
            e = launch_f64_fix(X, rows, cols, ldx, transpose, comps, ldcomp, plane, ws, slot, v_out, st, nlev);
        return e;
    }
    // an empty matrix: all levels zero, nothing to fix
    return launch_f64_fix_empty(ws, slot, v_out, st);
}


namespace {

// Cooperative launch of `kern` with as many blocks as fit on the device at once,
// at most `want` (the limit is found once per device and kernel).
template <typename... Args>
cudaError_t launch_cooperative(void (*kern)(Args...), int (&fits)[64], int64_t want, cudaStream_t st, Args... values)
{
    const size_t sm = smem_bytes(6) > kSpecTransposeSmem ? smem_bytes(6) : kSpecTransposeSmem;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    int most = fits[dev];
    if (most == 0) {
        int sms = 0, per = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kThreads, sm);
        if (e != cudaSuccess) return e;
        most = per * sms < 152 * 8 ? per * sms : 152 * 8;
        if (most < 1) return cudaErrorInvalidConfiguration;
        fits[dev] = most;
    }
    void *args[] = {(void *)&values...};
    return cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)(want < most ? want : most)), dim3(kThreads),
                                       args, sm, st);
}

template <int NLEV>
cudaError_t launch_small(const SplitOperand &a, const SplitOperand &b, int64_t ldcomp, int64_t tiles, WsHeader *ws,
                         cudaStream_t st)
{
    static int fits[64] = {};
    return launch_cooperative(f64_split_small_kernel<NLEV>, fits, tiles < 152 ? 152 : tiles, st, a, b, ldcomp, ws);
}

template <int NLEV>
cudaError_t launch_spec_pair(const SplitOperand &a, const SplitOperand &b, int64_t ldcomp, WsHeader *ws, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    for (int slot = 0; slot < 2 && e == cudaSuccess; ++slot) {
        const SplitOperand &o = slot ? b : a;
        const int gt = grid_for(((o.rows + kTile - 1) / kTile) * ((o.cols + kTile - 1) / kTile), 152 * 8);
        e = launch_spec<NLEV>(o.X, o.rows, o.cols, o.ldx, o.transpose, o.comps, ldcomp, o.plane, ws, slot, gt, st);
    }
    return e;
}

// Operands of together at most this many entries are split in one launch.
constexpr int64_t kSmallSplit = (int64_t)1 << 22;

}  // namespace

// Both operands of an FP64 GEMM: op(A) (M x K) into planes [s][M][ldcomp] and
// op(B) (K x N) into planes [s][N][ldcomp]; ta / tb: the stored matrix is read
// transposed to become the planes' rows (A stored K x M; B stored K x N).
// Small operands take one launch; larger ones the level maxima of both in one
// launch, a speculative pass each and the verifier of both.  Results are those
// of launch_split_f64 on A, then B.
cudaError_t launch_split_f64_gemm(const double *A, int64_t M, int64_t K, int64_t lda, const double *B, int64_t N,
                                  int64_t ldb, uint16_t *Ap, uint16_t *Bp, int64_t ldcomp, int32_t *vA_out,
                                  int32_t *vB_out, WsHeader *ws, cudaStream_t st, int nlev, bool ta, bool tb)
{
    if (nlev < 3 || nlev > 6) return cudaErrorInvalidValue;
    const SplitOperand a = {A, ta ? K : M, ta ? M : K, lda, Ap, M * ldcomp, vA_out, ta};
    const SplitOperand b = {B, tb ? K : N, tb ? N : K, ldb, Bp, N * ldcomp, vB_out, tb};
    if (M == 0 || N == 0 || K == 0) {
        cudaError_t e = launch_split_f64(A, a.rows, a.cols, lda, ta, Ap, ldcomp, vA_out, ws, 0, st, nlev);
        if (e == cudaSuccess) e = launch_split_f64(B, b.rows, b.cols, ldb, tb, Bp, ldcomp, vB_out, ws, 1, st, nlev);
        return e;
    }
    if ((M + N) * K <= kSmallSplit) {
        const int64_t tiles = ((M + kTile - 1) / kTile + (N + kTile - 1) / kTile) * ((K + kTile - 1) / kTile);
        switch (nlev) {
        case 3: return launch_small<3>(a, b, ldcomp, tiles, ws, st);
        case 4: return launch_small<4>(a, b, ldcomp, tiles, ws, st);
        case 5: return launch_small<5>(a, b, ldcomp, tiles, ws, st);
        default: return launch_small<6>(a, b, ldcomp, tiles, ws, st);
        }
    }
    // level-0 maxima: blocks shared in proportion to the entries, at most 152 x 8 in all
    const int64_t segA = a.rows * ((a.cols + 4 * kThreads - 1) / (4 * kThreads));
    const int64_t segB = b.rows * ((b.cols + 4 * kThreads - 1) / (4 * kThreads));
    const double fa = (double)(M * K) / (double)(M * K + K * N);
    int64_t nA = (int64_t)(152 * 8 * fa + 0.5), nB = 152 * 8 - nA;
    nA = nA < 1 ? 1 : (nA > segA ? segA : nA);
    nB = nB < 1 ? 1 : (nB > segB ? segB : nB);
    f64_max_gemm_kernel<<<(unsigned)(nA + nB), kThreads, 0, st>>>(A, a.rows, a.cols, lda, B, b.rows, b.cols, ldb, ws, nA,
                                                                  nB);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the speculative passes stay one launch per operand: in one launch the
    // row blocks would reserve the transposed blocks' shared memory (measured
    // 15-25 % slower)
    switch (nlev) {
    case 3: e = launch_spec_pair<3>(a, b, ldcomp, ws, st); break;
    case 4: e = launch_spec_pair<4>(a, b, ldcomp, ws, st); break;
    case 5: e = launch_spec_pair<5>(a, b, ldcomp, ws, st); break;
    default: e = launch_spec_pair<6>(a, b, ldcomp, ws, st); break;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    static int fits[64] = {};
    return launch_cooperative(f64_fix_pair_kernel, fits, (int64_t)152 * 8, st, a, b, ldcomp, ws, nlev);
}

}  // namespace emu
