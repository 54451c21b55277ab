// FP64-mode tensor-core product-sum, Eq. (fp64reconstruction) / Algorithm 2.
//
// Products are taken in Algorithm 2's diagonal order (outer loop); for each
// product K is walked in chunks of 256 (B_K of Section 6.1), every chunk
// partial fl32(A_i B_j) formed on the tensor cores in one of NBUF rotating
// TMEM buffers (all 512 columns).  Partials are exact: slice entries are
// integers times 2^(v-8) of magnitude <= 256, so a chunk partial is an
// integer of at most 2^24 units u = 2^(vA_i + vB_j - 16).
//
// Output tiles are 128 rows by BN = 256, 128 or 64 columns per CTA, or (PAIR)
// 256 x 256 or 256 x 128 on a cluster of two CTAs of one TPC with cta_group::2
// MMAs (M = 256): each CTA stages its 128 rows of the A slice and half of the B
// slice's BN rows, the leader (cluster rank 0) issues the MMAs for both, and each
// CTA's TMEM receives its 128 x BN part of the partials.  Every MMA brings
// its operands into the SM through shared memory and for one product at a
// time nothing is reused across MMAs, so wider tiles move fewer bytes per
// FLOP (per 2^20 FLOP: 8 KB as a pair, 12 KB at 256 columns, 16 KB at 128,
// 24 KB at 64); narrower ones give small results more CTAs.  All shapes share
// this source and give identical results.
//
// Eight or sixteen drain warps (two or four per TMEM lane quarter) sum
// partials exactly in FP32 registers: plain additions while the running sum
// stays below 2^24 u; past that the sum goes into the FP64 accumulator where
// that is exact (below), else a carry of the coarse part (multiples of 2^12 u)
// into a low word kept in C, or TwoSums whose errors are summed into that low
// word.
//
// Algorithm 2 adds every product once into the FP64 result, C <- fl64(C +
// A_i B_j), in diagonal order.  The accumulator is an FP64 buffer in the
// workspace, column-major within a 128-row stripe; a drain thread hands its
// exact sums (hi + lo) to the L2 as FP64 reductions (red.global.add.f64,
// round to nearest even; one thread's reductions to one address take effect
// in program order), so the SM's FP64 pipe (2 additions per clock) is not
// used.  An SM sends 25 bytes of reductions per clock (32 bytes of plain
// stores): 128 x 256 sums take 10,400 clocks, 4,000 of which the two TMEM
// buffers cover.  So products are grouped, and a group is reduced once, with
// the very bits that one reduction per product would give:
// - Products of one diagonal share their unit u when the levels fall in steps
//   of 8 (v_r = v_0 - 8r, the usual case), so their partials can run on in
//   one FP32 sum.
// - On the first diagonals every one of Algorithm 2's additions is exact
//   (all intermediate results are multiples of u below 2^53 u, known from K
//   alone: diag_exact), so their order does not matter and the sum of the
//   group is added instead.
// - On later diagonals each addition rounds to the unit in the last place g
//   of the result, which a group's products leave unchanged (except next to
//   a power of two, see below).  With H the accumulator before the group,
//   the running FP32 sum is rounded to multiples of g after each product, to
//   nearest, ties to even; the sum starts at g instead of 0 where H / g is
//   odd, so that even multiples of g in the sum are even multiples in the
//   result.  The last product's rounding is the reduction's own.  One byte
//   per element in shared memory holds g's rounding constant.
//   Elements of H within 2^-20 of a power of two (relative), or with too
//   coarse a g, are reduced after every product instead, and so are elements
//   whose running sum had to carry.
// Groups hold at most kGroupChunks chunk partials, so that running sums
// rarely reach 2^24 u (long K gains nothing: there a reduction is a small
// part of a product).  At 4096^3 with 21 products this takes 9 passes over
// the accumulator instead of 22.
//
// With levels per row / column (ROWCOL) every element has its own unit
// 2^(vA_i[row] + vB_j[col] - 16); columns' level exponents lie in shared
// memory and each running sum is compared with its own element's bound.
//
// Warp roles: warp 0 lane 0 issues TMA loads (64 of K of the A slice and the B
// slice per stage, 128 on 128 x 128 tiles), warp 1 owns TMEM and an elected lane
// of it issues the MMAs (PAIR: the leader's), warps 4-19 (4-11 on 256 columns)
// drain and reduce.  Every wait is bounded and reports EMU_FLAG_TIMEOUT instead
// of hanging.
#pragma once

#include "launchers.cuh"
#include "prodsum_f64_common.cuh"

namespace emu {

namespace {

template <int BN_, bool PAIR>
struct F64WCfgT {
    static constexpr int BN = BN_, KB = 64, NBUF = BN == 256 ? 2 : 4;
    static constexpr int BH = PAIR ? BN / 2 : BN;                       // B rows staged by this CTA
    static constexpr int A_TILE = kBM * KB * 2, B_TILE = BH * KB * 2;   // 16 KB + 8 to 32 KB
    // K-blocks of 64 per stage.  The 128 x 128 tiles run where few CTAs are at work and
    // wait for operands: with two blocks (adjacent 128-byte pieces of every plane
    // row requested together) 1024 x 1024 x 32768 / 21 takes 3090 us, with one 3620.
    static constexpr int SUB = BN == 128 && !PAIR ? 2 : 1, KSPAN = KB * SUB;
    static constexpr int STAGE = SUB * (A_TILE + B_TILE);
    static constexpr int STAGES = 196608 / STAGE;                        // 4 x 48, 3 x 64, 6 x 32 or 8 x 24 KB
    static constexpr int B_OFF = SUB * A_TILE;                           // A blocks, then B blocks
    static constexpr uint32_t SWZ = 2u, SBO = 1024u;                     // 128-byte swizzle
    // warpgroup 0: TMA producer (warp 0), MMA issuer + TMEM owner (warp 1), two
    // idle warps; then the drain warps: sixteen of BN / 4 columns each, or with
    // 256 columns eight of 128, whose threads have registers for their sums
    // (sixteen threads' worth of addresses and temporaries beside 64 sums did not
    // fit in 112 registers).  Spills: none but in the row/column instances (74
    // and 66 bytes at 256 columns, 16 at 256 x 128).
    static constexpr int FIRST_DRAIN = 4, DRAIN_WARPS = BN == 256 ? 8 : 16;
    static constexpr int DRAIN_THREADS = 32 * DRAIN_WARPS, THREADS = 128 + DRAIN_THREADS;
    static constexpr int COLS = BN / (DRAIN_WARPS / 4);                 // columns per drain thread
    // shared memory: stages; one rounding byte per element, [COLS / 4] words per
    // drain thread; level exponents of the columns; barriers (full/empty per
    // stage, tfull/tempty per buffer, done), the TMEM address slot and the
    // levels' summary
    static constexpr int CODE_OFF = STAGES * STAGE;
    static constexpr int LVL_OFF = CODE_OFF + kBM * BN;
    static constexpr int BAR_OFF = LVL_OFF + BN * 4;
    static constexpr int NBARS = 2 * STAGES + 2 * NBUF + 3;   // done, and two between the CTAs of a duo
    static constexpr int SMEM = BAR_OFF + 256 + 1024;
    // Register split: the launch reserves 384 x 168 = 128 x 40 (control) + 256 x
    // 232 (drain), or 640 x 96 = 128 x 32 + 512 x 112.
    static constexpr int REG_CTRL = BN == 256 ? 40 : 32, REG_DRAIN = BN == 256 ? 232 : 112,
                         REG_LAUNCH = BN == 256 ? 168 : 96;
    static_assert(NBUF * BN <= 512, "TMEM budget");
    static_assert(kKChunk % KSPAN == 0, "a K-chunk is a whole number of stages");
    static_assert(8 * NBARS + 8 + 20 <= 256, "barrier area");
    static_assert(SMEM <= 232448, "shared memory per CTA");
    static_assert(128 * REG_CTRL + DRAIN_THREADS * REG_DRAIN <= THREADS * REG_LAUNCH,
                  "setmaxnreg split exceeds the registers reserved at launch");
    static_assert(COLS % 16 == 0, "drain columns come in groups of 16");
    static_assert(DRAIN_WARPS * 8192 <= STAGES * STAGE, "TMA epilogue staging exceeds the stages");
};

// Largest number of chunk partials in one group of products: a sum of 192
// partials of uniform random slices stays below 2^24 u with 4.5 standard
// deviations to spare.
constexpr int kGroupChunks = 192;
// Coarsest g / u that a group's running sum is rounded to (log2): the start
// value g and a running sum below (1 - 2^-4) 2^24 u then sum to less than 2^24 u.
constexpr int kMaxRoundBits = 20;

// Every addition of Algorithm 2 up to the end of diagonal l is exact, with
// levels in steps of 8: the products' magnitudes sum to at most K 2^16 u_0
// (1 + 2 / 2^8 + 3 / 2^16 + ...) <= K 2^16 u_0 259 / 256, and all are multiples
// of u_l = u_0 / 2^(8 l), so results below 2^53 u_l are exact.
__device__ __forceinline__ bool diag_exact(int K, int l)
{
    return l <= 5 && (long long)K * 259 <= (1ll << (45 - 8 * l));
}

template <int THREADS>
__device__ __forceinline__ void drain_barrier()
{
    asm volatile("barrier.cta.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// max(|a|, |b|, |c|)
__device__ __forceinline__ float max3_abs(float a, float b, float c)
{
    float r;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// FP64 reduction in L2: *p <- fl64(*p + x), round to nearest even.
__device__ __forceinline__ void red_add_f64(double *p, double x)
{
    asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"(x) : "memory");
}

__device__ __forceinline__ double ld_cg_f64(const double *p)
{
    double x;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(x) : "l"(p) : "memory");
    return x;
}

// Summary of the level exponents a CTA's elements use (ROWCOL; shared memory).
struct LevelSummary {
    int lock;                    // every vector's levels fall in steps of 8
    int min_a, max_a, min_b, max_b;
};

__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[32]) { tmem_ld32(taddr, r); }
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[16]) { tmem_ld16(taddr, r); }

// Levels v[0 .. d-1] (stride apart) of one matrix or vector: how far the
// finest level lies below v_0 - 8r (0: steps of 8 until the residual is zero).
__device__ __forceinline__ int level_gap(const int32_t *v, int64_t stride, int d, int v0)
{
    int w = 0;
    for (int r = 1; r < d; ++r) {
        const int vr = v[r * stride];
        if (vr != kZeroLevel) w = max(w, v0 - 8 * r - vr);
    }
    return w;
}

// Levels per matrix in steps of 8 whose units, with the rounding constants (2^-25 u
// to 2^(23 + kMaxRoundBits) u), are normal; e0 = vA_0 + vB_0 then.
__device__ __forceinline__ bool matrix_lock(const int32_t *vA, const int32_t *vB, int d, int &e0)
{
    if (!vA || vA[0] == kZeroLevel || vB[0] == kZeroLevel) return false;
    e0 = vA[0] + vB[0];
    return level_gap(vA, 1, d, vA[0]) == 0 && level_gap(vB, 1, d, vB[0]) == 0 && e0 <= 100 && e0 + 8 - 8 * (d - 1) >= -76;
}

// Number of diagonals of nprod products.
__device__ __forceinline__ int diagonals_of(int nprod) { return nprod == 6 ? 3 : nprod == 10 ? 4 : nprod == 15 ? 5 : 6; }

// CTA of a duo that computes product q: whole diagonals each, 3 + 3 of 6 products,
// 5 + 5 of the first 10, and the first CTA any later ones.
__device__ __forceinline__ uint32_t duo_owner(int q, int nprod)
{
    return nprod == 6 ? (q < 3 ? 0u : 1u) : (q == 0 || q >= 6 ? 0u : 1u);
}

// Every lane's global writes and reductions so far become visible to the other
// CTA of the duo when its wait on `bar` (count: the drain warps) completes.
__device__ __forceinline__ void signal_duo(uint32_t bar, uint32_t rank)
{
    __threadfence();
    __syncwarp();
    if (lane_id() == 0)
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(peer_addr(bar, rank ^ 1u))
                     : "memory");
    __syncwarp();
}
// Bounded wait for phase 0 of a duo's barrier: mbar_wait's polling with an
// acquire at cluster scope, since the writes it orders are the other CTA's (a
// wait that acquires at CTA scope does not synchronise with that CTA's release).
__device__ __forceinline__ bool wait_duo(uint32_t bar, uint32_t *flags)
{
    auto poll = [bar] {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar)
            : "memory");
        return ok != 0;
    };
    bool ok = poll();
    const unsigned long long t0 = ok ? 0 : globaltimer_ns();
    for (uint32_t it = 1; !ok && it < (1u << 30); ++it) {
        ok = poll();
        if (!ok && (it & 63u) == 0u && globaltimer_ns() - t0 > kWaitLimitNs) break;
    }
    if (!ok) atomicOr(flags, (uint32_t)EMU_FLAG_TIMEOUT);
    ok = __all_sync(0xFFFFFFFFu, ok);
    __threadfence();
    return ok;
}

// Code byte of an element while its running sum is rounded to multiples of g =
// 2^n u: bits 0-6 hold n + 48 (kCodeKeep where g <= u: nothing to round;
// kCodeEach: reduced after every product), bit 7 says that the sum started
// at g.  bound_bits: bits of the FP32 value 2^24 u.  Adding and subtracting the
// constant 2^23 g rounds |x| < 2^24 u to the grid, to nearest, ties to even.
// kCodeKeep gives 2^-25 u, a quarter of the last place of the smallest nonzero
// sum u, which leaves every sum unchanged (2^-24 u and above would not: at the
// power of two of which it is half the last place, the subtraction steps
// below the binade).  A sum rounded to zero may become -0, which adds like +0.
constexpr uint32_t kCodeKeep = 0, kCodeEach = 1;
__device__ __forceinline__ uint32_t code_byte(uint32_t word, int k) { return (word >> (8 * k)) & 0xFFu; }
// Exponent fields of the four rounding constants of a code word: its bytes
// plus the field of 2^-25 u, bound_bits >> 23 minus 49.  No byte may borrow from or
// carry into the next, or be 255.  With lock, e0 + 8 - 8 (d - 1) >= -76 and e0 <= 100
// give 51 <= bound_bits >> 23 <= 227 on the diagonals that round (1 .. d - 1), and the
// largest byte is 227 - 49 + 48 + kMaxRoundBits = 246; the all-zero columns' word
// (level exponent 60, whatever the row) stays between 51 and 247 and its bytes are
// kCodeKeep, the all-zero rows take the level of another row.
__device__ __forceinline__ uint32_t round_fields(uint32_t word, uint32_t bound_bits)
{
    return (word & 0x7F7F7F7Fu) + ((bound_bits >> 23) - 49u) * 0x01010101u;
}
__device__ __forceinline__ float round_to(float x, uint32_t fields, int k)
{
    const float m = __uint_as_float((k == 3 ? fields >> 1 : fields << (23 - 8 * k)) & 0x7F800000u);
    const float r = __fsub_rn(__fadd_rn(fabsf(x), m), m);
    return __uint_as_float(__float_as_uint(r) | (__float_as_uint(x) & 0x80000000u));
}
// g of a code with bit 7 set (n >= 1), 0 otherwise: what the sum started at.
__device__ __forceinline__ float start_of(uint32_t code, uint32_t bound_bits)
{
    return (code & 0x80u) ? __uint_as_float(bound_bits - (72u << 23) + ((code & 0x7Fu) << 23)) : 0.0f;
}

// TAIL: add the merged tail T (an M x N FP32 matrix) once after the last product.
// vA, vB and T are written by the kernels before this one, which may still run when
// it starts: not __restrict__, so that no load of them moves above griddep_wait.
// wide_first >= 0 (pairs with BN = 128): this launch takes the 256 x 128 halves
// of the 256 x 256 tiles from raster index wide_first on.
// DUO: a cluster of two CTAs shares a tile's products.  While every addition up to
// the fourth diagonal is exact (diag_exact; levels in steps of 8), sums may reach
// the accumulator in any order, so the second CTA takes half of the first six or
// ten products; the first stores product 0 before the second reduces, the later
// diagonals (first CTA) wait for both halves, and each CTA writes half of the
// tile to C.  Otherwise the first CTA does everything.
template <int BN, bool ROWCOL, bool TAIL, bool PAIR, bool DUO>
__global__ void __launch_bounds__(F64WCfgT<BN, PAIR>::THREADS, 1)
prodsum_f64w_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmC, int c_tma, int M, int N, int K, int nprod,
                    const int32_t *vA, const int32_t *vB, double *__restrict__ C, int64_t ldc, double *__restrict__ acc,
                    uint32_t *flags, const float *T, int64_t ldt, int wide_first)
{
    using Cfg = F64WCfgT<BN, PAIR>;
    static_assert(!DUO || (!PAIR && !ROWCOL && !TAIL), "duos: one CTA per MMA, levels per matrix, no tail");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_raw + (base - raw);
    const uint32_t full0 = base + Cfg::BAR_OFF, empty0 = full0 + 8u * Cfg::STAGES;
    const uint32_t tfull0 = empty0 + 8u * Cfg::STAGES, tempty0 = tfull0 + 8u * Cfg::NBUF;
    const uint32_t done_bar = tempty0 + 8u * Cfg::NBUF;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + Cfg::BAR_OFF + 8 * Cfg::NBARS);
    LevelSummary *lsum = reinterpret_cast<LevelSummary *>(base_ptr + Cfg::BAR_OFF + 8 * Cfg::NBARS + 8);

    const int warp = threadIdx.x >> 5, lane = lane_id();
    const uint32_t rank = PAIR || DUO ? cluster_rank() : 0u;
    const uint32_t duo_first = done_bar + 8u, duo_done = done_bar + 16u;   // product 0 stored; the other CTA's sums reduced
    const int tiles_n = (N + BN - 1) / BN;
    int tm, tn;
    if constexpr (PAIR) {                             // the pair's 256 rows: this CTA takes half `rank`
        int tp;
        const int pair = (int)(blockIdx.x >> 1), tiles_p = (M + 2 * kBM - 1) / (2 * kBM);
        if (BN == 128 && wide_first >= 0) {
            // the two column halves of each 256 x 256 tile that a last, partial wave would have taken
            int tnw;
            tile_coords(wide_first + (pair >> 1), tiles_p, (N + 255) / 256, tp, tnw);
            tn = 2 * tnw + (pair & 1);
            if (tn >= tiles_n) return;                // past the last column (both CTAs)
        } else {
            tile_coords(pair, tiles_p, tiles_n, tp, tn);
        }
        tm = 2 * tp + (int)rank;
    } else {
        tile_coords((int)(DUO ? blockIdx.x >> 1 : blockIdx.x), (M + kBM - 1) / kBM, tiles_n, tm, tn);
    }
    const int m0 = tm * kBM, n0 = tn * BN;
    const int nch = (K + kKChunk - 1) / kKChunk;

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::STAGES; ++s) { mbar_init(full0 + 8u * s, 1); mbar_init(empty0 + 8u * s, 1); }
        // a pair's TMEM buffers are released by the drain warps of both CTAs,
        // on the leader's barriers
        for (int b = 0; b < Cfg::NBUF; ++b) {
            mbar_init(tfull0 + 8u * b, 1);
            mbar_init(tempty0 + 8u * b, (PAIR ? 2 : 1) * Cfg::DRAIN_WARPS);
        }
        mbar_init(done_bar, 1);
        mbar_init(duo_first, Cfg::DRAIN_WARPS);
        mbar_init(duo_done, Cfg::DRAIN_WARPS);
        fence_mbar_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        *lsum = {1, 0x7FFFFFFF, -0x7FFFFFFF, 0x7FFFFFFF, -0x7FFFFFFF};
    }
    if constexpr (PAIR) {
        __syncthreads();
        cluster_sync();                               // both CTAs' barriers initialised
        if (warp == 1) tmem_alloc_pair(smem_u32((const void *)tmem_slot), 512);
    } else {
        if (warp == 1) { tmem_alloc(smem_u32((const void *)tmem_slot), 512); tmem_relinquish(); }
    }
    if constexpr (DUO) {
        __syncthreads();
        cluster_sync();                               // both CTAs' barriers initialised
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // set-up above overlaps the end of the kernel that wrote the planes and levels
    // (launched as its programmatic dependent)
    griddep_wait();
    int e0 = 0;
    bool lock = false;
    if constexpr (!ROWCOL) lock = matrix_lock(vA, vB, diagonals_of(nprod), e0);
    const bool duo = DUO && lock && diag_exact(K, min(3, diagonals_of(nprod) - 1));
    // whether this CTA computes product q
    auto mine_q = [&](int q) { return !DUO || (duo ? duo_owner(q, nprod) == rank : rank == 0); };

    if (warp < Cfg::FIRST_DRAIN) {
      regs_dec<Cfg::REG_CTRL>();
      if (warp == 0 && lane == 0) {
        // ---------------- TMA producer: for product, for chunk, for stage (KSPAN of K) of the chunk
        int L = 0, s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int q = 0; q < nprod && ok; ++q) {
            if (!mine_q(q)) continue;
            const int ia = kDiag[q][0], jb = kDiag[q][1];
            for (int c = 0; c < nch && ok; ++c) {
                const int kbs = min(kKChunk / Cfg::KSPAN, (K - c * kKChunk + Cfg::KSPAN - 1) / Cfg::KSPAN);
                for (int u = 0; u < kbs; ++u, ++L) {
                    if (!(ok = mbar_wait(empty0 + 8u * s, ph ^ 1u, flags))) break;
                    const uint32_t st = base + (uint32_t)(s * Cfg::STAGE), fb = full0 + 8u * s;
                    const int k0 = c * kKChunk + u * Cfg::KSPAN;
                    if constexpr (PAIR) {
                        // both CTAs' copies are counted on the leader's full barrier
                        const uint32_t fl = peer_addr(fb, 0);
                        if (rank == 0) mbar_arrive_expect_tx(fb, 2 * Cfg::STAGE);
                        tma_load_3d_pair(st, &tmA, fl, k0, m0, ia);
                        tma_load_3d_pair(st + Cfg::B_OFF, &tmB, fl, k0, n0 + (int)rank * Cfg::BH, jb);
                    } else {
                        const int blocks = Cfg::SUB == 1 || k0 + Cfg::KB < K ? Cfg::SUB : 1;   // a block wholly past K is left out
                        mbar_arrive_expect_tx(fb, (uint32_t)(blocks * (Cfg::A_TILE + Cfg::B_TILE)));
                        for (int h = 0; h < blocks; ++h) {
                            tma_load_3d(st + h * Cfg::A_TILE, &tmA, fb, k0 + h * Cfg::KB, m0, ia);
                            tma_load_3d(st + Cfg::B_OFF + h * Cfg::B_TILE, &tmB, fb, k0 + h * Cfg::KB, n0, jb);
                        }
                    }
                    if (++s == Cfg::STAGES) { s = 0; ph ^= 1u; }
                }
            }
        }
        if (!ok) {
            if (!PAIR || rank == 0) {
                drain_inflight(full0, Cfg::STAGES, L, flags);
            } else {
                // the peer's copies complete on the leader's barriers, which it
                // cannot observe: give them 200 us before the CTA winds down
                const unsigned long long t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) {}
            }
        }
      } else if (warp == 1 && (!PAIR || rank == 0)) {
        // ---------------- MMA issuer (a pair's leader): one chunk partial into buffer t % NBUF.
        // The whole warp walks the loop (waits decided by vote), one elected lane
        // issues: control flow and operands are then uniform, and the descriptors
        // need no move from vector to uniform registers before every MMA.
        constexpr uint32_t idesc = make_idesc_bf16(PAIR ? 2 * kBM : kBM, BN);
        // descriptors of stage 0; stage s, block h and 16-wide K step kk of it add their byte
        // offsets / 16
        const uint64_t ad0 = make_sdesc(base, Cfg::SBO, Cfg::SWZ), bd0 = make_sdesc(base + Cfg::B_OFF, Cfg::SBO, Cfg::SWZ);
        int s = 0, b = 0, c = 0;
        uint32_t ph = 0, tph = 0;
        bool ok = true;
        int nmine = 0;                                // products of this CTA
        for (int q = 0; q < nprod; ++q) nmine += mine_q(q) ? 1 : 0;
        for (int t = 0; t < nmine * nch && ok; ++t) {
            const int kbs = min(kKChunk / Cfg::KSPAN, (K - c * kKChunk + Cfg::KSPAN - 1) / Cfg::KSPAN);
            if (!(ok = __all_sync(0xFFFFFFFFu, mbar_wait(tempty0 + 8u * b, tph ^ 1u, flags)))) break;
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(b * BN);
            for (int u = 0; u < kbs; ++u) {
                if (!(ok = __all_sync(0xFFFFFFFFu, mbar_wait(full0 + 8u * s, ph, flags)))) break;
                tc_fence_after();
                const uint32_t off = (uint32_t)(s * (Cfg::STAGE / 16));
                const uint64_t ad = ad0 + off, bd = bd0 + off;
                const bool second = Cfg::SUB == 1 || c * kKChunk + u * Cfg::KSPAN + Cfg::KB < K;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < Cfg::KSPAN / 16; ++kk) {
                        // K step kk lies 32 bytes a step into its 64-wide block
                        const int h = kk / (Cfg::KB / 16), o = 2 * (kk % (Cfg::KB / 16));
                        if (h > 0 && !second) break;
                        const uint64_t a = ad + h * (Cfg::A_TILE / 16) + o, w = bd + h * (Cfg::B_TILE / 16) + o;
                        if constexpr (PAIR) mma_bf16_pair(d, a, w, idesc, (u | kk) != 0);
                        else mma_bf16(d, a, w, idesc, (u | kk) != 0);
                    }
                    if constexpr (PAIR) mma_commit_pair(empty0 + 8u * s);
                    else mma_commit(empty0 + 8u * s);
                    if (u + 1 == kbs) {
                        if constexpr (PAIR) mma_commit_pair(tfull0 + 8u * b);
                        else mma_commit(tfull0 + 8u * b);
                    }
                }
                __syncwarp();
                if (++s == Cfg::STAGES) { s = 0; ph ^= 1u; }
            }
            if (++b == Cfg::NBUF) { b = 0; tph ^= 1u; }
            if (++c == nch) c = 0;
        }
        if (elect_one()) {
            if constexpr (PAIR) mma_commit_pair(done_bar);
            else mma_commit(done_bar);
        }
        __syncwarp();
        (void)mbar_wait(done_bar, 0, flags);
      }
    } else {
        regs_inc<Cfg::REG_DRAIN>();
        // ---------------- drain: exact sums of groups of products, reduced into the accumulator in L2
        const int quarter = warp & 3;                                    // TMEM lanes 32*quarter ..
        const int cq = (warp - Cfg::FIRST_DRAIN) >> 2;                   // column quarter
        const int r = quarter * 32 + lane;                               // tile row of this thread
        const int dt = (int)threadIdx.x - 32 * Cfg::FIRST_DRAIN;         // 0 .. DRAIN_THREADS - 1
        const uint32_t tcol = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(cq * Cfg::COLS);
        const int row = m0 + r;
        double *crow = C + (int64_t)row * ldc + n0 + cq * Cfg::COLS;
        const int lim = row < M ? N - (n0 + cq * Cfg::COLS) : 0;        // valid columns of this thread
        // this thread's elements of the accumulator: 128-row stripes, column-major, rows
        // of 256-column tiles whatever tile shape runs
        double *tacc = acc + ((size_t)tm * ((size_t)((N + 255) / 256) * 256u) + (size_t)(n0 + cq * Cfg::COLS)) * kBM + r;
        // a pair's second CTA may lie wholly below the last row, past the
        // accumulator's stripes: its threads touch neither the accumulator nor C
        const bool live = !PAIR || row < M;
        // where code_columns reads the accumulator: rows past M read the first stripe (any
        // address of it will do, the value is dropped)
        const double *hacc = live ? tacc : acc;
        // the low words live in one half of this thread's C words until their group is reduced
        float *lrow = reinterpret_cast<float *>(crow) + (DUO ? rank : 0u);
        uint32_t *codes = reinterpret_cast<uint32_t *>(base_ptr + Cfg::CODE_OFF) + dt;   // word w at w * DRAIN_THREADS
        int *lvl = reinterpret_cast<int *>(base_ptr + Cfg::LVL_OFF) + cq * Cfg::COLS;

        // Levels.  lock: the units of a diagonal's products agree, and they and the rounding
        // constants are normal (matrix_lock).
        const int d = diagonals_of(nprod);
        int row_e = 0, row_gap = 0, lvl_min = 0;
        if constexpr (ROWCOL) {
            // lvl[column]: (v_0 - gap + 68) << 23, so that adding (v_0 - gap + 67) << 23 of the
            // row gives the bits of the FP32 bound 2^24 u (integer order is the order of
            // magnitudes); an all-zero vector has no bound.  In the domain v_r >= -126 holds
            // for every level that is not zero; clamping at 60 only lowers the bound.
            for (int x = dt; x < BN; x += Cfg::DRAIN_THREADS) {
                const int col = n0 + x;
                int f = 0x40000000;
                if (col < N && vB[col] != kZeroLevel) {
                    const int v0 = vB[col], w = level_gap(vB + col, N, d, v0);
                    f = (min(max(v0 - w, -170), 60) + 68) << 23;
                    if (w > 0) atomicAnd(&lsum->lock, 0);
                    atomicMin(&lsum->min_b, v0);
                    atomicMax(&lsum->max_b, v0);
                }
                reinterpret_cast<int *>(base_ptr + Cfg::LVL_OFF)[x] = f;
            }
            const int v0 = row < M ? vA[row] : kZeroLevel;
            if (v0 != kZeroLevel) {
                row_gap = level_gap(vA + row, M, d, v0);
                row_e = v0;
                if (cq == 0) {
                    if (row_gap > 0) atomicAnd(&lsum->lock, 0);
                    atomicMin(&lsum->min_a, v0);
                    atomicMax(&lsum->max_a, v0);
                }
            }
            drain_barrier<Cfg::DRAIN_THREADS>();
            lock = lsum->lock != 0 && lsum->max_a <= 60 && lsum->max_b <= 60 && lsum->max_a + lsum->max_b <= 100 &&
                   lsum->max_a >= lsum->min_a && lsum->max_b >= lsum->min_b &&
                   lsum->min_a + lsum->min_b + 8 - 8 * (d - 1) >= -76;
            // An all-zero row has no level: take one of the range that lock has checked, so
            // that the row's bounds and rounding constants are normal numbers for every column
            // (with level 0 a constant's exponent could be all ones, and 0 + inf - inf a NaN).
            if (lock && v0 == kZeroLevel) row_e = lsum->min_a;
            lvl_min = 0x7FFFFFFF;
#pragma unroll 4
            for (int j = 0; j < Cfg::COLS; ++j) lvl_min = min(lvl_min, lvl[j]);
        }
        const int group = lock ? max(1, kGroupChunks / nch) : 1;          // most products in a group

        // low words of 16 columns from column h of this thread (zero where there are none)
        auto load_low = [&](int h, bool have, float (&lo)[16]) {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) lo[jj] = (have && h + jj < lim) ? lrow[2 * (h + jj)] : 0.0f;
        };

        float hi[Cfg::COLS];
        uint32_t dirty = 0;                                   // 16-column groups whose low part lives in C; from bit
                                                              // 16 on, those whose sums of product 0 have begun
                                                              // to be in the accumulator
        bool each = false;                                    // some element is reduced after every product
        int diag = 0, in_diag = 0, in_group = 0;              // product q: diagonal, place in it and in its group
        bool ok = true;
        int t0 = 0;                                           // chunk partials before product q
        bool first_in = !duo || rank == 0, others_in = !duo;  // what this CTA has waited for
        for (int q = 0; q < nprod && ok; ++q) {
            if (!mine_q(q)) {
                if (in_diag++ == diag) { ++diag; in_diag = 0; }
                continue;
            }
            if (DUO && diag >= 4 && !others_in) {
                // from here on the order of additions matters
                if (!(ok = wait_duo(duo_done, flags))) break;
                others_in = true;
            }
            const bool exact = diag_exact(K, diag);
            // rounding applies when the group goes on past its first product
            const bool rounds = !exact && group > 1 && diag > 0;
            if (in_group == 0) {
#pragma unroll
                for (int j = 0; j < Cfg::COLS; ++j) hi[j] = 0.0f;
                dirty = 0;
                each = false;
            }
            // row part of the bound's bits (ROWCOL), and the bound itself (the smallest of the
            // thread's elements for ROWCOL)
            const int abits = (min(max(row_e - row_gap, -170), 60) + 67 - 8 * diag) << 23;
            const float bound = ROWCOL ? __int_as_float(min(max(lvl_min + abits, 0), 0x7F800000))
                                       : exact_bound(vA, vB, kDiag[q][0], kDiag[q][1]);
            // bits of 2^24 u with element j's own unit on this diagonal (with lock)
            auto bits_of = [&](int j) { return (uint32_t)(ROWCOL ? lvl[j] + abits : (e0 + 135 - 8 * diag) << 23); };
            // while a group's sums are rounded they stay below (1 - 2^-4) 2^24 u (kMaxRoundBits)
            const float limit = rounds ? 0.9375f * bound : bound;
            const int abits_lim = rounds ? abits - 0x100000 : abits;
            // What happens to sums that would reach 2^24 u.
            // 2: they are reduced into the accumulator, while every addition to it is exact.
            // 1: a carry instead of TwoSums (0), when all elements share the unit u = 2^-24
            // bound (levels per matrix) and the split constant 1.5 * 2^35 u is finite.  A
            // carry splits the running sum and the partial (each at most 2^24 u) at
            // multiples of 2^12 u and moves both coarse parts (together at most
            // 2^25 u) to the low word in C, which stays exact below 2^36 u, i.e. for
            // up to 2^11 carries.
            const int past = exact && lock && first_in ? 2 : !ROWCOL && bound > 0.0f && bound <= 0x1p116f && nch <= 2048 ? 1 : 0;
            const int a_row = (ROWCOL && row < M) ? vA[(int64_t)kDiag[q][0] * M + row] : kZeroLevel;
            // The first product of a group whose sums are rounded: g of elements j0 .. j0 + HC - 1
            // from the accumulator H (every earlier product is in it; this thread's own
            // reductions, so they precede the loads).  HC columns per chunk, from the third
            // chunk on, in time the warp would wait for partials, and the rest after the
            // last chunk.  On pairs without branches: with a branch per element (a load
            // for live rows only, the cases of the code) the loads were not in flight
            // together and 128 columns took 64,000 clocks, now 20,000 (21 products of
            // 16384 x 256 x 256: 298 -> 259 us, of 3000 x 3000 x 300: 440 -> 358).  Elsewhere
            // every row is live, the loads stand together before the branches on the
            // codes, and without those branches ptxas spreads them (128 x 30000 x 300: 283 ->
            // 297 us).
            constexpr int HC = BN == 256 ? 16 : 8;
            auto code_columns = [&](int j0) {
                double hd[HC];
#pragma unroll
                for (int k = 0; k < HC; ++k) hd[k] = ld_cg_f64(hacc + (j0 + k) * kBM);
#pragma unroll
                for (int k = 0; k < HC; ++k) hd[k] = live ? hd[k] : 0.0;
#pragma unroll
                for (int w = 0; w < HC / 4; ++w) {
                    uint32_t cw = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const double h = hd[4 * w + k];
                        const uint32_t xh = (uint32_t)__double2hiint(h) & 0x7FFFFFFFu;
                        // g = 2^n u: exponent fields e - 1023 - 52 - (field of 2^24 u - 127 - 24)
                        const int n = (int)(xh >> 20) - 924 - (int)(bits_of(j0 + 4 * w + k) >> 23);
                        const uint32_t mh = xh & 0xFFFFFu;
                        const bool edge = ((n >= 0) & (mh == 0xFFFFFu)) | ((n > 0) & (mh == 0u)) | (n > kMaxRoundBits);
                        const uint32_t odd = ((uint32_t)__double2loint(h) & 1u) << 7;
                        uint32_t code = kCodeKeep;
                        if constexpr (PAIR) {
                            each |= edge;
                            code = edge ? kCodeEach : n > 0 ? (uint32_t)(n + 48) | odd : kCodeKeep;
                        } else if (edge) {
                            code = kCodeEach;
                            each = true;
                        } else if (n > 0) {
                            code = (uint32_t)(n + 48) | odd;
                        }
                        cw |= code << (8 * k);
                    }
                    codes[(j0 / 4 + w) * Cfg::DRAIN_THREADS] = cw;
                }
            };
            int coded = rounds && in_group == 0 && in_diag != diag ? 0 : Cfg::COLS;
            for (int c = 0; c < nch; ++c) {
                const int t = t0 + c, b = t % Cfg::NBUF;
                ok = mbar_wait(tfull0 + 8u * b, (uint32_t)((t / Cfg::NBUF) & 1), flags);
                __syncwarp();
                if (!ok) break;
                tc_fence_after();
                // LD columns at a time, the next LD on their way from TMEM meanwhile.  The sums
                // replace the partials in their registers; the largest magnitudes are found in
                // independent chains and voted on once (one chain of compares, each waiting
                // for the last, and a vote per 16 columns took as long as the MMAs).
                constexpr int LD = Cfg::COLS >= 32 ? 32 : 16;
                uint32_t pv[2][LD];
                tmem_ld_cols(tcol + (uint32_t)(b * BN), pv[0]);
#pragma unroll
                for (int hl = 0; hl < Cfg::COLS; hl += LD) {
                    uint32_t (&ps)[LD] = pv[(hl / LD) & 1];
                    tmem_ld_wait();
                    if (hl + LD < Cfg::COLS) tmem_ld_cols(tcol + (uint32_t)(b * BN + hl + LD), pv[(hl / LD + 1) & 1]);
                    bool big[LD / 16];
#pragma unroll
                    for (int g = 0; g < LD; g += 16) {
                        if constexpr (ROWCOL) {
                            int mx[4] = {-0x7FFFFFFF, -0x7FFFFFFF, -0x7FFFFFFF, -0x7FFFFFFF};
#pragma unroll
                            for (int j = g; j < g + 16; j += 4) {
                                const int4 f = *reinterpret_cast<const int4 *>(lvl + hl + j);
                                const int lv[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    ps[j + k] = __float_as_uint(__fadd_rn(hi[hl + j + k], __uint_as_float(ps[j + k])));
                                    mx[k] = max(mx[k], (int)(ps[j + k] & 0x7FFFFFFFu) - lv[k]);
                                }
                            }
                            big[g / 16] = max(max(mx[0], mx[1]), max(mx[2], mx[3])) >= abits_lim;
                        } else {
                            float mx[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                            for (int j = g; j < g + 16; j += 2) {
                                const float s0 = __fadd_rn(hi[hl + j], __uint_as_float(ps[j]));
                                const float s1 = __fadd_rn(hi[hl + j + 1], __uint_as_float(ps[j + 1]));
                                mx[(j >> 1) & 3] = max3_abs(mx[(j >> 1) & 3], s0, s1);
                                ps[j] = __float_as_uint(s0);
                                ps[j + 1] = __float_as_uint(s1);
                            }
                            big[g / 16] = !(max3_abs(max3_abs(mx[0], mx[1], mx[2]), mx[3], 0.0f) < limit);
                        }
                    }
                    if (!__any_sync(0xFFFFFFFFu, big[0] || big[LD / 16 - 1])) {
#pragma unroll
                        for (int j = 0; j < LD; ++j) hi[hl + j] = __uint_as_float(ps[j]);
                        continue;
                    }
#pragma unroll
                    for (int g = 0; g < LD; g += 16) {
                    const int h = hl + g;
                    uint32_t p16[16];                             // the partials again
                    if (!__any_sync(0xFFFFFFFFu, big[g / 16])) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) hi[h + j] = __uint_as_float(ps[g + j]);
                        continue;
                    }
                    if (past == 2) {
                        // some sum would reach 2^24 u, and every addition to the accumulator is
                        // exact up to this diagonal: reduce the sums now and go on from the
                        // partials (read again from TMEM).  Non-negative operands come here every
                        // few chunks of product 0; the accumulator's columns are 256 contiguous
                        // bytes of a warp, where the low words below are 32 sectors each way
                        // (4096 x 4096 x 2048 / 6, entries in [1/2, 1]: 2058 -> 580 us).
                        const bool store = q == 0 && !((dirty >> (16 + h / 16)) & 1u);
#pragma unroll
                        for (int j = h; j < h + 16; ++j) {
                            const double x = widen_normal(hi[j]);
                            if (live && store) tacc[j * kBM] = x;
                            if (live && !store) red_add_f64(tacc + j * kBM, x);
                        }
                        if (q == 0) dirty |= 0x10000u << (h / 16);
                        tmem_ld16(tcol + (uint32_t)(b * BN + h), p16);
                        tmem_ld_wait();
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj) hi[h + jj] = __uint_as_float(p16[jj]);
                        continue;
                    }
                    tmem_ld16(tcol + (uint32_t)(b * BN + h), p16);
                    tmem_ld_wait();
                    if (past == 1) {
                        // rare: some sum would reach 2^24 u.  Split the running sum and
                        // the partial (read again from TMEM) at multiples of 2^12 u by the add-subtract
                        // projection; the coarse parts go to the low word in C, the
                        // remainders (below 2^12 u) restart the running sum.  All exact.
                        const bool was = (dirty >> (h / 16)) & 1u;
                        dirty |= 1u << (h / 16);
                        const float cm = 3072.0f * bound;         // 1.5 * 2^35 u
                        float lo[16];                             // all loads before the first store
                        load_low(h, was, lo);
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj) {
                            const int j = h + jj;
                            const float p = __uint_as_float(p16[jj]);
                            const float h1 = __fsub_rn(__fadd_rn(hi[j], cm), cm), l1 = __fsub_rn(hi[j], h1);
                            const float h2 = __fsub_rn(__fadd_rn(p, cm), cm), l2 = __fsub_rn(p, h2);
                            hi[j] = __fadd_rn(l1, l2);
                            if (j < lim) lrow[2 * j] = __fadd_rn(lo[jj], __fadd_rn(h1, h2));
                        }
                    } else {
                        // rare: redo the 16 additions as TwoSums, the errors summed
                        // exactly into the low part; with levels per row / column an
                        // element whose own unit allows it takes the carry instead
                        // (its own split constant).
                        const bool was = (dirty >> (h / 16)) & 1u;
                        dirty |= 1u << (h / 16);
                        const float renorm = 0.5f * bound;        // lo is kept below 2^23 u
                        float lo[16];
                        load_low(h, was, lo);
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj) {
                            const int j = h + jj;
                            const float p = __uint_as_float(p16[jj]);
                            float be = 0.0f;
                            if (ROWCOL && j < lim && nch <= 2048)
                                be = bound_of_levels(a_row, vB[(int64_t)kDiag[q][1] * N + n0 + cq * Cfg::COLS + j]);
                            if (ROWCOL && isinf(be)) {
                                // a product of zero slices adds nothing
                            } else if (be > 0.0f && be <= 0x1p116f) {
                                const float cm = 3072.0f * be;
                                const float h1 = __fsub_rn(__fadd_rn(hi[j], cm), cm), l1 = __fsub_rn(hi[j], h1);
                                const float h2 = __fsub_rn(__fadd_rn(p, cm), cm), l2 = __fsub_rn(p, h2);
                                lo[jj] = __fadd_rn(lo[jj], __fadd_rn(h1, h2));
                                hi[j] = __fadd_rn(l1, l2);
                            } else {
                                float e;
                                const float sm = two_sum(hi[j], p, e);
                                lo[jj] = __fadd_rn(lo[jj], e);
                                hi[j] = (fabsf(lo[jj]) < renorm) ? sm : two_sum(sm, lo[jj], lo[jj]);   // renormalise (hi, lo)
                            }
                            if (j < lim) lrow[2 * j] = lo[jj];
                        }
                    }
                    }
                }
                tc_fence_before();                                // buffer free: all values are in registers
                __syncwarp();
                if (lane == 0) {
                    if constexpr (PAIR) mbar_arrive_peer(peer_addr(tempty0 + 8u * b, 0));
                    else mbar_arrive(tempty0 + 8u * b);
                }
                if (coded < Cfg::COLS && c >= 2) { code_columns(coded); coded += HC; }
            }
            if (!ok) break;
            t0 += nch;
            // The sums are integer multiples of the smallest unit of this thread's
            // elements, 2^-24 bound; when that unit is a normal FP32 number so is
            // every nonzero sum, and the short widening is exact.
            const bool normal_sums = bound >= 0x1p-102f;
            ++in_group;
            const bool last = in_diag == diag || in_group == group;      // last product of its group
            if (DUO && last && !first_in) {                              // product 0 is in the accumulator
                if (!(ok = wait_duo(duo_first, flags))) break;
                first_in = true;
            }
            if (last) {
                // C <- fl64(C + (hi + lo)) in L2, column by column (product 0: a plain store).
                // The common cases (no low words, normal unit) are branches of their own
                // with integer widening only: written as selects, the rare path's FP64
                // additions and general widening would run for every element (GB300's
                // FP64 pipe does about one warp-wide add per 32 clocks per SM
                // sub-partition).
                if (rounds && in_group > 1) {
                    // what the sums started at (exact).  All code words are read before the first
                    // reduction: a load behind queued reductions waits for them.
#pragma unroll
                    for (int w = 0; w < Cfg::COLS / 4; ++w) {
                        const uint32_t cw = codes[w * Cfg::DRAIN_THREADS];
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            hi[4 * w + k] = __fsub_rn(hi[4 * w + k], start_of(code_byte(cw, k), bits_of(4 * w + k)));
                    }
                }
#pragma unroll
                for (int h = 0; h < Cfg::COLS; h += 16) {
                    const bool low = (dirty >> (h / 16)) & 1u;
                    if (!__any_sync(0xFFFFFFFFu, low) && normal_sums) {
                        if (!live) continue;
                        if (q == 0 && !((dirty >> (16 + h / 16)) & 1u)) {
#pragma unroll
                            for (int j = h; j < h + 16; ++j) tacc[j * kBM] = widen_normal(hi[j]);
                        } else {
#pragma unroll
                            for (int j = h; j < h + 16; ++j) red_add_f64(tacc + j * kBM, widen_normal(hi[j]));
                        }
                    } else {
                        float lo[16];
                        load_low(h, low, lo);
#pragma unroll
                        for (int j = h; j < h + 16; ++j) {
                            const double sq = __dadd_rn(widen_exact(hi[j]), widen_exact(lo[j - h]));   // exact
                            if (live) {
                                if (q == 0) tacc[j * kBM] = sq;
                                else red_add_f64(tacc + j * kBM, sq);
                            }
                        }
                    }
                }
                in_group = 0;
                if (DUO && duo && q == 0) signal_duo(duo_first, rank);
            } else if (rounds) {
                // Round the running sums as the addition of this product to the result
                // rounds it.  (lock holds: the unit is normal.)
                const bool first = in_group == 1;
                for (; coded < Cfg::COLS; coded += HC) code_columns(coded);
                if (__any_sync(0xFFFFFFFFu, each)) {
                    // rare: elements reduced after every product
#pragma unroll
                    for (int w = 0; w < Cfg::COLS / 4; ++w) {
                        const uint32_t cw = codes[w * Cfg::DRAIN_THREADS], x = cw ^ (0x01010101u * kCodeEach);
                        if (!__any_sync(0xFFFFFFFFu, ((x - 0x01010101u) & ~x & 0x80808080u) != 0)) continue;   // no such byte
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (code_byte(cw, k) == kCodeEach && !((dirty >> (w / 4)) & 1u)) {
                                if (live) red_add_f64(tacc + (4 * w + k) * kBM, widen_normal(hi[4 * w + k]));
                                hi[4 * w + k] = 0.0f;
                            }
                        }
                    }
                }
                if (__any_sync(0xFFFFFFFFu, dirty != 0)) {
                    // rare: columns with low words, which are reduced after every product from now on
#pragma unroll
                    for (int h = 0; h < Cfg::COLS; h += 16) {
                        const bool low = (dirty >> (h / 16)) & 1u;
                        if (!__any_sync(0xFFFFFFFFu, low)) continue;
                        float lo[16];
                        load_low(h, low, lo);
#pragma unroll
                        for (int w = h / 4; w < h / 4 + 4; ++w) {
                            const uint32_t cw = codes[w * Cfg::DRAIN_THREADS];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int j = 4 * w + k;
                                double sq = __dadd_rn(widen_normal(hi[j]), widen_exact(lo[j - h]));        // exact
                                if (!first) sq = __dsub_rn(sq, widen_normal(start_of(code_byte(cw, k), bits_of(j))));
                                if (low) {
                                    if (live) red_add_f64(tacc + j * kBM, sq);
                                    hi[j] = 0.0f;
                                }
                            }
                            if (low) codes[w * Cfg::DRAIN_THREADS] = 0x01010101u * kCodeEach;
                        }
                    }
                    each |= dirty != 0;
                    dirty = 0;
                }
                if (first) {
#pragma unroll
                    for (int w = 0; w < Cfg::COLS / 4; ++w) {
                        const uint32_t cw = codes[w * Cfg::DRAIN_THREADS];
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            hi[4 * w + k] = __fadd_rn(hi[4 * w + k], start_of(code_byte(cw, k), bits_of(4 * w + k)));
                    }
                }
#pragma unroll
                for (int w = 0; w < Cfg::COLS / 4; ++w) {
                    const uint32_t cw = codes[w * Cfg::DRAIN_THREADS];
                    const uint32_t f = round_fields(cw, bits_of(0));      // ROWCOL: per element below
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int j = 4 * w + k;
                        hi[j] = round_to(hi[j], ROWCOL ? round_fields(cw, bits_of(j)) : f, k);
                    }
                }
            }
            if (in_diag++ == diag) { ++diag; in_diag = 0; }
        }
        // The warp takes the bulk-copy branch together (its __syncwarp and the
        // copies lane 0 issues need every lane) when no lane's wait timed out and
        // one of its rows is live (a pair's second CTA may reach past the last
        // row).  Lanes of rows past M read their accumulator elements (inside the
        // tile, never written) and the copies leave those rows out.
        if (DUO && duo && __all_sync(0xFFFFFFFFu, ok)) {
            signal_duo(duo_done, rank);
            if (!others_in) ok = wait_duo(duo_done, flags);
        }
        // the half of the tile's columns that this CTA of a duo writes
        const bool writes = !DUO || (duo ? (uint32_t)(cq >> 1) == rank : rank == 0);
        const bool warp_ok = __all_sync(0xFFFFFFFFu, ok), warp_live = __any_sync(0xFFFFFFFFu, live);
        if (warp_ok && warp_live && writes && c_tma && !TAIL) {
            // the accumulator holds every product now (this thread's own reductions,
            // same addresses, so they precede these loads): C <- acc through the TMA
            // engine.  Each 32 x 16 piece of the warp's rows (4 KB, two alternating
            // buffers per warp in the stage memory, which every MMA has finished
            // reading) is staged in the 128-byte-swizzled layout of the C map and
            // written by one bulk tensor store: whole 128-byte row segments, where
            // the per-lane stores below touch one cache line per row and lane.
            const uint32_t bufs = base + (uint32_t)(warp - Cfg::FIRST_DRAIN) * 8192u;
            fence_proxy_async_global();       // this thread's low-word writes to C precede the copies
            __syncwarp();
#pragma unroll 1
            // pieces wholly past the last column are neither staged nor copied
            for (int j0 = 0, g = 0; j0 < Cfg::COLS && n0 + cq * Cfg::COLS + j0 < N; j0 += 16, ++g) {
                const uint32_t buf = bufs + (uint32_t)(g & 1) * 4096u;
                if (g >= 2) {                 // the copy that last read this buffer
                    if (lane == 0) bulk_wait_read<1>();
                    __syncwarp();
                }
                const uint32_t srow = buf + (uint32_t)lane * 128u;
#pragma unroll
                for (int h = 0; h < 16; h += 8) {         // eight columns at a time: few live registers
                    double out[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) out[j] = ld_cg_f64(tacc + (j0 + h + j) * kBM);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned long long a = (unsigned long long)__double_as_longlong(out[2 * k]);
                        const unsigned long long b = (unsigned long long)__double_as_longlong(out[2 * k + 1]);
                        st_shared_v4(srow + ((uint32_t)((h / 2 + k) ^ (lane & 7)) << 4), (uint32_t)a,
                                     (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&tmC, buf, n0 + cq * Cfg::COLS + j0, m0 + quarter * 32);
                    bulk_commit();
                }
            }
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
        } else if (ok && live && writes && !(c_tma && !TAIL)) {
            // the accumulator holds every product now (this thread's own reductions,
            // same addresses, so they precede these loads): C <- acc (+ the merged tail)
            const float *trow = TAIL ? T + (int64_t)(row < M ? row : 0) * ldt + n0 + cq * Cfg::COLS : nullptr;
            const bool vec = ((ldc & 1) == 0) && ((reinterpret_cast<uintptr_t>(C) & 15u) == 0);
#pragma unroll 1
            for (int j0 = 0; j0 < Cfg::COLS; j0 += 8) {
                double out[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) out[j] = ld_cg_f64(tacc + (j0 + j) * kBM);
                if (TAIL) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j0 + j < lim) out[j] = __dadd_rn(out[j], widen_exact(trow[j0 + j]));
                }
                if (vec && lim >= j0 + 8) {
#pragma unroll
                    for (int j = 0; j < 8; j += 2)
                        *reinterpret_cast<double2 *>(crow + j0 + j) = make_double2(out[j], out[j + 1]);
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j0 + j < lim) crow[j0 + j] = out[j];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR || DUO) cluster_sync();        // the leader's MMAs, a duo's signals are done with both CTAs
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        if constexpr (PAIR) tmem_dealloc_pair(tmem, 512);
        else tmem_dealloc(tmem, 512);
    }
}

// tiles: the first `tiles` tiles in raster order (all of them, or the full
// waves when narrower tiles take the rest), one CTA each, or with PAIR one
// cluster of two CTAs each; or with wide_first >= 0 (pairs, BN = 128) `tiles`
// 256 x 128 halves of the 256 x 256 tiles from raster index wide_first on.
template <int BN, bool ROWCOL, bool TAIL, bool PAIR, bool DUO>
cudaError_t run_f64w(int64_t M, int64_t N, int64_t K, const uint16_t *Ap, const uint16_t *Bp, int64_t ldcomp,
                     const int32_t *vA, const int32_t *vB, int nprod, double *C, int64_t ldc, double *acc,
                     uint32_t *flags, cudaStream_t st, int64_t a_plane, const float *T, int64_t ldt, int64_t tiles,
                     int wide_first)
{
    using Cfg = F64WCfgT<BN, PAIR>;
    CUtensorMap ta, tb;
    if (!make_plane_map(&ta, Ap, K, M, 6, ldcomp, Cfg::KB, kBM, a_plane) ||
        !make_plane_map(&tb, Bp, K, N, 6, ldcomp, Cfg::KB, Cfg::BH))
        return cudaErrorInvalidValue;
    CUtensorMap tc = {};
    const int c_tma = make_c_map_f64(&tc, C, M, N, ldc) ? 1 : 0;
    auto kern = prodsum_f64w_kernel<BN, ROWCOL, TAIL, PAIR, DUO>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((PAIR || DUO ? 2 : 1) * tiles));
    cfg.blockDim = dim3(Cfg::THREADS);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 2;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = PAIR || DUO ? 2 : 1;
    e = cudaLaunchKernelEx(&cfg, kern, ta, tb, tc, c_tma, (int)M, (int)N, (int)K, nprod, vA, vB, C, ldc, acc, flags, T,
                           ldt, wide_first);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <int BN, bool PAIR>
cudaError_t dispatch_f64w(int64_t M, int64_t N, int64_t K, const uint16_t *Ap, const uint16_t *Bp, int64_t ldcomp,
                          const int32_t *vA, const int32_t *vB, int nprod, double *C, int64_t ldc, double *acc,
                          uint32_t *flags, cudaStream_t st, int64_t a_plane, bool rowcol, const float *T, int64_t ldt,
                          int64_t tiles, int wide_first, bool duo = false)
{
    if (T) {                                          // merged tail: whole-matrix levels only
        if (rowcol) return cudaErrorInvalidValue;
        return run_f64w<BN, false, true, PAIR, false>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane,
                                               T, ldt, tiles, wide_first);
    }
    if (rowcol)
        return run_f64w<BN, true, false, PAIR, false>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane,
                                               T, ldt, tiles, wide_first);
    if constexpr (BN < 256 && !PAIR) {
        if (duo)
            return run_f64w<BN, false, false, false, true>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st,
                                                           a_plane, T, ldt, tiles, wide_first);
    }
    return run_f64w<BN, false, false, PAIR, false>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane, T,
                                            ldt, tiles, wide_first);
}

}  // namespace
}  // namespace emu
