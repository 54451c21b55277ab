// Pieces shared by the FP32-mode product-sum kernels (the TMA-fed one and the
// one that splits inside its producer): tile configuration, the MMA issue
// loop of Eq. (fp32reuseorder) over a ring of stages.  The epilogues are in
// prodsum_f32.cu; the one-kernel GEMM's is store_tile of gemm_common.cuh.
#pragma once

#include "gemm_common.cuh"
#include "pair_common.cuh"

namespace emu {

namespace {

// FP32 chain, Eq. (fp32reuseorder): A1B1 A1B0 A2B0 A0B0 A0B1 A0B2.
__host__ __device__ constexpr int chain_a(int q) { return q == 2 ? 2 : q < 2 ? 1 : 0; }
__host__ __device__ constexpr int chain_b(int q) { return q == 0 || q == 4 ? 1 : q == 5 ? 2 : 0; }

// ===================================================================== FP32
template <int BN, int KB, int STAGES>
struct F32Cfg {
    static constexpr int A_TILE = kBM * KB * 2;
    static constexpr int B_TILE = BN * KB * 2;
    static constexpr int STAGE = 3 * A_TILE + 3 * B_TILE;
    static constexpr uint32_t SWZ = (KB == 64) ? 2u : 4u;       // 128-byte or 64-byte swizzle
    static constexpr uint32_t SBO = 8u * KB * 2u;               // bytes between 8-row groups
    static constexpr int BAR_OFF = STAGES * STAGE;
    static constexpr int CBAR = 128;                            // four barriers, after the pipeline's and the TMEM slot
    static constexpr int SMEM = BAR_OFF + 256 + 1024;           // + barriers + alignment slack
    static_assert(16 * STAGES + 12 <= CBAR, "barrier area");
    static constexpr int THREADS = 192;
    static_assert(KB == 32 || KB == 64, "K-block must fill one 64 B or 128 B swizzle row");
    static_assert(BN % 32 == 0 && BN >= 32 && BN <= 256, "UMMA N");
};

// The six products of Eq. (fp32reuseorder) for the K-block in one stage (at
// `st`), 16 of K at a time, into the TMEM accumulator, and the commit that
// releases the stage when they finish: called by a converged warp, issued by one
// elected lane.  PAIR: MMAs and commit of a CTA pair (M = 256).
template <class Cfg, int KB, int BTILE, bool PAIR>
__device__ __forceinline__ void issue_products(uint32_t tmem, uint32_t st, uint32_t idesc, bool accumulate,
                                               uint32_t empty_bar)
{
    // descriptors of the first slices; a slice, a tile or a K step further adds bytes / 16
    const uint64_t a0 = make_sdesc(st, Cfg::SBO, Cfg::SWZ), b0 = make_sdesc(st + 3 * Cfg::A_TILE, Cfg::SBO, Cfg::SWZ);
    if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < KB / 16; ++kk) {
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const uint64_t ad = a0 + (uint32_t)((chain_a(q) * Cfg::A_TILE + kk * 32) / 16);
                const uint64_t bd = b0 + (uint32_t)((chain_b(q) * BTILE + kk * 32) / 16);
                if constexpr (PAIR) mma_bf16_pair(tmem, ad, bd, idesc, accumulate || (kk | q) != 0);
                else mma_bf16(tmem, ad, bd, idesc, accumulate || (kk | q) != 0);
            }
        }
        if constexpr (PAIR) mma_commit_pair(empty_bar);
        else mma_commit(empty_bar);
    }
    __syncwarp();
}

// MMA issuer (a whole warp, converged): for every K-block, wait for its stage,
// issue the six products of Eq. (fp32reuseorder) from it into the one TMEM
// accumulator, and release the stage when those MMAs finish.  Then wait for
// all MMAs.  The warp walks the loop together (waits decided by vote), so
// control flow and descriptors are uniform: issued from one lane's own
// branch, every MMA had to wait for its operands' moves to uniform registers.
template <int BN, int KB, int STAGES>
__device__ __forceinline__ void mma_loop(uint32_t tmem, uint32_t base, uint32_t full0, uint32_t empty0,
                                         uint32_t accum_bar, int nkb, uint32_t *flags)
{
    using Cfg = F32Cfg<BN, KB, STAGES>;
    constexpr uint32_t idesc = make_idesc_bf16(kBM, BN);
    for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % STAGES;
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(full0 + 8u * s, (kb / STAGES) & 1, flags))) break;
        tc_fence_after();
        issue_products<Cfg, KB, Cfg::B_TILE, false>(tmem, base + (uint32_t)(s * Cfg::STAGE), idesc, kb != 0,
                                                    empty0 + 8u * s);
    }
    if (elect_one()) mma_commit(accum_bar);  // all MMAs issued so far are done
    __syncwarp();
    (void)mbar_wait(accum_bar, 0, flags);
}

}  // namespace

}  // namespace emu
