// FP64-mode product-sum on 256-column tiles: 128 x 256 tiles, one CTA each,
// and 256 x 256 tiles on CTA pairs (the kernel and its notes are in
// prodsum_f64w_kernel.cuh; prodsum_f64n.cu compiles its narrower tiles).
#include "prodsum_f64w_kernel.cuh"

namespace emu {

cudaError_t launch_prodsum_f64_wide(int64_t M, int64_t N, int64_t K, const uint16_t *Ap, const uint16_t *Bp,
                                     int64_t ldcomp, const int32_t *vA, const int32_t *vB, int nprod, double *C,
                                     int64_t ldc, double *acc, uint32_t *flags, cudaStream_t st, int64_t a_plane,
                                     bool rowcol, const float *T, int64_t ldt, bool pair, int64_t tiles)
{
    if (f64_diagonals(nprod) == 0) return cudaErrorInvalidValue;
    return pair ? dispatch_f64w<256, true>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane,
                                           rowcol, T, ldt, tiles, -1)
                : dispatch_f64w<256, false>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane,
                                            rowcol, T, ldt, tiles, -1);
}

}  // namespace emu
