// FP64-mode product-sum on tiles of 128 or 64 columns (128 rows, or 256 x 128 on
// CTA pairs), for results too small to fill the GPU with wider ones and for the
// last, partial wave of those (the kernel and its notes are in prodsum_f64w_kernel.cuh).
#include "prodsum_f64w_kernel.cuh"

namespace emu {

cudaError_t launch_prodsum_f64_narrow(int64_t M, int64_t N, int64_t K, const uint16_t *Ap, const uint16_t *Bp,
                                     int64_t ldcomp, const int32_t *vA, const int32_t *vB, int nprod, double *C,
                                     int64_t ldc, double *acc, uint32_t *flags, cudaStream_t st, int64_t a_plane,
                                     bool rowcol, const float *T, int64_t ldt, int cols, bool pair, int64_t tiles,
                                      int wide_first, bool duo)
{
    if (f64_diagonals(nprod) == 0) return cudaErrorInvalidValue;
    if (pair)
        return dispatch_f64w<128, true>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st, a_plane, rowcol, T,
                                        ldt, tiles, wide_first);
    return cols == 128 ? dispatch_f64w<128, false>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st,
                                                   a_plane, rowcol, T, ldt, tiles, wide_first, duo)
                       : dispatch_f64w<64, false>(M, N, K, Ap, Bp, ldcomp, vA, vB, nprod, C, ldc, acc, flags, st,
                                                  a_plane, rowcol, T, ldt, tiles, wide_first, duo);
}

}  // namespace emu
