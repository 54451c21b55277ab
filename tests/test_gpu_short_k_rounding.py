"""FP64 products of one or two chunks whose later diagonals round: the
accumulator is read for the rounding codes after the last chunk, none of it in
the shadow of the partials, and rows past the last one (a ragged second CTA of a
pair) read the first stripe and drop it."""
import numpy as np
import pytest

import oracle
import paper_2609_04663_gb300 as emu
import synth
from helpers import device, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [32, 256, 513])
@pytest.mark.parametrize("M,N", [(300, 2500), (4000, 1300), (5000, 700)])
def test_rounded_products_of_few_chunks(M, N, K):
    dev = device()
    A, B = synth.gemm_inputs("f64", M, N, K, 31)
    A[7] *= 2.0 ** -30                               # results far below the largest, and a zero one
    A[M - 2] = 0.0
    B[:, N - 1] = -B[:, 0]
    C, ws = emu.gemm_f64(to_dev(A, dev), to_dev(B, dev), 21)
    assert emu.read_flags(ws) == 0
    Cn = C.cpu().numpy()
    for r in (0, 7, 128, 255, M // 2, M - 2, M - 1):
        assert np.array_equal(Cn[r], oracle.gemm_f64(A, B, 21, rows=(r, r + 1))[0][0]), r
