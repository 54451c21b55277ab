"""The FP64 split of both operands of a GEMM: one launch for small operands, a
few for larger ones, either way as the single-operand split does each
(planes and levels identical), with the speculative levels failing in
neither, one or both operands, and for every orientation of the general
GEMM."""
import numpy as np
import pytest

import paper_2609_04663_gb300 as emu
from helpers import device, to_dev

pytestmark = pytest.mark.gpu


def _operand(shape, gap, seed):
    rng = np.random.default_rng(seed)
    X = rng.random(shape) * 2 - 1
    if gap:                                   # entries whose residuals skip binades
        X = np.round(X * 128) / 128
        X[rng.random(shape) < 0.01] += 2.0 ** -31
    return X


# 64-bit sizes around one tile, ragged ones, and past the one-launch limit of 2^22 entries
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (64, 64, 64), (65, 130, 257), (300, 77, 1025), (2100, 1000, 1500)])
@pytest.mark.parametrize("gap", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("nslices", [3, 6])
def test_pair_equals_single_operand_splits(M, N, K, gap, nslices):
    import torch
    dev = device()
    A, B = to_dev(_operand((M, K), gap[0], 1), dev), to_dev(_operand((K, N), gap[1], 2), dev)
    ldk = emu.gemm_ldk(K)
    Ap = torch.zeros((6, M, ldk), dtype=torch.int16, device=dev)
    Bp = torch.zeros((6, N, ldk), dtype=torch.int16, device=dev)
    v = torch.zeros((2, 6), dtype=torch.int32, device=dev)
    ws = emu.workspace(emu.emu_split_workspace_bytes(64), dev)
    r = emu.emu_split_f64_pair(M, N, K, A.data_ptr(), K, B.data_ptr(), N, Ap.data_ptr(), Bp.data_ptr(), ldk, nslices,
                               v.data_ptr(), v.data_ptr() + 24, ws.data_ptr(), ws.numel(), emu._stream(None))
    assert r == 0 and emu.read_flags(ws) == 0
    Ar, va, wa = emu.split_f64(A, ldcomp=ldk, nslices=nslices)
    Br, vb, wb = emu.split_f64(B, transpose=True, ldcomp=ldk, nslices=nslices)
    assert torch.equal(v[0, :nslices], va[:nslices]) and torch.equal(v[1, :nslices], vb[:nslices])
    assert torch.equal(Ap[:nslices], Ar[:nslices]) and torch.equal(Bp[:nslices], Br[:nslices])


@pytest.mark.parametrize("M,N,K", [(70, 65, 129), (2100, 1000, 1500)])
@pytest.mark.parametrize("gap", [False, True])
def test_every_orientation_gives_the_same_product(M, N, K, gap):
    import torch
    dev = device()
    A, B = to_dev(_operand((M, K), gap, 3), dev), to_dev(_operand((K, N), False, 4), dev)
    want, ws = emu.gemm_f64(A, B, 10)
    assert emu.read_flags(ws) == 0
    for opA in (emu.OP_N, emu.OP_T):
        for opB in (emu.OP_N, emu.OP_T):
            As = A.t().contiguous() if opA == emu.OP_T else A
            Bs = B.t().contiguous() if opB == emu.OP_T else B
            C, ws = emu.gemm_ex(As, Bs, opA, opB, nprod=10)
            assert emu.read_flags(ws) == 0
            assert torch.equal(C, want), (opA, opB)
