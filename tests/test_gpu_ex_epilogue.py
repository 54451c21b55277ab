"""The general FP32 GEMM applies alpha and beta in the product-sum's epilogue:
C must equal the product (one accumulator per element) scaled and added in
separate roundings, bit for bit, for every tile shape, edge and orientation;
and a C that no tensor map describes (odd sizes and pitches) must equal the
same product in an aligned C."""
import pytest

import paper_2609_04663_gb300 as emu
from helpers import device, gemm_f32_one_accumulator

pytestmark = pytest.mark.gpu


def _rand(torch, rows, cols, seed, pad=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.rand((rows, cols + pad), generator=g, device="cuda") * 2 - 1)[:, :cols]


# narrow tiles, one column, ragged pairs, the quarters launch with a partial last tile row
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (70, 65, 129), (300, 333, 700), (1537, 2050, 100), (4000, 4096, 96)])
@pytest.mark.parametrize("alpha,beta", [(-1.0, 1.0), (0.75, 0.0), (1.0, 0.3), (1.25, -0.5)])
def test_alpha_beta_in_the_epilogue(M, N, K, alpha, beta):
    import torch
    device()
    A, B, C0 = _rand(torch, M, K, 1), _rand(torch, K, N, 2), _rand(torch, M, N, 3, pad=3)
    P, flags = gemm_f32_one_accumulator(A, B)
    assert flags == 0
    want = P * torch.tensor(alpha, dtype=torch.float32, device="cuda")
    if beta != 0.0:
        want = want + C0 * torch.tensor(beta, dtype=torch.float32, device="cuda")
    for opA, opB in [(0, 0), (1, 0), (0, 1), (1, 1)]:
        C = torch.full((M, N + 3), float("nan"), device="cuda")[:, :N]
        if beta != 0.0:
            C.copy_(C0)
        As = A.t().contiguous() if opA else A
        Bs = B.t().contiguous() if opB else B
        _, ws = emu.gemm_ex(As, Bs, opA, opB, alpha=alpha, beta=beta, C=C)
        assert emu.read_flags(ws) == 0
        assert torch.equal(C, want), (opA, opB)
        assert bool(torch.isnan(C.as_strided((M, 3), (N + 3, 1), N)).all())          # padding untouched


@pytest.mark.parametrize("M,N,K,pad", [(300, 333, 700, 0), (257, 64, 40, 1), (2048, 2050, 64, 0), (130, 515, 33, 2)])
def test_c_without_a_tensor_map(M, N, K, pad):
    import torch
    device()
    A, B = _rand(torch, M, K, 4), _rand(torch, K, N, 5)
    Np = (N + 3) // 4 * 4
    Ap, _ = emu.split_f32(A, ldcomp=emu.gemm_ldk(K))
    Bp, _ = emu.split_f32(B, transpose=True, ldcomp=emu.gemm_ldk(K))
    odd = torch.zeros((M, N + pad), device="cuda")[:, :N]
    emu.prodsum_f32(Ap, Bp, M, N, K, C=odd)
    Bw = torch.zeros((K, Np), device="cuda")
    Bw[:, :N] = B
    Bpw, _ = emu.split_f32(Bw, transpose=True, ldcomp=emu.gemm_ldk(K))
    full, _ = emu.prodsum_f32(Ap, Bpw, M, Np, K)
    assert torch.equal(odd, full[:, :N])
