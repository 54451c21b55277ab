"""The general FP32 GEMM's alpha and beta with a C that a tensor map describes
(sizes and pitches in multiples of 4): C is read and written by bulk tensor
copies in the product-sum's epilogue, and must equal the product scaled and
added in separate roundings, bit for bit, with nothing written past its
columns or rows."""
import pytest

import paper_2609_04663_gb300 as emu
from helpers import device, gemm_f32_one_accumulator

pytestmark = pytest.mark.gpu


def _rand(torch, rows, cols, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand((rows, cols), generator=g, device="cuda") * 2 - 1


# one piece, partial pieces and tiles, narrow tiles, ragged pairs, a second launch of quarters
@pytest.mark.parametrize("M,N,K", [(1, 4, 1), (33, 36, 65), (70, 300, 129), (129, 256, 64), (1537, 2052, 100),
                                   (4000, 4096, 96), (16, 4100, 32)])
@pytest.mark.parametrize("alpha,beta", [(-1.0, 1.0), (0.75, 0.0), (1.25, -0.5)])
@pytest.mark.parametrize("pad", [0, 4])
def test_alpha_beta_through_bulk_copies(M, N, K, alpha, beta, pad):
    import torch
    device()
    A, B, C0 = _rand(torch, M, K, 1), _rand(torch, K, N, 2), _rand(torch, M, N, 3)
    P, flags = gemm_f32_one_accumulator(A, B)
    assert flags == 0
    want = P * torch.tensor(alpha, dtype=torch.float32, device="cuda")
    if beta != 0.0:
        want = want + C0 * torch.tensor(beta, dtype=torch.float32, device="cuda")
    guard = torch.full((M + 2, N + pad), float("nan"), device="cuda")
    C = guard[1:M + 1, :N]
    if beta != 0.0:
        C.copy_(C0)
    _, ws = emu.gemm_ex(A, B, alpha=alpha, beta=beta, C=C)
    assert emu.read_flags(ws) == 0
    assert torch.equal(C, want)
    assert bool(torch.isnan(guard[0]).all() and torch.isnan(guard[M + 1]).all() and torch.isnan(guard[:, N:]).all())
