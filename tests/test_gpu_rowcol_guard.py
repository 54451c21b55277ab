"""The calls with levels per row / column write nothing past the workspace size
they ask for: a band of canaries after it stays intact, on the speculative
path and on the literal passes (a vector whose levels do not fall in steps of
8), with results equal to the oracle's."""
import numpy as np
import pytest

import oracle
import paper_2609_04663_gb300 as emu
from helpers import device, planes_np, to_dev

pytestmark = pytest.mark.gpu

CANARY, BAND = 0xA5, 64 * 1024


def _ws(nbytes, dev):
    import torch
    return torch.full((nbytes + BAND,), CANARY, dtype=torch.uint8, device=dev)


def _intact(ws, nbytes):
    return bool(np.all(ws[nbytes:].cpu().numpy() == CANARY))


def _input(rows, cols, gap, seed):
    rng = np.random.default_rng(seed)
    X = rng.random((rows, cols)) * 2 - 1
    if gap:
        X[rows // 2] = np.where(rng.random(cols) < 0.5, 1.0, 2.0 ** -30 * rng.random(cols))
    return X


@pytest.mark.parametrize("gap", [False, True])
@pytest.mark.parametrize("rows", [1, 64, 1000, 4096])
def test_split_rowcol_workspace_band(rows, gap):
    dev = device()
    X = _input(rows, 40, gap, rows)
    need = emu.emu_split_f64_rowcol_workspace_bytes(rows)
    ws = _ws(need, dev)
    planes, v, _ = emu.split_f64_rowcol(to_dev(X, dev), ws=ws[:need])
    P, V, _ = oracle.split_f64_rows(X)
    assert _intact(ws, need)
    assert np.array_equal(planes_np(planes), P.view(np.uint16))
    assert np.array_equal(v.cpu().numpy().T, np.asarray(V))


@pytest.mark.parametrize("M,N", [(1000, 64), (64, 1000), (2048, 130)])
def test_gemm_rowcol_workspace_band(M, N):
    dev = device()
    K = 40
    A, B = _input(M, K, True, M), _input(K, N, False, N)
    need = emu.emu_gemm_f64_rowcol_workspace_bytes(M, N, K)
    ws = _ws(need, dev)
    C, _ = emu.gemm_f64_rowcol(to_dev(A, dev), to_dev(B, dev), 6, ws=ws[:need])
    assert emu.read_flags(ws) == 0
    assert _intact(ws, need)
    assert np.array_equal(C.cpu().numpy(), oracle.gemm_f64_rowcol(A, B, 6)[0])
