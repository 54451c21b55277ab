"""GEMM calls captured in a CUDA graph and run on several streams: cooperative
splits, product-sums launched as programmatic dependents and two-launch
schedules must replay as they run, on changed inputs, and calls with buffers of
their own must not disturb each other."""
import pytest

import paper_2609_04663_gb300 as emu
from helpers import device

pytestmark = pytest.mark.gpu


# small split and duos, large split, two launches, levels per vector, alpha and beta
@pytest.mark.parametrize("kind,M,N,K,nprod", [
    ("f64", 256, 256, 256, 21), ("f64", 1024, 1024, 1100, 10), ("f64", 2100, 2048, 1040, 6), ("f64", 4096, 4096, 72, 10),
    ("rowcol", 300, 400, 500, 15), ("ex64", 300, 333, 700, 10), ("f32", 512, 512, 512, None), ("f32", 4000, 4096, 96, None),
    ("ex32", 300, 332, 700, None), ("ex32", 300, 333, 700, None)])
def test_captured_and_concurrent_calls(kind, M, N, K, nprod):
    import torch
    device()
    f32 = kind.endswith("32")
    dt = torch.float32 if f32 else torch.float64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    A = torch.rand((M, K), generator=gen, dtype=dt, device="cuda") * 2 - 1
    B = torch.rand((K, N), generator=gen, dtype=dt, device="cuda") * 2 - 1
    mode = 32 if f32 else 64
    nbytes = emu.emu_gemm_f64_rowcol_workspace_bytes(M, N, K) if kind == "rowcol" else \
        emu.emu_gemm_ex_workspace_bytes(mode, M, N, K) if kind.startswith("ex") else \
        emu.emu_gemm_workspace_bytes(mode, M, N, K)

    def call(C, ws):
        if kind == "f32":
            emu.gemm_f32(A, B, C=C, ws=ws)
        elif kind == "f64":
            emu.gemm_f64(A, B, nprod, C=C, ws=ws)
        elif kind == "rowcol":
            emu.gemm_f64_rowcol(A, B, nprod, C=C, ws=ws)
        else:
            emu.gemm_ex(A, B, alpha=-1.5, beta=0.0, C=C, nprod=nprod, ws=ws)

    C, ws = torch.zeros((M, N), dtype=dt, device="cuda"), emu.workspace(nbytes)
    call(C, ws)
    torch.cuda.synchronize()
    want = C.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(C, ws)
        call(C, ws)
    C.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(C, want) and emu.read_flags(ws) == 0
    A.mul_(0.5)                                          # exact: the result halves
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(C, want * 0.5)
    outs = []
    for s in (torch.cuda.Stream(), torch.cuda.Stream()):
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            out, w = torch.zeros((M, N), dtype=dt, device="cuda"), emu.workspace(nbytes)
            for _ in range(5):
                call(out, w)
            outs.append((out, w))
    torch.cuda.synchronize()
    for out, w in outs:
        assert torch.equal(out, want * 0.5) and emu.read_flags(w) == 0
