"""Performance cases: emulated GEMM calls as a user's program makes them.

Every case is one call of a public entry point on matrices that are already on
the GPU, with the output and the workspace allocated once beforehand, as a
program that multiplies in a loop keeps them.  The calls cover both modes
(FP32 with 6 products, FP64 with 6, 10, 15 or 21), the plain GEMM, the general
GEMM (transposed operands, alpha and beta) and the GEMM with levels per row
and column, from 256^3, where launches count, to 16384^3.

A case is a dict of plain values:
  call    "f32", "f64", "ex_f32", "ex_f64" or "rowcol"
  M, N, K sizes of the result and of the sum
  nprod   products kept (FP64 mode)
  opA/opB 1 when the stored operand is the transpose (general GEMM)
  alpha, beta  general GEMM
  phi     0: entries uniform in [-1, 1]; otherwise the scaled class
          (u - 0.5) exp(phi g), g standard normal
  pad     extra columns in each matrix's row pitch (a view of a wider matrix)
"""
import math

import torch

import paper_2609_04663_gb300 as emu


def listed():
    return [
        # -- FP32 mode: C = A B with 6 products
        # a small layer or block update: the call's launches and set-up dominate
        {"name": "f32_256", "call": "f32", "M": 256, "N": 256, "K": 256},
        # a mid-size product with fewer output tiles than the GPU has SMs
        {"name": "f32_1024", "call": "f32", "M": 1024, "N": 1024, "K": 1024},
        # residual R <- R0 - A^T B of a least-squares step: odd sizes, a transposed
        # operand, alpha and beta, and matrices that are views of wider ones
        {"name": "f32_residual_ragged", "call": "ex_f32", "M": 1537, "N": 2050, "K": 1100, "opA": 1, "opB": 0,
         "alpha": -1.0, "beta": 1.0, "pad": 3},
        # the top of the square sweep: two 1 GiB operands
        {"name": "f32_16384", "call": "f32", "M": 16384, "N": 16384, "K": 16384},
        # -- FP64 mode
        # a small block in full precision
        {"name": "f64_256_p21", "call": "f64", "M": 256, "N": 256, "K": 256, "nprod": 21},
        # a mid-size product at the middle accuracy
        {"name": "f64_1024_p10", "call": "f64", "M": 1024, "N": 1024, "K": 1024, "nprod": 10},
        # R <- R0 - A X for a block of right-hand sides in iterative refinement: a tall,
        # narrow result, odd sizes and row pitches, full precision
        {"name": "f64_residual_skinny", "call": "ex_f64", "M": 3001, "N": 203, "K": 2999, "nprod": 21, "opA": 0,
         "opB": 0, "alpha": -1.0, "beta": 1.0, "pad": 0},
        # operands with levels per row and per column, the second one stored transposed in use
        # by programs whose rows and columns differ widely in magnitude
        {"name": "f64_rowcol_2048_p15", "call": "rowcol", "M": 2048, "N": 2048, "K": 2048, "nprod": 15, "phi": 1.0},
        # the square size of the accuracy tables, cheapest and most accurate product set
        {"name": "f64_4096_p6", "call": "f64", "M": 4096, "N": 4096, "K": 4096, "nprod": 6},
        {"name": "f64_4096_p21", "call": "f64", "M": 4096, "N": 4096, "K": 4096, "nprod": 21},
        # a large product of operands with entries spread over many binades
        {"name": "f64_8192_scaled_p21", "call": "f64", "M": 8192, "N": 8192, "K": 8192, "nprod": 21, "phi": 4.0},
        # a long sum into a small result (Gram matrices, correlations)
        {"name": "f64_long_k_p10", "call": "f64", "M": 2048, "N": 2048, "K": 65536, "nprod": 10},
    ]


# the largest listed case, 6 products of 16384^3, in multiply-adds
_MOST = 6 * 16384.0 ** 3


def _size(rng, lo, hi):
    """A size between lo and hi, spread over the logarithm; one in three is rounded to a multiple of 64."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 1 / 3:
        n = max(lo, n // 64 * 64)
    return n


def draw(rng):
    call = rng.choice(["f32", "f32", "f64", "f64", "f64", "ex_f32", "ex_f64", "rowcol"])
    f32 = call.endswith("f32")
    nprod = 6 if f32 else rng.choice([6, 10, 15, 21])
    while True:
        hi = 16384 if f32 else 8192
        M, N = _size(rng, 200, hi), _size(rng, 200, hi)
        K = _size(rng, 200, 65536)
        if nprod * float(M) * N * K <= _MOST and (M + N) * float(K) <= 2.0 * 16384 ** 2:
            break
    case = {"call": call, "M": M, "N": N, "K": K}
    if not f32:
        case["nprod"] = nprod
        case["phi"] = rng.choice([0.0, 0.0, 0.5, 2.0, 4.0])
    if call.startswith("ex"):
        case.update(opA=rng.randrange(2), opB=rng.randrange(2), pad=rng.choice([0, 1, 3, 8]))
        case["alpha"], case["beta"] = rng.choice([(1.0, 0.0), (-1.0, 1.0), (0.75, 0.0), (1.25, -0.5)])
    return case


def _is_f32(case):
    return case["call"].endswith("f32")


def _matrix(gen, rows, cols, dtype, phi, pad):
    """rows x cols entries on the GPU, a view of a matrix with `pad` more columns."""
    full = torch.rand((rows, cols + pad), generator=gen, dtype=dtype, device="cuda")
    if phi == 0.0:
        full.mul_(2.0).sub_(1.0)
    else:
        g = torch.randn((rows, cols + pad), generator=gen, dtype=dtype, device="cuda")
        full.sub_(0.5).mul_(g.mul_(phi).exp_())
        tiny, top = 2.0 ** -126, (2.0 - 2.0 ** -7) * 2.0 ** 127
        full = torch.where(full == 0, full, torch.sign(full) * full.abs().clamp_(tiny, top))
    return full[:, :cols]


def _inputs(case, seed):
    """A and B as stored, and the C the general GEMM updates (None otherwise)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    M, N, K = case["M"], case["N"], case["K"]
    dtype = torch.float32 if _is_f32(case) else torch.float64
    phi, pad = case.get("phi", 0.0), case.get("pad", 0)
    a = (K, M) if case.get("opA", 0) else (M, K)
    b = (N, K) if case.get("opB", 0) else (K, N)
    A, B = _matrix(gen, *a, dtype, phi, pad), _matrix(gen, *b, dtype, phi, pad)
    if case["call"] == "rowcol":
        # rows of A and columns of B of very different magnitudes
        A = A * torch.exp(2.0 * torch.randn((M, 1), generator=gen, dtype=dtype, device="cuda"))
        B = B * torch.exp(2.0 * torch.randn((1, N), generator=gen, dtype=dtype, device="cuda"))
    C0 = _matrix(gen, M, N, dtype, 0.0, pad) if case["call"].startswith("ex") else None
    return A, B, C0


def prepare(case, seed):
    A, B, C0 = _inputs(case, seed)
    M, N, K = case["M"], case["N"], case["K"]
    mode = 32 if _is_f32(case) else 64
    pad = case.get("pad", 0)
    C = torch.zeros((M, N + pad), dtype=A.dtype, device="cuda")[:, :N]
    nbytes = {"ex_f32": emu.emu_gemm_ex_workspace_bytes, "ex_f64": emu.emu_gemm_ex_workspace_bytes,
              "f32": emu.emu_gemm_workspace_bytes, "f64": emu.emu_gemm_workspace_bytes}
    if case["call"] == "rowcol":
        ws = emu.workspace(emu.emu_gemm_f64_rowcol_workspace_bytes(M, N, K))
    else:
        ws = emu.workspace(nbytes[case["call"]](mode, M, N, K))
    return {"case": case, "A": A, "B": B, "C0": C0, "C": C, "ws": ws}


def run(state):
    case, A, B, C, ws = state["case"], state["A"], state["B"], state["C"], state["ws"]
    call = case["call"]
    if call == "f32":
        emu.gemm_f32(A, B, C=C, ws=ws)
    elif call == "f64":
        emu.gemm_f64(A, B, case["nprod"], C=C, ws=ws)
    elif call == "rowcol":
        emu.gemm_f64_rowcol(A, B, case["nprod"], C=C, ws=ws)
    else:
        # the program keeps the right-hand side and updates a copy of it
        if case["beta"] != 0.0:
            C.copy_(state["C0"])
        emu.gemm_ex(A, B, opA=case["opA"], opB=case["opB"], alpha=case["alpha"], beta=case["beta"], C=C,
                    nprod=case.get("nprod"), ws=ws)
    return C


def work(case):
    """A, B (and the C that beta reads) read once, C written once; the kept products on the tensor cores."""
    M, N, K = case["M"], case["N"], case["K"]
    word = 4 if _is_f32(case) else 8
    nbytes = word * (M * K + K * N + M * N)
    if case.get("beta", 0.0) != 0.0:
        nbytes += word * M * N
    return {"bytes": nbytes, "flops": 2 * M * N * K * case.get("nprod", 6)}


def exact(case, seed):
    A, B, C0 = _inputs(case, seed)
    # above about 20 seconds of FP64 multiplication
    if 2.0 * case["M"] * case["N"] * case["K"] > 1e13:
        return None
    A, B = A.double(), B.double()
    A = A.t() if case.get("opA", 0) else A
    B = B.t() if case.get("opB", 0) else B
    P = A @ B
    if C0 is None:
        return P
    R = case["alpha"] * P
    if case["beta"] != 0.0:
        R = R + case["beta"] * C0.double()
    return R
