"""The FP64 product-sum adds products of a diagonal in groups (one FP32 sum,
rounded as Algorithm 2's FP64 additions round): inputs at which that could go
wrong, on every tile shape, against the oracle bit for bit.  The tile switch
is read once per process, so each shape runs in a child process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, {root!r})
sys.path.insert(0, {tests!r})
import numpy as np
import oracle
import paper_2609_04663_gb300 as emu
from helpers import device, to_dev
dev = device()
rng = np.random.default_rng(5)

def check(tag, A, B, nprod, rows=None, rowcol=False):
    f = emu.gemm_f64_rowcol if rowcol else emu.gemm_f64
    C, ws = f(to_dev(A, dev), to_dev(B, dev), nprod)
    assert emu.read_flags(ws) == 0, tag
    Cn = C.cpu().numpy()
    if rowcol:
        assert np.array_equal(Cn, oracle.gemm_f64_rowcol(A, B, nprod)[0]), tag
        return
    for r in (rows if rows is not None else range(A.shape[0])):
        assert np.array_equal(Cn[r], oracle.gemm_f64(A, B, nprod, rows=(r, r + 1))[0][0]), (tag, r)

def slices(shape, draw, sign):
    # entries whose slices are the integers draw() gives, in units of their level
    return sum(draw(shape) * sign(shape) * 2.0 ** (-7 - 8 * r) for r in range(6))

def signs(s): return rng.choice([-1.0, 0.0, 0.0, 1.0], s)
def ones(s): return np.ones(s)
def pow2(s): return 2.0 ** rng.integers(5, 7, s)
def big(s): return rng.integers(64, 128, s).astype(float)

M, N = 140, 300
# sparse power-of-two slices: sums that are powers of two units
for K, nprod in [(64, 15), (300, 21)]:
    check("pow2", slices((M, K), pow2, signs), slices((K, N), pow2, signs), nprod, rows=range(0, M, 9))
# all slices positive: every product's sum passes 2^24 units, so groups carry
for K, nprod in [(600, 21), (1100, 15)]:
    check("carry", slices((M, K), big, ones), slices((K, N), big, ones), nprod, rows=(0, 127, 128, M - 1))
# one chunk, partial chunks, and a K whose fourth diagonal rounds (K above 8097)
for K, nprod in [(1, 21), (255, 21), (257, 10), (8200, 10)]:
    check("uniform", rng.random((M, K)) * 2 - 1, rng.random((K, N)) * 2 - 1, nprod, rows=(0, 64, 139))
# groups of fewer products than the diagonal has (long K)
check("long", rng.random((3, 20000)) * 2 - 1, rng.random((20000, N)) * 2 - 1, 21)
# results that cancel: last places far below the products' magnitude
A = rng.random((M, 200)) * 2 - 1
B = rng.random((200, N)) * 2 - 1
check("cancel", np.hstack([A, A]), np.vstack([B, -B * (1 + 2.0 ** -20)]), 21, rows=range(0, M, 7))
# operands of small and of large magnitude: the last products' units near the ends of the
# range in which the tensor cores' FP32 sums are exact (2^-126 is the smallest)
for ea, eb in [(-40, -30), (-30, -20), (-20, -20), (60, 40), (45, 60)]:
    check("scale", (rng.random((M, 300)) * 2 - 1) * 2.0 ** ea, (rng.random((300, N)) * 2 - 1) * 2.0 ** eb, 21, rows=(0, 139))
# levels per row / column of very different sizes, then with a zero vector and integer vectors
# (levels that end early) among them
A = (rng.random((M, 500)) * 2 - 1) * np.exp2(rng.integers(-20, 20, (M, 1)))
B = (rng.random((500, N)) * 2 - 1) * np.exp2(rng.integers(-20, 20, (1, N)))
check("rowcol", A, B, 21, rowcol=True)
A[3] = 0.0
A[5] = rng.integers(-8, 9, 500)
B[:, 7] = 0.0
B[:, 70] = rng.integers(-8, 9, 500)
check("rowcol zero", A, B, 21, rowcol=True)
check("rowcol zero", A, B, 10, rowcol=True)
# a vector whose levels do not fall in steps of 8
A[9] = np.where(rng.random(500) < 0.5, 1.0, 2.0 ** -30 * rng.random(500))
check("rowcol gap", A, B, 15, rowcol=True)
print("ok")
"""


@pytest.mark.parametrize("tile", ["128x64", "128x128", "128x256", "256x256"])
def test_groups_on_every_tile_shape(tile):
    env = dict(os.environ, EMU_F64_TILE=tile)
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr[-2000:]
