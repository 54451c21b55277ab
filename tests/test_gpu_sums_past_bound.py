"""FP64 products whose running sums pass 2^24 units: entries of one sign, on every
tile shape (the switch is read once per process).  While every addition is exact
the sums are reduced into the accumulator as they fill up, by both CTAs of a
duo (K up to 8097), with levels per matrix and per vector; operands whose
levels do not fall in steps of 8 keep the low words."""
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
rng = np.random.default_rng(7)
M, N, rows = 290, 270, [0, 77, 128, 255, 256, 289]
for K, nprod in [(300, 6), (2000, 10), (2000, 21), (9000, 15)]:
    A = rng.uniform(0.5, 1.0, (M, K))
    B = rng.uniform(0.5, 1.0, (K, N))
    A[77] = -A[77]
    A[255, ::2] = 1.0                                 # the largest partials: a whole number of bounds
    B[:, 130] = 1.0
    C, ws = emu.gemm_f64(to_dev(A, dev), to_dev(B, dev), nprod)
    assert emu.read_flags(ws) == 0
    Cn = C.cpu().numpy()
    for r in rows:
        assert np.array_equal(Cn[r], oracle.gemm_f64(A, B, nprod, rows=(r, r + 1))[0][0]), (K, nprod, r)
    A *= np.exp2(rng.integers(-9, 10, (M, 1)))
    B *= np.exp2(rng.integers(-9, 10, (1, N)))
    A[128] = 0.0
    C, ws = emu.gemm_f64_rowcol(to_dev(A, dev), to_dev(B, dev), nprod)
    assert emu.read_flags(ws) == 0
    assert np.array_equal(C.cpu().numpy()[rows], oracle.gemm_f64_rowcol(A[rows], B, nprod)[0]), (K, nprod, "rowcol")
# levels with a gap: 1 or a value far below
A = np.where(rng.random((M, 1500)) < 0.5, 1.0, 2.0 ** -30 * rng.random((M, 1500)))
B = rng.uniform(0.5, 1.0, (1500, N))
C, ws = emu.gemm_f64(to_dev(A, dev), to_dev(B, dev), 15)
assert emu.read_flags(ws) == 0
Cn = C.cpu().numpy()
for r in rows:
    assert np.array_equal(Cn[r], oracle.gemm_f64(A, B, 15, rows=(r, r + 1))[0][0]), ("gap", r)
print("ok")
"""


@pytest.mark.parametrize("tile", [None, "128x64", "128x128", "256x128", "128x256", "256x256"])
def test_sums_past_the_exact_bound(tile):
    env = dict(os.environ)
    env.pop("EMU_F64_TILE", None)
    if tile:
        env["EMU_F64_TILE"] = tile
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr[-2000:]
