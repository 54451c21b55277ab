"""Levels per row / column: all-zero vectors beside vectors whose levels lie far
from zero.  An all-zero row or column has no level; its elements of C must be
zero whatever levels the other operand's vectors have, on every tile shape (the
switch is read once per process, so each shape runs in a child process).  The
columns' levels here, -47, -55 and -63, are the ones at which a rounding
constant formed with level 0 for a zero row had an all-ones exponent field on
the diagonals 5, 4 and 3."""
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
rng = np.random.default_rng(6)

def vectors(rows, cols, exps, zero):
    # row i: entries of magnitude 2^(e-1) to 2^e, so its first level is e = exps[i % len(exps)]
    X = rng.uniform(0.5, 1.0, (rows, cols)) * rng.choice([-1.0, 1.0], (rows, cols))
    X *= np.exp2(np.resize(exps, rows))[:, None]
    X[zero] = 0.0
    return X

M, N = 140, 76
low, high = [-47, -63, -55, 2, -55, -47, -63], [20, 30, 25]    # seven levels: each meets every column index mod 4
for K, nprod in [(64, 15), (300, 21), (8200, 15), (8200, 10)]:
    for ea, eb in [(high, low), (low, high)]:
        A = vectors(M, K, ea, [3, 131])
        B = vectors(N, K, eb, [8, 70]).T.copy()
        C, ws = emu.gemm_f64_rowcol(to_dev(A, dev), to_dev(B, dev), nprod)
        Cn = C.cpu().numpy()
        assert not Cn[[3, 131]].any() and not Cn[:, [8, 70]].any(), (K, nprod, ea)
        want, flags = oracle.gemm_f64_rowcol(A, B, nprod)
        assert emu.read_flags(ws) == flags == 0
        assert np.array_equal(Cn, want), (K, nprod, ea)
print("ok")
"""


@pytest.mark.parametrize("tile", [None, "128x64", "256x128", "256x256"])
def test_zero_rows_and_columns_beside_distant_levels(tile):
    env = dict(os.environ)
    env.pop("EMU_F64_TILE", None)
    if tile:
        env["EMU_F64_TILE"] = tile
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr[-2000:]
