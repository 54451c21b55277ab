"""The FP64 product-sum's 256 x 128 tiles on CTA pairs: forced for every result
(the inputs of the other shapes' tests), and as the halves that a second launch
takes of the last, partial wave of 256 x 256 tiles."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import paper_2609_04663_gb300 as emu
import synth
from helpers import device, to_dev
from test_gpu_groups import CHILD as GROUPS
from test_gpu_tile_option import _run64

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_groups_on_256x128_tiles():
    env = dict(os.environ, EMU_F64_TILE="256x128")
    code = GROUPS.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr[-2000:]


def test_every_path_on_the_remaining_shapes():
    ref = _run64(None)
    for tile in ("256x128", "128x64"):
        assert _run64(tile) == ref, tile


@pytest.mark.parametrize("rowcol", [False, True])
@pytest.mark.parametrize("K,nprod", [(40, 21), (300, 15)])
def test_halves_past_the_last_column(K, nprod, rowcol):
    """Two launches, an odd number of 128-column tiles (the last 256 x 256 tile has
    one half only), a ragged last pair, and diagonals that round (K > 31)."""
    M, N = 4090, 3900
    dev = device()
    assert emu.emu_prodsum_f64_launches(M, N) == 2 and emu.emu_prodsum_f64_tile_rows(M, N) == 256
    assert ((N + 127) // 128) % 2 == 1
    A, B = synth.gemm_inputs("f64", M, N, K, 21)
    C, ws = (emu.gemm_f64_rowcol if rowcol else emu.gemm_f64)(to_dev(A, dev), to_dev(B, dev), nprod)
    assert emu.read_flags(ws) == 0
    Cn = C.cpu().numpy()
    rows = [0, 127, 2047, 2048, 3333, 3967, 3968, 4089]
    if rowcol:                                       # a row's levels are its own
        want = oracle.gemm_f64_rowcol(np.ascontiguousarray(A[rows]), B, nprod)[0]
    else:
        want = np.vstack([oracle.gemm_f64(A, B, nprod, rows=(r, r + 1))[0] for r in rows])
    assert np.array_equal(Cn[rows], want)
