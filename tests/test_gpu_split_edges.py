"""The persistent split kernels at their edges, against the FP64 apply of the same
operands (itself against the oracle in test_gpu_tile_edges).

Tile edges: sectors one below, at and above 8, 16, 32 and 64 of the split-BF16
kernel's tiles, 16-wide K steps, pieces of 64 and fold groups of two.  Many items: an
MPO bond of 2500 channels on small sectors, 6594 tiles in S1 or 43 per CTA, beyond the
40 whose records are kept in shared memory, and S3 chains of 2500 segments shared by
several CTAs.

Per right-sector group, error over the group's largest |y|.  A product is short by
the dropped level pairs, 3 2^-16 of it (x3) or 3 2^-24 (x6), in both GEMMs, and adds
in random sign like the products themselves (and T1 is rounded to FP32): some 1e-4
and 4e-7, ten times that allowed.  Exact split: 1e-8 as in test_gpu_tile_edges."""
import os
import subprocess
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import _layout as lay  # noqa: E402

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHARGES = [(-1, -1), (-1, 1), (0, -2), (0, 0), (0, 2), (1, -1), (1, 1), (2, 0)]
TABLES = [(1, 1, 1, 1, 1, 1, 1, 1), (7, 8, 9, 3, 4, 5, 1, 2), (15, 16, 17, 33, 8, 1, 7, 9), (31, 32, 33, 65, 63, 64, 16, 2),
          (129, 1, 64, 128, 127, 2, 65, 130)]
TOL = {1: 1e-3, 2: 4e-6, 3: 1e-8}

CHILD = r"""
import sys, numpy as np
sys.path[:0] = [{root!r}, {tests!r}]
import test_gpu_split_edges as t
from paper_2212_11973_gb300 import tantrg as tt
t.check(tt, {case!r}, {precs!r})
"""


def edge_case(left, right):
    from oracle import model as om
    from oracle import mpo as ompo
    Ws = ompo.hubbard_mpo(om.Model(6, 2, False, 1.0, 6.0, -0.4, 1))
    ch = lay.mpo_channel_charges(Ws)
    sec = [[(n, s, d) for (n, s), d in zip(CHARGES, TABLES[k])] for k in (left, right)]
    return ch[5], ch[6], lay.mpo_terms(Ws[5]), *sec


def many_items():
    nw = 2500
    chan = [(0, 0)] * nw
    terms = [(w, w, s, s, 1.0 + 0.25 * ((7 * w + s) % 5)) for w in range(nw) for s in range(4)]
    sec = [(n, s, 8) for n, s in CHARGES]
    return chan, chan, terms, sec, sec


def check(tt, case, precs):
    from paper_2212_11973_gb300 import workloads as wl
    chl, chr_, terms, SL, SR = many_items() if case is None else edge_case(*case)
    nx, nl, nr = tt.layout_sizes_terms(chl, chr_, SL, SR)
    L, R, x = (wl.random_vector(n, 40 + k) for k, n in enumerate((nl, nr, nx)))
    ctx = tt.Context()
    want = tt.heff_apply_terms_host(ctx, chl, chr_, terms, 0, SL, SR, L, R, x)
    groups, _ = lay.right_groups(SL, SR)
    for prec in precs:
        y = tt.heff_apply_terms_host(ctx, chl, chr_, terms, prec, SL, SR, L, R, x)
        for off, rows, dr in groups:
            a, b = y[off:off + rows * dr], want[off:off + rows * dr]
            assert np.abs(a - b).max() <= TOL[prec] * np.abs(b).max(), (case, prec, off, rows, dr)
    ctx.close()


def _run(case, precs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"), case=case, precs=precs)
    p = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, TT_GEMM="tcp"), capture_output=True, text=True,
                       timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]


@pytest.mark.parametrize("left", range(5))
@pytest.mark.parametrize("right", [1, 3, 4])
def test_split_bf16_tile_edges(left, right):
    _run((left, right), (1, 2))


def test_more_items_than_the_table_holds():
    _run(None, (1, 2, 3))
