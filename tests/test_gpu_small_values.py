"""Outputs below the FP32 normal range: a split-BF16 apply whose operands are scaled
by powers of two so that the result is 2^-135 of the unscaled one, its two-float
sums FP32 subnormals.  They keep their values (multiples of 2^-149, some fifty
roundings of half of one against results of up to 2^-130: below 1e-3 of the largest)
and are not dropped.  The persistent kernel is forced in a child process (the
choice is read once per process)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys, numpy as np
sys.path.insert(0, {root!r})
from paper_2212_11973_gb300 import tantrg as tt, workloads as wl
ctx = tt.Context()
mpo = tt.Mpo(ctx, 4, 2, False, t=1.0, U=8.0, mu=-1.0, form=1)
SL = wl.gaussian_sectors(60, 1.0, wl.SECTOR_CHARGES, 5)
SR = wl.gaussian_sectors(57, 1.0, wl.SECTOR_CHARGES, 6)
nx, nl, nr = tt.layout_sizes(mpo, 3, SL, SR)
L, R, x = wl.random_vector(nl, 7), wl.random_vector(nr, 8), wl.random_vector(nx, 9)
y = [tt.heff_apply_host(ctx, mpo, 3, {prec}, SL, SR, L * 2.0 ** a, R * 2.0 ** b, x * 2.0 ** c)
     for a, b, c in ((0, 0, 0), (-40, -55, -40))]
np.save({out!r}, np.stack(y))
"""


@pytest.mark.parametrize("kernel", ["tcp", "mma"])
@pytest.mark.parametrize("prec", [1, 2])
def test_subnormal_sums_are_kept(tmp_path, kernel, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = str(tmp_path / "y.npy")
    p = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, out=out, prec=prec)],
                       env=dict(os.environ, TT_GEMM=kernel), capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    y, small = np.load(out)
    assert np.abs(small * 2.0 ** 135 - y).max() <= 1e-3 * np.abs(y).max()
