"""Waits that run out in the middle of a persistent tcgen05 GEMM: limits from
below to above what a chain of segments takes, so that the roles of a CTA see the
abort at any of their steps.  Every apply ends, with its result or with
TT_ERR_TIMEOUT, and the next one with the usual limit is right."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys, numpy as np
sys.path.insert(0, {root!r})
from paper_2212_11973_gb300 import tantrg as tt, workloads as wl
ctx = tt.Context()
mpo = tt.Mpo(ctx, 6, 4, True, t=1.0, U=4.0, mu=-0.3, form=1)
SL = wl.gaussian_sectors(300, 1.5, wl.SECTOR_CHARGES, 1)
SR = wl.gaussian_sectors(300, 1.5, wl.SECTOR_CHARGES, 2)
nx, nl, nr = tt.layout_sizes(mpo, 11, SL, SR)
L, R, x = wl.random_vector(nl, 3), wl.random_vector(nr, 4), wl.random_vector(nx, 5)
y0 = tt.heff_apply_host(ctx, mpo, 11, {prec}, SL, SR, L, R, x)
ended = [0, 0]
for wait in [1e-7 * 1.6 ** k for k in range(16)]:
    ctx.set_wait_limit(wait)
    try:
        y = tt.heff_apply_host(ctx, mpo, 11, {prec}, SL, SR, L, R, x)
        assert np.array_equal(y, y0)
        ended[0] += 1
    except tt.TTError as e:
        assert e.status == 5, e
        ended[1] += 1
    ctx.set_wait_limit(2.0)
    assert np.array_equal(tt.heff_apply_host(ctx, mpo, 11, {prec}, SL, SR, L, R, x), y0)
print("OK", ended)
"""


@pytest.mark.parametrize("kernel,prec", [("tcp", 2), ("tcz", 3)])
def test_apply_ends_under_any_limit(kernel, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, prec=prec)], env=dict(os.environ, TT_GEMM=kernel),
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0 and p.stdout.startswith("OK"), (p.stdout[-1000:], p.stderr[-2000:])
