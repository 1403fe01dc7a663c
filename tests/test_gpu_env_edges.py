"""Environment updates on the exact split at the edges of the 64 x 64 x 32
tiles: a beta-step of a 3x2 ladder whose bonds carry sectors one below, at and
above 8, 32 and 64 states (ragged rows, columns and K, tiles with idle warps),
against the same step in FP64.  Each digit GEMM is within about 2^-32 = 2.3e-10
of its rows' bounds; some ten updates and eight applies of it adding in random
sign stay below 1e-8 in the observables."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import test_gpu_cholqr_edges as edges  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = {"one tile": {(0, 0): 33, (1, 1): 32, (1, -1): 31, (-1, 1): 7, (-1, -1): 8, (2, 0): 9, (0, 2): 1},
         "several": {(0, 0): 129, (1, 1): 65, (1, -1): 64, (-1, 1): 63, (-1, -1): 72, (2, 0): 2, (0, 2): 17}}


@pytest.mark.parametrize("size", sorted(SIZES))
def test_beta_step_against_fp64(size, tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11973_gb300 import tantrg as tt
    path = str(tmp_path / "s.ttck")
    edges._checkpoint(path, edges._tables(SIZES[size]))
    got = []
    for prec in (0, 3):
        ctx = tt.Context()
        mpo = tt.Mpo(ctx, 3, 2, False, t=1.0, U=4.0, mu=-0.3, form=1)
        rho = tt.Rho.load(ctx, mpo, path, tt.run_opts(600, 4, prec))
        rho.step(0.05, 1)
        got.append(rho.measure())
        rho.close()
        mpo.close()
        ctx.close()
    for k in ("energy_per_site", "density", "double_occ", "lnZ"):
        a, b = got[1][k], got[0][k]
        assert abs(a - b) <= 1e-8 * max(1.0, abs(b)), (k, a, b)
