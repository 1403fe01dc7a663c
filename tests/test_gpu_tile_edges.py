"""Site H_eff apply at the edges of the GEMM tiles: sector dimensions one below,
at and one above the 8, 16, 32 and 64 of the tile sizes, against the oracle's
dense definition.  Per right-sector group the error over the group's largest
|y| stays below 1e-12 in FP64 (sums of at most ~1500 products of order one:
1500 2^-53 = 1.7e-13 of the largest product sum) and below 1e-8 for the
exact-accumulation split (2^-32 of each row's bound per operand, ~1e3 of them
adding in random sign)."""
import os
import sys

import numpy as np
import pytest

from paper_2212_11973_gb300 import workloads as wl

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import _layout as lay  # noqa: E402

pytestmark = pytest.mark.gpu

CHARGES = [(-1, -1), (-1, 1), (0, -2), (0, 0), (0, 2), (1, -1), (1, 1), (2, 0)]
TABLES = [(1, 1, 1, 1, 1, 1, 1, 1), (7, 8, 9, 3, 4, 5, 1, 2), (15, 16, 17, 33, 8, 1, 7, 9), (31, 32, 33, 65, 63, 64, 16, 2)]


@pytest.mark.parametrize("left", range(4))
@pytest.mark.parametrize("right", [1, 3])
def test_heff_apply_at_tile_edges(left, right):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import model as om
    from oracle import mpo as ompo
    from oracle import tantrg as ot
    from paper_2212_11973_gb300 import tantrg as tt
    Ws = ompo.hubbard_mpo(om.Model(6, 2, False, 1.0, 6.0, -0.4, 1))
    j, ch = 5, lay.mpo_channel_charges(Ws)
    SL = [(n, s, d) for (n, s), d in zip(CHARGES, TABLES[left])]
    SR = [(n, s, d) for (n, s), d in zip(CHARGES, TABLES[right])]
    nx, nl, nr = tt.layout_sizes_terms(ch[j], ch[j + 1], SL, SR)
    L, R, x = (wl.random_vector(n, 900 + 10 * left + right + k) for k, n in enumerate((nl, nr, nx)))
    Y = ot.heff_site(lay.env_to_dense(L, SL, ch[j]), Ws[j], lay.env_to_dense(R, SR, ch[j + 1]),
                     lay.site_to_dense(x, SL, SR))
    want = lay.dense_to_site(Y, SL, SR)
    groups, _ = lay.right_groups(SL, SR)
    ctx = tt.Context()
    for prec, tol in ((0, 1e-12), (3, 1e-8)):
        y = tt.heff_apply_terms_host(ctx, ch[j], ch[j + 1], lay.mpo_terms(Ws[j]), prec, SL, SR, L, R, x)
        for off, rows, dr in groups:
            a, b = y[off:off + rows * dr], want[off:off + rows * dr]
            assert np.abs(a - b).max() <= tol * np.abs(b).max(), (prec, off, rows, dr)
    ctx.close()
