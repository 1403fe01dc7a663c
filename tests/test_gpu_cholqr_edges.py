"""The CholeskyQR gauge at the edges of its blocks: a beta-step of a 3x2 ladder
whose middle bonds carry sectors of one below, at and above the 8-row blocks of
the factorisation, one larger than shared memory holds (233 and more, FP64
scratch path) and one of a single state, against the same step with the
Householder gauge (TT_QR=householder).  The state is a random right-canonical
one (all sectors well conditioned), so both gauges give the same factors up to
rounding: observables to 1e-11 in FP64 (sums of ~1e5 products), 1e-8 on the
exact split (digits to 2^-32, double-float factor)."""
import os
import struct
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import _layout as lay  # noqa: E402

pytestmark = pytest.mark.gpu

PAIRS = lay.pair_table()
SIZES = {"small": {(0, 0): 9, (1, 1): 8, (1, -1): 7, (-1, 1): 17, (-1, -1): 16, (2, 0): 1, (0, 2): 15},
         "large": {(0, 0): 240, (1, 1): 100, (1, -1): 33, (-1, 1): 31, (-1, -1): 64, (2, 0): 3, (0, 2): 5}}


def _tables(mid):
    """Bond tables of a 6-site chain: `mid` wherever the neighbours can hold it."""
    tab = [{(0, 0): 1}] + [dict(mid) for _ in range(5)] + [{(0, 0): 1}]
    while True:
        old = [dict(t) for t in tab]
        for k in (1, 2, 3, 4, 5, 4, 3, 2, 1):
            new = {}
            for q, d in tab[k].items():
                left = sum(len(s) * tab[k - 1].get((q[0] - p[0], q[1] - p[1]), 0) for p, s in PAIRS.items())
                right = sum(len(s) * tab[k + 1].get((q[0] + p[0], q[1] + p[1]), 0) for p, s in PAIRS.items())
                if min(d, left, right) > 0:
                    new[q] = min(d, left, right)
            tab[k] = new
        if tab == old:
            return [[(n, s, d) for (n, s), d in sorted(t.items())] for t in tab]


def _checkpoint(path, tab):
    rng = np.random.default_rng(2212)
    with open(path, "wb") as f:
        f.write(b"TTRHO001" + struct.pack("<iddd", 6, 0.4, 0.0, 0.0))
        for t in tab:
            f.write(struct.pack("<i", len(t)))
            for v in t:
                f.write(struct.pack("<iii", *v))
        for j in range(6):
            blocks, total = lay.site_blocks(tab[j], tab[j + 1])
            x = np.zeros(total)
            for l, (_, _, dl) in enumerate(tab[j]):
                mine = [(o, len(PAIRS[p]) * tab[j + 1][r][2]) for o, ll, p, r in blocks if ll == l]
                M = rng.standard_normal((dl, sum(c for _, c in mine)))
                if j > 0:
                    M = np.linalg.qr(M.T)[0].T
                at = 0
                for o, c in mine:
                    x[o:o + dl * c] = M[:, at:at + c].reshape(-1)
                    at += c
            if j == 0:
                x /= np.linalg.norm(x)
            f.write(struct.pack("<q", total) + x.tobytes())


@pytest.mark.parametrize("size,prec,tol", [("small", 0, 1e-11), ("large", 0, 1e-11), ("small", 3, 1e-8),
                                           ("large", 3, 1e-8)])
def test_beta_step_against_householder(size, prec, tol, tmp_path, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11973_gb300 import tantrg as tt
    tab = _tables(SIZES[size])
    path = str(tmp_path / "s.ttck")
    _checkpoint(path, tab)
    got = {}
    for gauge in ("cholesky", "householder"):
        monkeypatch.setenv("TT_QR", gauge)
        ctx = tt.Context()
        mpo = tt.Mpo(ctx, 3, 2, False, t=1.0, U=4.0, mu=-0.3, form=1)
        rho = tt.Rho.load(ctx, mpo, path, tt.run_opts(600, 4, prec))
        rho.step(0.05, 1)
        got[gauge] = rho.measure()
        assert gauge == "householder" or rho.stats()["qr_fallbacks"] == 0
        rho.close()
        mpo.close()
        ctx.close()
    for k in ("energy_per_site", "density", "double_occ", "lnZ"):
        a, b = got["cholesky"][k], got["householder"][k]
        assert abs(a - b) <= tol * max(1.0, abs(b)), (k, a, b)
