"""The double-float GEMM (32 x 32 tiles, two chunks of 16 K in flight) at the edges
of its tiles.  Gauge products (TT_QR_GEMM=df: at these sizes the rule would take the
FP64 kernel): a beta-step of a 3x2 ladder whose sectors lie one below, at and above 8,
16, 32, 64 and 232, rows and K ragged, against the Householder gauge; observables to
1e-8 in the exact split (double-float 2^-46 is far below its 2^-32).  Environment
updates (env_precision 2) on the same states against FP64 ones: the same bound, as
test_gpu_env_edges has it for the digit kernel."""
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import test_gpu_cholqr_edges as edges  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = dict(edges.SIZES, tile={(0, 0): 129, (1, 1): 65, (1, -1): 64, (-1, 1): 63, (-1, -1): 33, (2, 0): 31, (0, 2): 32})
KEYS = ("energy_per_site", "density", "double_occ", "lnZ")


def _step(tt, path, prec, save=None, **opts):
    ctx = tt.Context()
    mpo = tt.Mpo(ctx, 3, 2, False, t=1.0, U=4.0, mu=-0.3, form=1)
    rho = tt.Rho.load(ctx, mpo, path, tt.run_opts(600, 4, prec, **opts))
    rho.step(0.05, 1)
    o = rho.measure()
    assert rho.stats()["qr_fallbacks"] == 0
    if save:
        rho.save(save)
    rho.close()
    mpo.close()
    ctx.close()
    return [o[k] for k in KEYS]


def _near(a, b):
    assert all(abs(x - y) <= 1e-8 * max(1.0, abs(y)) for x, y in zip(a, b)), (a, b)


@pytest.fixture()
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11973_gb300 import tantrg
    return tantrg


@pytest.mark.parametrize("size", sorted(SIZES))
def test_gauge_products_in_double_float(tt, size, tmp_path, monkeypatch):
    path = str(tmp_path / "s.ttck")
    edges._checkpoint(path, edges._tables(SIZES[size]))
    out, bits = {}, {}
    for gemm in ("df", "f64"):
        monkeypatch.setenv("TT_QR_GEMM", gemm)
        out[gemm] = _step(tt, path, 3, save=str(tmp_path / gemm))
        bits[gemm] = np.fromfile(str(tmp_path / gemm), np.uint8)
    monkeypatch.setenv("TT_QR", "householder")
    _near(out["df"], _step(tt, path, 3))
    _near(out["df"], out["f64"])
    assert not np.array_equal(bits["df"], bits["f64"])  # (two kernels ran)


@pytest.mark.parametrize("size", sorted(SIZES))
def test_environments_in_double_float(tt, size, tmp_path):
    path = str(tmp_path / "s.ttck")
    edges._checkpoint(path, edges._tables(SIZES[size]))
    _near(_step(tt, path, 3, env_precision=2), _step(tt, path, 3, env_precision=1))
