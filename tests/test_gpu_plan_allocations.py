"""Plans come to the device whole: once a state's plans are built (a call of zero
steps builds them), the first step allocates its environments and counters, at
most one buffer per bond and a few more, and nothing per gauge product (FP64 mode
with the double-float kernel preferred for them: it must not matter there)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import test_gpu_cholqr_edges as edges  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gemm", [None, "df"])
def test_first_step_allocates_no_tile_lists(gemm, tmp_path, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11973_gb300 import tantrg as tt
    if gemm:
        monkeypatch.setenv("TT_QR_GEMM", gemm)
    path = str(tmp_path / "s.ttck")
    edges._checkpoint(path, edges._tables(edges.SIZES["small"]))
    count = [0]
    alloc = torch.cuda.caching_allocator_alloc

    def counted(*a):
        count[0] += 1
        return alloc(*a)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", counted)
    ctx = tt.Context()
    mpo = tt.Mpo(ctx, 3, 2, False, t=1.0, U=4.0, mu=-0.3, form=1)
    rho = tt.Rho.load(ctx, mpo, path, tt.run_opts(600, 4, 0))
    rho.step(0.05, 0)
    before = count[0]
    rho.step(0.05, 1)
    assert count[0] - before <= 6 + 4, count[0] - before
    rho.close()
    mpo.close()
    ctx.close()
