"""States padded with directions of weight zero: their first beta-step chooses the
null directions by rounding, so it runs in a fixed arithmetic (tt_settle.cu) and
gives what it gave before the kernels of the later steps were rewritten.

Golden values (tests/golden/padded_ladders.json): six 2x8 ladders of D = 64 to
128 in each precision after one step and after five.  One step: the same state
to the last bit, only the order of the measurement's sums differs (~1e5 terms:
1e-12).  Five: four steps of the precision's own rounding on top, per apply
1e-15 in FP64, 6e-6 (x3), 2e-7 (x6), 2e-9 (exact split) of the norm, some 60 of
them a step adding in random sign in the energy of order one: 1e-11, 1e-4, 4e-6,
4e-8."""
import json
import os

import pytest

from paper_2212_11973_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "padded_ladders.json")
KEYS = ("energy_per_site", "lnZ", "double_occ")


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11973_gb300 import tantrg
    tantrg.load_library()
    return tantrg


@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (1, 1e-4), (2, 4e-6), (3, 4e-8)])
def test_golden_energies(tt, prec, tol):
    import torch
    with open(GOLDEN) as f:
        gold = json.load(f)["values"][str(prec)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = tt.Context(stream=stream)
        ws = wl.batch_ladders(6, wl.BATCH_SEED + 100)
        b = tt.Batch(ctx, ws, ws[0].beta0, tt.run_opts(0, 8, prec))
        b.pad()
        for steps, total, bound in ((1, "1", 1e-12), (4, "5", tol)):
            b.step(0.05, steps)
            for i, o in enumerate(b.measure()):
                for k in KEYS:
                    want = gold[total][k][i]
                    assert abs(o[k] - want) <= bound * max(1.0, abs(want)), (total, i, k, o[k], want)
        b.close()
        ctx.close()


def _single(tt, ctx, w, prec, calls, path=None):
    """Observables after each call of `calls` steps of one padded ladder."""
    mpo = tt.Mpo(ctx, w.Lx, w.Wy, w.periodic, t=w.t, U=w.U, mu=w.mu, form=w.form)
    opts = tt.run_opts(w.D, 8, prec)
    rho = tt.Rho(ctx, mpo, w.beta0, opts)
    rho.pad(w.D)
    if path:
        rho.save(path)
        rho.close()
        rho = tt.Rho.load(ctx, mpo, path, opts)
    out = []
    for n in calls:
        rho.step(0.05, n)
        out.append([rho.measure()[k] for k in KEYS])
    rho.close()
    mpo.close()
    return out


@pytest.mark.parametrize("prec", [0, 3])
def test_saved_before_the_first_step(tt, prec, tmp_path):
    """A padded state that is saved and loaded before its first step takes the
    same step."""
    import torch
    w = wl.batch_ladders(1, wl.BATCH_SEED + 7)[0]
    with torch.cuda.stream(torch.cuda.Stream()) as _:
        ctx = tt.Context()
        a = _single(tt, ctx, w, prec, (1, 2))
        b = _single(tt, ctx, w, prec, (1, 2), str(tmp_path / "p.ttck"))
        ctx.close()
    assert a == b


def test_batch_and_single_in_any_call_pattern(tt):
    """One step of a call, several, and the batch's graphs give the same bits (the
    first step is never captured, the second may be)."""
    import torch
    ws = wl.batch_ladders(2, wl.BATCH_SEED + 11)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = tt.Context(stream=stream)
        ends = []
        for calls in ((6,), (1, 1, 1, 3), (2, 4)):
            b = tt.Batch(ctx, ws, ws[0].beta0, tt.run_opts(0, 8, 3))
            b.pad()
            for n in calls:
                b.step(0.05, n)
            ends.append([[o[k] for k in KEYS] for o in b.measure()])
            b.close()
        ends.append([_single(tt, ctx, w, 3, (1, 5))[-1] for w in ws])
        ctx.close()
    assert all(e == ends[0] for e in ends[1:])
