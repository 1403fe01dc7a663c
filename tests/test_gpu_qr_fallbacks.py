"""tt_qr_device where the grid-wide kernel does not apply, gives up, or must not
disturb what else lives in the context: outputs that overlap the input, more
columns than the CTAs' shared memory holds, a wait limit of zero, and a captured
beta-step beside it.  Householder: |A - Q R|_F <= c n u |A|_F and |Q^T Q - I|_max
with c a few (n = 609: 3 x 609 x 1.1e-16 = 2e-13)."""
import time

import numpy as np
import pytest

from paper_2212_11973_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11973_gb300 import tantrg
    tantrg.load_library()
    return tantrg


def _good(A, Q, R, tol):
    assert np.array_equal(R, np.triu(R)) and (np.diag(R) >= 0).all()
    assert np.linalg.norm(A - Q @ R) <= tol * np.linalg.norm(A)
    assert np.abs(Q.T @ Q - np.eye(A.shape[1])).max() <= tol


def test_output_over_the_input(tt):
    import torch
    m, n = 300, 20
    A = np.random.default_rng(1).standard_normal((m, n))
    ctx = tt.Context()
    buf = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()  # column-major
    R = torch.empty((n, n), dtype=torch.float64, device="cuda")
    tt._check(ctx.h, tt.load_library().tt_qr_device(ctx.h, buf.data_ptr(), m, n, buf.data_ptr(), R.data_ptr()))
    _good(A, buf.cpu().numpy().T, R.cpu().numpy().T, 1e-13)
    ctx.close()


def test_more_columns_than_shared_memory_holds(tt):
    import torch
    A = np.random.default_rng(2).standard_normal((4096, 609))
    ctx = tt.Context()
    Q, R = tt.qr_device(ctx, torch.from_numpy(A).cuda())
    _good(A, Q.cpu().numpy(), R.cpu().numpy(), 3e-13)
    ctx.close()


def test_accepted_under_a_wait_limit_of_zero(tt):
    import torch
    A = np.random.default_rng(3).standard_normal((700, 160))
    ctx = tt.Context()
    ctx.set_wait_limit(0.0)
    Q, R = tt.qr_device(ctx, torch.from_numpy(A).cuda())
    _good(A, Q.cpu().numpy(), R.cpu().numpy(), 1e-13)
    ctx.set_wait_limit(2.0)
    Q, R = tt.qr_device(ctx, torch.from_numpy(A).cuda())
    _good(A, Q.cpu().numpy(), R.cpu().numpy(), 1e-13)
    ctx.close()


@pytest.mark.parametrize("m,n", [(333, 37), (4097, 9)])
def test_captured_step_survives(tt, m, n):
    """A QR between the steps of a state leaves its captured step as it is: queueing
    a replay takes some 0.1 ms of the host, capturing again several ms."""
    import torch
    cfg = wl.LADDER_2x4
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = tt.Context(stream=stream)
        mpo = tt.Mpo(ctx, cfg.Lx, cfg.Wy, cfg.periodic, t=cfg.t, U=cfg.U, mu=cfg.mu, form=cfg.form)
        rho = tt.Rho(ctx, mpo, cfg.beta0, tt.run_opts(cfg.D, cfg.krylov, 0))
        rho.grow(cfg.dtau, 0.2)
        A = torch.randn((m, n), dtype=torch.float64, device="cuda")

        def host_ms(qr):
            out = []
            for _ in range(5):
                if qr:
                    tt.qr_device(ctx, A)
                rho.stats()  # (ends the statistics window and waits)
                t0 = time.perf_counter()
                rho.step(cfg.dtau, 1)
                out.append(1e3 * (time.perf_counter() - t0))
            return sorted(out)[2]

        rho.step(cfg.dtau, 2)
        alone = host_ms(False)
        beside = host_ms(True)
        assert beside <= 3 * alone + 0.5, (alone, beside)
        rho.close()
        mpo.close()
        ctx.close()
