"""tt_qr_device over the whole GPU, at the edges of its layout: 256 rows per
register step, one to several columns per CTA (152 SMs), the size beyond which
one CTA factorises, rank-deficient and zero columns, output that overlaps the
input.  Householder: |A - Q R|_F <= c n u |A|_F and |Q^T Q - I|_max small with c
a few; n <= 310 gives 310 x 1.1e-16 x 3 = 1e-13."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_11973_gb300 import tantrg
    tantrg.load_library()
    return tantrg


def _check(tt, A):
    import torch
    ctx = tt.Context()
    Q, R = tt.qr_device(ctx, torch.from_numpy(A).cuda())
    Q, R = Q.cpu().numpy(), R.cpu().numpy()
    assert np.array_equal(R, np.triu(R)) and (np.diag(R) >= 0).all()
    assert np.linalg.norm(A - Q @ R) <= 1e-13 * max(np.linalg.norm(A), 1e-300)
    assert np.abs(Q.T @ Q - np.eye(A.shape[1])).max() <= 1e-13
    ctx.close()


@pytest.mark.parametrize("m,n", [(1, 1), (5, 5), (255, 1), (257, 2), (512, 151), (513, 153), (700, 310), (1025, 64),
                                 (2304, 160), (2305, 40), (4096, 9), (4097, 9)])
def test_sizes(tt, m, n):
    _check(tt, np.random.default_rng(m + 7 * n).standard_normal((m, n)))


def test_deficient_columns(tt):
    A = np.random.default_rng(3).standard_normal((300, 12))
    A[:, 4] = A[:, 1]
    A[:, 7] = 0.0
    A[:, 9] = np.eye(300)[9] * -2.0
    _check(tt, A)


def test_upper_triangular_input(tt):
    A = np.vstack([-np.triu(np.random.default_rng(4).uniform(1, 2, (20, 20))), np.zeros((9, 20))])
    _check(tt, A)
