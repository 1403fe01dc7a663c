"""The CholeskyQR gauge where a sector's triangle just fits shared memory (232
states) and just does not (233), with smaller ones and a larger one in the same
launch: a beta-step against the Householder gauge, as in test_gpu_cholqr_edges
(1e-11 in FP64, 1e-8 on the exact split)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import test_gpu_cholqr_edges as edges  # noqa: E402

pytestmark = pytest.mark.gpu
SIZES = {(0, 0): 256, (1, 1): 233, (1, -1): 232, (-1, 1): 216, (-1, -1): 192, (2, 0): 24, (0, 2): 8}


def test_the_state_has_these_sectors():
    assert {(n, s): d for n, s, d in edges._tables(SIZES)[3]} == SIZES


@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (3, 1e-8)])
def test_beta_step_against_householder(prec, tol, monkeypatch, tmp_path):
    monkeypatch.setitem(edges.SIZES, "limit", SIZES)
    edges.test_beta_step_against_householder("limit", prec, tol, tmp_path, monkeypatch)
