"""The preparation at the edges of its blocks (64-wide pieces of a cluster's
block of up to 512 columns, 512-wide blocks beyond): the factor against fp64
on the host, its structure, and the failing column of a Hessian that is not
positive definite.

Tolerance: U = R^-1 of a damped H with condition number at most about 1 / damp
= 100 n / n: fp32 arithmetic with sums of at most 512 terms taken in fp32
gives a few units of 2^-24 times the growth of the inverse; 2e-6 of max |U| is
twenty times the error that fp32 rounding of H alone makes (1e-7)."""
import numpy as np
import pytest
import torch

import paper_2609_00049_gb300 as rq
from paper_2609_00049_gb300 import layer

pytestmark = pytest.mark.gpu


def _case(n, seed=5):
    r = np.random.default_rng(seed + n)
    X = r.standard_normal((max(64, 2 * n), n)).astype(np.float32)
    X[:, :: max(1, n // 3)] *= 5.0
    return (X.T.astype(np.float64) @ X.astype(np.float64)).astype(np.float32), X.shape[0]


def _exact(H, T, damp):
    Hb = (H / np.float32(T)).astype(np.float64)
    Hd = Hb + damp * np.mean(np.diag(Hb)) * np.eye(len(Hb))
    L = np.linalg.cholesky(Hd[::-1, ::-1])
    return np.linalg.inv(L)[::-1, ::-1]


@pytest.mark.parametrize("n", [1, 33, 64, 65, 127, 200, 511, 512, 513, 577, 1001, 1024, 1030, 1537, 2052])
def test_factor_matches_fp64_at_block_edges(n):
    H, T = _case(n)
    p = layer.prepare(torch.from_numpy(H).cuda(), T, 0.01)
    U = p.U.cpu().numpy().astype(np.float64)
    want = _exact(H, T, 0.01)
    assert np.array_equal(U, np.triu(U))
    err = np.abs(U - want).max() / np.abs(want).max()
    print(f"\nn = {n}: {err:.2e} of max |U|")
    assert err <= 2e-6


@pytest.mark.parametrize("n,bad", [(96, 70), (300, 5), (512, 448), (700, 650), (700, 100), (1300, 513)])
def test_a_bad_pivot_reports_its_column(n, bad):
    # diagonal H: the pivot of column j is H_jj + lambda whatever came before
    H = np.eye(n, dtype=np.float32)
    H[bad, bad] = -3.0
    with pytest.raises(rq.RealqError) as e:
        layer.prepare(torch.from_numpy(H).cuda(), 1, 0.01)
    assert e.value.status == rq.REALQ_ERR_NOT_SPD and e.value.fail_col == bad
