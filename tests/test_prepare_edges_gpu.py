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


# The allocation-free entry point: blocks of 512, 256, 128 and 64 columns by
# what its scratch holds, at the widths around each change.
def _no_alloc(H, T):
    n = H.shape[0]
    U, Hbar = torch.empty_like(H), torch.empty_like(H)
    dead = torch.empty(n, dtype=torch.uint8, device="cuda")
    assert rq.realq_hessian_prepare_noalloc(H, T, 0.01, U, Hbar, dead) == -1
    return U


@pytest.mark.parametrize("n", [513, 577, 1024, 1030, 2224, 2225])
def test_no_alloc_factor_matches_fp64_at_block_edges(n):
    H, T = _case(n)
    U = _no_alloc(torch.from_numpy(H).cuda(), T).cpu().numpy().astype(np.float64)
    want = _exact(H, T, 0.01)
    assert np.array_equal(U, np.triu(U))
    assert np.abs(U - want).max() / np.abs(want).max() <= 2e-6


@pytest.mark.parametrize("n", [5216, 5217, 10816, 10817])
def test_no_alloc_factor_matches_fp64_at_wider_blocks(n):
    # (inputs as _case's and its bound; the exact factor on the GPU)
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(2 * n, n, generator=g, device="cuda")
    X[:, :: n // 3] *= 5.0
    H = X.T @ X
    U = _no_alloc(H, 2 * n)
    Hd = (H / float(2 * n)).double()
    Hd.diagonal().add_(0.01 * Hd.diagonal().mean())
    want = torch.linalg.inv(torch.linalg.cholesky(Hd.flip((0, 1)))).flip((0, 1))
    assert torch.equal(U, torch.triu(U))
    assert (U - want).abs().max().item() <= 2e-6 * want.abs().max().item()


@pytest.mark.parametrize("n,bad", [(700, 650), (700, 100), (2300, 2047), (2300, 255), (5300, 130)])
def test_no_alloc_reports_a_bad_pivot(n, bad):
    H = torch.eye(n, device="cuda")
    H[bad, bad] = -3.0
    with pytest.raises(rq.RealqError) as e:
        _no_alloc(H, 1)
    assert e.value.status == rq.REALQ_ERR_NOT_SPD and e.value.fail_col == bad


@pytest.mark.parametrize("n", [1024, 4096])
def test_no_alloc_updates_run_on_the_tensor_cores(n):
    H, T = torch.eye(n, device="cuda"), 1
    rq.realq_profile_enable(True)
    try:
        _no_alloc(H, T)
        kernels = rq.realq_profile_collect()
    finally:
        rq.realq_profile_enable(False)
    assert "chol_update_tc" in kernels and "trtri_update_tc" in kernels and "chol_update" not in kernels
