"""The tensor-core Hessian and cross moment at the edges of their 256-channel
tiles (a last block of 8 to 248 channels, computed as the columns of its tiles
and stored transposed where it belongs on the rows), of the token stages and of
the token splits, with and without room for the splits' partial sums.  Inputs
are small integers, so that every sum is exact in fp32: equality."""
import numpy as np
import pytest
import torch

import paper_2609_00049_gb300 as rq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits", [True, False])
@pytest.mark.parametrize("n,T", [(64, 1), (72, 100), (248, 1030), (256, 2049), (264, 5000), (384, 3000), (520, 9000),
                                 (1000, 7777), (1288, 4096)])
def test_exact_on_integers_at_tile_edges(n, T, splits):
    g = torch.Generator().manual_seed(n + T)
    Xh = torch.randint(-3, 4, (T, n), generator=g).to(torch.bfloat16).cuda()
    Xf = torch.randint(-3, 4, (T, n), generator=g).to(torch.bfloat16).cuda()
    ws = rq.workspace(rq.realq_hessian_workspace_size(n, T, rq.REALQ_BF16, True)) if splits else None
    H0 = torch.randint(-5, 6, (n, n), generator=g).float().cuda()
    H0 = H0 + H0.T
    D0 = torch.randint(-5, 6, (n, n), generator=g).float().cuda()
    H, D, P = H0.clone(), D0.clone(), H0.clone()
    rq.realq_hessian_accumulate(Xh, H, D, Xf, ws=ws)
    rq.realq_hessian_accumulate(Xh, P, ws=ws)
    a, b = Xh.double().cpu(), Xf.double().cpu()
    assert torch.equal(H.double().cpu(), H0.double().cpu() + a.T @ a)
    assert torch.equal(D.double().cpu(), D0.double().cpu() + a.T @ a - b.T @ a)
    assert torch.equal(P, H)


@pytest.mark.parametrize("off", [(1, 0), (0, 2), (3, 1)])
def test_moments_at_any_word(off):
    """H and D as views that begin at any 4-byte word of their buffers."""
    n, T = 264, 5000
    g = torch.Generator().manual_seed(off[0] * 4 + off[1])
    Xh = torch.randint(-3, 4, (T, n), generator=g).to(torch.bfloat16).cuda()
    Xf = torch.randint(-3, 4, (T, n), generator=g).to(torch.bfloat16).cuda()
    H, D = (torch.zeros(n * n + 4, device="cuda")[o:o + n * n].view(n, n) for o in off)
    ws = rq.workspace(rq.realq_hessian_workspace_size(n, T, rq.REALQ_BF16, True))
    rq.realq_hessian_accumulate(Xh, H, D, Xf, ws=ws)
    a, b = Xh.double().cpu(), Xf.double().cpu()
    assert torch.equal(H.double().cpu(), a.T @ a)
    assert torch.equal(D.double().cpu(), a.T @ a - b.T @ a)


@pytest.mark.parametrize("splits", [True, False])
@pytest.mark.parametrize("n,T", [(128, 65536), (264, 9000), (512, 20000), (2056, 3000)])
def test_h_has_the_same_bits_with_and_without_d(n, T, splits):
    """Real-valued activations over several accumulator passes, where another
    order of the sums gives other bits (above, every order is exact)."""
    g = torch.Generator().manual_seed(n + T)
    Xh = torch.randn(T, n, generator=g).to(torch.bfloat16).cuda()
    Xf = torch.randn(T, n, generator=g).to(torch.bfloat16).cuda()
    ws = rq.workspace(rq.realq_hessian_workspace_size(n, T, rq.REALQ_BF16, True)) if splits else None
    H, D, P = (torch.zeros(n, n, device="cuda") for _ in range(3))
    rq.realq_hessian_accumulate(Xh, H, D, Xf, ws=ws)
    rq.realq_hessian_accumulate(Xh, P, ws=ws)
    assert torch.equal(P, H)


@pytest.mark.parametrize("n,T", [(264, 9000), (512, 20000)])
def test_h_has_the_same_bits_in_a_workspace_sized_without_d(n, T):
    """Room for one product's partial sums only: H as without D, and D within
    the bound of its two parts' fp32 sums (each about sqrt(T) units of 2^-24 of
    the diagonal's scale T; 1e-5 T leaves a factor of ten)."""
    g = torch.Generator().manual_seed(n + T)
    Xh = torch.randn(T, n, generator=g).to(torch.bfloat16).cuda()
    Xf = torch.randn(T, n, generator=g).to(torch.bfloat16).cuda()
    ws = rq.workspace(rq.realq_hessian_workspace_size(n, T, rq.REALQ_BF16, False))
    H, D, P = (torch.zeros(n, n, device="cuda") for _ in range(3))
    rq.realq_hessian_accumulate(Xh, H, D, Xf, ws=ws)
    rq.realq_hessian_accumulate(Xh, P, ws=ws)
    assert torch.equal(P, H)
    a, b = Xh.double().cpu(), Xf.double().cpu()
    assert (D.double().cpu() - (a.T @ a - b.T @ a)).abs().max().item() <= 1e-5 * T
