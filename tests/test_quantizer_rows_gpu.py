"""The column-serial quantizer's eight-lanes-per-row kernel against the
pipelined one, bit for bit: row counts around its CTAs (16 rows, 32 from 4864
rows on), last blocks of every remainder, blocks of 32 and 64, group parameters
before, at the start of and inside a block, symmetric grids, scales far outside
the range of its division-free rounding, and weights on rounding ties."""
import pytest
import torch

import paper_2609_00049_gb300 as rq
from paper_2609_00049_gb300 import layer

pytestmark = pytest.mark.gpu


def _run(W0, U, q, mode):
    n = U.shape[0]
    prep = layer.Prepared(U, None, torch.zeros(n, dtype=torch.uint8, device="cuda"), 1)
    try:
        rq.realq_set_quant_kernel(mode)
        return layer.quantize(W0, prep, q, None)
    finally:
        rq.realq_set_quant_kernel(0)


@pytest.mark.parametrize("m,n,group,block,sym,scale", [
    (1, 40, 0, 128, 0, 1.0), (15, 129, 128, 128, 0, 1.0), (17, 160, 0, 128, 1, 1.0), (33, 300, 128, 128, 1, 1.0),
    (64, 333, 64, 64, 0, 1.0), (100, 96, 32, 32, 0, 1.0), (260, 384, 256, 128, 0, 1.0), (4863, 131, 128, 128, 0, 1.0),
    (4900, 257, 0, 128, 0, 1.0), (48, 256, 128, 128, 0, 1e-33), (48, 256, 128, 128, 0, 1e32), (64, 256, 128, 128, 0, 0.0)])
def test_rows_kernel_matches_the_pipelined_kernel(m, n, group, block, sym, scale):
    g = torch.Generator().manual_seed(m * 1000 + n)
    if scale == 0.0:
        # multiples of half a step of a fixed grid, and U = I: every code is a tie
        W0 = (torch.randint(-15, 16, (m, n), generator=g).float() * 0.5).cuda()
        W0[:, ::block] = 7.5
        W0[:, 1::block] = -7.5
        U = torch.eye(n, device="cuda")
    else:
        W0 = (torch.randn(m, n, generator=g) * scale).cuda()
        U = (torch.triu(torch.randn(n, n, generator=g), 1) * 0.05 + torch.diag(torch.rand(n, generator=g) + 0.5)).cuda()
    q = rq.quant_cfg(4, group, block, sym, 0.01)
    a, b = _run(W0, U, q, 0), _run(W0, U, q, 1)
    for x, y in ((a.codes, b.codes), (a.scale, b.scale), (a.zero, b.zero), (a.W, b.W)):
        assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))


def test_a_non_finite_weight_is_reported():
    W0 = torch.randn(20, 256).cuda()
    W0[7, 200] = float("nan")
    n = 256
    ws = rq.workspace(rq.realq_quantize_workspace_size(20, n, rq.quant_cfg()))
    prep = layer.Prepared(torch.eye(n, device="cuda"), None, torch.zeros(n, dtype=torch.uint8, device="cuda"), 1)
    layer.quantize(W0, prep, rq.quant_cfg(), None, ws=ws)
    with pytest.raises(rq.RealqError) as e:
        rq.realq_workspace_status(ws)
    assert e.value.status == rq.REALQ_ERR_NONFINITE
