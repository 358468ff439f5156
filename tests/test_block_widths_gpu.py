"""The block ops at one head width after another in one process: the attention
kernels serve a range of widths each, and a call at a narrower one must leave
the wider one's shared-memory limit alone."""
import pytest
import torch

import paper_2609_00049_gb300 as rq

pytestmark = pytest.mark.gpu


def _window(dh):
    g = torch.Generator().manual_seed(dh)
    d, f, S, L = 64, 96, 1, 70
    shape = {"g1": (d,), "Wq": (dh, d), "Wk": (dh, d), "Wv": (dh, d), "Wo": (d, dh), "g2": (d,), "Wg": (f, d), "Wu": (f, d),
             "Wd": (d, f)}
    W = {k: (torch.randn(s, generator=g) * 0.1).cuda() for k, s in shape.items()}
    dims = rq.block_dims(d, 1, 1, dh, f)
    ws = rq.workspace(rq.realq_block_workspace_size(dims, S, L))
    x, dx = torch.randn(S, L, d, generator=g).cuda(), (0.1 * torch.randn(S, L, d, generator=g)).cuda()
    y, gx = torch.empty_like(x), torch.empty_like(x)
    rq.realq_block_forward(dims, W, x, y, ws)
    rq.realq_block_window(dims, W, x, dx, torch.eye(d).cuda(), gx, ws)
    rq.realq_workspace_status(ws)
    return y, gx


@pytest.mark.parametrize("wide,narrow", [(256, 132), (32, 20), (62, 38), (126, 70)])
def test_a_wide_head_after_a_narrow_one(wide, narrow):
    first = _window(wide)
    _window(narrow)
    again = _window(wide)
    assert torch.equal(first[0], again[0]) and torch.equal(first[1], again[1])
