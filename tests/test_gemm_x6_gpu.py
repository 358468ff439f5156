"""The block ops' products as bf16x6 on the tensor cores (gemm_x6.cu) at the
edges of their tiles: a decoder block's forward with one token per sequence
(the attention is then v itself, so every output is a chain of products)
against the fp64 oracle.  Tolerance as the forward's in
test_zy_window_block_gpu.py: 1e-5 of the output's scale, for fp32 operands
with fp32-level products (each product within about 3e-7 of its scale)."""
import numpy as np
import pytest
import torch

from oracle import block as ob
import paper_2609_00049_gb300 as rq
from test_zy_window_block_gpu import _case, _dev, _f32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", [
    # (tokens, d, heads, kv heads, head dim, ffn): the smallest product that
    # takes the tensor cores and one token fewer; K slices of 32 with a
    # remainder, rows and columns one off a 128 tile; 256-wide tiles with
    # ragged edges; K of several ring rounds
    (64, 64, 1, 1, 64, 64), (63, 64, 1, 1, 64, 64), (65, 72, 1, 1, 66, 100), (127, 130, 2, 1, 64, 129),
    (129, 257, 2, 2, 128, 255), (260, 264, 4, 2, 66, 1000), (2500, 520, 8, 4, 64, 1544)])
def test_products_at_tile_edges_match_the_oracle(case):
    T, d, H, Hkv, dh, f = case
    r, P, W, dims, ws = _case(31, T, 1, d, H, Hkv, dh, f)
    x = _f32(r.standard_normal((T, 1, d)))
    want, _ = ob.block_forward(x, P)
    y = torch.empty((T, 1, d), dtype=torch.float32, device="cuda")
    rq.realq_block_forward(dims, W, _dev(x), y, ws)
    rq.realq_workspace_status(ws)
    got = y.cpu().numpy()
    err = np.abs(got - want).max() / np.abs(want).max()
    print(f"\n{case}: {err:.2e} of the output's scale")
    assert err <= 1e-5
