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


# Each of the small products of a bf16x6 product alone decides the result:
# columns in pairs (a b - a b', b' = b without its last plane) or fours
# ((a1 + a2)(b1 + b2) - a1 (b1 + b2) - (a1 + a2) b1 + a1 b1 = a2 b2) whose other
# products cancel.  The products go through o_proj's inputs with one token per
# sequence (attention is then v = RMSNorm(x) Wv^T) and x = +-1, so that the
# operands are +-g and Wv themselves.
#
# Tolerance: a column's large products are below 4 and cancel, and what the
# accumulator cuts off is at most about one unit of 2^-23 of them per MMA of the
# large products (two per 32 terms): 2 (K / 32) 2^-21 in all, 2^-19 at K = 64, against
# sums of K / 2 terms of 2^-17.5 (K / 4 of 2^-17 for a2 b2), whose largest is about
# 2^-12.5: a hundredth.  A quarter of the largest is allowed; a missing
# product is off by all of it.
def _bf16(v):
    u = np.asarray(v, dtype=np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32)


def _planes(r, shape):
    """Three bf16 values of falling size whose sum is exact in fp32 and splits
    back into them."""
    p1 = _bf16(r.uniform(1.02, 2.0, shape) * r.choice([-1.0, 1.0], shape))
    p2 = _bf16(np.ldexp(r.integers(65, 128, shape) * r.choice([-1.0, 1.0], shape), -15))
    p3 = _bf16(np.ldexp(r.integers(16, 32, shape) * r.choice([-1.0, 1.0], shape), -22))
    v = (p1 + p2 + p3).astype(np.float32)
    assert np.array_equal(v.astype(np.float64), p1.astype(np.float64) + p2 + p3)
    q1 = _bf16(v)
    q2 = _bf16(v - q1)
    assert np.array_equal(q1, p1) and np.array_equal(q2, p2) and np.array_equal(_bf16(v - q1 - q2), p3)
    return p1, (p1 + p2).astype(np.float32), v


@pytest.mark.parametrize("K", [64, 256])
@pytest.mark.parametrize("which", ["a1b2", "a2b1", "a1b3", "a3b1", "a2b2"])
def test_every_small_product_counts(which, K):
    r = np.random.default_rng(K)
    T, N = 128, 64
    per = 4 if which == "a2b2" else 2
    p = K // per
    a1, a12, a123 = _planes(r, p)
    b1, b12, b123 = _planes(r, (N, p))
    cols = {"a1b2": ([a1, a1], [b12, b1], [1, -1]), "a2b1": ([a12, a1], [b1, b1], [1, -1]),
            "a1b3": ([a1, a1], [b123, b12], [1, -1]), "a3b1": ([a123, a12], [b1, b1], [1, -1]),
            "a2b2": ([a12, a1, a12, a1], [b12, b12, b1, b1], [1, -1, -1, 1])}[which]
    g = np.stack(cols[0], axis=-1).reshape(K)
    Wv = np.stack(cols[1], axis=-1).reshape(N, K)
    x = (r.choice([-1.0, 1.0], (T, p))[:, :, None] * np.array(cols[2])).reshape(T, K)
    want = (x * g) @ Wv.astype(np.float64).T
    f = 64
    W = {"g1": g, "Wq": np.zeros((N, K)), "Wk": np.zeros((N, K)), "Wv": Wv, "Wo": np.zeros((K, N)), "g2": np.ones(K),
         "Wg": np.zeros((f, K)), "Wu": np.zeros((f, K)), "Wd": np.zeros((K, f))}
    dims = rq.block_dims(K, 1, 1, N, f, rms_eps=1e-12)   # (1 + eps rounds to 1)
    ws = rq.workspace(rq.realq_block_workspace_size(dims, T, 1))
    out = torch.empty((T, N), dtype=torch.float32, device="cuda")
    rq.realq_block_module_inputs(dims, {k: _dev(v) for k, v in W.items()}, _dev(x.reshape(T, 1, K)), "o_proj", out, ws)
    rq.realq_workspace_status(ws)
    err = np.abs(out.cpu().numpy() - want).max() / np.abs(want).max()
    print(f"\n{which}, K = {K}: {err:.2e} of the largest")
    assert err <= 0.25
