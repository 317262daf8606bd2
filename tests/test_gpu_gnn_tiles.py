"""GPU: the network at the edges of its kernels' tiles: row counts around the
64-row tiles and 32-row warps, a hub row around the 64-entry chunk, against
the float64 network with the same storage rounding. The bars are those of
test_gpu_gnn.py: 1e-2 in norm per parameter block and for the logits (bf16
operands, fp32 sums)."""

import numpy as np
import pytest

import synth
from oracle import gnn_oracle as go
from test_gpu_gnn import _norm_rel, effective_params

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_1807_10750_gb300")


@pytest.mark.parametrize("n,hub", [(31, 30), (33, 32), (63, 62), (64, 63), (65, 64), (127, 65), (128, 127),
                                   (129, 128), (257, 129), (320, 319), (4097, 640),
                                   (19500, 129), (25000, 700)])
def test_logits_and_gradients_at_tile_edges(n, hub):
    rng = np.random.default_rng(n)
    src = np.concatenate([np.zeros(hub, np.int64), rng.integers(1, n, 2 * n)])
    dst = np.concatenate([rng.permutation(np.arange(1, n))[:hub], rng.integers(1, n, 2 * n)])
    keep = src != dst
    src, dst = src[keep].astype(np.int32), dst[keep].astype(np.int32)
    w = rng.integers(-100, 101, src.size)
    w = np.where(w == 0, 1, w).astype(np.int32)
    s = rng.choice(np.array([-1, 1], np.int8), size=n)
    y = np.where(rng.random(n) < 0.8, s, -s).astype(np.int8)
    params = synth.gnn_init_params(5)
    with P.ising_create(n, src, dst, w) as h, P.ising_gnn_create(params) as net:
        P.ising_set_spins(h, s)
        z = P.ising_gnn_forward(net, h)
        loss, grad = P.ising_gnn_gradients(net, h, y)
    G = go.Graph(n, src, dst, w)
    pe = effective_params(params)
    z_rd, cache = go.forward(G, go.features(G, s), pe, storage="bf16")
    assert _norm_rel(z, z_rd) <= 1e-2
    yf = y.astype(np.float64)
    assert loss == pytest.approx(go.loss(z_rd, yf), rel=1e-3)
    g_rd = go.backward(G, pe, cache, z_rd, yf, storage="bf16")
    k = 0
    for blk, shape in go.SHAPES:
        sl = slice(k, k + int(np.prod(shape)))
        assert _norm_rel(grad[sl], g_rd[sl]) <= 1e-2, blk
        k = sl.stop
