"""Tile edges, remainders and rarely taken branches of the GPU kernels, against fp64 references."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d_in,hidden", [(1, 1, 1), (33, 17, 63), (129, 64, 65), (700, 165, 130), (260, 33, 300)])
def test_mlp_gradients_at_tile_edges(soar, B, d_in, hidden):
    g = torch.Generator().manual_seed(B)
    n1, n2 = hidden * d_in, hidden * hidden
    params = 0.3 * torch.randn(soar.soar_mlp_param_count(d_in, hidden), generator=g)
    Z, target = torch.randn(B, d_in, generator=g), torch.randn(B, generator=g)
    G, loss = soar.soar_mlp_backward(params.cuda(), d_in, hidden, Z.cuda(), target.cuda())
    y = soar.soar_mlp_forward(params.cuda(), d_in, hidden, Z.cuda())

    def passes(p, z, t, abs_=False):
        """(y, loss, gradient); with abs_, every term replaced by its magnitude (the scale of the rounding errors)."""
        W1, b1, W2, b2, w3, b3 = torch.split(p, [n1, hidden, n2, hidden, hidden, 1])
        W1, W2 = W1.view(hidden, d_in), W2.view(hidden, hidden)
        a1 = z @ W1.T + b1
        h1 = a1 if abs_ else a1.relu()
        a2 = h1 @ W2.T + b2
        h2 = a2 if abs_ else a2.relu()
        out = h2 @ w3 + b3
        e = out + t if abs_ else out - t
        gy = 2 * e / B
        ga2 = gy[:, None] * w3 * (1 if abs_ else (a2 > 0))
        ga1 = (ga2 @ W2) * (1 if abs_ else (a1 > 0))
        grad = [ga1.T @ z, ga1.sum(0), ga2.T @ h1, ga2.sum(0), gy @ h2, gy.sum()[None]]
        return out, (e * e).mean(), torch.cat([v.reshape(-1) for v in grad])

    p, z, t = params.double(), Z.double(), target.double()
    want = passes(p, z, t)
    scale = passes(p.abs(), z.abs(), t.abs(), True)
    # at most this many roundings lie on the way from an input to a gradient entry
    tol = 2.0 ** -24 * (d_in + 4 * hidden + 2 * B + 40)
    for got, w, s in zip((y, loss[0], G), want, scale):
        assert ((got.cpu().double() - w).abs() <= tol * s).all()
