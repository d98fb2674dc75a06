"""The training step's tiled kernels at the edges of their tiles: loss and
gradient against the oracle for sample counts around the 64-sample tile, around
the smallest scratch that holds rows of partial sums, and above one tile per
resident CTA.

Inputs, weights and biases are multiples of 2^-6 small enough that every hidden
value is exact in fp32 and bfloat16 rounding sees the oracle's values, so the
only differences are the rounding of the sigmoid, the deltas and the sums.  A
gradient entry is a sum over samples of products; with u = 2^-24, a term
carries at most 70 u of relative error (the sigmoid and its argument's 66
terms, the delta's 64-term chain counted by the magnitude of its terms) and the
sum at most (64 t + r / 8 + 16) u, t tiles per CTA and r rows: the tolerance is
that bound times the sum of the terms' magnitudes (times two for the terms of
second order).
"""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def dyadic(rng, shape, scale):
    return (rng.integers(-scale, scale + 1, size=shape) / 64.0).astype(np.float32)


@pytest.mark.parametrize("n", [1, 29, 30, 63, 64, 65, 128, 129, 1000, 40001])
def test_loss_and_gradient_at_tile_edges(n):
    import torch
    import paper_1708_00783_gb300 as itm
    rng = np.random.default_rng(n)
    nf, nh = 52, 64
    W1, b1 = dyadic(rng, (nh, nf), 16), dyadic(rng, nh, 16)
    W2, b2 = dyadic(rng, (nh, nh), 16), dyadic(rng, nh, 16)
    w3, b3 = dyadic(rng, nh, 8), dyadic(rng, 1, 8)
    P = np.concatenate([x.ravel() for x in (W1, b1, W2, b2, w3, b3)])
    X = dyadic(rng, (n, nf), 32)
    y = (rng.uniform(size=n) > 0.4).astype(np.float32)
    used = n * itm.ITM_MLP_SCRATCH_PER_SAMPLE
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    grad = torch.full((oracle.N_PARAMS + 8,), 7.0, device="cuda")
    loss = torch.full((4,), 7.0, device="cuda")
    scratch = torch.full((used + 64,), 7.0, device="cuda")
    itm.itm_mlp_loss_grad(dev(P), dev(X), dev(y), n, scratch, grad, loss)
    torch.cuda.synchronize()
    # nothing is written behind the caller's buffers
    assert bool((scratch[used:] == 7.0).all()) and bool((grad[oracle.N_PARAMS:] == 7.0).all())
    assert bool((loss[1:] == 7.0).all())

    lo, go = oracle.mlp_loss_grad(P, X.astype(np.float64), y, round_bf16=True)
    # the magnitudes of the terms of every sum, in fp64
    bf = lambda a: torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16).double().numpy()  # noqa: E731
    h1 = bf(np.maximum(X.astype(np.float64) @ W1.T.astype(np.float64) + b1, 0))
    h2 = np.maximum(h1 @ W2.T.astype(np.float64) + b2, 0)
    o = h2 @ w3.astype(np.float64) + b3[0]
    do = np.abs(1 / (1 + np.exp(-o)) - y) / n + 2.0 ** -24 / n
    d2 = (h2 > 0) * do[:, None] * np.abs(w3)
    d1 = (h1 > 0) * (d2 @ np.abs(W2))
    mag = np.concatenate([(d1.T @ np.abs(X)).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), do @ h2, [do.sum()]])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-n // 64)
    rows = min(tiles, sms)                  # at least this many CTAs when there are as many tiles
    u, per_cta = 2.0 ** -24, -(-tiles // rows)
    # the output's own error enters through the sigmoid's slope, absolutely
    o_err = 66 * u * (np.abs(w3) @ h2.T + abs(b3[0])).max()
    tol = 2 * ((70 + 64 * per_cta + 2 * sms / 8 + 16) * u * mag + o_err * mag / np.maximum(do.min() * n, 2.0 ** -24))
    diff = np.abs(grad[:oracle.N_PARAMS].cpu().numpy().astype(np.float64) - go)
    small = np.abs(diff) <= np.minimum(tol, 1e-3 * mag + 1e-12)
    assert small.all(), (diff / np.maximum(mag, 1e-30)).max()
    assert abs(loss[0].item() - lo) <= 2 * (o_err + (64 * per_cta + 2 * sms + 70) * u * max(1.0, abs(lo)))
