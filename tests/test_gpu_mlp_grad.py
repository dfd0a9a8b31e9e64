"""The tiled gradient (32 rows per tile, at most 608 blocks, sums over a block's tiles in registers) at row counts
around a tile, around one tile per block and with several tiles per block, every parameter against the FP64
gradient with the same rounding points."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


def _reference(p, X, Y, bf16):
    """Loss, gradient and, per parameter, the sum of the absolute contributions (FP64)."""
    W1, b1, W2, b2, W3, b3 = omlp.unpack(p)
    r = omlp.bf16_round if bf16 else (lambda a: a)
    y, (a0, z1, a1, z2, a2) = omlp.forward(p, X, bf16=bf16)
    n = len(Y)
    res = y - Y
    # the sum that gives a row's output: its rounding enters every contribution of the row
    mag = np.abs(a2) @ np.abs(r(W3)) + (np.abs(a1) @ np.abs(r(W2)).T + np.abs(b2)) @ np.abs(r(W3)) + abs(b3) + np.abs(Y)
    dy, ady = 2.0 * res / n, 2.0 * (np.abs(res) + mag) / n
    d2, ad2 = np.outer(dy, r(W3)) * (z2 > 0), np.outer(ady, np.abs(r(W3))) * (z2 > 0)
    d1, ad1 = (d2 @ r(W2)) * (z1 > 0), (ad2 @ np.abs(r(W2))) * (z1 > 0)
    g, s = [], []
    for out, e, ae, a in ((g, d1, ad1, a0), (g, d2, ad2, a1)):
        out += [(e.T @ a).ravel(), e.sum(axis=0)]
        s += [(ae.T @ np.abs(a)).ravel(), ae.sum(axis=0)]
    g += [a2.T @ dy, [dy.sum()]]
    s += [np.abs(a2).T @ ady, [ady.sum()]]
    return np.mean(res * res), np.mean((np.abs(res) + mag) ** 2), np.concatenate(g), np.concatenate(s)


# FP32: a parameter is a sum of at most 32 * 4 terms per thread, 608 blocks and some 70 roundings of the terms
# themselves, 806 * 2^-24 = 5e-5 of the absolute contributions at 60,001 rows (3e-5 up to 30,000): 1e-4 allowed.
# BF16: besides, an activation within FP32 rounding of a BF16 boundary may round to the other side, 2^-8 of its
# row's contribution; up to 33 rows a single such row may show, beyond it is averaged: 5e-3 and 2e-4 allowed.
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 3000, 19456, 19457, 30000, 60001])
@pytest.mark.parametrize("bf16", [False, True])
def test_gradient_at_every_tile_count(n, bf16):
    import torch
    from paper_1608_06577_gb300.binding import mlp_grad
    rng = np.random.default_rng(n + 7)
    p = (rng.normal(size=omlp.NPARAM) * 0.3).astype(np.float32)
    X = rng.normal(size=(n, 6)).astype(np.float32)
    Y = rng.normal(size=n).astype(np.float32)
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    g, loss = mlp_grad(dev(p), dev(X), dev(Y), bf16_forward=bf16)
    g = g.cpu().numpy().astype(np.float64)
    lr, ls, gr, s = _reference(p.astype(np.float64), X.astype(np.float64), Y.astype(np.float64), bf16)
    tol = 1e-4 if not bf16 else (5e-3 if n <= 64 else 2e-4)
    assert abs(loss.item() - lr) <= tol * ls
    err = np.abs(g - gr) / np.where(s > 0, s, 1.0)
    print(f"n {n} bf16 {bf16}: largest error {err.max():.2e} of the absolute contributions")
    names = ("W1", "b1", "W2", "b2", "W3", "b3")
    at = np.cumsum([0, 192, 32, 1024, 32, 32, 1])
    for k, name in enumerate(names):
        assert err[at[k]:at[k + 1]].max() <= tol, (name, err[at[k]:at[k + 1]].max())
