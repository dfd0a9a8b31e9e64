"""kt_mlp_predict over row counts around its groups of 32 rows and its grid, and rows that are not 8-byte
aligned: the same values whatever the count and the alignment."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [1, 7, 31, 32, 33, 255, 257, 2432 * 32 + 5, 200001])
def test_counts_and_alignment(n):
    import torch
    from oracle import mlp as omlp
    from paper_1608_06577_gb300.binding import mlp_predict
    rng = np.random.default_rng(2)
    p = torch.as_tensor((rng.normal(size=omlp.NPARAM) * 0.3).astype(np.float32), device="cuda")
    X = rng.normal(size=(n, 6)).astype(np.float32)
    x = torch.as_tensor(X, device="cuda")
    scratch = torch.zeros(3396, dtype=torch.uint8, device="cuda")
    y = mlp_predict(p, x, scratch)
    # the packed weights are in the caller's scratch afterwards (biases as they are: words 784.. of 849)
    words = scratch.cpu().numpy().view(np.float32)
    assert np.array_equal(words[784:816], p.cpu().numpy()[192:224])
    odd = torch.empty(6 * n + 1, dtype=torch.float32, device="cuda")[1:].view(n, 6)  # 4-byte aligned rows
    odd.copy_(x)
    assert odd.data_ptr() % 8 == 4
    assert torch.equal(mlp_predict(p, odd), y)
    # a row's value does not depend on its neighbours or the count
    k = min(n, 100)
    assert torch.equal(mlp_predict(p, x[n - k:].clone()), y[n - k:])
    # against the FP64 forward with the same BF16 rounding points: FP32 accumulation order, and rarely an
    # activation on the other side of a BF16 rounding (the bounds of the inference test)
    yb, _ = omlp.forward(p.cpu().numpy(), X, bf16=True)
    scale = max(np.max(np.abs(yb)), 1e-3)
    err = np.abs(y.cpu().numpy() - yb) / scale
    assert (err > 1e-6).sum() <= max(3, 3 * n // 1000) and err.max() < 4e-3
