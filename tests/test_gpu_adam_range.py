"""Adam's update where gradients vanish: a feature that is nonzero in the first
step only leaves its weights a first moment that decays through the denormal
range (0.9^900 = 6e-42), and one that is always zero moments of exactly zero."""
import numpy as np
import pytest

from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2302_13524_gb300 as tmr  # noqa: E402


# products on the tensor cores (Adam as their epilogue) and on the generic kernel (Adam on its own)
@pytest.mark.parametrize("dims,B", [((256, 136, 128, 320), 133), ((40, 24, 24, 16), 9)])
def test_vanished_gradients(dims, B):
    steps, lr = 900, 1e-3
    rng = np.random.default_rng(B)
    X = rng.standard_normal((B, dims[0])).astype(np.float32)
    X[:, 1] = 0.0
    later = X.copy()
    later[:, 0] = 0.0
    T = to_dev(rng.standard_normal((B, dims[3])).astype(np.float32))
    with tmr.tmr_mlp_create(*dims, seed=1) as m:
        start, end = np.empty(m.n_params, np.float32), np.empty(m.n_params, np.float32)
        G = torch.empty(m.n_params, dtype=torch.float32, device="cuda")
        loss = torch.empty(1, dtype=torch.float32, device="cuda")
        tmr.tmr_mlp_get_params(m, start)
        tmr.tmr_mlp_grad(m, to_dev(X), T, B, loss, G)
        X, later = to_dev(X), to_dev(later)
        for t in range(steps):
            tmr.tmr_mlp_train_step(m, X if t == 0 else later, T, B, lr, loss)
        tmr.tmr_mlp_get_params(m, end)
        torch.cuda.synchronize()
    n = dims[0] * dims[1]
    w0, w1, g = (a[:n].reshape(dims[1], dims[0]).astype(np.float64) for a in (start, end, to_np(G)))
    assert np.all(np.isfinite(end)) and np.array_equal(w1[:, 1], w0[:, 1])
    t = np.arange(1, steps + 1)[:, None]
    mt, vt = 0.1 * g[:, 0] * 0.9 ** (t - 1), 0.001 * g[:, 0] ** 2 * 0.999 ** (t - 1)
    moves = lr * mt / (1 - 0.9 ** t) / (np.sqrt(vt / (1 - 0.999 ** t)) + 1e-8)
    # FP32: half an ulp of w for each of the about 200 steps that still move it, the step itself to 1e-5
    tol = 200 * 2.0 ** -24 * np.abs(w0[:, 0]) + 1e-5 * np.abs(moves).sum(0)
    assert np.all(np.abs(w1[:, 0] - (w0[:, 0] - moves.sum(0))) <= tol)
