"""The fused training step at the edges of its tiles (64 rows), its split-K
chunks (up to 32 of at most 256 rows, longer beyond 8192 rows, some not whole
tiles) and its ring of rounds, by the bars and for the reasons of
test_surrogate_parity_gpu."""
import numpy as np
import pytest

from oracle import mlp
from test_surrogate_parity_gpu import P, gpu_gradient, problem, tensors  # noqa: F401 (P is the fixture)

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 31, 64, 65, 448, 600, 777, 8191, 8193, 20011])
def test_gradient_at_the_edges(P, M):  # noqa: F811
    params, X, t = problem(M)
    g, loss = gpu_gradient(P, params, X, t, 2)
    g2, loss2 = gpu_gradient(P, params, X, t, 2)
    assert np.array_equal(g, g2) and loss == loss2
    loss_ref, ref = mlp.loss_and_grads(params, X, t, emulate_bf16=True)
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    for name, got, r in tensors(g, ref):
        d = np.abs(got - r)
        assert (d / np.maximum(np.abs(r), np.sqrt(np.mean(r * r)))).max() <= 1e-2, name
        assert np.linalg.norm(d) <= 1e-3 * np.linalg.norm(r), name
