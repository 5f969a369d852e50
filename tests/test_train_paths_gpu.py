"""Training of a 48-256x4 network by the fused step (gemm path 2) against the
same steps taken layer by layer on gemm_tc_kernel (training on path 3) and
against gradient + optimiser calls: the arithmetic and its order are the same,
so everything is equal bit for bit, for any batch (64 rows a tile, chunks of
rows, beyond 8192 rows longer chunks) and over many dependent steps.

And gemm_tc_kernel at width 256 on the depths that the fused step leaves to
it, by the bars of test_surrogate_gemm_tc_gpu."""
import numpy as np
import pytest

from oracle import mlp
from test_surrogate_gemm_tc_gpu import P, dev, layer_blocks  # noqa: F401 (P is the fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS = 20011


@pytest.fixture(scope="module")
def data():
    X = np.random.default_rng(8).uniform(-1, 1, (ROWS, 48)).astype(np.float32)
    t = (np.sin(3 * X[:, 0]) + X[:, 1] * X[:, 2] + 0.5 * X[:, 40]).astype(np.float32)
    return dev(X), dev(t)


def state(S):
    (p, norm), (m1, m2, taken) = S.params(), S.adam_state()
    return [p, norm, m1, m2, np.array(taken)]


def same(a, b):
    return len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("steps", [1, 2, 50])
@pytest.mark.parametrize("batch", [1, 63, 65, 777, 8192, 8193])
def test_fused_step_equals_layer_by_layer(P, data, batch, steps):  # noqa: F811
    got = []
    for path in (2, 3, 2):
        with P.Surrogate(256, 4, seed=3) as S:
            S.set_gemm_path(path)
            hist = S.train(*data, batch=batch, steps=steps, lr=2e-3, weight_decay=1e-2, seed=4)
            hist2 = S.train(*data, batch=batch, steps=1, lr=2e-3, seed=5)  # (from a used state)
            assert S.status() == 0
            got.append([hist, hist2] + state(S))
    assert same(got[0], got[2])  # run to run
    assert same(got[0], got[1])


@pytest.mark.parametrize("batch", [65, 777])
def test_fused_step_is_gradient_and_optimiser_step(P, orc, data, batch):  # noqa: F811
    """The rows of step k are drawn by the first word of the Philox block
    (row, k, 0x5AFE, 0); its gradient and one AdamW step (both checked against
    the oracle elsewhere) are the training step."""
    x, t = data
    steps, seed = 3, 11
    words = orc.philox_words(seed, 0x5AFE, 0, batch, 4 * steps).reshape(batch, steps, 4)[:, :, 0]
    with P.Surrogate(256, 4, seed=3) as A, P.Surrogate(256, 4, seed=3) as B:
        hist = A.train(x, t, batch=batch, steps=steps, lr=2e-3, weight_decay=1e-2, seed=seed, normalize=False)
        losses = []
        for k in range(steps):
            row = torch.as_tensor(((words[:, k].astype(np.uint64) * np.uint64(ROWS)) >> np.uint64(32)).astype(np.int64)).cuda()
            g, loss = B.gradient(x[row].contiguous(), t[row].contiguous())
            B.adamw_step(g, 2e-3, 1e-2)
            losses.append(loss)
        assert same(state(A), state(B))
        assert np.array_equal(hist, np.float32(losses))


@pytest.mark.parametrize("M,depth", [(256, 3), (3001, 3), (777, 5)])
def test_width_256_at_other_depths(P, M, depth):  # noqa: F811
    params = mlp.init_params(48, 256, depth, seed=M + depth)
    X = np.random.default_rng(M).uniform(-1, 1, (M, 48))
    t = np.sin(X[:, 0] * 2) + X[:, 1] * X[:, 2]
    got = {}
    with P.Surrogate(256, depth) as S:
        S.set_params(mlp.flatten(params), np.array([0.0, 1.0]))
        for path in (1, 2):
            S.set_gemm_path(path)
            got[path] = S.gradient(dev(X), dev(t))
        assert S.status() == 0
    loss_ref, grads = mlp.loss_and_grads(params, X, t)
    for g, loss in got.values():
        assert abs(loss - loss_ref) <= 2e-2 * loss_ref
        for a, ref in layer_blocks(g, grads):
            assert np.linalg.norm(a - ref) <= 3e-2 * np.linalg.norm(ref) + 1e-7
    (g1, l1), (g2, l2) = got[1], got[2]
    assert abs(l1 - l2) <= 1e-3 * abs(l1)
    for (a, _), (b, _) in zip(layer_blocks(g1, grads), layer_blocks(g2, grads)):
        assert np.linalg.norm(a - b) <= 1e-2 * np.linalg.norm(a) + 1e-7


def test_training_of_width_256_depth_3(P, data):  # noqa: F811
    hist, out = {}, []
    for path in (1, 2, 2):
        with P.Surrogate(256, 3, seed=3) as S:
            S.set_gemm_path(path)
            hist[path] = S.train(*data, batch=2048, steps=150, lr=2e-3, seed=4)
            assert S.status() == 0
            out.append(S.params()[0])
    assert np.array_equal(out[1], out[2])
    for path in (1, 2):
        assert hist[path][-10:].mean() < 0.3 * hist[path][:3].mean()
    np.testing.assert_allclose(hist[1][:3], hist[2][:3], rtol=1e-2)
