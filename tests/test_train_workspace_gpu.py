"""The fused training step's workspace stays with its handle when the row
workspace (screening, unaligned rows, the layer-by-layer paths) grows, and
gives way to it where the device has no room for both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_11571_gb300 as P
    from paper_2512_11571_gb300 import build

    build.build()
    P.load()
    return P


def rows(n, seed):
    x = torch.as_tensor(np.random.default_rng(seed).uniform(-1, 1, (n, 48)).astype(np.float32)).cuda()
    return x, torch.sin(2 * x[:, 0]) + x[:, 1]


def unaligned(x):
    """The same rows 4 bytes past a 16-byte boundary: they go through the row workspace."""
    buf = torch.empty(x.numel() + 1, device="cuda")
    out = buf[1:].view(x.shape)
    out.copy_(x)
    return out


def test_training_allocates_nothing_after_the_rows_grew(P):
    x, t = rows(3001, 1)
    small = unaligned(x[:64])
    big = unaligned(x)
    with P.Surrogate(256, 4, seed=1) as S:
        want = S.gradient(x[:700], t[:700])
        for some in (small, big):
            S.forward(some)
            P.cem_test_fail_allocation(1)
            try:
                got = S.gradient(x[:700], t[:700])
            finally:
                P.cem_test_fail_allocation(0)
            assert np.array_equal(got[0], want[0]) and got[1] == want[1]


@pytest.mark.parametrize("k", [1, 5])
def test_the_training_block_gives_way(P, k):
    """An allocation of the row workspace fails while the block is held: the
    block is given up for it, and the call goes through."""
    x, t = rows(3001, 2)
    with P.Surrogate(256, 4, seed=1) as S:
        want_g, want_y = S.gradient(x, t), S.forward(x)
        torch.cuda.synchronize()
        P.cem_test_fail_allocation(k)
        try:
            y = S.forward(unaligned(x))
        finally:
            P.cem_test_fail_allocation(0)
        assert torch.equal(y, want_y)
        got = S.gradient(x, t)
        assert np.array_equal(got[0], want_g[0]) and got[1] == want_g[1]
