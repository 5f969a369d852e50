"""The fused training step's bounded waits: one that runs out (the test hook
leaves a copy or an arrival out, so the wait has nothing in flight) ends the call with
CEM_ERR_TIMEOUT and its code, changes no parameter, moment or counter, and the
next call on the same handle is the one that never failed."""
import time

import numpy as np
import pytest

import workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# hook value -> status: the first weights of the rows launch, the first operands of the weights launch, its last MMAs
WAITS = [(1, 2), (2, 12), (3, 14)]


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
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1, 1, (n, 48)).astype(np.float32)
    t = (np.sin(2 * x[:, 0]) + x[:, 1] * x[:, 2]).astype(np.float32)
    return torch.as_tensor(x).cuda(), torch.as_tensor(t).cuda()


def state(S):
    p, norm = S.params()
    m1, m2, taken = S.adam_state()
    return [p, norm, m1, m2, np.array(taken)]


def timed_out(P, call):
    """Runs call, which has to end in CEM_ERR_TIMEOUT after one wait's time: the
    launches after the expired one do not wait again."""
    t0 = time.time()
    with pytest.raises(P.CemError) as err:
        call()
    assert err.value.code == -3
    assert 0.9 < time.time() - t0 < 3.5


@pytest.mark.parametrize("hook,code", WAITS)
def test_expired_training_wait_changes_nothing(P, hook, code):
    x, t = rows(900, 1)
    with P.Surrogate(256, 4, seed=2) as S, P.Surrogate(256, 4, seed=2) as never:
        for net in (S, never):
            net.train(x, t, batch=200, steps=3, seed=5)
        before = state(S)
        P.cem_surrogate_test_expire_wait(S.h, hook)
        timed_out(P, lambda: S.train(x, t, batch=200, steps=5, seed=6, normalize=False))
        assert S.status() == code and S.status() == 0
        for a, b in zip(before, state(S)):
            assert np.array_equal(a, b)
        P.cem_surrogate_test_expire_wait(S.h, 0)
        h1 = S.train(x, t, batch=200, steps=5, seed=7)
        h2 = never.train(x, t, batch=200, steps=5, seed=7)
        assert S.status() == 0 and np.array_equal(h1, h2)
        for a, b in zip(state(never), state(S)):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("hook,code", WAITS)
def test_expired_gradient_wait(P, hook, code):
    x, t = rows(300, 3)
    with P.Surrogate(256, 4, seed=2) as S:
        g, loss = S.gradient(x, t)
        P.cem_surrogate_test_expire_wait(S.h, hook)
        timed_out(P, lambda: S.gradient(x, t))
        assert S.status() == code
        P.cem_surrogate_test_expire_wait(S.h, 0)
        g2, loss2 = S.gradient(x, t)
        assert S.status() == 0 and np.array_equal(g, g2) and loss == loss2


def test_the_limit_does_not_grow_with_the_rows(P):
    """64 rounds a CTA have one limit together (and CTAs that start later leave at once)."""
    x, t = rows(32 * 64 * 64, 4)
    with P.Surrogate(256, 4, seed=2) as S:
        P.cem_surrogate_test_expire_wait(S.h, 3)
        timed_out(P, lambda: S.gradient(x, t))
        assert S.status() == 14


def test_fine_tuning_reports_it_once(P):
    """The screened loop reports an expired wait of its fine-tuning and clears
    the word, as it does for its scoring: the next run is not held to it."""
    sc, sk, _ = workload.config(2, seed=1, T=200)
    f16 = workload.scene_features(sc)
    run = dict(seed=1, N=128, K=16, iters=2, n_pool=256)
    with P.Scene(sc, sk) as Sc, P.Surrogate(256, 4, seed=2) as S:
        want = Sc.solve_screened(S, f16, **run)
        P.cem_surrogate_test_expire_wait(S.h, 2)
        with pytest.raises(P.CemError) as err:
            Sc.solve_screened(S, f16, finetune=dict(every=1, steps=2, batch=64, capacity=1280), **run)
        assert err.value.code == -3 and "training" in str(err.value)
        P.cem_surrogate_test_expire_wait(S.h, 0)
        got = Sc.solve_screened(S, f16, **run)
        assert S.status() == 0
    assert got["best_J"] == want["best_J"] and np.array_equal(got["mean"], want["mean"])
