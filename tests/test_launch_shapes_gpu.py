"""Rollout launches: CTAs smaller than a warp for randomised samples (a CTA
holds whole environment groups), and reach skeletons of several moves (the
next action is loaded where its predecessor ends)."""
import numpy as np
import pytest

import workload

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


def population(sk, N, seed):
    lo, hi = np.array(sk["lo"]), np.array(sk["hi"])
    th = (lo + hi) / 2 + np.random.default_rng(seed).standard_normal((N, len(lo))) * (hi - lo) / 4
    return torch.as_tensor(th.astype(np.float32)).cuda()


@pytest.mark.parametrize("M", [2, 8, 32])
@pytest.mark.parametrize("task", ["reach", "push", "pickplace"])
def test_randomised_rollouts_do_not_depend_on_the_cta(P, task, M):
    sc, sk = {"reach": workload.reach_scene, "push": workload.push_scene, "pickplace": workload.pickplace_scene}[task](2)
    sc = dict(sc, T=150)
    th = population(sk, 37, 4)
    with P.Scene(sc, sk) as S:
        S.set_randomization(M, 0.3, 0.4, 9)
        got = []
        for block in (256, 32, 16, 8, 2, 0):
            P.cem_set_launch(S.h, block)
            got.append([t.cpu() for t in S.rollout(th)])
    for J, cls in got[1:]:
        assert torch.equal(J, got[0][0]) and torch.equal(cls, got[0][1])


@pytest.mark.parametrize("n", [1, 2, 3])
def test_reach_of_several_moves(P, n):
    """The cost without its time term is the distance of the traced final state
    (one state, a few FP32 roundings apart); the class follows from the traced
    count of ended actions."""
    sc, sk = workload.reach_scene(5)
    sc = dict(sc, w_time=0.0, T=900)
    first = sk["actions"][0]
    goal = np.array(first["nominal"])
    acts = [dict(first, nominal=tuple((goal * (i + 1) / n).tolist())) for i in range(n)]
    sk = dict(sk, actions=acts, lo=list(sk["lo"]) * n, hi=list(sk["hi"]) * n)
    th = population(sk, 300, 3)
    with P.Scene(sc, sk) as S:
        J, cls = S.rollout(th)
        last = S.trace(th, 900)[:, -1].cpu().numpy().astype(np.float64)
    dist = np.linalg.norm(last[:, :2] - np.float32(sc["goal_center"])[:2], axis=1)
    np.testing.assert_allclose(J.cpu().numpy(), sc["w_goal"] * dist, rtol=2e-6, atol=2e-6)
    clear = np.abs(dist - sc["eps"]) > 1e-6
    want = np.where(last[:, 12] == n, np.where(dist <= sc["eps"], 0, 1), 2)
    assert np.array_equal(cls.cpu().numpy()[clear], want[clear])
    assert n == 1 or len(np.unique(last[:, 12])) > 1
