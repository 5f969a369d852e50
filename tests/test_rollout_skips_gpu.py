"""The pick-and-place rollout leaves out work that cannot change its result:
contact queries while a mover is provably clear of every body, the step of
an object at rest, and the steps of a sample whose whole state is at rest.

The traced rollout takes every step, so its last state gives the cost that a
rollout which left early must report; the contact queries are checked
against the FP64 oracle on movers that meet bodies after free motion.
"""
import numpy as np
import pytest

import workload
from pickplace_common import ATT, BX, BY, OX, OY, OZ

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


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, np.float32)).cuda()


def initial(sk, N, seed, spread=1.0):
    lo, hi = np.array(sk["lo"]), np.array(sk["hi"])
    return (lo + hi) / 2 + spread * np.random.default_rng(seed).standard_normal((N, len(lo))) * (hi - lo) / 4


@pytest.mark.parametrize("controller", ["pd", "astar"])
@pytest.mark.parametrize("T", [1, 7, 8, 9, 3000])
def test_final_state_is_the_traced_one(P, T, controller):
    """J without its time term is the distances of the final state: FP32
    arithmetic on one state, a few roundings apart."""
    sc, sk = workload.pickplace_scene(3, T=T, controller=controller)
    sc = dict(sc, w_time=0.0)
    th = dev(initial(sk, 333, 5))
    with P.Scene(sc, sk) as S:
        J, cls = S.rollout(th)
        last = S.trace(th, T)[:, -1].cpu().numpy().astype(np.float64)
    e = np.abs(last[:, [OX, OY, OZ]] - np.float32(sc["obj_region_center"])) - np.float32(sc["obj_region_half"])
    b = np.abs(last[:, [BX, BY]] - np.float32(sc["base_region_center"])[:2]) - np.float32(sc["base_region_half"])[:2]
    want = sc["w_obj"] * np.linalg.norm(np.maximum(e, 0), axis=1) + sc["w_base"] * np.linalg.norm(np.maximum(b, 0), axis=1)
    np.testing.assert_allclose(J.cpu().numpy(), want, rtol=2e-6, atol=1e-5)
    done = last[:, 16] == len(sk["actions"])
    goal = (e <= 0).all(1) & (b <= 0).all(1) & (last[:, ATT] == 0)
    assert np.array_equal(cls.cpu().numpy(), np.where(done, np.where(goal, 0, 1), 2))


@pytest.mark.parametrize("lanes", [8, 32])
def test_lane_groups_leave_alike(P, lanes):
    sc, sk = workload.pickplace_scene(11)
    th = dev(initial(sk, 203, 6))
    with P.Scene(sc, sk) as S:
        J1, c1 = S.rollout(th)
        S.set_threads_per_rollout(lanes)
        J2, c2 = S.rollout(th)
    assert torch.equal(J1, J2) and torch.equal(c1, c2)


@pytest.mark.parametrize("seed", range(4))
def test_contacts_after_free_motion(P, orc, seed):
    """A thrown object and a fast base fly freely, hit walls, ground, tables
    and boxes, and slide on.  A query left out for one step too many lets a
    body in by v dt = 4 mm, k depth dt / m = 0.3 m/s (object) and 0.016 m/s
    (base); the paths below agree with FP64 to well under 1 mm otherwise."""
    rng = np.random.default_rng(seed)
    sc, sk = workload.pickplace_scene(seed, T=400)
    ang = rng.uniform(0, 2 * np.pi, 2)
    sc = dict(sc, obj_start=(rng.uniform(-0.5, 0.2), rng.uniform(-0.8, 0.2), rng.uniform(0.4, 1.2)),
              obj_v0=(2 * np.cos(ang[0]), 2 * np.sin(ang[0]), rng.uniform(-1, 1)),
              base_v0=(2 * np.cos(ang[1]), 2 * np.sin(ang[1]), 0.0))
    th = initial(sk, 8, seed)
    with P.Scene(sc, sk) as S:
        got = S.trace(dev(th), 400).cpu().numpy()
    for i in range(len(th)):
        ref = orc.trace(sc, sk, th[i].astype(np.float32).astype(np.float64), 400)
        assert np.abs(got[i][:, [BX, BY, OX, OY, OZ]] - ref[:, [BX, BY, OX, OY, OZ]]).max() < 1e-3
