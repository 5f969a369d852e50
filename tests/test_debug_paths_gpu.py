"""The bounds-checked debug build on the paths with contact queries, selection
and row drawing of their own: the A* base, randomised environments, 8 and 32
lanes a rollout, refits at the edges of their sizes, the screening's top-k in
one to eight CTAs, the fused training step.  No check fires (among them codes
10 and 11: a contact query left out that would have found something), and
every result equals the release library's bit for bit."""
import json
import os
import subprocess
import sys

import pytest
from test_debug_build_gpu import P, ROOT  # noqa: F401 (P is the fixture)

pytestmark = pytest.mark.gpu

WORK = r'''
import hashlib, json
import numpy as np
import torch
import workload
import paper_2512_11571_gb300 as P


def dev(a, t=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a)).to("cuda", t)


def digest(*parts):
    h = hashlib.sha256()
    for p in parts:
        p = p.cpu().numpy() if isinstance(p, torch.Tensor) else np.asarray(p)
        h.update(np.ascontiguousarray(p).tobytes())
    return h.hexdigest()


def population(sk, N, seed):
    lo, hi = np.array(sk["lo"]), np.array(sk["hi"])
    return dev((lo + hi) / 2 + np.random.default_rng(seed).standard_normal((N, len(lo))) * (hi - lo) / 4)


def run():
    out = {}
    for ctrl, seed in (("pd", 3), ("astar", 1), ("astar", 7)):
        sc, sk = workload.pickplace_scene(seed, n_actions=5, T=900, controller=ctrl)
        th = population(sk, 200, seed)
        with P.Scene(sc, sk) as S:
            for lanes in (1, 8, 32):
                S.set_threads_per_rollout(lanes)
                out[f"rollout {ctrl} {seed} {lanes}"] = digest(*S.rollout(th))
    for task, make in (("push", workload.push_scene), ("pickplace", workload.pickplace_scene)):
        sc, sk = make(4)
        with P.Scene(dict(sc, T=600), sk) as S:
            S.set_randomization(8, 0.3, 0.4, 9)
            out[f"randomised {task}"] = digest(*S.rollout(population(sk, 150, 5)))
    probs = []
    for i, ctrl in enumerate(("pd", "astar", "pd")):
        sc, sk = workload.pickplace_scene(20 + i, n_actions=4, T=500, controller=ctrl)
        probs.append(dict(scene=sc, skel=sk, N=300 + i, K=20, seed=8, problem=i))
    with P.Batch(probs) as B:
        B.iterate(2, use_graph=True)
        out["batch"] = digest(*[np.asarray(g[k]) for g in B.read() for k in ("best_J", "mean", "cov", "best_theta")])
    rng = np.random.default_rng(6)
    for N, K, D in ((512, 25, 3), (16385, 512, 14), (65537, 4096, 6)):
        theta, J = rng.standard_normal((N, D)).astype(np.float32), np.round(rng.uniform(0, 9, N), 2).astype(np.float32)
        J[::97] = np.nan
        sc, sk = workload.quadratic_scene(0, D)
        mean, cov, chol = (torch.zeros(n, device="cuda") for n in (D, (D, D), (D, D)))
        with P.Scene(sc, sk) as S:
            idx, keff = S.refit(dev(theta), dev(J), dev(rng.integers(0, 3, N), torch.uint8), K, mean, cov, chol)
        out[f"refit {N}"] = digest(idx[:int(keff.item())], mean, cov, chol)
    sc, sk, _ = workload.config(2, seed=4)
    lo, hi = np.array(sk["lo"]), np.array(sk["hi"])
    with P.Scene(sc, sk) as Sc, P.Surrogate(256, 4, seed=7) as S:
        for pool, keep in ((4000, 100), (16384, 4097), (65537, 8192)):
            kept = torch.empty((keep, len(lo)), device="cuda")
            idx = torch.empty(keep, dtype=torch.int32, device="cuda")
            P.cem_surrogate_screen(Sc.h, S.h, dev((lo + hi) / 2), dev(np.diag((hi - lo) / 4)), 9, 1, 0, pool, keep,
                                   workload.scene_features(sc), kept, idx)
            out[f"screen {pool}"] = digest(kept, idx)
        x = dev(rng.uniform(-1, 1, (5001, 48)))
        t = torch.sin(2 * x[:, 0]) + x[:, 1]
        out["train"] = digest(S.train(x, t, batch=777, steps=20, seed=2), S.params()[0])
        out["gradient"] = digest(S.gradient(x, t)[0])
    return out
'''

CHILD = WORK + r'''
P.load(P.DEBUG_LIB_PATH)
res = run()
print(json.dumps([res, P.cem_debug_status()]))
'''


def test_no_check_fires_and_no_result_changes(P):  # noqa: F811
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    got, code = json.loads(r.stdout.strip().splitlines()[-1])
    assert code == 0
    scope = {}
    exec(compile(WORK, "work", "exec"), scope)
    assert got == scope["run"]()
