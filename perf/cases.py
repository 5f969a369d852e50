"""What this library is measured on: calls that a planner or a training
script makes, each through the public binding, at the sizes of the
repository's configurations, tests and benchmark.

Kinds of case (the "kind" of a case's dict):

solve     a whole CE search on one scene (``Scene.solve``): what a planner
          calls for one plan skeleton.
batch     CE iterations of many problems at once (``Batch``): reset, iterate,
          read; the benchmark's workload.
rollout   one batch of samples through the simulator (``Scene.rollout``):
          what a program with its own optimiser, and the surrogate's data
          generation, call.  With the A* base or a randomised environment as
          options.
update    elite selection + refit of a scored population, then the next
          population drawn from the new distribution (``Scene.refit``,
          ``Scene.sample``): an ask/tell step around another simulator.
forward   surrogate scores of feature rows (``Surrogate.forward``).
gradient  loss gradient of the surrogate on a set of rows.
train     AdamW steps of the surrogate on a training set.
screen    draw a pool, score it, keep the best (``cem_surrogate_screen``).

Trajectories with contacts (push, pick-place) part from any other rounding
of themselves after a few hundred steps, and a CE search follows its elite
sets, so rollouts with contacts and whole searches have no value in 64 bits
here; the others have.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2512_11571_gb300 as P
import workload

WIDTH, DEPTH, IN = 256, 4, 48


def listed():
    return [
        # the smallest search: one moveTo, N = 256; every launch and copy shows
        dict(name="solve reach N=256", kind="solve", task="reach", scene=0, N=256, K=25, iters=10),
        # move-and-push at its configured size: contacts, 4096 rollouts a step
        dict(name="solve push N=4096", kind="solve", task="push", scene=0, N=4096, K=200, iters=20),
        # one evaluation of the pick-and-place configuration (N = 16384, T = 3000)
        dict(name="rollout pickplace N=16384", kind="rollout", task="pickplace", scene=0, actions=5, N=16384,
             controller="pd", envs=1),
        # the A* base controller, ragged population
        dict(name="rollout astar N=4001", kind="rollout", task="pickplace", scene=1, actions=5, N=4001,
             controller="astar", envs=1),
        # domain randomisation: every sample in 8 environments
        dict(name="rollout randomised N=1000x8", kind="rollout", task="push", scene=2, actions=2, N=1000,
             controller="pd", envs=8),
        # the benchmark's batch: 64 problems, 1 to 6 actions, uneven N; ten CE iterations of one run
        dict(name="batch 64 problems", kind="batch", scene=0, problems=64, iters=10),
        # refit + next draw at the pick-and-place configuration's N, D and K
        dict(name="update N=16384", kind="update", D=14, N=16384, K=512),
        # a screening pool's worth of scores
        dict(name="forward 65536", kind="forward", rows=65536),
        # a handful of candidates, ragged
        dict(name="forward 777", kind="forward", rows=777),
        # a validation gradient, ragged
        dict(name="gradient 3001", kind="gradient", rows=3001),
        # the surrogate's training settings (batch 8192 of a million rollouts), a stretch of steps
        dict(name="train batch 8192", kind="train", rows=1 << 20, batch=8192, steps=50),
        # screening as configured: the best 8192 of 65536
        dict(name="screen 65536", kind="screen", scene=0, pool=65536, keep=8192),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of lo .. hi."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "batch", "rollout", "rollout", "update", "forward", "gradient", "train", "screen"])
    scene = rng.randrange(1000)
    if kind == "solve":
        N = _log(rng, 64, 4096)
        return dict(kind=kind, task=rng.choice(["reach", "push"]), scene=scene, N=N, K=max(2, N // rng.choice([8, 20])),
                    iters=rng.randrange(3, 16))
    if kind == "batch":
        return dict(kind=kind, scene=scene, problems=_log(rng, 2, 48), iters=rng.randrange(2, 6))
    if kind == "rollout":
        task = rng.choice(["reach", "push", "pickplace", "pickplace"])
        envs = rng.choice([1, 1, 4, 8])
        N = _log(rng, 100, 16384 // envs)
        controller = rng.choice(["pd", "pd", "astar"]) if task == "pickplace" else "pd"
        actions = rng.randrange(3, 7) if task == "pickplace" else 1 if task == "reach" else 2
        return dict(kind=kind, task=task, scene=scene, actions=actions, N=N, controller=controller, envs=envs)
    if kind == "update":
        N = _log(rng, 200, 65536)
        return dict(kind=kind, D=rng.randrange(3, 19), N=N, K=min(4096, max(4, N // rng.choice([10, 20, 32]))))
    if kind == "forward":
        return dict(kind=kind, rows=_log(rng, 64, 65536))
    if kind == "gradient":
        return dict(kind=kind, rows=_log(rng, 256, 8192))
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 30000, 500000), batch=_log(rng, 512, 8192), steps=rng.randrange(10, 41))
    pool = _log(rng, 1000, 65536)
    return dict(kind=kind, scene=scene, pool=pool, keep=max(1, pool // rng.choice([4, 8])))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _problem(case):
    if case["task"] == "reach":
        return workload.reach_scene(case["scene"])
    if case["task"] == "push":
        return workload.push_scene(case["scene"])
    return workload.pickplace_scene(case["scene"], n_actions=case["actions"], controller=case["controller"])


def _initial(lo, hi):
    """The initial sampling distribution of a skeleton: mid-bounds, range / 4."""
    lo, hi = np.asarray(lo), np.asarray(hi)
    return (lo + hi) / 2, np.diag((hi - lo) / 4)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, np.float32)).cuda()


def _theta(lo, hi, N, seed):
    """A population of the initial distribution."""
    mean, chol = _initial(lo, hi)
    return _dev(mean) + torch.randn((N, len(lo)), generator=_gen(seed), device="cuda") @ _dev(chol)


def _mlp(seed):
    """Parameters of a surrogate, flat (per layer the weights [out, in], then the
    biases), FP32: the usual Linear-layer initialisation with the weights at
    twice its scale, so that scores spread as a trained network's do."""
    rng = np.random.default_rng(seed)
    parts = []
    for l in range(DEPTH + 1):
        fi, fo = (IN if l == 0 else WIDTH), (1 if l == DEPTH else WIDTH)
        parts.append(rng.uniform(-2, 2, fi * fo) / math.sqrt(fi))
        parts.append(rng.uniform(-1, 1, fo) / math.sqrt(fi))
    return np.concatenate(parts).astype(np.float32)


NORM = (1.9, 0.7)  # score mean and deviation of trained pick-and-place surrogates


def _rows(n, seed):
    """Feature rows: 14 normalised parameters, 18 zeros, 16 scene values."""
    g = _gen(seed)
    x = torch.zeros((n, IN), device="cuda")
    x[:, :14] = (torch.randn((n, 14), generator=g, device="cuda") * 0.5).clamp_(-1, 1)
    x[:, 32:46] = torch.rand((n, 14), generator=g, device="cuda") * 2 - 1
    return x


def _targets(x, seed):
    """log(1 + cost + 10 class) of a smooth cost with classes 0 to 2."""
    g = _gen(seed + 1)
    u = (x[:, :14] - 0.2).square().sum(1)
    cost = 2.5 + u + 0.3 * torch.sin(4 * x[:, 0] + x[:, 33]) + 0.05 * torch.randn(x.shape[0], generator=g, device="cuda")
    cls = (u > 2.5).float() + (x[:, 4].abs() > 0.4).float()
    return torch.log1p(cost.clamp_(min=0) + 10 * cls)


def _population(case, seed):
    """A scored population of the update kind: parameters, costs, classes."""
    D, N = case["D"], case["N"]
    lo, hi = np.linspace(-1.0, -0.2, D), np.linspace(0.3, 2.0, D)
    theta = _theta(lo, hi, N, seed)
    g = _gen(seed + 1)
    mid = _dev((lo + hi) / 2 + 0.1)
    J = 2.0 + (theta - mid).square().sum(1) + 0.2 * torch.rand(N, generator=g, device="cuda")
    cls = torch.where(torch.rand(N, generator=g, device="cuda") < 0.2, 0, 2).to(torch.uint8)
    cls[torch.rand(N, generator=g, device="cuda") < 0.1] = 1
    return lo, hi, theta, J, cls


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed)
    if kind == "solve":
        s["scene"] = P.Scene(*_problem(case))
    elif kind == "batch":
        probs = workload.batch_problems(case["scene"], case["problems"])
        s["batch"] = P.Batch([dict(p, seed=seed) for p in probs])
    elif kind == "rollout":
        sc, sk = _problem(case)
        s["scene"] = P.Scene(sc, sk)
        if case["envs"] > 1:  # friction +-30 %, mass +-40 %, as in the tests
            s["scene"].set_randomization(case["envs"], 0.3, 0.4, seed)
        s["theta"] = _theta(sk["lo"], sk["hi"], case["N"], seed)
    elif kind == "update":
        lo, hi, s["theta"], s["J"], s["cls"] = _population(case, seed)
        sc, sk = workload.quadratic_scene(0, case["D"])
        s["scene"] = P.Scene(sc, dict(sk, lo=lo.tolist(), hi=hi.tolist()))
        D = case["D"]
        s["dist"] = [torch.zeros(D, device="cuda"), torch.zeros((D, D), device="cuda"), torch.zeros((D, D), device="cuda")]
    elif kind == "screen":
        sc, sk = workload.pickplace_scene(case["scene"])
        s["scene"], s["f16"] = P.Scene(sc, sk), workload.scene_features(sc)
        s["mean"], s["chol"] = (_dev(a) for a in _initial(sk["lo"], sk["hi"]))
        s["keep"] = torch.empty((case["keep"], len(sk["lo"])), device="cuda")
        s["idx"] = torch.empty(case["keep"], dtype=torch.int32, device="cuda")
    else:
        s["x"] = _rows(case["rows"], seed)
        if kind != "forward":
            s["t"] = _targets(s["x"], seed)
    if kind in ("forward", "gradient", "train", "screen"):
        s["net"] = P.Surrogate(WIDTH, DEPTH)
        s["net"].set_params(_mlp(seed), NORM)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "solve":
        r = s["scene"].solve(s["seed"], case["N"], case["K"], case["iters"])
        r.pop("elapsed_ms")
        return r
    if kind == "batch":
        b = s["batch"]
        b.reset()
        b.iterate(case["iters"])
        got = b.read()
        return {k: np.concatenate([np.asarray(r[k]).reshape(-1) for r in got]) for k in got[0]}
    if kind == "rollout":
        return s["scene"].rollout(s["theta"])
    if kind == "update":
        mean, cov, chol = s["dist"]
        idx, keff = s["scene"].refit(s["theta"], s["J"], s["cls"], case["K"], mean, cov, chol)
        return dict(idx=idx, k_eff=keff, mean=mean, cov=cov, chol=chol,
                    theta=s["scene"].sample(mean, chol, s["seed"], 1, case["N"]))
    if kind == "forward":
        return s["net"].forward(s["x"])
    if kind == "gradient":
        return s["net"].gradient(s["x"], s["t"])
    if kind == "train":
        loss = s["net"].train(s["x"], s["t"], batch=case["batch"], steps=case["steps"], seed=s["seed"])
        params, norm = s["net"].params()
        return dict(loss=loss, params=params, norm=norm)
    P.cem_surrogate_screen(s["scene"].h, s["net"].h, s["mean"], s["chol"], s["seed"], 0, 0, case["pool"], case["keep"],
                           s["f16"], s["keep"], s["idx"])
    return dict(theta=s["keep"], idx=s["idx"])


# -------------------------------------------------------------------- work
# adds + multiplies per simulated step and sample, by skeleton length
# (workload/flops_per_step.json), and per row of the surrogate's forward
STEP_FLOPS = {1: 47.0, 2: 73.7, 3: 303.7, 4: 315.8, 5: 316.9, 6: 303.7}
ROW_FLOPS = 2 * (IN * WIDTH + (DEPTH - 1) * WIDTH * WIDTH + WIDTH)
PARAMS = IN * WIDTH + (DEPTH - 1) * WIDTH * WIDTH + WIDTH + DEPTH * WIDTH + 1


def work(case):
    kind = case["kind"]
    if kind in ("solve", "rollout"):
        L = 1 if case["task"] == "reach" else 2 if case["task"] == "push" else case["actions"]
        T = {1: 400, 2: 1000}.get(L, 3000)
        D = {1: 3, 2: 6, 3: 8, 4: 11, 5: 14, 6: 17}[L]
        flops = case["N"] * T * STEP_FLOPS[L] * case.get("iters", 1) * case.get("envs", 1)
        return dict(flops=flops, bytes=2 * 4 * D * (1 + D) if kind == "solve" else case["N"] * (4 * D + 5))
    if kind == "batch":
        probs = workload.batch_problems(case["scene"], case["problems"])
        return dict(flops=case["iters"] * sum(p["N"] * p["scene"]["T"] * STEP_FLOPS[p["L"]] for p in probs),
                    bytes=sum(4 * (1 + 2 * len(p["skel"]["lo"])) * len(p["skel"]["lo"]) for p in probs))
    if kind == "update":
        D, N, K = case["D"], case["N"], case["K"]
        return dict(flops=K * D * (D + 1) + N * D * (D + 1), bytes=5 * N + 4 * K * (D + 1) + 4 * N * D)
    if kind == "forward":
        return dict(flops=case["rows"] * ROW_FLOPS, bytes=case["rows"] * 4 * (IN + 1) + 2 * PARAMS)
    if kind == "gradient":
        return dict(flops=3 * case["rows"] * ROW_FLOPS, bytes=case["rows"] * 4 * (IN + 1) + 6 * PARAMS)
    if kind == "train":
        return dict(flops=3 * case["batch"] * case["steps"] * ROW_FLOPS,
                    bytes=case["rows"] * 4 * (IN + 1) + case["steps"] * case["batch"] * 2 * IN + 8 * PARAMS)
    D = 14
    return dict(flops=case["pool"] * (ROW_FLOPS + D * (D + 1)), bytes=case["keep"] * 4 * (D + 1) + 2 * PARAMS)


# ------------------------------------------------------------------- exact
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words of whole-number arrays of counters."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.asarray(v, np.uint64) & m32 for v in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _normals(N, D, seed, it):
    z = np.zeros((N, (D + 3) // 4 * 4))
    for c in range((D + 3) // 4):
        u = [(w.astype(np.float64) + 1) * 2.0 ** -32 for w in _philox(np.arange(N), np.full(N, c), np.full(N, it),
                                                                      np.zeros(N), seed)]
        for p in (0, 2):
            r = np.sqrt(-2 * np.log(u[p]))
            z[:, 4 * c + p], z[:, 4 * c + p + 1] = r * np.cos(2 * np.pi * u[p + 1]), r * np.sin(2 * np.pi * u[p + 1])
    return z[:, :D]


def _exact_reach(case, seed):
    """The moveTo rollout (its scene has no contacts): unit-mass PD, Coulomb
    clamp of the trial velocity, interpolated crossing time."""
    sc, sk = workload.reach_scene(case["scene"])
    lo, hi = np.float32(sk["lo"]), np.float32(sk["hi"])
    th = _theta(sk["lo"], sk["hi"], case["N"], seed).cpu().numpy()
    th = np.clip(th, lo, hi).astype(np.float64)
    nom, dt, eps = np.array([2.0, 1.0]), sc["dt"], sc["eps"]
    mu = np.full(case["N"], sc["base_mu"])
    J = np.zeros(case["N"])
    for m in range(case["envs"]):
        if case["envs"] > 1:
            w = _philox(m, 256, 0, 0, seed)
            mu = np.full(case["N"], sc["base_mu"] * (1 + 0.3 * (2 * (float(w[0]) + 1) * 2.0 ** -32 - 1)))
        p, v = np.zeros((case["N"], 2)), np.zeros((case["N"], 2))
        goal, kp = nom + th[:, :2], th[:, 2:3]
        t = np.full(case["N"], sc["T"] * dt)
        open_ = np.ones(case["N"], bool)
        d0 = np.linalg.norm(p - nom, axis=1)
        for k in range(sc["T"]):
            v = v + dt * (kp * (goal - p) - 2 * np.sqrt(kp) * v)
            n = np.linalg.norm(v, axis=1)
            cap = mu * sc["g"] * dt
            v = v * np.where(n > cap, 1 - cap / np.maximum(n, 1e-300), 0.0)[:, None]
            p = p + v * dt
            d = np.linalg.norm(p - nom, axis=1)
            hit = open_ & (d <= eps)
            frac = np.where(d0 > eps, (d0 - eps) / np.where(d0 > d, d0 - d, 1), 0.0)
            t[hit] = (k + np.clip(frac[hit], 0, 1)) * dt
            open_ &= ~hit
            d0 = d
        J += sc["w_time"] * t + sc["w_goal"] * d
    return J / case["envs"], None


def _layers(flat):
    W, o = [], 0
    for l in range(DEPTH + 1):
        fi, fo = (IN if l == 0 else WIDTH), (1 if l == DEPTH else WIDTH)
        W.append((flat[o:o + fi * fo].view(fo, fi), flat[o + fi * fo:o + fi * fo + fo]))
        o += fi * fo + fo
    return W


def _raw(flat, x):
    a = x
    W = _layers(flat)
    for w, b in W[:-1]:
        z = a @ w.T + b
        a = 0.5 * z * (1 + torch.erf(z / math.sqrt(2)))
    return (a @ W[-1][0].T + W[-1][1])[:, 0]


def _loss(flat, x, t, mu, sd):
    return (_raw(flat, x) - (t - mu) / sd).square().mean()


def exact(case, seed):
    kind = case["kind"]
    if kind == "rollout":
        return _exact_reach(case, seed) if case["task"] == "reach" else None
    if kind == "update":
        lo, hi, theta, J, cls = _population(case, seed)
        th, J, cls = theta.cpu().numpy().astype(np.float64), J.cpu().numpy(), cls.cpu().numpy()
        best = min(set(cls.tolist()))
        sel = np.flatnonzero(cls == best)
        e = th[sel[np.lexsort((sel, J[sel]))][:case["K"]]]
        lo, hi = np.float32(lo).astype(np.float64), np.float32(hi).astype(np.float64)
        mean, c = e.mean(0), e - e.mean(0)
        cov = c.T @ c / len(e) + np.diag((1e-4 * (hi - lo)) ** 2) if len(e) > 1 else np.diag((0.05 * (hi - lo)) ** 2)
        chol = np.linalg.cholesky(cov)
        return dict(idx=None, k_eff=None, mean=mean, cov=cov, chol=chol,
                    theta=mean + _normals(case["N"], case["D"], seed, 1) @ chol.T)
    if kind not in ("forward", "gradient", "train"):
        return None
    flat = torch.as_tensor(_mlp(seed)).double().cuda()
    mu, sd = NORM
    x32 = _rows(case["rows"], seed)
    if kind == "forward":
        return mu + sd * _raw(flat, x32.double())
    t32 = _targets(x32, seed)
    if kind == "gradient":
        flat.requires_grad_(True)
        loss = _loss(flat, x32.double(), t32.double(), mu, sd)
        loss.backward()
        return flat.grad, float(loss)
    t = t32.double()
    mu, sd = float(t.mean()), float(t.std(unbiased=False))
    decay, o = torch.zeros_like(flat), 0
    for l in range(DEPTH + 1):
        fi, fo = (IN if l == 0 else WIDTH), (1 if l == DEPTH else WIDTH)
        decay[o:o + fi * fo] = 1e-4
        o += fi * fo + fo
    m1, m2, losses = torch.zeros_like(flat), torch.zeros_like(flat), []
    for k in range(case["steps"]):
        w = _philox(np.arange(case["batch"]), k, 0x5AFE, 0, seed)[0]
        row = torch.as_tensor(((w * np.uint64(case["rows"])) >> np.uint64(32)).astype(np.int64)).cuda()
        f = flat.clone().requires_grad_(True)
        loss = _loss(f, x32[row].double(), t[row], mu, sd)
        loss.backward()
        losses.append(float(loss))
        m1 = 0.9 * m1 + 0.1 * f.grad
        m2 = 0.999 * m2 + 0.001 * f.grad.square()
        step = (m1 / (1 - 0.9 ** (k + 1))) / ((m2 / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        flat = flat - 1e-3 * decay * flat - 1e-3 * step
    return dict(loss=np.array(losses), params=flat, norm=np.array([mu, sd]))
