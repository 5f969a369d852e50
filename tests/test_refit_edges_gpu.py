"""Elite selection and refit at the edges of its sizes (16,384 keys in registers,
512 elites staged, 1024 sorted in registers), with ties and costs that are not
finite, against the oracle: indices exact,
statistics within the roundings of their FP32 results (2^-24 relative, the
covariance and its factor relative to their largest entry, with the factor's
condition number allowed for)."""
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


def dev(a, t=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a)).to("cuda", t)


def population(N, D, costs, seed):
    rng = np.random.default_rng(seed)
    theta = rng.standard_normal((N, D)).astype(np.float32)
    J = rng.uniform(0, 10, N).astype(np.float32)
    cls = rng.integers(0, 3, N).astype(np.uint8)
    if costs == "ties":
        J = np.round(J).astype(np.float32)
    elif costs == "equal":
        J[:] = 1.5
        cls[:] = 1
    elif costs == "bad":  # infinities, NaN and signed zeros among few good ones
        J[rng.random(N) < 0.5] = np.nan
        J[rng.random(N) < 0.2] = -np.inf
        J[rng.random(N) < 0.2] = -0.0
        J[rng.random(N) < 0.1] = 0.0
    return theta, J, cls


@pytest.mark.parametrize("costs", ["spread", "ties", "equal", "bad"])
@pytest.mark.parametrize("N,K,D", [(1, 1, 3), (31, 40, 3), (512, 25, 3), (513, 25, 6), (4096, 511, 14), (4097, 512, 14),
                                   (16384, 513, 17), (16385, 512, 18), (65537, 4096, 6)])
def test_matches_oracle(P, orc, N, K, D, costs):
    theta, J, cls = population(N, D, costs, N + D)
    sc, sk = workload.quadratic_scene(0, D)
    mean, cov, chol = torch.zeros(D, device="cuda"), torch.zeros((D, D), device="cuda"), torch.zeros((D, D), device="cuda")
    with P.Scene(sc, sk) as S:
        idx, keff = S.refit(dev(theta), dev(J), dev(cls, torch.uint8), K, mean, cov, chol)
    k = int(keff.item())
    want = orc.select(J, cls, K)
    assert k == len(want) and np.array_equal(idx.cpu().numpy()[:k], want)
    if k == 0:
        return
    e = theta[want].astype(np.float64)
    span = np.array(sk["hi"]) - np.array(sk["lo"])
    m = e.mean(0)
    C = (e - m).T @ (e - m) / k + np.diag((1e-4 * span) ** 2) if k > 1 else np.diag((0.05 * span) ** 2)
    L = np.linalg.cholesky(C)
    ulp = 2.0 ** -23
    assert np.abs(mean.cpu().numpy() - m).max() <= ulp * max(1.0, np.abs(m).max())
    assert np.abs(cov.cpu().numpy() - C).max() <= ulp * np.abs(C).max()
    assert np.abs(chol.cpu().numpy() - L).max() <= ulp * np.abs(L).max() + 1e-15 * np.linalg.cond(C)
