"""Screening keeps exactly the lowest scores, ties by index, in index order,
at the edges of the selecting cluster's shares (4096 candidates in one CTA,
16,384 in four, eight beyond; 65,536 keys in registers) and with many or only
tied scores.  Whole numbers: no tolerance."""
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


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, np.float32)).cuda()


@pytest.mark.parametrize("scores", ["spread", "clamped", "equal", "nan"])
@pytest.mark.parametrize("n_pool,n_keep", [(1, 1), (33, 32), (4096, 511), (4097, 4096), (16384, 1), (16385, 8000),
                                           (65536, 8192), (65537, 65537), (1 << 20, 131073)])
def test_keeps_the_lowest(P, n_pool, n_keep, scores):
    sc, sk, _ = workload.config(2, seed=4)
    f16 = workload.scene_features(sc)
    lo, hi = np.array(sk["lo"]), np.array(sk["hi"])
    # clamped: most samples lie on their bounds, so that few scores differ
    mean, chol = dev((lo + hi) / 2), dev(np.diag((hi - lo) * (1e4 if scores == "clamped" else 0.25)))
    with P.Scene(sc, sk) as Sc, P.Surrogate(256, 4, seed=7) as S:
        p, norm = S.params()
        if scores in ("equal", "nan"):
            S.set_params(np.full_like(p, 0.0 if scores == "equal" else np.nan), norm)
        keep = torch.empty((n_keep, len(lo)), device="cuda")
        idx = torch.full((n_keep,), -1, dtype=torch.int32, device="cuda")
        P.cem_surrogate_screen(Sc.h, S.h, mean, chol, 9, 1, 0, n_pool, n_keep, f16, keep, idx)
        pool = Sc.sample(mean, chol, 9, 1, n_pool, problem=0)
        score = S.forward(S.features(pool, lo, hi, f16)).cpu().numpy()
    score = np.where(np.isfinite(score), score, np.inf)
    expect = np.sort(np.lexsort((np.arange(n_pool), score))[:n_keep])
    assert np.array_equal(idx.cpu().numpy(), expect)
    assert np.array_equal(keep.cpu().numpy(), pool.cpu().numpy()[expect])
