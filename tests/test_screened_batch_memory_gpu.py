"""A screened batch whose surrogate lost its rows (a larger call on the same
handle found no memory) gets them again, or reports that there is no room."""
import numpy as np
import pytest

from test_screened_batch_gpu import P, scenes  # noqa: F401 (P is the fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_rows_are_reserved_again(P):  # noqa: F811
    probs = [dict(scene=sc, skel=sk, N=300, K=20, seed=i) for i, (sc, sk, _) in enumerate(scenes(2, T=200))]
    f16 = np.stack([f for _, _, f in scenes(2, T=200)])
    x = torch.zeros(5000 * 48 + 1, device="cuda")[1:].view(5000, 48)  # (unaligned: scored through the row workspace)
    with P.Surrogate(256, 4, seed=3) as S, P.Batch(probs) as B:
        B.set_screening(S, f16, 1024, 100)
        B.iterate_screened(2)
        want = B.read()
        B.reset()
        P.cem_test_fail_allocation(3)
        with pytest.raises(P.CemError):
            S.forward(x)
        P.cem_test_fail_allocation(1)
        with pytest.raises(P.CemError) as err:
            B.iterate_screened(2)
        assert P.STATUS[err.value.code] == "CEM_ERR_NO_MEMORY"
        B.iterate_screened(2)
        for g, w in zip(B.read(), want):
            assert g["best_J"] == w["best_J"] and np.array_equal(g["mean"], w["mean"]) and np.array_equal(g["chol"], w["chol"])
