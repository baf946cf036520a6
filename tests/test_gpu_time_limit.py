"""A time limit that strikes on the attempt before a check leaves the decision to that check:
the returned pair is the candidate of the last record, whatever attempt the limit meets.

Every second iteration is followed by a check here, so that many of the stops meet it."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("halpern", [0, 1])
@pytest.mark.parametrize("m,n", [(300, 700), (6000, 15000)])
def test_pair_of_the_last_check(oracle_mod, m, n, halpern):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    rng = np.random.default_rng(m)
    lp = synth.random_planted(m, n, lengths=rng.integers(3, 15, m), seed=m)
    prob = L.Problem(lp)
    for limit in np.linspace(0.002, 0.02, 24):
        x, y, info, tr = prob.solve(tol=1e-14, max_iters=10**9, time_limit_s=float(limit), halpern=halpern,
                                    check_every=2, trace_cap=100000)
        assert info["status"] == L.LP_TIME_LIMIT
        k = oracle_mod.kkt(lp, x, y)
        for f in ("rel_gap", "rel_pres", "rel_dres"):
            assert tr[-1][f] == info[f]
            if halpern:
                assert k[f] == pytest.approx(info[f], rel=1e-6, abs=1e-12)
    prob.close()
