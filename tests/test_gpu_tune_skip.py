"""The schedule autotuner times nothing that a solve does not run, and the launch counts of
a sliced batch are those of its launches."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    L.load()
    return L


def _lp(m, n, seed):
    rng = np.random.default_rng(seed)
    return synth.random_planted(m, n, lengths=rng.integers(5, 13, m), seed=seed)


# resident; both sides in slices; rows too long for slices, no split rows (tuned: two sides of
# six candidates, a warm-up and three timed launches each)
@pytest.mark.parametrize("m,n,row,extra", [(2000, 4000, 0, 0), (120000, 240000, 0, 0),
                                           (20000, 30000, 120, 48)])
def test_launches_of_the_tuner(L, m, n, row, extra):
    lp = _lp(m, n, m) if not row else synth.random_planted(m, n, lengths=np.full(m, row), seed=m)
    count = []
    for tune in (0, 1):
        prob = L.Problem(lp)
        count.append(prob.solve(tol=1e-14, max_iters=8, adaptive_step=0, autotune=tune)[2]["kernel_launches"])
        prob.close()
    assert count[1] - count[0] == extra


def test_launches_of_a_sliced_batch(L):
    """A check period more: 64 attempts of four launches, and a check of nine (one of them
    lists the slices of the unfinished LPs)."""
    batch = L.Batch([_lp(13000, 26000, 1), _lp(14000, 28000, 2)])
    # (the first solve builds the slices)
    _, a, b = (batch.solve(tol=1e-14, max_iters=k, adaptive_step=0)[0][2]["kernel_launches"]
               for k in (64, 64, 128))
    batch.close()
    assert b - a == 64 * 4 + 9
