"""A batch in sliced rows whose LPs finish at different times: from then on the products
walk the slices of the unfinished ones alone (csrc/batch.cu, kb_compact_slices).

An LP's sums do not depend on which list its slices come from, nor on the LPs beside it:
every LP returns the bits of a batch of its own."""
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


def _planted(m, seed, longest=20):
    rng = np.random.default_rng(seed)
    return synth.random_planted(m, 2 * m, lengths=rng.integers(4, longest + 1, m), seed=seed + 1)


def _solved_at_start(m, seed):
    """x = 0, y = 0 is optimal: done at the check of the start point."""
    lp = _planted(m, seed)
    lp.sense[:] = 1
    lp.c[:], lp.q[:], lp.l[:], lp.u[:] = 1.0, -1.0, 0.0, 5.0
    return lp


# every LP by itself is in sliced rows too (both vectors beyond what L1 holds)
@pytest.mark.parametrize("prec,sizes", [(0, [12400, 20000, 13001, 16000, 12500]),
                                        (1, [25000, 31007, 24600])])
def test_bits_of_a_batch_of_its_own(L, prec, sizes):
    # rows of other lengths: other numbers of iterations
    lps = [_planted(m, 7 * m, 6 + 9 * k) for k, m in enumerate(sizes)] + [_solved_at_start(25001, 3)]
    opts = dict(precision=[L.LP_PREC_FP64, L.LP_PREC_MIXED][prec], tol=1e-3, max_iters=1200,
                check_every=16)
    batch = L.Batch(lps)
    out = batch.solve(**opts)
    again = batch.solve(**opts)
    batch.close()
    assert len({r[2]["iters"] for r in out}) > 2 and out[-1][2]["iters"] == 0
    for lp, (x, y, info), second in zip(lps, out, again):
        alone = L.Batch([lp])
        (xa, ya, ia), = alone.solve(**opts)
        alone.close()
        for k in ("iters", "attempts", "restarts", "status"):
            assert info[k] == ia[k] == second[2][k]
        assert np.array_equal(x, xa) and np.array_equal(y, ya)
        assert np.array_equal(x, second[0]) and np.array_equal(y, second[1])


def test_finished_lps_cost_an_iteration_little(L):
    """An iteration of one 13,000-row LP beside 1,600 LPs that finished at the start point:
    the products and their launches stay, walking all slices would treble it (19 us -> 57 us
    on a GB300; 27 us with the finished ones left out)."""
    slow, done = _planted(13000, 1), _solved_at_start(2000, 2)

    def per_iteration(lps):
        batch = L.Batch(lps)
        best = []
        for iters in (128, 2176):
            opts = dict(tol=1e-15, max_iters=iters, adaptive_step=0)
            times = [batch.solve(**opts)[0][2] for _ in range(4)]
            assert all(t["iters"] == iters for t in times)
            best.append(min(t["solve_s"] for t in times[1:]))
        batch.close()
        return (best[1] - best[0]) / 2048

    assert per_iteration([slow] + [done] * 1600) < 2.0 * per_iteration([slow])
