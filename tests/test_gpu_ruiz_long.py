"""Ruiz passes on rows and columns of thousands of nonzeros (csrc/setup.cu, k_ruiz_pass):
the first 32 of a block's are finished by the whole block, any more by a warp each."""
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


def _transposed(lp):
    """The LP with K^T for K (its own costs and sides; only the iterates matter)."""
    rows = np.repeat(np.arange(lp.m), np.diff(lp.row_ptr))
    order = np.lexsort((rows, lp.col_idx))
    rp = np.zeros(lp.n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(lp.col_idx, minlength=lp.n))
    rng = np.random.default_rng(9)
    return synth.LP(lp.n, lp.m, rp, rows[order].astype(np.int32), lp.vals[order],
                    (np.arange(lp.n) % 2).astype(np.uint8), rng.standard_normal(lp.m),
                    rng.standard_normal(lp.n), np.full(lp.m, -1.0), np.full(lp.m, 2.0))


@pytest.mark.parametrize("side", [0, 1])
def test_scaling_against_the_oracle(L, oracle_mod, side):
    """Forty such rows (columns) in one block and one of 20,000; fixed steps on the scaled
    LP agree with the oracle's to 1e-10, as the other solves do."""
    rng = np.random.default_rng(side)
    lengths = rng.integers(2, 8, 20000)
    lengths[100:140] = np.arange(1040, 1840, 20)
    lengths[140:144] = [1024, 1025, 1088, 1089]
    lengths[9000] = 20000
    lp = synth.random_planted(20000, 30000, lengths=lengths, seed=side)
    lp.vals[:] *= 10.0 ** rng.integers(-2, 3, lp.vals.size)
    if side:
        lp = _transposed(lp)
    opts = dict(tol=1e-14, max_iters=40, adaptive_step=0)
    xo, yo, io, _ = oracle_mod.solve(lp, **opts)
    prob = L.Problem(lp)
    x, y, info, _ = prob.solve(**opts)
    x2, y2, _, _ = prob.solve(**opts)
    prob.close()
    assert abs(info["norm_K"] - io["norm_K"]) <= 1e-10 * io["norm_K"]
    for a, b in ((x, xo), (y, yo)):
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
    assert np.array_equal(x, x2) and np.array_equal(y, y2)


def test_a_pass_does_not_wait_for_one_warp(L):
    """Ten passes on a row of 500,000 nonzeros among 5,000 short ones: 96 times the time of
    the short ones alone when one warp walks the row."""
    def ten_passes(longest):
        rng = np.random.default_rng(5)
        lengths = rng.integers(3, 9, 5000)
        lengths[1666] = longest
        prob = L.Problem(synth.random_planted(5000, 600000, lengths=lengths, seed=6))
        best = [min(prob.solve(max_iters=0, ruiz_iters=k, ruiz_tol=0.0, power_iters=0)[2]["setup_s"]
                    for _ in range(6)) for k in (0, 10)]
        prob.close()
        return best[1] - best[0]

    assert ten_passes(500000) < 30 * ten_passes(20)
