"""A row of thousands of nonzeros among short ones: no product waits for one warp's walk
along it (the rule of csrc/sliced.cu, slices_pay; FP32 iterations, where slices gain least).

Iterations of a 100,000 x 200,000 LP on a GB300: 24 us; with one row of 8,000 nonzeros
48 us in slices, 30 us in the CSR ring."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


def test_iterations_with_a_long_row():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L

    def per_iteration(longest):
        rng = np.random.default_rng(1)
        lengths = rng.integers(5, 21, 100000)
        lengths[33333] = longest
        prob = L.Problem(synth.random_planted(100000, 200000, lengths=lengths, seed=2))
        opts = dict(precision=L.LP_PREC_MIXED, adaptive_step=0, tol=1e-30, polish_switch_tol=1e-30)
        best = [min(prob.solve(max_iters=k, **opts)[2]["solve_s"] for _ in range(4)) for k in (64, 576)]
        prob.close()
        return (best[1] - best[0]) / 512

    assert per_iteration(8000) < 1.6 * per_iteration(20)


def test_sliced_products_up_to_the_longest_row_taken():
    """Rows of every lane count of a slice, up to the longest that slices take in both
    precisions; one unrolled step against NumPy, bounds as in the other test of slices: a
    row of n terms errs by n 2^-53 (FP32: 2^-24) of its magnitudes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import autograd as A
    from paper_2508_16806_gb300 import lp as L
    rng = np.random.default_rng(3)
    m, n = 190003, 130017
    lengths = rng.integers(1, 16, m)
    special = [0, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025, 2047, 2048]
    lengths[rng.permutation(m)[: len(special)]] = special
    lp = synth.random_planted(m, n, lengths=lengths, seed=4)
    prob = L.Problem(lp)
    for prec, tol in ((L.LP_PREC_FP64, 1e-12), (L.LP_PREC_MIXED, 2e-4)):
        x, y, (tau, sigma) = A.unroll(prob, 1, precision=prec)
        x0 = np.clip(0.0, lp.l, lp.u)
        x1 = np.clip(x0 - tau * lp.c, lp.l, lp.u)
        y1 = sigma * (lp.q - lp.matvec(2.0 * x1 - x0))
        y1[lp.sense == 1] = np.maximum(y1[lp.sense == 1], 0.0)
        for a, b in ((x, x1), (y, y1)):
            assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)
    prob.close()
