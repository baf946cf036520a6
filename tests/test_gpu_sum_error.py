"""Rounding of the products' row sums, in slices and in resident iterations: no longer a
chain of additions than the CSR ring's lane groups have.

One Halpern step from x = 0, K x^ with x^ = u known exactly, costs far below zero: y^ =
-2 sigma K u.  Rows of n equal-sized random terms; the error against 64-bit mantissas or
wider, in units of 2^-52 (2^-23) times the sum of the terms' magnitudes, root mean square.
Simulated orders, n = 12 | 24 | 32: one chain 0.199 | 0.199 | 0.197; four chains up to 15,
eight (or two lanes of four) above 0.163 | 0.131 | 0.118; the ring in FP64 0.172 | 0.135 |
0.119.  Bound: the ring's plus a tenth."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


# resident in a cluster and in the grid, slices
@pytest.mark.parametrize("m,n", [(3000, 6000), (20000, 30000), (120000, 240000)])
@pytest.mark.parametrize("row,bound", [(6, 0.222), (12, 0.19), (24, 0.149), (32, 0.131)])
def test_row_sums(m, n, row, bound):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    wide = np.longdouble
    assert np.finfo(wide).nmant >= 63
    rng = np.random.default_rng(row)
    for prec, f in ((L.LP_PREC_FP64, np.float64), (L.LP_PREC_MIXED, np.float32)):
        if f == np.float32 and m > 20000 and row >= 16:
            continue      # in the ring
        lp = synth.random_planted(m, n, lengths=np.full(m, row), seed=row)
        lp.sense[:], lp.q[:], lp.c[:], lp.l[:] = 0, 0.0, -1e6, 0.0
        lp.vals[:] = lp.vals.astype(f)
        lp.u[:] = (0.5 + rng.random(n)).astype(f)
        prob = L.Problem(lp)
        y = prob.solve(precision=prec, halpern=1, tol=0.0, max_iters=1, check_every=1, ruiz_iters=0,
                       eta0=0.5, omega0=1.0)[1]
        prob.close()
        terms = lp.vals.astype(wide).reshape(m, row) * lp.u.astype(wide)[lp.col_idx].reshape(m, row)
        err = (y.astype(wide) + terms.sum(1)) / np.abs(terms).sum(1)
        assert float(np.sqrt(np.mean(err ** 2))) <= bound * np.finfo(f).eps
