"""FP32 sums of a KKT check: no thread adds more rows or columns in FP32 than 1,216 blocks
of 256 threads do (csrc/common.cuh, kCheckGrid).

As many rows and columns as those threads, in two halves of 1 and of 2^-25, which FP32
loses beside a 1: each must reach FP64 by itself.  Both sums are then exact in doubles."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


def test_every_term_reaches_fp64():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    N = 1216 * 256
    one = np.ones(N)
    v = np.where(np.arange(N) < N // 2, 1.0, 2.0 ** -25)
    lp = synth.LP(N, N, np.arange(N + 1, dtype=np.int64), np.arange(N, dtype=np.int32), one.copy(),
                  np.zeros(N, np.uint8), one.copy(), one.copy(), np.zeros(N), 2.0 * one)
    prob = L.Problem(lp)
    info = prob.solve(precision=L.LP_PREC_MIXED, tol=0.0, max_iters=0, ruiz_iters=0, x0=v, y0=v)[2]
    prob.close()
    assert info["status"] == L.LP_ITERATION_LIMIT
    # c^T x, and q^T y + l^T lambda^+ + u^T lambda^- with lambda = c - y >= 0, l = 0
    assert info["pobj"] == v.sum() and info["dobj"] == v.sum()
