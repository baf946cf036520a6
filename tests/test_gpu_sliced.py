"""Sliced rows (csrc/sliced.cuh) against a NumPy FP64 product, through lp_unroll and
lp_solve: LPs too large for the resident form, with the edges of the slices in their
rows and columns (none, 1, 31 to 33, 64 / 65, 127 to 129, 1,023 to 1,025 nonzeros and
thousands; row and column counts that are no multiple of 32 or of a window).

FP64: one unrolled step is two products and elementwise operations; a row's sum of n
terms differs from NumPy's by at most n 2^-53 times the sum of the terms' magnitudes:
1e-12 relative to the vector's norm for the longest rows here."""
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


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _lp(m, n, seed):
    rng = np.random.default_rng(seed)
    lengths = rng.integers(1, 24, m)
    special = [0, 1, 31, 32, 33, 64, 65, 127, 128, 129, 1023, 1024, 1025, 5000]
    lengths[rng.permutation(m)[: len(special)]] = special
    return synth.random_planted(m, n, lengths=lengths, seed=seed + 1)


@pytest.mark.parametrize("m,n", [(150001, 290017), (260000, 70003)])
def test_sliced_products(L, m, n):
    from paper_2508_16806_gb300 import autograd as A
    lp = _lp(m, n, m + n)
    prob = L.Problem(lp)
    # x1 = clamp(x0 - tau c), y1 = proj(sigma (q - K (2 x1 - x0))), then K^T y1 enters x2
    for prec, tol in ((L.LP_PREC_FP64, 1e-12), (L.LP_PREC_MIXED, 2e-4)):
        x, y, (tau, sigma) = A.unroll(prob, 2, precision=prec)
        x0 = np.clip(0.0, lp.l, lp.u)
        x1 = np.clip(x0 - tau * lp.c, lp.l, lp.u)
        y1 = sigma * (lp.q - lp.matvec(2.0 * x1 - x0))
        y1[lp.sense == 1] = np.maximum(y1[lp.sense == 1], 0.0)
        x2 = np.clip(x1 - tau * (lp.c - lp.rmatvec(y1)), lp.l, lp.u)
        y2 = y1 + sigma * (lp.q - lp.matvec(2.0 * x2 - x1))
        y2[lp.sense == 1] = np.maximum(y2[lp.sense == 1], 0.0)
        assert rel(x, x2) <= tol and rel(y, y2) <= tol
    # bitwise repeatable, and the solver's own reductions see every row
    a = prob.solve(tol=1e-14, max_iters=20)
    b = prob.solve(tol=1e-14, max_iters=20)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    prob.close()


@pytest.mark.parametrize("rows", [[2, 31, 255, 256, 257, 9000, 20011], [30000, 1, 30001]])
def test_sliced_batch_tracks_single_solves(L, rows):
    """Slices of several LPs side by side (windows cut at LP ends): 64 fixed steps of each LP
    are those of its own solve, to the bound of the batch's other tests (1e-10)."""
    rng = np.random.default_rng(len(rows))
    lps = [synth.random_planted(m, 2 * m, lengths=rng.integers(1, min(2 * m, 21) + 1, m), seed=m)
           for m in rows]
    batch = L.Batch(lps)
    out = batch.solve(tol=1e-13, max_iters=64, adaptive_step=0)
    for lp, (x, y, info) in zip(lps, out):
        prob = L.Problem(lp)
        xs, ys, si, _ = prob.solve(tol=1e-13, max_iters=64, adaptive_step=0)
        assert info["status"] == si["status"] and info["iters"] == si["iters"]
        assert rel(x, xs) <= 1e-10 and rel(y, ys) <= 1e-10
        prob.close()
    batch.close()
