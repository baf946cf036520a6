"""Block products of fishnet casting with few points: a row's terms are added in 32 / P
groups, whose sums then meet in pairs, with a warp per row (few rows: k_spmm_warp in
csrc/fishnet.cu) and with lanes (many: k_spmm) alike.

Rows of 128 nonzeros, the first so large that a 1 added to it is lost, the others 1: the
group of the first keeps it alone, every other group its 128 / G ones.  No steps: the dual
point is the product of the cast point (all ones), exactly."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 6200])
@pytest.mark.parametrize("P", [1, 2, 4])
@pytest.mark.parametrize("mixed", [0, 1])
def test_groups_of_a_row(m, P, mixed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    opts = dict(precision=L.LP_PREC_MIXED if mixed else L.LP_PREC_FP64, ruiz_iters=0, power_iters=0)
    big, terms = (2.0 ** 24 if mixed else 2.0 ** 53), 128 - 128 // (32 // P)
    for n in range(128, 160):
        lp = synth.LP(m, n, 128 * np.arange(m + 1, dtype=np.int64),
                      np.tile(np.arange(128, dtype=np.int32), m),
                      np.tile(np.concatenate([[big], np.ones(127)]), m), np.zeros(m, np.uint8),
                      np.ones(n), np.ones(m), np.zeros(n), np.full(n, 2.0))
        prob = L.Problem(lp)
        # the points are cast as ||K|| / sqrt(n) times the draws: draws that give ones
        rad = prob.solve(max_iters=0, **opts)[2]["norm_K"] / np.sqrt(n)
        if rad * (1.0 / rad) == 1.0:
            break
        prob.close()
    else:
        pytest.fail("no size casts ones")
    x, y, _, _ = prob.fishnet(P, 0, np.full((n, P), 1.0 / rad), np.ones(64), **opts)
    prob.close()
    assert np.array_equal(x, np.ones(n)) and np.array_equal(y, np.full(m, big + terms))


@pytest.mark.parametrize("P", [2, 4, 8, 16, 32, 64])
def test_products_of_many_rows(oracle_mod, P):
    """Every width and group count of the lanes' form at the edges of its rounds of eight;
    bounds as in the other comparisons with the oracle: 1e-9 (FP64) and 1e-3 (FP32)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    edges = [0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 127, 128, 129, 300]
    lengths = np.array(edges + [5] * (6400 - len(edges)))
    lp = synth.random_planted(lengths.size, 7000, lengths=lengths, seed=P)
    rng = np.random.default_rng(P)
    G = rng.standard_normal((lp.n, P))
    Z = rng.standard_normal(max(oracle_mod.fishnet_draws(P), 1))
    ox, oy, og, orounds = oracle_mod.fishnet(lp, P, 4, G, Z)
    for prec, tol in ((L.LP_PREC_FP64, 1e-9), (L.LP_PREC_MIXED, 1e-3)):
        gx, gy, gg, rounds = L.Problem(lp).fishnet(P, 4, G, Z, precision=prec)
        assert rounds == orounds
        fin = np.isfinite(og)
        np.testing.assert_allclose(gg[fin], og[fin], rtol=tol, atol=tol * 1e-3)
        assert np.linalg.norm(gx - ox) <= tol * np.linalg.norm(ox)
        assert np.linalg.norm(gy - oy) <= tol * np.linalg.norm(oy)
