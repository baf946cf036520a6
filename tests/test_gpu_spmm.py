"""Block products of fishnet casting at the edges of their lanes: rows of 0, 1, 7 to 9
(eight gathers in flight), 127 to 129 (a block per row above 128) and hundreds of
nonzeros, every width of a lane's load (2, 4 and 64 points, both precisions).  Bounds
as in the comparisons with the oracle elsewhere: 1e-9 (FP64) and 1e-3 (FP32) of a
fixed-step trajectory."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [2, 4, 64])
def test_block_products(oracle_mod, P):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    lengths = np.array([0, 1, 7, 8, 9, 15, 16, 17, 127, 128, 129, 300] + [5] * 289)
    lp = synth.random_planted(lengths.size, 700, lengths=lengths, seed=P)
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
