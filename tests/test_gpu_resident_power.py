"""Algorithm 2 in one resident launch (csrc/resident.cu, k_res_power): its last barrier
follows a deciding barrier directly, so both take their sums from sets of their own.

One block, clusters of 2, 4, 8 and 16, and the grid.  A product's row of at most 20
terms errs by 20 x 2^-53 in its magnitudes; 2 x 100 products and their norms: 1e-12
bounds the quotient ||K b|| / ||b||."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(9, 30), (31, 64), (40, 100), (65, 200), (150, 400), (1500, 3001),
                                 (20000, 9000)])
def test_norm_of_resident_lps(oracle_mod, m, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    rng = np.random.default_rng(m)
    lp = synth.random_planted(m, n, lengths=rng.integers(1, min(n, 20) + 1, m), seed=n)
    prob = L.Problem(lp)
    for iters in (0, 1, 2, 3, 100):
        norms = {prob.solve(max_iters=1, ruiz_iters=0, power_iters=iters)[2]["norm_K"]
                 for _ in range(10)}
        assert len(norms) == 1
        want = oracle_mod.power_norm(lp, iters)
        assert abs(norms.pop() - want) <= 1e-12 * want
    prob.close()


@pytest.mark.parametrize("m,n", [(9, 30), (31, 64), (150, 400), (20000, 9000)])
@pytest.mark.parametrize("halpern", [0, 1])
def test_iterations_are_resident(oracle_mod, m, n, halpern):
    """One block, clusters of 2 and 16, the grid: a check period more is one launch and the
    nine of a check, and 70 fixed steps are the oracle's to 1e-10."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    rng = np.random.default_rng(m)
    lp = synth.random_planted(m, n, lengths=rng.integers(1, min(n, 20) + 1, m), seed=n)
    prob = L.Problem(lp)
    opts = dict(tol=1e-30, adaptive_step=0, halpern=halpern)
    _, a, b = (prob.solve(max_iters=k, **opts)[2]["kernel_launches"] for k in (64, 64, 128))
    assert b - a == 10
    x, y, info, _ = prob.solve(max_iters=70, **opts)
    xo, yo, io, _ = oracle_mod.solve(lp, max_iters=70, **opts)
    prob.close()
    assert info["iters"] == io["iters"] == 70
    for u, v in ((x, xo), (y, yo)):
        assert np.linalg.norm(u - v) <= 1e-10 * max(np.linalg.norm(v), 1e-300)
