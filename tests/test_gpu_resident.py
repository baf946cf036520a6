"""Resident iterations (csrc/resident.cuh) against the FP64 oracle: every form of
the plan (one block, clusters of 2 to 16, the cooperative grid, an LP that is too
large for it) and the edges of its row classes (empty rows, 31 to 33 and 64 / 65
nonzeros, rows of 1,023 to 1,025 and of thousands, an empty column, dense columns).

FP64 runs of the fixed step agree with the oracle to 1e-10 over 70 iterations (one
full check period, a restart decision and a part of the next), as the other paths
do.  FP32 runs: an entry's relative error grows by at most the length of a dot
product (a few dozen terms for all but a handful of rows) times 2^-24 a step, and
the map does not expand: 70 steps x 64 x 6e-8 = 2.7e-4 in norm."""
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


@pytest.fixture(scope="module")
def oracle_mod():
    import oracle
    oracle.build()
    return oracle


def rel(a, b):
    a, b = np.asarray(a, float), np.asarray(b, float)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _lp(m, n, seed):
    rng = np.random.default_rng(seed)
    lengths = rng.integers(1, min(n, 14) + 1, m)
    special = [0, 31, 32, 33, 64, 65, 1023, 1024, 1025, 3000]
    special = [s for s in special if s <= n // 2 and m >= 200]
    lengths[rng.permutation(m)[: len(special)]] = special
    return synth.random_planted(m, n, lengths=lengths, seed=seed + 1)


# one block; clusters of 2, 4, 8, 16; FP64 grid; both on the grid; too large for either
SIZES = [(1, 1), (7, 3), (40, 100), (65, 129), (200, 400), (1500, 3001), (7001, 6500),
         (12000, 9000), (90000, 200001)]
FIXED = dict(adaptive_step=0)


@pytest.mark.parametrize("m,n", SIZES)
@pytest.mark.parametrize("halpern", [0, 1])
def test_resident_iterations_against_the_oracle(L, oracle_mod, m, n, halpern):
    lp = _lp(m, n, 17 * m + n)
    opts = dict(tol=1e-14, max_iters=70, halpern=halpern, **FIXED)
    xo, yo, io, _ = oracle_mod.solve(lp, **opts)
    prob = L.Problem(lp)
    x, y, info, _ = prob.solve(**opts)
    assert info["iters"] == io["iters"] and info["restarts"] == io["restarts"]
    assert rel(x, xo) <= 1e-10 and rel(y, yo) <= 1e-10
    # the same solve again on the same handle: the same bits
    x2, y2, _, _ = prob.solve(**opts)
    assert np.array_equal(x, x2) and np.array_equal(y, y2)
    xm, ym, im, _ = prob.solve(precision=L.LP_PREC_MIXED, polish_switch_tol=1e-14, **opts)
    if not halpern:      # (FP32 Halpern iterations take another reflection)
        assert im["iters"] == info["iters"]
        assert rel(xm, xo) <= 2.7e-4 and rel(ym, yo) <= 2.7e-4
    prob.close()


@pytest.mark.parametrize("m,n", [(200, 400), (1500, 3001), (12000, 9000)])
def test_resident_adaptive_steps(L, oracle_mod, m, n):
    """Algorithm 5 inside the launch: the attempts, decisions and iterates of the first
    check period (32 iterations) are the oracle's."""
    lp = _lp(m, n, 3 * m + n)
    opts = dict(tol=1e-14, max_iters=32, check_every=32)
    xo, yo, io, _ = oracle_mod.solve(lp, **opts)
    prob = L.Problem(lp)
    x, y, info, _ = prob.solve(attempt_cap=200, **opts)
    assert info["iters"] == io["iters"] and info["attempts"] == io["attempts"]
    assert len(info["attempt_log"]) == info["attempts"]
    assert rel(x, xo) <= 1e-10 and rel(y, yo) <= 1e-10
    prob.close()
