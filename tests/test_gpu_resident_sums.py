"""The sums of Algorithm 5 of FP32 iterations inside a resident launch lose nothing that a
reduction in doubles keeps (csrc/resident.cuh, warp_fixed_sum).

The first step goes to the upper bounds (costs far below zero, x = 0), so ||x' - x||^2 is
the sum of the squares of 31 chosen FP32 values, each rounded to FP32, a value to a lane.
Its double may be off by the two roundings that form it and the scaling's none: 3 x 2^-53."""
import math

import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spread", [0, 3, 15, 30])
def test_step_sums_in_full(spread):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    for seed in range(10):
        rng = np.random.default_rng(seed)
        lp = synth.random_planted(3, 31, lengths=np.array([2, 3, 4]), seed=seed)
        lp.l[:] = 0.0
        lp.u[:] = ((1.0 + rng.random(31)) * 2.0 ** rng.integers(-spread, spread + 1, 31)).astype(np.float32)
        lp.c[:] = -1e18
        prob = L.Problem(lp)
        info = prob.solve(precision=L.LP_PREC_MIXED, tol=0.0, max_iters=1, ruiz_iters=0, omega0=1.0,
                          eta0=1.0, attempt_cap=4)[2]
        prob.close()
        u = lp.u.astype(np.float32)
        want = math.fsum(float(v) for v in u * u)
        assert abs(info["attempt_log"][0]["dx2"] - want) <= 3 * 2.0 ** -53 * want
