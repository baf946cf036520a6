"""The first solve of a new LP whose products run in slices builds no task lists of the CSR
ring (csrc/setup.cu, schedule_side): host work, copies and allocations that nothing reads."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


def test_setup_of_a_new_lp():
    """200,000 x 400,000 with FP32 iterations on a GB300: the setup of a first solve beside
    that of a second one on the same handle: 1.6 times, 3.4 with the lists."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import lp as L
    rng = np.random.default_rng(1)
    lp = synth.random_planted(200000, 400000, lengths=rng.integers(5, 21, 200000), seed=2)
    opts = dict(precision=L.LP_PREC_MIXED, adaptive_step=0, tol=1e-30, polish_switch_tol=1e-30,
                max_iters=16)
    ratio = []
    for _ in range(6):
        prob = L.Problem(lp)
        first, second = (prob.solve(**opts)[2]["setup_s"] for _ in range(2))
        prob.close()
        ratio.append(first / second)
    assert min(ratio) < 2.5
