"""Gradient of unrolled iterations where the reverse steps are taken in packs of eight:
segments below, at and above a pack and its remainders, on rows in the CSR form (small
vectors) and in slices, against the FP64 oracle.

Tolerance: a step's rounding is about 1e-16 times the row lengths (up to 20) and does not
grow (the steps are non-expansive), over at most 24 steps and their reverse: 1e-13; 1e-10
leaves room for gradients that cancel."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("m,K,ckpt", [(50, 8, 8), (50, 9, 9), (50, 16, 16), (50, 17, 20), (50, 24, 7),
                                      (50, 5, 2), (13001, 18, 9)])
def test_reverse_steps_in_packs(oracle_mod, m, K, ckpt):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import autograd as AG
    from paper_2508_16806_gb300 import lp as L
    lp, xt = synth.adjoint_lp(m, 2 * m, 8, seed=11)
    eta = 0.9 / oracle_mod.power_norm(lp, 200)
    prob = L.Problem(lp)
    xK, _, (tau, sigma) = AG.unroll(prob, K, eta=eta, omega=1.0)
    assert rel(xK, oracle_mod.unrolled_forward(lp, tau, sigma, K)[0][-1]) < 1e-12
    g = 2.0 * (xK - xt)
    dc, dq, dv, xK2, _ = AG.grad(prob, K, ckpt, g, eta=eta, omega=1.0)
    assert np.array_equal(xK, xK2)
    for a, b in zip((dc, dq, dv), oracle_mod.unrolled_adjoint(lp, tau, sigma, K, g)):
        assert rel(a, b) < 1e-10
