"""Gradient packs on an LP whose products run in slices (too large for the resident form, which
keeps the CSR ring for gradients): segments below, at and above a pack of eight reverse steps,
against the FP64 oracle, with the bound of the other pack tests (1e-10)."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


def test_reverse_steps_in_packs_on_slices(oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_16806_gb300 import autograd as AG
    from paper_2508_16806_gb300 import lp as L
    lp, xt = synth.adjoint_lp(100000, 200000, 8, seed=12)
    eta = 0.9 / oracle_mod.power_norm(lp, 50)
    prob = L.Problem(lp)
    # slices: the loop's launches are one per product (a resident solve takes one a check)
    few, more = (prob.solve(tol=1e-30, max_iters=k, adaptive_step=0)[2]["kernel_launches"] for k in (64, 128))
    assert more - few > 64
    for K, ckpt in ((5, 2), (8, 8), (9, 20), (17, 9)):
        xK, _, (tau, sigma) = AG.unroll(prob, K, eta=eta, omega=1.0)
        g = 2.0 * (xK - xt)
        dc, dq, dv, xK2, _ = AG.grad(prob, K, ckpt, g, eta=eta, omega=1.0)
        assert np.array_equal(xK, xK2)
        for a, b in zip((dc, dq, dv), oracle_mod.unrolled_adjoint(lp, tau, sigma, K, g)):
            assert rel(a, b) < 1e-10
    prob.close()
