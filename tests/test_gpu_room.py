"""Second copies of the matrix and little device memory (csrc/sliced.cu, csrc/capi.cu): the
form of the products does not follow what is free, and a call that does not fit beside the
copies runs without them.

The memory left is counted from the buffers that the calls hold; 150 MB is the room for the
2 MB granules of some forty allocations."""
import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu
M, N, CKPT = 500000, 1000000, 100
MB = 1 << 20


@pytest.fixture(scope="module")
def lp():
    rng = np.random.default_rng(1)
    return synth.random_planted(M, N, lengths=rng.integers(5, 21, M), seed=2)


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


class _Left:
    """All device memory but `left` bytes is taken."""

    def __init__(self, torch, left):
        self.torch = torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        self.hog = torch.empty(free - int(left), dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *_):
        self.hog = None
        self.torch.cuda.empty_cache()


def _engine_bytes(torch, prob, call):
    before = torch.cuda.mem_get_info()[0]
    out = call()
    torch.cuda.synchronize()
    return out, before - torch.cuda.mem_get_info()[0]


def test_same_bits_with_little_memory(torch, lp):
    from paper_2508_16806_gb300 import lp as L
    opts = dict(tol=1e-14, max_iters=20, adaptive_step=0)
    prob = L.Problem(lp)
    (x, y, _, _), held = _engine_bytes(torch, prob, lambda: prob.solve(**opts))
    prob.close()
    prob = L.Problem(lp)
    with _Left(torch, held + 150 * MB):
        x2, y2, _, _ = prob.solve(**opts)
    prob.close()
    assert np.array_equal(x, x2) and np.array_equal(y, y2)


def test_gradient_runs_without_the_copies(torch, lp):
    from paper_2508_16806_gb300 import autograd as A
    from paper_2508_16806_gb300 import lp as L
    g = np.ones(N)
    args = (CKPT, CKPT, g)
    prob = L.Problem(lp)
    want, held = _engine_bytes(torch, prob, lambda: A.grad(prob, *args, eta=0.05, omega=1.0))
    prob.close()
    # what the call holds by itself: checkpoints, the ring of iterates and masks, adjoints,
    # one step's factors, the derivatives and their staging
    s, c, z = 8 * (N + M), N + M, lp.nnz
    call = s + (CKPT + 1) * s + CKPT * c + 2 * s + 2 * s + s + 2 * 8 * z
    copies = 32 * z          # values, columns and nonzeros of both sides, without padding
    prob = L.Problem(lp)
    with _Left(torch, held - copies + call + 150 * MB):
        got = A.grad(prob, *args, eta=0.05, omega=1.0)
        again = A.grad(prob, *args, eta=0.05, omega=1.0)
    prob.close()
    for a, b, d in zip(got[:4], want[:4], again[:4]):
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
        assert np.array_equal(a, d)


def test_a_call_that_never_fits_leaves_the_handle_usable(torch, lp):
    from paper_2508_16806_gb300 import lp as L
    opts = dict(tol=1e-14, max_iters=4, adaptive_step=0)
    prob = L.Problem(lp)
    want = prob.solve(**opts)
    prob.close()
    prob = L.Problem(lp)
    with _Left(torch, 200 * MB):
        for _ in range(2):
            with pytest.raises(L.LpError):
                prob.solve(**opts)
    got = prob.solve(**opts)
    prob.close()
    for a, b in zip(got[:2], want[:2]):
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
