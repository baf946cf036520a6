"""An LP on a stream that has a part of the device's SMs (a green context): no launch whose
blocks wait for one another, and the results of the whole device (csrc/resident.cu,
stream_sms)."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2508_16806_gb300 import synth

pytestmark = pytest.mark.gpu
HELPER = r"""
#include <cuda.h>
static CUgreenCtx ctx;
static CUstream stream;
void* part_stream(int sms, int* got)
{
    CUdevResource all, part, rest, mine;
    CUdevResourceDesc desc;
    CUdevice dev;
    unsigned int n = 1;
    if (cuCtxGetDevice(&dev) || cuDeviceGetDevResource(dev, &all, CU_DEV_RESOURCE_TYPE_SM) ||
        cuDevSmResourceSplitByCount(&part, &n, &all, &rest, 0, sms) ||
        cuDevResourceGenerateDesc(&desc, &part, 1) ||
        cuGreenCtxCreate(&ctx, desc, dev, CU_GREEN_CTX_DEFAULT_STREAM) ||
        cuGreenCtxStreamCreate(&stream, ctx, CU_STREAM_NON_BLOCKING, 0) ||
        cuGreenCtxGetDevResource(ctx, &mine, CU_DEV_RESOURCE_TYPE_SM))
        return 0;
    *got = (int)mine.sm.smCount;
    return stream;
}
void part_free(void) { cuStreamDestroy(stream); cuGreenCtxDestroy(ctx); }
"""


@pytest.fixture(scope="module")
def part(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("part")
    (d / "part.c").write_text(HELPER)
    r = subprocess.run(["gcc", "-shared", "-fPIC", "-I/usr/local/cuda/include", str(d / "part.c"), "-o",
                        str(d / "part.so"), "-L/usr/local/cuda/lib64/stubs", "-lcuda"])
    if r.returncode:
        pytest.skip("no driver header or stub to build the helper with")
    torch.zeros(1, device="cuda")
    lib, got = C.CDLL(str(d / "part.so")), C.c_int(0)
    lib.part_stream.restype = C.c_void_p
    s = lib.part_stream(64, C.byref(got))
    if not s or got.value >= torch.cuda.get_device_properties(0).multi_processor_count:
        pytest.skip("the driver gives no part of the device")
    yield torch.cuda.ExternalStream(s)
    torch.cuda.synchronize()
    lib.part_free()


# a cluster of the whole device, its grid, slices
@pytest.mark.parametrize("m,n", [(1500, 3000), (20000, 30000), (120000, 240000)])
def test_solve_and_gradient_on_a_part(part, m, n):
    from paper_2508_16806_gb300 import autograd as A
    from paper_2508_16806_gb300 import lp as L
    rng = np.random.default_rng(m)
    lp = synth.random_planted(m, n, lengths=rng.integers(5, 13, m), seed=m)
    out = []
    for stream in (None, part):
        prob = L.Problem(lp, stream=stream)
        x, y, info, _ = prob.solve(tol=1e-14, max_iters=70, adaptive_step=0, loop_mode=1)
        assert info["iters"] == 70
        out.append((x, y, *A.grad(prob, 10, 5, np.ones(n))[:4]))
        prob.close()
    for a, b in zip(*out):
        assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
