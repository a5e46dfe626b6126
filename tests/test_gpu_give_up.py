"""The FP32 kernels' pipeline waits that run out (an operand copy that never arrives): the call
ends, raises GFIP_STATUS_WAIT_TIMEOUT, and the next call on the handle is right.  The wait's limit
is 20 ms, nothing faults."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2302_08417_gb300 import gemmfip as g  # noqa: E402
from paper_2302_08417_gb300 import inputs  # noqa: E402
from tests import gpu_util as gu  # noqa: E402
from tests.test_gpu_trsm import residual_check, system  # noqa: E402

WAIT_NS = 20_000_000


@pytest.fixture(scope="module")
def runner():
    import __graft_entry__
    __graft_entry__.build()
    return gu.Runner()


# tensor-core tile core (whole and split tiles), the kernel for few rows, and the FFMA core behind
# both (an element outside the split's range; few tiles split along k, and whole ones)
@pytest.mark.parametrize("m,n,k,big", [(2000, 1500, 300, 0.0), (300, 290, 7001, 0.0),
                                       (8200, 100, 1499, 0.0), (700, 690, 900, 1e30),
                                       (2100, 2300, 200, 1e30)])
def test_gemm(runner, m, n, k, big):
    p = inputs.problem(m + n + k, "N", "T", m, n, k, 1.0, 0.5, 0, 0, 0, dtype=np.float32)
    if big:
        p.A[3] = big
    assert g.gfip_debug_f32_timeout(runner.h.h, True, WAIT_NS) == 0
    try:
        runner.run(p)
        assert runner.h.status() == g.GFIP_STATUS_WAIT_TIMEOUT
    finally:
        assert g.gfip_debug_f32_timeout(runner.h.h, False, 0) == 0
    got, guard = runner.run(p)
    gu.assert_close(p, got)
    gu.assert_gap_untouched(p, got, guard)
    assert runner.h.status() == 0


def test_trsm_panel(runner):
    rng = np.random.Generator(np.random.PCG64(3))
    na, nv = 300, 40
    A = system(rng, na, na, "L", "N", np.float32)
    B0 = inputs.colmajor(rng, na, nv, na, np.float32)
    dA, dB = (torch.from_numpy(x).to(runner.dev) for x in (A, B0))
    runner.h.ensure_trsm_workspace("L", "L", "N", "N", na, nv, 4)

    def solve():
        rc = g.gfip_trsm(4, runner.h.h, "L", "L", "N", "N", na, nv, 1.0, dA.data_ptr(), na,
                         dB.data_ptr(), na)
        assert rc == 0
        torch.cuda.synchronize()
        return dB.cpu().numpy()

    assert g.gfip_debug_f32_timeout(runner.h.h, True, WAIT_NS) == 0
    try:
        X = solve()
        assert runner.h.status() == g.GFIP_STATUS_WAIT_TIMEOUT
    finally:
        assert g.gfip_debug_f32_timeout(runner.h.h, False, 0) == 0
    # the CTA of the first 16 right-hand sides gave up and left them as they were
    assert np.array_equal(X[: 16 * na].view(np.uint8), B0[: 16 * na].view(np.uint8))
    dB.copy_(torch.from_numpy(B0))
    residual_check("L", "L", "N", "N", na, nv, 1.0, A, na, B0, na, solve())
    assert runner.h.status() == 0
