"""FP64 products of few rows and columns and many terms: on either side of the line between the
small kernels and the persistent core, in every order, against the oracle; and the choice itself,
by the launch's grid."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2302_08417_gb300 import gemmfip as g  # noqa: E402
from paper_2302_08417_gb300 import inputs  # noqa: E402
from tests import gpu_util as gu  # noqa: E402


@pytest.fixture(scope="module")
def runner():
    import __graft_entry__
    __graft_entry__.build()
    return gu.Runner()


@pytest.mark.parametrize("m,n,k", [(8, 8, 8191), (8, 8, 8192), (1, 33, 20001), (64, 64, 8193),
                                   (3, 5, 400000), (20, 17, 131073)])
def test_orders(runner, m, n, k):
    for ta, tb in itertools.product("NT", "NT"):
        p = inputs.problem(m + k, ta, tb, m, n, k, -0.5, 0.5, 3, 1, 2)
        got, guard = runner.run(p)
        gu.assert_close(p, got)
        gu.assert_gap_untouched(p, got, guard)
    assert runner.h.status() == 0


def test_few_tiles_and_a_long_k_take_all_sms(runner):
    """8 x 8 x 4000000: one tile of the small kernels is a cluster of eight CTAs, a third of the
    speed of the core that splits k over all SMs; up to k = 200000 the cluster is faster."""
    m = n = 8
    for k, all_sms in ((30000, False), (4000000, True)):
        A = torch.rand(m * k, dtype=torch.float64, device="cuda")
        B = torch.rand(k * n, dtype=torch.float64, device="cuda")
        C = g.gemm(torch.as_strided(A, (m, k), (1, m)), torch.as_strided(B, (k, n), (1, k)),
                   handle=runner.h)
        assert (g.gfip_last_launch_info(runner.h.h)[1] > 8) == all_sms
        want = torch.as_strided(A, (m, k), (1, m)) @ torch.as_strided(B, (k, n), (1, k))
        assert torch.all((C - want).abs() <= 2 * k * 2.0**-53 * want)   # entries in [0, 1]
