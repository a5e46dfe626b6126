"""The small-product kernels (csrc/gfip_small.cu) at the edges of their tiles, k groups and
slabs, with one CTA or a cluster per tile and one tile per warp or per CTA, against the oracle
within 2 max(k, 2) u (|alpha||op(A)||op(B)| + |beta||C0|)."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2302_08417_gb300 import inputs  # noqa: E402
from tests import gpu_util as gu  # noqa: E402


@pytest.fixture(scope="module")
def runner():
    import __graft_entry__
    __graft_entry__.build()
    return gu.Runner()


# one element; tile and group remainders; clusters of 2, 4 and 8 with ragged k; many tiles
SHAPES = [(1, 1, 1), (8, 8, 16), (9, 7, 19), (33, 31, 63), (32, 32, 65), (1, 40, 3000),
          (64, 64, 1001), (100, 90, 333), (250, 240, 129), (450, 440, 35)]


@pytest.mark.parametrize("dtype", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_shapes_and_orders(runner, dtype, m, n, k):
    for (ta, tb), (alpha, beta) in zip(itertools.product("NT", "NT"),
                                       ((1.0, 0.5), (-0.75, 0.0), (1.0, 0.0), (2.0, -1.0))):
        p = inputs.problem(m + n + k, ta, tb, m, n, k, alpha, beta, 7, 3, 5, dtype=dtype)
        c0 = np.full_like(p.C0, np.nan) if beta == 0.0 else None   # not read
        got, guard = runner.run(p, C_init=c0)
        gu.assert_close(p, got)
        gu.assert_gap_untouched(p, got, guard, C_init=c0)
    assert runner.h.status() == 0
