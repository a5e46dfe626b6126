"""FP32 triangular solves at the edges of the panel kernel's blocks (32 unknowns), of its CTAs
(16 right-hand sides) and of a panel (512 unknowns), both sides and directions, within the
residual bound of test_gpu_trsm.py; and a zero diagonal entry in a later block, whose special
values must match the oracle's IEEE classes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2302_08417_gb300 import inputs  # noqa: E402
from tests import gpu_util as gu  # noqa: E402
from tests.test_gpu_trsm import residual_check, run, system  # noqa: E402


@pytest.fixture(scope="module")
def runner():
    import __graft_entry__
    __graft_entry__.build()
    return gu.Runner()


@pytest.mark.parametrize("na,nv", [(31, 16), (32, 15), (64, 17), (97, 1), (511, 33), (513, 16)])
def test_block_edges(runner, na, nv):
    rng = np.random.Generator(np.random.PCG64(na + nv))
    for side, uplo, ta, diag in (("L", "L", "N", "N"), ("L", "U", "N", "U"), ("R", "L", "N", "N"),
                                 ("R", "U", "T", "N"), ("L", "L", "T", "N")):
        m, n = (na, nv) if side == "L" else (nv, na)
        lda, ldb = na + 3, m + 1
        A = system(rng, na, lda, uplo, diag, np.float32)
        B0 = inputs.colmajor(rng, m, n, ldb, np.float32)
        X, guard = run(runner, side, uplo, ta, diag, m, n, 1.0, A, lda, B0, ldb)
        assert np.all(np.isnan(guard))
        residual_check(side, uplo, ta, diag, m, n, 1.0, A, lda, B0, ldb, X)


def test_zero_diagonal_in_a_later_block(runner):
    rng = np.random.Generator(np.random.PCG64(7))
    na, nv = 100, 20
    A = system(rng, na, na, "L", "N", np.float32)
    A[70 * na + 70] = 0.0
    B0 = inputs.colmajor(rng, na, nv, na, np.float32)
    X, _ = run(runner, "L", "L", "N", "N", na, nv, 1.0, A, na, B0, na)
    with np.errstate(all="ignore"):
        ref = oracle.trsm_result("L", "L", "N", "N", na, nv, 1.0, A.astype(np.float64), na,
                                 B0.astype(np.float64), na)
    got, want = X.astype(np.float64), ref
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(np.isinf(got), np.isinf(want))
    assert np.array_equal(np.sign(got[np.isinf(got)]), np.sign(want[np.isinf(want)]))
