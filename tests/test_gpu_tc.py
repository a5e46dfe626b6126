"""The tensor-core tile core (csrc/gfip_tc.cuh) where it can go wrong: tile and k-block
remainders, accumulation-chunk boundaries and every digit count of the emulated FP64 GEMM,
against the oracle with the splitting bound of test_gpu_ozaki.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2302_08417_gb300 import inputs  # noqa: E402
from tests import gpu_util as gu  # noqa: E402
from tests.test_gpu_ozaki import run_ozaki, split_bound  # noqa: E402


@pytest.fixture(scope="module")
def runner():
    import __graft_entry__
    __graft_entry__.build()
    return gu.Runner()


@pytest.mark.parametrize("slices", range(1, 11))
def test_digit_counts_and_chunk_edges(runner, slices):
    """k one block and a bit past the shortest accumulation chunk (16384 / slices terms, in
    32-wide blocks), so every group of classes has a full and a ragged chunk."""
    k = 16384 // slices // 32 * 32 + 33 if slices > 2 else 190
    for ta, tb, m, n in (("N", "T", 129, 257), ("T", "N", 250, 70)):
        p = inputs.problem(300 + slices, ta, tb, m, n, k, -1.25, 0.5, 7, 3, 5)
        got, guard = run_ozaki(runner, p, slices)
        ref, _ = gu.reference(p)
        err = np.abs(inputs.as_matrix(got, m, n, p.ldc) - inputs.as_matrix(ref, m, n, p.ldc))
        assert np.all(err <= split_bound(p, slices)), (slices, ta, tb, m, n, k)
        gu.assert_gap_untouched(p, got, guard)
        assert runner.h.status() == 0
