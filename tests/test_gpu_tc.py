"""The tensor-core tile core (csrc/gfip_tc.cuh) where it can go wrong: tile and k-block
remainders, accumulation-chunk boundaries, every digit count, split k, and FP32 operands at the
edges of the range the BF16 planes hold.  Against the oracle, with the bounds of the routines
these products belong to: 2 max(k, 2) u (|alpha||op(A)||op(B)| + |beta||C0|) in FP32, the
splitting bound of test_gpu_ozaki.py for the emulated FP64 GEMM."""
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


@pytest.mark.parametrize("m,n,k", [(700, 650, 600), (2000, 1500, 16), (1030, 1100, 289),
                                   (900, 700, 1024), (900, 700, 1025),
                                   (130, 8000, 255), (2100, 129, 1025), (300, 290, 7001)])
def test_fp32_shapes(runner, m, n, k):
    for ta, tb in (("N", "N"), ("T", "T")):
        p = inputs.problem(m + n + k, ta, tb, m, n, k, -0.75, 0.5, 7, 3, 5, dtype=np.float32)
        got, guard = runner.run(p)
        gu.assert_close(p, got)
        gu.assert_gap_untouched(p, got, guard)
        q = inputs.problem(m + n + k, ta, tb, m, n, k, 1.0, 0.0, 1, 0, 2, dtype=np.float32)
        got, _ = runner.run(q, C_init=np.full_like(q.C0, np.nan))   # beta == 0: C not read
        gu.assert_close(q, got)
    assert runner.h.status() == 0


SKINNY = [("N", "T", 64, 8200, 1500), ("T", "T", 120, 9001, 1027), ("N", "N", 8200, 100, 1499),
          ("N", "T", 9000, 128, 1090)]


@pytest.mark.parametrize("ta,tb,m,n,k", SKINNY)
def test_fp32_skinny(runner, ta, tb, m, n, k):
    """At most 128 rows or columns: the large operand is split on its way to the MMA."""
    p = inputs.problem(m + n + k, ta, tb, m, n, k, -0.75, 0.5, 7, 3, 5, dtype=np.float32)
    got, guard = runner.run(p)
    gu.assert_close(p, got)
    gu.assert_gap_untouched(p, got, guard)
    # an element outside the split's range in the large operand: the whole product is the FFMA
    # kernel's, beta * C applied once
    q = inputs.problem(m + n + k, ta, tb, m, n, k, 1.0, 0.5, 1, 1, 1, dtype=np.float32)
    big, ld = (q.A, q.lda) if n <= m else (q.B, q.ldb)
    big[40 + 900 * ld] = 1e25
    got, _ = runner.run(q)
    gu.assert_close(q, got)
    assert runner.h.status() == 0


@pytest.mark.parametrize("ea,eb", [(-99, 55), (-101, 30), (-115, 115), (-60, -60), (20, 56)])
def test_fp32_magnitudes(runner, ea, eb):
    """Operands whose low planes are still normal BF16 numbers, and ones that would leave the
    range: the error bound holds on both sides of the line."""
    p = inputs.problem(500 + ea, "N", "T", 700, 680, 660, 1.0, 0.0, 3, 1, 2, dtype=np.float32)
    # magnitudes in [1/2, 1) times the power of two
    p.A, p.B = (np.ldexp(np.copysign(0.5 + np.abs(x) / 2, x), e).astype(np.float32)
                for x, e in ((p.A, ea), (p.B, eb)))
    got, _ = runner.run(p)
    gu.assert_close(p, got)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38, 1e-42])
def test_fp32_special_operands(runner, value):
    """One infinity, NaN, near-overflow or subnormal entry of A: its row of C has the oracle's
    IEEE classes, every other row is within the bound; and the next call is unaffected."""
    p = inputs.problem(77, "N", "N", 700, 680, 660, 1.0, 0.0, 0, 0, 0, dtype=np.float32)
    clean = p.A.copy()
    p.A[5 + 17 * p.lda] = value
    got, _ = runner.run(p)
    ref, ab = gu.reference(p)
    g = inputs.as_matrix(got.astype(np.float64), p.m, p.n, p.ldc)
    with np.errstate(over="ignore"):
        r = inputs.as_matrix(ref, p.m, p.n, p.ldc).astype(np.float32).astype(np.float64)
    if not np.isfinite(value):
        assert np.array_equal(np.isnan(g[5]), np.isnan(r[5]))
        assert np.array_equal(np.sign(g[5][np.isinf(g[5])]), np.sign(r[5][np.isinf(r[5])]))
        assert np.array_equal(np.isinf(g[5]), np.isinf(r[5]))
    rows = np.arange(p.m) != 5 if not np.isfinite(value) else np.ones(p.m, dtype=bool)
    tol = gu.tolerance(p, ab)
    err = np.abs(g[rows] - r[rows])
    assert np.all(err <= tol[rows] + np.spacing(np.abs(r[rows]).astype(np.float32)))
    p.A = clean
    got, _ = runner.run(p)
    gu.assert_close(p, got)
    assert runner.h.status() == 0
