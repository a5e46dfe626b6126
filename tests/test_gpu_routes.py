"""Every path a product can take, whatever the size: the routines' own tests (variants, policies
and packers bit for bit, special values, graph replay, stale workspaces, ragged edges, triangles
and masks), sent through one path by the test hook gfip_debug_route.  By size alone these shapes
would all take the small kernels or the tensor cores.  And FP32 operands outside the range of the
BF16 planes, whose product must have the bits of the core the tensor-core paths fall back to."""
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
from tests import test_gpu_graph as graph  # noqa: E402
from tests import test_gpu_parity as parity  # noqa: E402
from tests import test_gpu_syrk as syrk  # noqa: E402
from tests import test_gpu_trmm as trmm  # noqa: E402
from tests import test_gpu_trsm as trsm  # noqa: E402

F64, F32 = np.float64, np.float32
BOTH = [("core", F64), ("core", F32), ("small", F64), ("small", F32), ("tensor", F32),
        ("skinny", F32)]
MASKED = BOTH[:-1]   # the kernel for few rows takes dense operands only


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture
def routed(monkeypatch):
    """A function route -> Runner; handles made afterwards in the test take the route as well."""
    class Routed(g.Handle):
        route = "auto"

        def __init__(self, *args):
            super().__init__(*args)
            assert g.gfip_debug_route(self.h, Routed.route) == 0

    monkeypatch.setattr(g, "Handle", Routed)

    def runner(route):
        Routed.route = route
        return gu.Runner()
    return runner


def ids(cases):
    return [f"{r}-{'f64' if d is F64 else 'f32'}" for r, d in cases]


@pytest.mark.parametrize("route,dtype", BOTH, ids=ids(BOTH))
def test_gemm_ragged(routed, route, dtype):
    runner = routed(route)
    for variant in gu.VARIANTS if route == "core" else ("fused",):
        parity.test_medium_ragged_all_trans(runner, dtype, variant)
    parity.test_integer_inputs_bit_exact(runner, dtype)
    assert runner.h.status() == 0


@pytest.mark.parametrize("route", ["core", "small", "tensor", "skinny"])
def test_gemm_special_values(routed, route):
    for variant in gu.VARIANTS:
        parity.test_blas_special_values(routed(route), variant)


@pytest.mark.parametrize("dtype", [F64, F32], ids=["f64", "f32"])
def test_core_policies_and_packers(routed, dtype):
    parity.test_variants_and_policies_bitwise_identical(routed("core"), dtype)
    parity.test_shared_packer_sizes_and_codes(routed("core"), dtype)


def test_core_stale_workspace_and_repeats(routed):
    runner = routed("core")
    parity.test_workspace_reuse_across_shapes_and_garbage(runner)
    parity.test_repeated_calls_identical(runner)
    graph.test_first_call_under_capture_is_refused_then_capture_works(runner)


@pytest.mark.parametrize("variant", ["fused", "pack_then_compute"])
@pytest.mark.parametrize("case", range(len(graph.CASES)))
def test_core_graph_replay(routed, case, variant):
    graph.test_replayed_graph_matches_eager_and_oracle(routed("core"), *graph.CASES[case], variant)


@pytest.mark.parametrize("route,dtype", MASKED, ids=ids(MASKED))
def test_syrk(routed, route, dtype):
    runner = routed(route)
    for uplo, trans in itertools.product("LU", "NT"):
        syrk.test_ragged_and_policies_bitwise(runner, dtype, uplo, trans)
    syrk.test_integer_bit_exact(runner, dtype)


@pytest.mark.parametrize("route,dtype", MASKED, ids=ids(MASKED))
def test_trmm(routed, route, dtype):
    runner = routed(route)
    for combo in trmm.COMBOS:
        trmm.test_ragged_and_policies_bitwise(runner, dtype, *combo)
    trmm.test_integer_bit_exact(runner, dtype)


@pytest.mark.parametrize("route,dtype", [("core", F64), ("core", F32), ("tensor", F32)],
                         ids=["core-f64", "core-f32", "tensor-f32"])
def test_triangles_over_several_rounds(routed, route, dtype):
    """More tiles than SMs, ragged: the tensor cores' triangular operands take their longest tiles
    first and every other round backwards, the core packs panels that later rounds read."""
    runner = routed(route)
    rng = np.random.Generator(np.random.PCG64(31))
    u = inputs.unit_roundoff(dtype)

    def close(got, X, Y, C, alpha, beta, part=slice(None)):
        # numpy's FP64 products and the result are each within (k + 2) u of the exact one
        want = alpha * (X @ Y) + beta * C
        bound = abs(alpha) * (np.abs(X) @ np.abs(Y)) + abs(beta) * np.abs(C)
        assert np.all(np.abs(got - want)[part] <= (2 * (X.shape[1] + 2) * u * bound)[part])

    for side, uplo, ta, diag in trmm.COMBOS:
        m, n = (1650, 1910) if side == "L" else (1910, 1650)
        A = trmm.poisoned(rng, 1650, 1653, uplo, diag, dtype)
        B0 = inputs.colmajor(rng, m, n, m + 1, dtype)
        got, guard = trmm.run(runner, side, uplo, ta, diag, m, n, 1.25, A, 1653, B0, m + 1)
        assert np.all(np.isnan(guard))
        D = trmm.dense_op(A.astype(np.float64), 1653, 1650, uplo, ta, diag)
        B = inputs.as_matrix(B0.astype(np.float64), m, n, m + 1)
        close(inputs.as_matrix(got.astype(np.float64), m, n, m + 1),
              *((D, B) if side == "L" else (B, D)), np.zeros((m, n)), 1.25, 0.0)
    for uplo, trans in itertools.product("LU", "NT"):
        n, k = 2500, 333
        A, lda, C0, ldc = syrk.make(17, uplo, trans, n, k, 7, dtype)
        got, guard = syrk.run(runner, uplo, trans, n, k, 0.75, A, lda, 0.5, C0, ldc)
        assert np.all(np.isnan(guard))
        X = inputs.as_matrix(A.astype(np.float64), *((n, k) if trans == "N" else (k, n)), lda)
        X = X if trans == "N" else X.T
        C = inputs.as_matrix(C0.astype(np.float64), n, n, ldc)
        G = inputs.as_matrix(got.astype(np.float64), n, n, ldc)
        tri = np.tri(n, dtype=bool) if uplo == "L" else np.tri(n, dtype=bool).T
        close(np.where(tri, G, 0), X, X.T, np.where(tri, C, 0), 0.75, 0.5, tri)
        assert np.array_equal(G[~tri], C[~tri], equal_nan=True)   # the other triangle


@pytest.mark.parametrize("route,dtype", MASKED, ids=ids(MASKED))
def test_trsm(routed, route, dtype):
    runner = routed(route)
    for combo in (("L", "L", "N", "N"), ("L", "U", "T", "U"), ("R", "U", "N", "N"),
                  ("R", "L", "T", "U")):
        trsm.test_several_panels(runner, dtype, *combo)


def test_the_hook_reaches_each_path(routed):
    """Launches per call: the split, tile core and gated core; one more for few rows; grids."""
    p = inputs.problem(1, "N", "T", 500, 120, 300, 1.0, 0.0, dtype=F32)
    seen = {}
    for route in ("core", "small", "tensor", "skinny"):
        runner = routed(route)
        runner.run(p)
        seen[route] = g.gfip_last_launch_info(runner.h.h)
    assert [seen[r][0] for r in ("core", "small", "tensor", "skinny")] == [1, 1, 3, 4]
    assert seen["small"][1] % (16 * 4) == 0 and seen["core"][1] != seen["small"][1]


# an entry of A that the planes cannot hold: too large, too small, not a number
@pytest.mark.parametrize("value", [1e30, 1e-42, np.nan])
def test_outside_the_planes_range_equals_the_core(routed, value):
    def bits(x):
        return x.view(np.uint8)

    core, tensor, skinny = routed("core"), routed("tensor"), routed("skinny")
    for variant, policy, packer in itertools.product(
            gu.VARIANTS, (g.GFIP_PACK_AUTO, g.GFIP_PACK_BOTH),
            (g.GFIP_PACKER_LINE, g.GFIP_PACKER_SHARED)):
        p = inputs.problem(5, "N", "T", 390, 260, 300, -1.5, 0.5, 7, 0, 7, dtype=F32)
        p.A[100 + 40 * p.lda] = value
        want, _ = core.run(p, variant, policy=policy, packer=packer)
        got, _ = tensor.run(p, variant, policy=policy, packer=packer)
        assert np.array_equal(bits(got), bits(want)), (variant, policy, packer)
    for m, n in ((390, 100), (100, 390)):
        p = inputs.problem(6, "N", "T", m, n, 300, -1.5, 0.5, 7, 0, 7, dtype=F32)
        p.A[50 + 40 * p.lda] = value
        assert np.array_equal(bits(skinny.run(p)[0]), bits(core.run(p)[0]))
    for uplo, trans in itertools.product("LU", "NT"):
        A, lda, C0, ldc = syrk.make(9, uplo, trans, 300, 200, 7, F32)
        A[150 + 60 * lda] = value
        args = (uplo, trans, 300, 200, 0.75, A, lda, 0.5, C0, ldc)
        assert np.array_equal(bits(syrk.run(tensor, *args)[0]), bits(syrk.run(core, *args)[0]))
    rng = np.random.Generator(np.random.PCG64(12))
    for side, uplo, ta, diag in trmm.COMBOS:
        m, n = (300, 200) if side == "L" else (200, 300)
        A = trmm.poisoned(rng, 300, 303, uplo, diag, F32)
        A[(150 + 60 * 303) if uplo == "L" else (60 + 150 * 303)] = value   # in the kept triangle
        B0 = inputs.colmajor(rng, m, n, m + 5, F32)
        args = (side, uplo, ta, diag, m, n, 1.25, A, 303, B0, m + 5)
        assert np.array_equal(bits(trmm.run(tensor, *args)[0]), bits(trmm.run(core, *args)[0]))
    # the gate is open again: the next product is the tensor cores'
    p = inputs.problem(7, "N", "N", 300, 280, 260, 1.0, 0.5, 7, 7, 7, dtype=F32)
    gu.assert_close(p, tensor.run(p)[0])
    assert core.h.status() == tensor.h.status() == skinny.h.status() == 0


@pytest.mark.parametrize("at", [0, 700, 3499, "many", "small operand"])
def test_few_rows_stop_at_an_element_outside(routed, at):
    """The kernel for few rows stops where its CTAs next look (units of several looks, more units
    than CTAs): the core's bits, C scaled once, no status, and the next call is right."""
    core, skinny = routed("core"), routed("skinny")
    for m, n, k in ((2000, 64, 3500), (25000, 16, 3500)):
        p = inputs.problem(3, "N", "N", m, n, k, 1.0, 0.5, 0, 0, 0, dtype=F32)
        clean_A, clean_B = p.A.copy(), p.B.copy()
        if at == "small operand":
            p.B[5] = 1e-42
        elif at == "many":
            p.A[::1001] = 1e-42
        else:
            p.A[m // 2 + at * m] = 1e-42
        got, _ = skinny.run(p)
        assert np.array_equal(got.view(np.uint8), core.run(p)[0].view(np.uint8))
        p.A, p.B = clean_A, clean_B
        gu.assert_close(p, skinny.run(p)[0])
        assert skinny.h.status() == 0
