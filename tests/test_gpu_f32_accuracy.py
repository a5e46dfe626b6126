"""How exact the FP32 tensor-core paths are: sums of one product, which pin every plane product of
the split, and the relative error of whole products against the FP32 core's on the same inputs,
for entries of both signs and of one sign (where the tensor cores' truncation shows)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2302_08417_gb300 import gemmfip as g  # noqa: E402


@pytest.fixture(scope="module")
def multiply():
    """A function (route, A, B) -> A B in FP32 through that path, A and B row-major arrays."""
    import __graft_entry__
    __graft_entry__.build()
    handles = {r: g.Handle() for r in ("core", "tensor", "skinny")}
    for r, h in handles.items():
        assert g.gfip_debug_route(h.h, r) == 0

    def run(route, A, B):
        # the large operand along memory: the kernel for few rows reads it so
        if A.shape[0] >= B.shape[1]:
            dA = torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t()
            dB, tb = torch.from_numpy(np.ascontiguousarray(B.T)).cuda().t(), "N"
        else:
            dA = torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t()
            dB, tb = torch.from_numpy(np.ascontiguousarray(B)).cuda().t(), "T"
        C = g.gemm(dA, dB, transb=tb, handle=handles[route])
        assert handles[route].status() == 0
        return C.cpu().numpy().astype(np.float64)
    return run


@pytest.mark.parametrize("route,m,n,k", [("tensor", 300, 260, 40), ("tensor", 300, 260, 900),
                                         ("tensor", 700, 650, 300), ("tensor", 520, 2000, 1300),
                                         ("skinny", 900, 100, 300), ("skinny", 90, 2000, 1300),
                                         ("skinny", 128, 500, 40)])
def test_sums_of_one_product(multiply, route, m, n, k):
    """A has one entry a row, of 24 significant bits like all of B's, at every k in turn.  The
    product is rounded once (half an ulp, 2^-24); of the nine plane products one, below 2^-32, is
    left out, and seven are added below 2^-7 of the product by additions that may truncate: each
    loses at most 2^-30."""
    rng = np.random.Generator(np.random.PCG64(k))
    mant = lambda *s: (rng.integers(2**23, 2**24, s) * rng.choice([-1.0, 1.0], s)  # noqa: E731
                       * 2.0**-23 * 2.0**rng.integers(-6, 7, s)).astype(np.float32)
    A = np.zeros((m, k), dtype=np.float32)
    at = np.arange(m) * (k / m) if k > m else np.arange(m) % k
    at = at.astype(int)
    A[np.arange(m), at] = mant(m)
    B = mant(k, n)
    want = A[np.arange(m), at].astype(np.float64)[:, None] * B[at].astype(np.float64)
    if route == "skinny" and m < n:   # the large operand's turn to be the sparse one
        A, B, want = B.T.copy(), A.T.copy(), want.T
    err = np.abs(multiply(route, A, B) - want) / np.abs(want)
    assert err.max() <= 2.0**-24 + 2.0**-32 + 7 * 2.0**-30


@pytest.mark.parametrize("sign", ["one", "both"])
@pytest.mark.parametrize("route,m,n", [("tensor", 512, 512), ("tensor", 1030, 1100),
                                       ("skinny", 2000, 100), ("skinny", 64, 8192)])
def test_error_no_larger_than_the_cores(multiply, route, m, n, sign):
    """The 2-norm of the error against 64 bits, k from one accumulation chunk to many and on
    both sides of every change of the chunk's length."""
    for k in (64, 129, 300, 700, 1024, 1025, 1500, 2500, 4096):
        rng = np.random.Generator(np.random.PCG64(m + k))
        A, B = ((rng.random(s) * (1 if sign == "one" else 2) - (sign == "both"))
                .astype(np.float32) for s in ((m, k), (k, n)))
        want = A.astype(np.float64) @ B.astype(np.float64)
        err = {r: np.linalg.norm(multiply(r, A, B) - want) for r in ("core", route)}
        assert err[route] <= err["core"], (k, err[route] / np.linalg.norm(want),
                                           err["core"] / np.linalg.norm(want))


@pytest.mark.parametrize("ea,eb", [(-60, -60), (-65, -65), (-70, -70), (-99, -30), (-90, -50),
                                   (-99, 46)])
@pytest.mark.parametrize("route,m,n,k", [("tensor", 700, 690, 660), ("skinny", 2000, 100, 1499)])
def test_small_products_lose_no_more_than_the_cores(multiply, route, m, n, k, ea, eb):
    """Products near and below FP32's normal range: the largest and the mean error, in absolute
    terms, are at most the core's, whose every multiply-add rounds to a multiple of 2^-149."""
    rng = np.random.Generator(np.random.PCG64(k - ea))
    A, B = ((rng.uniform(0.5, 1.0, s) * rng.choice([-1.0, 1.0], s) * 2.0**e).astype(np.float32)
            for s, e in (((m, k), ea), ((k, n), eb)))
    want = A.astype(np.float64) @ B.astype(np.float64)
    err = {r: np.abs(multiply(r, A, B) - want) for r in ("core", route)}
    assert err[route].max() <= err["core"].max()
    assert err[route].mean() <= err["core"].mean()
