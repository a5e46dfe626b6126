"""TRSM and the workspace's control words: a first call on a workspace leaves its header clear, a
solve captured before any eager call replays without touching the words that later calls keep
there, and a solve that has to clear control words while its stream is capturing is refused with
nothing enqueued."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2302_08417_gb300 import gemmfip as g  # noqa: E402
from paper_2302_08417_gb300 import inputs  # noqa: E402
from tests.test_gpu_trsm import residual_check, system  # noqa: E402

HEADER = 64 * 1024   # the control region's first granule


@pytest.fixture(scope="module")
def dev():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    return torch.device("cuda", 0)


class Solve:
    """op(A) X = B, A lower triangular, na unknowns, 40 right-hand sides, on a fresh workspace
    whose bytes are all set."""

    def __init__(self, dev, na, dtype, uplo="L"):
        rng = np.random.Generator(np.random.PCG64(na))
        self.na, self.nv, self.uplo, self.esz = na, 40, uplo, np.dtype(dtype).itemsize
        self.A = system(rng, na, na, uplo, "N", dtype)
        self.B0 = inputs.colmajor(rng, na, self.nv, na, dtype)
        self.dA, self.dB0 = (torch.from_numpy(x).to(dev) for x in (self.A, self.B0))
        self.dB = self.dB0.clone()
        self.h = g.Handle()
        self.h.bind_stream()
        self.h.ensure_trsm_workspace("L", uplo, "N", "N", na, self.nv, self.esz)
        # room for a later product with more control words
        self.h._set_ws(self.h.workspace.numel() + (64 << 20))
        self.h.workspace.fill_(255)
        torch.cuda.synchronize()

    def call(self):
        return g.gfip_trsm(self.esz, self.h.h, "L", self.uplo, "N", "N", self.na, self.nv, 1.0,
                           self.dA.data_ptr(), self.na, self.dB.data_ptr(), self.na)

    def capture(self):
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.stream(stream):
            self.h.bind_stream(stream)
            with torch.cuda.graph(graph, stream=stream):
                rc = self.call()
                torch.cuda._sleep(1)     # keeps the captured graph non-empty
        self.h.bind_stream()
        torch.cuda.synchronize()
        return rc, graph

    def check(self):
        torch.cuda.synchronize()
        X = self.dB.cpu().numpy()
        residual_check("L", self.uplo, "N", "N", self.na, self.nv, 1.0, self.A, self.na,
                       self.B0, self.na, X)
        return X


@pytest.mark.parametrize("na", [97, 200, 512])
def test_first_call_leaves_the_header_clear(dev, na):
    s = Solve(dev, na, np.float32)
    assert s.call() == 0
    s.check()
    assert not s.h.workspace[:HEADER].any()
    assert s.h.status() == 0


@pytest.mark.parametrize("dtype", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("na", [96, 97, 200, 512])
def test_single_panel_captured_first(dev, dtype, na):
    """One panel needs no control words, so it is captured on a workspace no call has used.  Its
    replays leave the words of the products in between alone: those keep their bits."""
    s = Solve(dev, na, dtype)
    rc, graph = s.capture()
    assert rc == 0, g.error_string(rc)
    graph.replay()
    first = s.check()
    # a product on the kernel that counts launches in the header: an infinity among FP32 operands
    p = inputs.problem(na, "N", "N", 300, 280, 500, 1.0, 0.0, dtype=np.float32)
    p.A[0] = np.inf
    A, B = (torch.from_numpy(x).to(dev) for x in (p.A, p.B))
    C = torch.empty(p.m * p.n, dtype=torch.float32, device=dev)

    def product():
        C.fill_(np.nan)
        assert g._gemm_call("gfip_sgemm", s.h.h, "N", "N", p.m, p.n, p.k, 1.0, A.data_ptr(),
                            p.lda, B.data_ptr(), p.ldb, 0.0, C.data_ptr(), p.ldc) == 0
        torch.cuda.synchronize()
        return C.cpu().numpy().view(np.uint8)

    before = product()
    header = s.h.workspace[:HEADER].clone()
    for _ in range(3):
        s.dB.copy_(s.dB0)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(s.h.workspace[:HEADER], header)
        assert np.array_equal(s.check().view(np.uint8), first.view(np.uint8))
        assert np.array_equal(product(), before)
        header = s.h.workspace[:HEADER].clone()
    s.dB.copy_(s.dB0)
    assert s.call() == 0     # eager, staged by bulk copies: the same operations
    assert np.array_equal(s.check().view(np.uint8), first.view(np.uint8))
    assert s.h.status() == 0


@pytest.mark.parametrize("dtype", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("na,uplo", [(600, "L"), (1040, "U")])
def test_several_panels_refused_before_anything_is_enqueued(dev, dtype, na, uplo):
    s = Solve(dev, na, dtype, uplo)
    rc, graph = s.capture()
    assert rc == g.GFIP_ERR_CAPTURE, g.error_string(rc)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(s.dB, s.dB0)
    assert s.call() == 0
    first = s.check()
    rc, graph = s.capture()
    assert rc == 0
    s.dB.copy_(s.dB0)
    graph.replay()
    assert np.array_equal(s.check().view(np.uint8), first.view(np.uint8))
    assert s.h.status() == 0
