"""FP32 products whose split planes do not fit device memory still run: the handle falls back to
the workspace the FP32 kernel needs.  Memory is made short by a stand-in for the allocation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2302_08417_gb300 import gemmfip as g  # noqa: E402
from paper_2302_08417_gb300 import inputs  # noqa: E402
from tests import gpu_util as gu  # noqa: E402


@pytest.fixture
def short(monkeypatch):
    """A Runner whose handle gets workspaces of fewer than runner.limit bytes only; runner.tries
    lists the sizes asked for."""
    import __graft_entry__
    __graft_entry__.build()
    runner = gu.Runner()
    runner.limit, runner.tries = 1 << 40, []
    set_ws = runner.h._set_ws

    def limited(nbytes):
        runner.tries.append(nbytes)
        if nbytes >= runner.limit:
            raise torch.cuda.OutOfMemoryError("no room")
        set_ws(nbytes)
    monkeypatch.setattr(runner.h, "_set_ws", limited)
    return runner


def sizes(h, query, *args):
    assert g.gfip_set_planes(h, False) == 0
    without = query(h, *args)
    assert g.gfip_set_planes(h, True) == 0
    return without, query(h, *args)


def test_gemm(short):
    # 304 whole tiles, two per SM: the FP32 kernel needs packed panels only, fewer bytes than planes
    p = inputs.problem(3, "N", "T", 2400, 2040, 900, 1.0, 0.5, 3, 1, 2, dtype=np.float32)
    floor, need = sizes(short.h.h, g.gfip_workspace_size, "N", "T", p.m, p.n, p.k, 4)
    assert floor < need
    short.limit = need
    for _ in range(2):     # the second call asks for no memory again
        gu.assert_close(p, short.run(p)[0])
        assert g.gfip_last_launch_info(short.h.h)[0] == 1      # the FP32 kernel's launch
        assert short.h.workspace.numel() == floor and len(short.tries) == 3
    # smaller products have their planes
    q = inputs.problem(4, "N", "T", 2400, 2040, 300, 1.0, 0.5, 3, 1, 2, dtype=np.float32)
    gu.assert_close(q, short.run(q)[0])
    assert g.gfip_last_launch_info(short.h.h)[0] > 1
    # exactly as much as the planes take
    short.limit = need + 1
    short.h._short = None
    gu.assert_close(p, short.run(p)[0])
    assert g.gfip_last_launch_info(short.h.h)[0] > 1 and short.h.workspace.numel() == need
    # too little for any path
    short.limit = 1000
    r = inputs.problem(5, "N", "T", 2500, 2400, 900, 1.0, 0.5, 3, 1, 2, dtype=np.float32)
    with pytest.raises(torch.cuda.OutOfMemoryError):
        short.run(r)
    short.limit = 1 << 40
    gu.assert_close(r, short.run(r)[0])
    assert short.h.status() == 0


@pytest.mark.parametrize("ensure,query,args", [
    ("ensure_syrk_workspace", g.gfip_syrk_workspace_size, ("L", "N", 4000, 6000, 4)),
    ("ensure_trmm_workspace", g.gfip_trmm_workspace_size, ("L", "L", "N", "N", 8000, 6000, 4)),
    ("ensure_trsm_workspace", g.gfip_trsm_workspace_size, ("L", "L", "N", "N", 60000, 40000, 4))])
def test_other_routines(short, ensure, query, args):
    floor, need = sizes(short.h.h, query, *args)
    assert floor < need
    short.limit = need
    getattr(short.h, ensure)(*args)
    getattr(short.h, ensure)(*args)
    assert short.h.workspace.numel() == floor and len(short.tries) == 3
