"""The work that is measured: calls of the library's public entry points over the range they
are used in, from one 16 x 16 product to products of a few thousand rows, in both element
types, with every operand order, aligned and odd leading dimensions.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes the
inputs a user has in hand, ``run`` is one pass, ``work`` what a pass cannot do without and
``exact`` the same result in 64 bits by plain torch.
"""
import math
import random

import torch

from paper_2302_08417_gb300 import autograd, gemmfip, grouped

DTYPES = {"f32": torch.float32, "f64": torch.float64}
# cost limits of a drawn case (multiply-adds of the largest listed case of each kind)
MAX_MADDS = {"f32": 4096 ** 3, "f64": 2900 * 3100 * 3000, "ozaki": 4096 ** 3,
             "trsm": 2048 ** 3, "trmm": 2048 ** 3, "syrk": 2048 ** 3}


def listed():
    return [
        # the smallest call of the size spectrum: latency, launches and host path only
        dict(name="dgemm_16", kind="gemm", dtype="f64", ta="N", tb="N", m=16, n=16, k=16,
             pad=7, alpha=1.0, beta=0.5),
        # the 256^3 FP64 workload with tight leading dimensions
        dict(name="dgemm_256", kind="gemm", dtype="f64", ta="N", tb="N", m=256, n=256, k=256,
             pad=0, alpha=1.0, beta=0.5),
        # an ordinary small FP32 product of ragged size, A stored transposed
        dict(name="sgemm_ragged_512", kind="gemm", dtype="f32", ta="T", tb="N", m=517, n=500,
             k=509, pad=7, alpha=1.0, beta=0.5),
        # a large square FP32 product with odd leading dimensions
        dict(name="sgemm_4096", kind="gemm", dtype="f32", ta="N", tb="N", m=4096, n=4096,
             k=4096, pad=7, alpha=1.0, beta=0.5),
        # a skinny product: few rows against a large matrix, C only written
        dict(name="sgemm_skinny", kind="gemm", dtype="f32", ta="N", tb="T", m=64, n=8192,
             k=8192, pad=7, alpha=1.0, beta=0.0),
        # a large ragged FP64 product, both operands stored transposed
        dict(name="dgemm_3000", kind="gemm", dtype="f64", ta="T", tb="T", m=2900, n=3100,
             k=3000, pad=7, alpha=1.0, beta=0.5),
        # the symmetric rank-k update, one triangle
        dict(name="ssyrk_2048", kind="syrk", dtype="f32", uplo="L", ta="N", n=2048, k=2048,
             pad=7, alpha=1.0, beta=0.5),
        # triangular product in place
        dict(name="strmm_2048", kind="trmm", dtype="f32", side="L", uplo="L", ta="N", diag="N",
             m=2048, n=2048, pad=7, alpha=1.0),
        # triangular solve in place, many right-hand sides
        dict(name="strsm_2048", kind="trsm", dtype="f32", side="L", uplo="L", ta="N", diag="N",
             m=2048, n=2048, pad=7, alpha=1.0),
        # FP64 emulated from digit products on the tensor cores, 7 digits
        dict(name="ozaki_4096_s7", kind="ozaki", dtype="f64", ta="N", tb="N", m=4096, n=4096,
             k=4096, slices=7, pad=7, alpha=1.0, beta=0.5),
        # a batch of uneven small products in one grouped call
        dict(name="sgrouped_4096", kind="grouped", dtype="f32", count=4096, lo=4, hi=256,
             sizes_seed=1, alpha=1.0, beta=0.5),
        # a training step's products: forward and both gradients
        dict(name="sgemm_fwd_bwd", kind="autograd", dtype="f32", ta="N", tb="N", m=4096,
             n=4096, k=1024, alpha=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "syrk", "trmm", "trsm", "ozaki", "grouped",
                       "autograd"])
    dtype = rng.choice(["f32", "f64"])
    trans = lambda: rng.choice("NT")  # noqa: E731
    pad = rng.choice([0, 1, 4, 7])
    beta = rng.choice([0.0, 0.5])
    while True:
        m, n, k = (_log_int(rng, 16, 8192) for _ in range(3))
        if kind == "gemm" and m * n * k <= MAX_MADDS[dtype]:
            return dict(kind="gemm", dtype=dtype, ta=trans(), tb=trans(), m=m, n=n, k=k, pad=pad,
                        alpha=rng.choice([1.0, -0.75]), beta=beta)
        if kind == "autograd" and 3 * m * n * k <= MAX_MADDS[dtype]:
            return dict(kind="autograd", dtype=dtype, ta=trans(), tb=trans(), m=m, n=n, k=k,
                        alpha=1.0)
        if kind == "syrk" and n * n * k <= MAX_MADDS["syrk"]:
            return dict(kind="syrk", dtype=dtype, uplo=rng.choice("LU"), ta=trans(), n=n, k=k,
                        pad=pad, alpha=1.0, beta=beta)
        if kind in ("trmm", "trsm"):
            side = rng.choice("LR")
            na = m if side == "L" else n
            if na <= 4096 and m * n * na <= MAX_MADDS[kind]:
                return dict(kind=kind, dtype=dtype, side=side, uplo=rng.choice("LU"), ta=trans(),
                            diag=rng.choice("NU"), m=m, n=n, pad=pad, alpha=1.0)
        if kind == "ozaki" and min(m, n, k) >= 128 and m * n * k <= MAX_MADDS["ozaki"]:
            return dict(kind="ozaki", dtype="f64", ta=trans(), tb=trans(), m=m, n=n, k=k,
                        slices=rng.randint(3, 9), pad=pad, alpha=1.0, beta=beta)
        if kind == "grouped":
            return dict(kind="grouped", dtype=dtype, count=_log_int(rng, 64, 4096), lo=4,
                        hi=rng.choice([64, 128, 256]), sizes_seed=rng.randrange(1 << 30),
                        alpha=1.0, beta=beta)


# ---- inputs -----------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _colmajor(gen, rows, cols, ld, dtype):
    """rows x cols column-major view of leading dimension ld, entries uniform in [-1, 1]."""
    buf = torch.rand((cols, ld), generator=gen, device="cuda", dtype=dtype).mul_(2).sub_(1)
    return buf.t()[:rows, :]


def _shape(trans, rows, cols):
    return (rows, cols) if trans == "N" else (cols, rows)


def _grouped_sizes(case):
    rng = random.Random(case["sizes_seed"])
    out = []
    for _ in range(case["count"]):
        m, n, k = (_log_int(rng, case["lo"], case["hi"]) for _ in range(3))
        ta, tb = rng.choice("NT"), rng.choice("NT")
        out.append((m, n, k, ta, tb, [rng.randint(0, 7) for _ in range(3)]))
    return out


def _flat_views(gen, shapes, dtype):
    """One flat buffer of uniform [-1, 1] entries and the column-major views of (rows, cols, ld)."""
    total = sum(ld * cols for _, cols, ld in shapes)
    flat = torch.rand(total, generator=gen, device="cuda", dtype=dtype).mul_(2).sub_(1)
    views, off = [], 0
    for rows, cols, ld in shapes:
        views.append(flat.as_strided((rows, cols), (1, ld), off))
        off += ld * cols
    return flat, views


def _grouped_shapes(sizes):
    a = [_shape(ta, m, k) for m, n, k, ta, tb, p in sizes]
    b = [_shape(tb, k, n) for m, n, k, ta, tb, p in sizes]
    pads = [s[5] for s in sizes]
    A = [(r, c, r + p[0]) for (r, c), p in zip(a, pads)]
    B = [(r, c, r + p[1]) for (r, c), p in zip(b, pads)]
    C = [(s[0], s[1], s[0] + p[2]) for s, p in zip(sizes, pads)]
    return A, B, C


def _grouped_plan(batch):
    """A plan by size: small warp tiles for small problems, 32 x 32 from 65 rows or columns on."""
    tiles = (gemmfip.GFIP_GROUP_TILE_TINY, gemmfip.GFIP_GROUP_TILE_TINY,
             gemmfip.GFIP_GROUP_TILE_SMALL, gemmfip.GFIP_GROUP_TILE_DEFAULT,
             gemmfip.GFIP_GROUP_TILE_DEFAULT)
    choice = {b: (tiles[b[0]], 1) for b in {grouped.bucket_of(*s) for s in batch.sizes}}
    return grouped.Plan.from_buckets(batch, choice)


def _operands(case, seed):
    """The tensors of a case, by name, from the seed alone."""
    gen, dtype, kind = _gen(seed), DTYPES[case["dtype"]], case["kind"]
    if kind in ("gemm", "ozaki"):
        m, n, k, pad = case["m"], case["n"], case["k"], case["pad"]
        ra, ca = _shape(case["ta"], m, k)
        rb, cb = _shape(case["tb"], k, n)
        return dict(A=_colmajor(gen, ra, ca, ra + pad, dtype),
                    B=_colmajor(gen, rb, cb, rb + pad, dtype),
                    C=_colmajor(gen, m, n, m + pad, dtype))
    if kind == "autograd":
        m, n, k = case["m"], case["n"], case["k"]
        ra, ca = _shape(case["ta"], m, k)
        rb, cb = _shape(case["tb"], k, n)
        return dict(A=_colmajor(gen, ra, ca, ra, dtype), B=_colmajor(gen, rb, cb, rb, dtype),
                    dC=_colmajor(gen, m, n, m, dtype))
    if kind == "syrk":
        n, k, pad = case["n"], case["k"], case["pad"]
        ra, ca = _shape(case["ta"], n, k)
        return dict(A=_colmajor(gen, ra, ca, ra + pad, dtype),
                    C=_colmajor(gen, n, n, n + pad, dtype))
    if kind in ("trmm", "trsm"):
        m, n, pad = case["m"], case["n"], case["pad"]
        na = m if case["side"] == "L" else n
        A = _colmajor(gen, na, na, na + pad, dtype)
        if kind == "trsm":    # well conditioned: small off-diagonal entries, diagonal near 2
            A.div_(na)
            A.diagonal().mul_(na * 0.25).add_(2.0)
        return dict(A=A, B=_colmajor(gen, m, n, m + pad, dtype))
    sizes = _grouped_sizes(case)
    sa, sb, sc = _grouped_shapes(sizes)
    fa, A = _flat_views(gen, sa, dtype)
    fb, B = _flat_views(gen, sb, dtype)
    fc, C = _flat_views(gen, sc, dtype)
    return dict(A=A, B=B, C=C, flat=fc, sizes=sizes)


def prepare(case, seed):
    s = _operands(case, seed)
    s["case"] = case
    kind = case["kind"]
    esz = 8 if case["dtype"] == "f64" else 4
    if kind == "autograd":
        s["A"] = s["A"].requires_grad_()
        s["B"] = s["B"].requires_grad_()
    if kind in ("trmm", "trsm", "ozaki"):     # entry points that take a handle
        h = gemmfip.Handle()
        h.bind_stream()
        if kind == "ozaki":
            h.ensure_ozaki_workspace(case["m"], case["n"], case["k"], case["slices"])
        else:
            ensure = h.ensure_trmm_workspace if kind == "trmm" else h.ensure_trsm_workspace
            ensure(case["side"], case["uplo"], case["ta"], case["diag"], case["m"], case["n"],
                   esz)
            s["X"] = torch.empty_strided(s["B"].shape, s["B"].stride(), dtype=s["B"].dtype,
                                         device="cuda")
        s["handle"] = h
    if kind == "grouped":
        sizes = s["sizes"]
        count = len(sizes)
        s["batch"] = grouped.Batch([x[3] for x in sizes], [x[4] for x in sizes], s["A"], s["B"],
                                   s["C"], [case["alpha"]] * count, [case["beta"]] * count)
        s["plan"] = _grouped_plan(s["batch"])
    return s


# ---- one pass ----------------------------------------------------------------------------------

def _ok(rc, name):
    if rc != gemmfip.GFIP_OK:
        raise gemmfip.GemmError(rc, name)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "gemm":
        return gemmfip.gemm(s["A"], s["B"], s["C"], case["alpha"], case["beta"], case["ta"],
                            case["tb"])
    if kind == "syrk":
        return gemmfip.syrk(s["A"], s["C"], case["alpha"], case["beta"], case["uplo"],
                            case["ta"])
    if kind == "autograd":
        C = autograd.gemm(s["A"], s["B"], case["ta"], case["tb"], case["alpha"])
        dA, dB = torch.autograd.grad(C, (s["A"], s["B"]), s["dC"])
        return C.detach(), dA, dB
    esz = 8 if case["dtype"] == "f64" else 4
    A, B = s["A"], s["B"]
    if kind == "ozaki":
        C = s["C"]
        _ok(gemmfip.gfip_dgemm_ozaki(
            s["handle"].h, case["ta"], case["tb"], case["m"], case["n"], case["k"],
            case["alpha"], A.data_ptr(), A.stride(1), B.data_ptr(), B.stride(1), case["beta"],
            C.data_ptr(), C.stride(1), case["slices"]), "gfip_dgemm_ozaki")
        return C
    if kind in ("trmm", "trsm"):
        X = s["X"]
        X.copy_(B)        # the operation works in place: every pass has its right-hand sides
        call = gemmfip.gfip_trmm if kind == "trmm" else gemmfip.gfip_trsm
        _ok(call(esz, s["handle"].h, case["side"], case["uplo"], case["ta"], case["diag"],
                 case["m"], case["n"], case["alpha"], A.data_ptr(), A.stride(1), X.data_ptr(),
                 X.stride(1)), "gfip_" + kind)
        return X
    grouped.run(s["batch"], s["plan"])
    return s["flat"]


# ---- what a pass cannot do without --------------------------------------------------------------

def work(case):
    es = 8 if case["dtype"] == "f64" else 4
    kind = case["kind"]
    if kind in ("gemm", "ozaki"):
        m, n, k = case["m"], case["n"], case["k"]
        c = 2 if case["beta"] != 0.0 else 1
        return {"bytes": es * (m * k + k * n + c * m * n), "flops": 2 * m * n * k}
    if kind == "autograd":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": es * (2 * m * k + 2 * k * n + 2 * m * n), "flops": 6 * m * n * k}
    if kind == "syrk":
        n, k = case["n"], case["k"]
        c = 2 if case["beta"] != 0.0 else 1
        tri = n * (n + 1) // 2
        return {"bytes": es * (n * k + c * tri), "flops": 2 * tri * k}
    if kind in ("trmm", "trsm"):
        m, n = case["m"], case["n"]
        na, nb = (m, n) if case["side"] == "L" else (n, m)
        return {"bytes": es * (na * (na + 1) // 2 + 2 * m * n), "flops": na * na * nb}
    c = 2 if case["beta"] != 0.0 else 1
    sizes = _grouped_sizes(case)
    return {"bytes": es * sum(m * k + k * n + c * m * n for m, n, k, *_ in sizes),
            "flops": sum(2 * m * n * k for m, n, k, *_ in sizes)}


# ---- the same results in 64 bits -----------------------------------------------------------------

def _op(x, trans):
    return x if trans == "N" else x.t()


def _triangle(A, case):
    A = torch.tril(A) if case["uplo"] == "L" else torch.triu(A)
    if case["diag"] == "U":
        A = A - torch.diag(A.diagonal()) + torch.eye(A.shape[0], dtype=A.dtype, device=A.device)
    return _op(A, case["ta"])


def exact(case, seed):
    s = _operands(case, seed)
    kind = case["kind"]
    if kind == "grouped":
        C = s["flat"].double()
        off = 0
        for a, b, (m, n, k, ta, tb, p) in zip(s["A"], s["B"], s["sizes"]):
            ld = m + p[2]
            c = C.as_strided((m, n), (1, ld), off)
            off += ld * n
            ab = _op(a.double(), ta) @ _op(b.double(), tb)
            c.copy_(case["alpha"] * ab + (case["beta"] * c if case["beta"] != 0.0 else 0.0))
        return C
    A = s["A"].double()
    if kind in ("gemm", "ozaki"):
        r = case["alpha"] * (_op(A, case["ta"]) @ _op(s["B"].double(), case["tb"]))
        return r + case["beta"] * s["C"].double() if case["beta"] != 0.0 else r
    if kind == "autograd":
        B, dC = s["B"].double(), s["dC"].double()
        opA, opB = _op(A, case["ta"]), _op(B, case["tb"])
        dA, dB = dC @ opB.t(), opA.t() @ dC
        return (case["alpha"] * (opA @ opB), case["alpha"] * _op(dA, case["ta"]),
                case["alpha"] * _op(dB, case["tb"]))
    if kind == "syrk":
        opA = _op(A, case["ta"])
        C = s["C"].double()
        r = case["alpha"] * (opA @ opA.t()) + case["beta"] * C
        tri = torch.tril if case["uplo"] == "L" else torch.triu
        keep = tri(torch.ones_like(C, dtype=torch.bool))
        return torch.where(keep, r, C)
    T, B = _triangle(A, case), s["B"].double()
    if kind == "trmm":
        return case["alpha"] * (T @ B if case["side"] == "L" else B @ T)
    lower = (case["uplo"] == "L") == (case["ta"] == "N")
    return torch.linalg.solve_triangular(T, case["alpha"] * B, upper=not lower,
                                         left=case["side"] == "L")
