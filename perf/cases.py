"""The calls a user of gbgemm makes, as cases that can be timed and checked.

Every case goes through the public binding (``gbgemm.Handle``,
``gbgemm.GroupedPlan``) with device buffers the caller owns.  Matrices are
column-major: a rows x cols matrix with leading dimension ld is a (cols, ld)
tensor, and its logical form is ``buf[:, :rows].T``.
"""

import math

import torch

from paper_1608_05265_gb300 import gbgemm


def listed():
    return [
        # The smallest call: one 256^3 product inside a larger program, where
        # the launches and the latency of one pass decide.
        {"name": "sgemm_256", "kind": "sgemm", "ta": "N", "tb": "N", "m": 256, "n": 256, "k": 256, "pad": 0,
         "alpha": 1.0, "beta": 0.5, "dist": "uniform"},
        # A short inner dimension (below the tensor path's k), odd leading
        # dimensions: the update with a narrow panel.
        {"name": "sgemm_short_k", "kind": "sgemm", "ta": "N", "tb": "T", "m": 2048, "n": 1777, "k": 64, "pad": 1,
         "alpha": -1.0, "beta": 1.0, "dist": "uniform"},
        # Ordinary square products of the sweep, padded by 8: the smallest,
        # the middle and the largest.
        {"name": "sgemm_1024_tn", "kind": "sgemm", "ta": "T", "tb": "N", "m": 1024, "n": 1024, "k": 1024, "pad": 8,
         "alpha": 1.5, "beta": -0.25, "dist": "uniform"},
        # No dimension a multiple of anything, odd leading dimensions.
        {"name": "sgemm_ragged", "kind": "sgemm", "ta": "N", "tb": "N", "m": 1931, "n": 1207, "k": 877, "pad": 2,
         "alpha": 1.0, "beta": 0.0, "dist": "uniform"},
        {"name": "sgemm_4096_nt", "kind": "sgemm", "ta": "N", "tb": "T", "m": 4096, "n": 4096, "k": 4096, "pad": 8,
         "alpha": 1.5, "beta": -0.25, "dist": "uniform"},
        {"name": "sgemm_8192", "kind": "sgemm", "ta": "N", "tb": "N", "m": 8192, "n": 8192, "k": 8192, "pad": 8,
         "alpha": 1.5, "beta": -0.25, "dist": "uniform"},
        # The trailing update of a Linpack run, C := C - A B with k = nb, rows
        # scaled by 2^-20 .. 2^20: bound by reading and writing C.
        {"name": "linpack_update", "kind": "sgemm", "ta": "N", "tb": "N", "m": 8192, "n": 8192, "k": 128, "pad": 0,
         "alpha": -1.0, "beta": 1.0, "dist": "rowscaled"},
        # A small result with a very long inner dimension.
        {"name": "sgemm_long_k", "kind": "sgemm", "ta": "N", "tb": "N", "m": 512, "n": 512, "k": 65536, "pad": 0,
         "alpha": 1.0, "beta": 0.0, "dist": "uniform"},
        # A strided batch of the paper's micro-kernel problem (Table I).
        {"name": "batched", "kind": "batched", "ta": "N", "tb": "N", "m": 192, "n": 256, "k": 4096, "batch": 64,
         "alpha": 1.0, "beta": 0.0},
        # The uneven batch: thousands of independent products of random
        # shapes and transposes, tight leading dimensions, one plan.
        {"name": "grouped_4096", "kind": "grouped", "count": 4096, "lo": 16, "hi": 1024, "shapes": 3, "alpha": 1.0,
         "beta": 0.0},
        # A matrix-vector product, bound by reading the matrix.
        {"name": "sgemv_16384", "kind": "sgemv", "trans": "N", "m": 16384, "n": 16384, "pad": 0, "alpha": 1.0,
         "beta": 0.0},
        # The paper's Linpack order: factor and solve with one right-hand side.
        {"name": "lu_4608", "kind": "lu", "n": 4608, "nrhs": 1},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["square", "any", "any", "short", "update", "long", "batched", "grouped", "sgemv", "lu"])
    ta, tb = rng.choice("NT"), rng.choice("NT")
    scale = rng.choice([(1.0, 0.0), (1.5, -0.25), (1.0, 0.5)])
    pad = rng.choice([0, 1, 3, 8])
    if kind in ("square", "any", "short", "update", "long"):
        dist, (alpha, beta) = "uniform", scale
        if kind == "square":
            m = n = k = _log(rng, 128, 6000)
        elif kind == "any":
            m, n, k = (_log(rng, 100, 5000) for _ in range(3))
        elif kind == "short":
            m, n, k = _log(rng, 256, 4096), _log(rng, 256, 4096), _log(rng, 16, 127)
        elif kind == "update":
            m, n, k = _log(rng, 1024, 8192), _log(rng, 1024, 8192), rng.choice([128, 256])
            ta, tb, dist, alpha, beta = "N", "N", "rowscaled", -1.0, 1.0
        else:
            m, n, k = _log(rng, 128, 640), _log(rng, 128, 640), _log(rng, 8192, 65536)
        return {"kind": "sgemm", "ta": ta, "tb": tb, "m": m, "n": n, "k": k, "pad": pad, "alpha": alpha,
                "beta": beta, "dist": dist}
    if kind == "batched":
        return {"kind": "batched", "ta": ta, "tb": tb, "m": _log(rng, 64, 512), "n": _log(rng, 64, 512),
                "k": _log(rng, 128, 4096), "batch": _log(rng, 8, 96), "alpha": scale[0], "beta": scale[1]}
    if kind == "grouped":
        return {"kind": "grouped", "count": _log(rng, 128, 4096), "lo": 16, "hi": rng.choice([256, 512, 1024]),
                "shapes": rng.randrange(1 << 20), "alpha": scale[0], "beta": scale[1]}
    if kind == "sgemv":
        return {"kind": "sgemv", "trans": ta, "m": _log(rng, 256, 16384), "n": _log(rng, 256, 16384), "pad": pad,
                "alpha": scale[0], "beta": scale[1]}
    return {"kind": "lu", "n": _log(rng, 500, 4608), "nrhs": rng.choice([1, 1, 16])}


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _op_rows(trans, rows, cols):
    """Stored (rows, cols) of a matrix whose op() is rows x cols."""
    return (rows, cols) if trans == "N" else (cols, rows)


def _matrix(g, rows, cols, ld, dist="uniform"):
    x = torch.empty(cols, ld, device="cuda")
    if dist == "uniform":
        return x.uniform_(-1.0, 1.0, generator=g)
    x.normal_(generator=g)
    e = torch.randint(-20, 21, (ld,), device="cuda", generator=g)
    return x.mul_(torch.ldexp(torch.ones((), device="cuda"), e)[None, :])


def _handle():
    h = gbgemm.Handle(0)
    h.set_stream(torch.cuda.current_stream())
    return h


def _sgemm_inputs(c, seed):
    g = _gen(seed)
    (ar, ac), (br, bc) = _op_rows(c["ta"], c["m"], c["k"]), _op_rows(c["tb"], c["k"], c["n"])
    lda, ldb, ldc = ar + c["pad"], br + c["pad"], c["m"] + c["pad"]
    return (_matrix(g, ar, ac, lda, c["dist"]), lda, _matrix(g, br, bc, ldb, c["dist"]), ldb,
            _matrix(g, c["m"], c["n"], ldc, c["dist"]), ldc)


def _batched_inputs(c, seed):
    g = _gen(seed)
    shape = lambda rows, cols: torch.empty(c["batch"], cols, rows, device="cuda").uniform_(-1.0, 1.0, generator=g)
    return (shape(*_op_rows(c["ta"], c["m"], c["k"])), shape(*_op_rows(c["tb"], c["k"], c["n"])),
            shape(c["m"], c["n"]))


def _grouped_shapes(c):
    """Flags, dimensions and operand offsets of every problem of the batch,
    the operands one after the other with tight leading dimensions, and the
    three totals."""
    r = torch.Generator()
    r.manual_seed(c["shapes"])
    lo, hi = c["lo"], c["hi"]
    u = torch.rand(c["count"], 3, generator=r, dtype=torch.float64)
    dims = torch.exp(math.log(lo) + u * (math.log(hi + 1) - math.log(lo))).long().clamp(lo, hi).tolist()
    flags = torch.randint(0, 2, (c["count"], 2), generator=r).tolist()
    probs, a, b, o = [], 0, 0, 0
    for (m, n, k), (fa, fb) in zip(dims, flags):
        probs.append(("NT"[fa], "NT"[fb], m, n, k, a, b, o))
        a, b, o = a + m * k, b + k * n, o + m * n
    return probs, (a, b, o)


def _grouped_inputs(c, seed):
    probs, sizes = _grouped_shapes(c)
    g = _gen(seed)
    return probs, *(torch.empty(s, device="cuda").uniform_(-1.0, 1.0, generator=g) for s in sizes)


def _sgemv_inputs(c, seed):
    g = _gen(seed)
    lx, ly = (c["n"], c["m"]) if c["trans"] == "N" else (c["m"], c["n"])
    vec = lambda s: torch.empty(s, device="cuda").uniform_(-1.0, 1.0, generator=g)
    return _matrix(g, c["m"], c["n"], c["m"] + c["pad"]), vec(lx), vec(ly)


def _lu_inputs(c, seed):
    """A = P^T L U with |l_ij| <= 0.5 / sqrt(n) and a dominant diag(U), so
    that every pivot wins by a wide margin whatever the rounding, and B."""
    n, g = c["n"], _gen(seed)
    uni = lambda *s: torch.empty(*s, device="cuda").uniform_(-1.0, 1.0, generator=g)
    s = 1.0 / math.sqrt(n)
    low = torch.tril(uni(n, n) * (0.5 * s), -1) + torch.eye(n, device="cuda")
    up = torch.triu(uni(n, n) * s, 1) + torch.diag(1.5 + 0.5 * uni(n))
    rows = torch.randperm(n, device="cuda", generator=g)
    a = torch.empty(n, n, device="cuda")
    a[rows] = low @ up
    return a.T.contiguous(), uni(c["nrhs"], n)  # both column-major


def prepare(case, seed):
    c, h = dict(case), _handle()
    s = {"case": c, "h": h}
    if c["kind"] == "sgemm":
        s["A"], s["lda"], s["B"], s["ldb"], s["C"], s["ldc"] = _sgemm_inputs(c, seed)
        h.reserve_workspace(gbgemm.split_workspace_bytes(c["m"], c["n"], c["k"]))
    elif c["kind"] == "batched":
        s["A"], s["B"], s["C"] = _batched_inputs(c, seed)
    elif c["kind"] == "grouped":
        probs, s["A"], s["B"], s["C"] = _grouped_inputs(c, seed)
        pa, pb, pc = s["A"].data_ptr(), s["B"].data_ptr(), s["C"].data_ptr()
        s["plan"] = gbgemm.GroupedPlan(h, [
            gbgemm.problem(ta, tb, m, n, k, c["alpha"], pa + 4 * a, _op_rows(ta, m, k)[0], pb + 4 * b,
                           _op_rows(tb, k, n)[0], c["beta"], pc + 4 * o, m)
            for ta, tb, m, n, k, a, b, o in probs])
    elif c["kind"] == "sgemv":
        s["A"], s["x"], s["y"] = _sgemv_inputs(c, seed)
    else:
        s["A"], s["B"] = _lu_inputs(c, seed)
        s["LU"], s["X"] = torch.empty_like(s["A"]), torch.empty_like(s["B"])
        s["ipiv"] = torch.zeros(c["n"], dtype=torch.int32, device="cuda")
        s["info"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return s


def run(s):
    c, h = s["case"], s["h"]
    if c["kind"] == "sgemm":
        h.sgemm(c["ta"], c["tb"], c["m"], c["n"], c["k"], c["alpha"], s["A"], s["lda"], s["B"], s["ldb"], c["beta"],
                s["C"], s["ldc"])
        return s["C"][:, :c["m"]]
    if c["kind"] == "batched":
        (ar, ac), (br, bc) = _op_rows(c["ta"], c["m"], c["k"]), _op_rows(c["tb"], c["k"], c["n"])
        h.sgemm_strided_batched(c["ta"], c["tb"], c["m"], c["n"], c["k"], c["alpha"], s["A"], ar, ar * ac, s["B"], br,
                                br * bc, c["beta"], s["C"], c["m"], c["m"] * c["n"], c["batch"])
        return s["C"]
    if c["kind"] == "grouped":
        s["plan"].run()
        return s["C"]
    if c["kind"] == "sgemv":
        h.sgemv(c["trans"], c["m"], c["n"], c["alpha"], s["A"], c["m"] + c["pad"], s["x"], 1, c["beta"], s["y"], 1)
        return s["y"]
    n = c["n"]
    s["LU"].copy_(s["A"])  # the factors overwrite the matrix, and the program keeps A
    s["X"].copy_(s["B"])
    h.sgetrf(n, s["LU"], n, s["ipiv"], s["info"])
    h.sgetrs(n, c["nrhs"], s["LU"], n, s["ipiv"], s["X"], n)
    return {"lu": s["LU"], "ipiv": s["ipiv"], "info": s["info"], "x": s["X"]}


def work(case):
    c = case
    beta = 1 if c.get("beta", 0.0) != 0.0 else 0
    if c["kind"] in ("sgemm", "batched"):
        m, n, k, z = c["m"], c["n"], c["k"], c.get("batch", 1)
        return {"bytes": 4.0 * z * (m * k + k * n + (1 + beta) * m * n), "flops": 2.0 * z * m * n * k}
    if c["kind"] == "grouped":
        probs, (a, b, o) = _grouped_shapes(c)
        return {"bytes": 4.0 * (a + b + (1 + beta) * o), "flops": sum(2.0 * p[2] * p[3] * p[4] for p in probs)}
    if c["kind"] == "sgemv":
        m, n = c["m"], c["n"]
        ly = m if c["trans"] == "N" else n
        return {"bytes": 4.0 * (m * n + m + n + beta * ly), "flops": 2.0 * m * n}
    n, r = c["n"], c["nrhs"]
    return {"bytes": 4.0 * (3 * n * n + 2 * n * r), "flops": 2.0 / 3.0 * n ** 3 + 2.0 * n * n * r}


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "sgemm":
        A, _, B, _, C, _ = _sgemm_inputs(c, seed)
        a, b = A[:, :_op_rows(c["ta"], c["m"], c["k"])[0]], B[:, :_op_rows(c["tb"], c["k"], c["n"])[0]]
        a, b = (a.T if c["ta"] == "N" else a).double(), (b.T if c["tb"] == "N" else b).double()
        out = c["alpha"] * (a @ b)
        return ((out + c["beta"] * C[:, :c["m"]].T.double()) if c["beta"] != 0.0 else out).T.contiguous()
    if c["kind"] == "batched":
        A, B, C = _batched_inputs(c, seed)
        a, b = (A.mT if c["ta"] == "N" else A).double(), (B.mT if c["tb"] == "N" else B).double()
        out = c["alpha"] * (a @ b)
        return ((out + c["beta"] * C.mT.double()) if c["beta"] != 0.0 else out).mT.contiguous()
    if c["kind"] == "grouped":
        probs, A, B, C = _grouped_inputs(c, seed)
        A, B, out = A.double(), B.double(), C.double() * c["beta"]
        for ta, tb, m, n, k, a, b, o in probs:
            x = A[a:a + m * k].view(k, m).T if ta == "N" else A[a:a + m * k].view(m, k)
            y = B[b:b + k * n].view(n, k).T if tb == "N" else B[b:b + k * n].view(k, n)
            out[o:o + m * n].view(n, m).add_((x @ y).T, alpha=c["alpha"])
        return out
    if c["kind"] == "sgemv":
        A, x, y = _sgemv_inputs(c, seed)
        a = A[:, :c["m"]].double()
        out = c["alpha"] * ((a.T if c["trans"] == "N" else a) @ x.double())
        return out + c["beta"] * y.double() if c["beta"] != 0.0 else out
    A, B = _lu_inputs(c, seed)
    a = A.T.double()
    lu, _ = torch.linalg.lu_factor(a)
    x = torch.linalg.solve(a, B.T.double())
    return {"lu": lu.T.contiguous(), "ipiv": None, "info": None, "x": x.T.contiguous()}
