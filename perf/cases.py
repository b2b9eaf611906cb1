"""Performance cases: what a user of this library runs, through its public
Python entry points, over the range of sizes, precisions and call forms that
it is used with.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` builds a case's inputs and handle on the GPU, ``run`` makes one
pass, ``work`` states the bytes and flops a pass cannot do without, and
``exact`` computes the same outputs with plain torch in 64 bits.

A case is one of

* ``kind = "solo"``: one matrix (``nt``, ``b``, ``w``, ``a``) in precision
  ``prec``, by ``op``: ``fused`` (factor + selected inversion), ``factor``
  (factor and logdet, a likelihood evaluation), ``selinv`` (from a given L),
  ``selected`` (Sigma from tile column ``first`` on), ``host`` (end to end on
  page-locked host buffers);
* ``kind = "batch"``: uneven matrices (``shapes``) in one graph launch;
* ``kind = "serve"``: a request server started, given ``requests`` sweep
  points of its pool (``shapes``), drained and stopped.
"""
import random

import numpy as np
import torch

from paper_2504_19171_gb300 import stiles as S
from paper_2504_19171_gb300 import workloads as W

DEV = "cuda"
PREC = {"fp64": S.STILES_FP64, "emu64": S.STILES_EMU64, "fp32x": S.STILES_FP32X}


def solo(name, op, prec, nt, b, w, a, values="random", first=0):
    c = {"kind": "solo", "op": op, "prec": prec, "nt": nt, "b": b, "w": w, "a": a, "values": values, "first": first}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small model (n = 1040): a single evaluation inside an optimiser's
        # loop, where latency is everything
        solo("small fp64", "fused", "fp64", 16, 64, 1, 16),
        # a longer model with odd tile and arrow sizes (ragged 64-blocks)
        solo("ragged fp64", "fused", "fp64", 40, 100, 2, 37),
        # the benchmark matrix: spatio-temporal, n = 204,864, true FP64
        solo("spatiotemporal fp64", "fused", "fp64", 200, 1024, 1, 64, "spatiotemporal"),
        # the same model in emulated FP64 (120 of its 200 time steps)
        solo("spatiotemporal emu64", "fused", "emu64", 120, 1024, 1, 64, "spatiotemporal"),
        # the same at tile bandwidth 4 (higher-order autoregression)
        solo("band 4 emu64", "fused", "emu64", 28, 1024, 4, 64, "spatiotemporal"),
        # FP32-class precision, for a quick look at marginal variances
        solo("spatiotemporal fp32x", "fused", "fp32x", 64, 1024, 1, 64, "spatiotemporal"),
        # a likelihood evaluation: factor and logdet only, mid-size, odd sizes
        solo("likelihood fp64", "factor", "fp64", 60, 250, 2, 50),
        # the selected inversion of a factor kept from before
        solo("selinv emu64", "selinv", "emu64", 48, 512, 2, 100),
        # the fixed effects' covariance only (the arrow block of Sigma)
        solo("arrow block emu64", "selected", "emu64", 80, 529, 1, 64, "spatiotemporal", 80),
        # a matrix that lives in host memory, end to end
        solo("host fp64", "host", "fp64", 60, 256, 1, 32),
        # uneven models of one study in one launch
        {"name": "batch emu64", "kind": "batch", "prec": "emu64",
         "shapes": "96,256,1,61 40,128,4,17 64,512,2,90 31,256,3,8 110,128,2,120 52,512,1,33 20,256,4,75 77,128,1,44"},
        # a hyperparameter sweep through the request server
        {"name": "serve emu64", "kind": "serve", "prec": "emu64", "shapes": "40,128,1,20 24,256,1,64 30,200,2,33",
         "requests": 9},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


# A drawn case costs no more than the largest listed one: its flops, and the
# length of its chain of pivots, stay below these.
MAX_FLOPS = {"fp64": 1.2e12, "emu64": 1.6e12, "fp32x": 1.6e12}
MAX_COLUMNS = 120000


def _draw_shape(rng, nt, b, w, a):
    return _log_int(rng, *nt), _log_int(rng, *b), rng.randint(*w), rng.choice([0, rng.randint(*a), rng.randint(*a)])


def draw(rng):
    kind = rng.choice(["solo"] * 6 + ["batch", "serve"])
    prec = rng.choice(["fp64", "fp64", "emu64", "emu64", "fp32x"])
    if kind == "solo":
        while True:
            nt, b, w, a = _draw_shape(rng, (6, 200), (16, 1024), (1, 4), (1, 128))
            op = rng.choice(["fused", "fused", "fused", "factor", "selinv", "selected", "host"])
            first = rng.randint(1, nt if a else nt - 1) if op == "selected" else 0
            values = "spatiotemporal" if op != "selinv" and rng.random() < 0.4 else "random"
            if values == "spatiotemporal":  # the space is a square grid
                b = round(b ** 0.5) ** 2
            c = solo(None, op, "emu64" if op == "selinv" and prec == "fp32x" else prec, nt, b, w, a, values, first)
            if work(c)["flops"] <= MAX_FLOPS[prec] and nt * b <= MAX_COLUMNS:
                return c
    if kind == "batch":
        while True:
            shapes = [_draw_shape(rng, (20, 120), (64, 512), (1, 4), (8, 128)) for _ in range(rng.randint(3, 10))]
            c = {"kind": "batch", "prec": prec, "shapes": _text(shapes)}
            if work(c)["flops"] <= 0.5 * MAX_FLOPS[prec]:
                return c
    shapes = [_draw_shape(rng, (10, 60), (40, 300), (1, 2), (8, 128)) for _ in range(rng.randint(1, 3))]
    return {"kind": "serve", "prec": "emu64" if prec == "fp32x" else prec, "shapes": _text(shapes),
            "requests": rng.randint(2, 10)}


def _text(shapes):
    return " ".join(",".join(str(v) for v in sh) for sh in shapes)


def _shapes(case):
    return [tuple(int(v) for v in sh.split(",")) for sh in case["shapes"].split()]


# ------------------------------------------------------------- the layout ----
class Grid:
    """Packed band + arrow layout of one matrix."""

    def __init__(self, nt, b, w, a):
        self.nt, self.b, self.w, self.a = nt, b, min(w, nt - 1), a
        self.stride = (1 + self.w) * b * b + a * b
        self.doubles = nt * self.stride + a * a
        self.cols = nt + (1 if a else 0)
        self.n = nt * b + a

    def rows(self, i):
        return self.a if i == self.nt else self.b

    def below(self, k):
        """Off-diagonal tile rows of tile column k."""
        if k == self.nt:
            return []
        return list(range(k + 1, min(k + self.w, self.nt - 1) + 1)) + ([self.nt] if self.a else [])

    def tile(self, flat, i, k):
        if k == self.nt:
            off = self.nt * self.stride
        elif i == self.nt:
            off = k * self.stride + (1 + self.w) * self.b * self.b
        else:
            off = k * self.stride + (i - k) * self.b * self.b
        r, c = self.rows(i), self.rows(k)
        return flat[off:off + r * c].view(c, r).t()

    def parts(self, flat):
        """The written part of a packed buffer (the last columns' slots beyond
        the matrix are never written): contiguous pieces that cover it."""
        got, start = [], 0
        for k in range(max(0, self.nt - self.w), self.nt):
            end = k * self.stride + (self.nt - k) * self.b * self.b
            got.append(flat[start:end])
            start = k * self.stride + (1 + self.w) * self.b * self.b
        got.append(flat[start:])
        return [g for g in got if g.numel()]


def _spatiotemporal(g, seed, out):
    """AR(1)^w in time, 5-point Laplacian plus identity in space, dense N(0,1)
    arrow with a dominant corner; (tau, rho) vary with the seed, as in a
    sweep over hyperparameters."""
    side = int(round(g.b ** 0.5))
    r = random.Random(seed)
    rho, tau = r.uniform(0.6, 0.95), r.uniform(0.5, 2.0)
    qt = np.linalg.matrix_power(W.ar1_precision(g.nt, rho), max(1, g.w))
    qs = torch.from_numpy(W.laplacian2d_plus_identity(side)).to(out.device)
    eye = torch.eye(g.b, dtype=torch.float64, device=out.device)
    gen = torch.Generator(device=out.device)
    gen.manual_seed(int(seed))
    rowabs = torch.zeros(g.a, dtype=torch.float64, device=out.device)
    for k in range(g.nt):
        g.tile(out, k, k).copy_(float(qt[k, k]) * qs + tau * eye)
        for i in g.below(k):
            if i == g.nt:
                t = torch.randn((g.a, g.b), generator=gen, dtype=torch.float64, device=out.device)
                rowabs += t.abs().sum(dim=1)
                g.tile(out, i, k).copy_(t)
            else:
                g.tile(out, i, k).copy_(float(qt[i, k]) * qs)
    if g.a:
        t = torch.tril(torch.randn((g.a, g.a), generator=gen, dtype=torch.float64, device=out.device), -1)
        t = t + t.t()
        t.diagonal().copy_(1.0 + rowabs + t.abs().sum(dim=1))
        g.tile(out, g.nt, g.nt).copy_(t)


def _matrix(case, g, seed):
    A = torch.zeros(g.doubles, dtype=torch.float64, device=DEV)
    if case.get("values") == "spatiotemporal":
        _spatiotemporal(g, seed, A)
    else:
        W.random_arrowhead_packed(g.nt, g.b, g.w, g.a, seed, A)
    return A


# ------------------------------------------------------ prepare and run ----
def prepare(case, seed):
    if case["kind"] == "batch":
        shapes = _shapes(case)
        bt = S.StilesBatch(shapes, device=DEV, precision=PREC[case["prec"]])
        bt.A = torch.zeros(bt.doubles, dtype=torch.float64, device=DEV)
        bt.L.zero_()
        bt.S.zero_()
        for m, sh in enumerate(shapes):
            W.random_arrowhead_packed(*sh, 64 * seed + m, bt.A[int(bt.off[m]):])
        return {"case": case, "batch": bt}
    if case["kind"] == "serve":
        return _prepare_server(case, seed)
    g = Grid(case["nt"], case["b"], case["w"], case["a"])
    st = S.Stiles(g.nt, g.b, g.w, g.a, device=DEV, precision=PREC[case["prec"]], first_column=case["first"])
    st.L.zero_()
    st.S.zero_()
    st.A = _matrix(case, g, seed)
    state = {"case": case, "st": st}
    if case["op"] == "selinv":
        st.L.copy_(_factor(g, st.A))
    elif case["op"] == "host":
        state["A_host"] = st.A.cpu().pin_memory()
        state["S_host"] = torch.zeros(g.doubles, dtype=torch.float64).pin_memory()
    return state


def _prepare_server(case, seed):
    shapes = _shapes(case)
    grids = [Grid(*sh) for sh in shapes]
    count = case["requests"]
    data = sum(3 * 8 * (grids[q % len(grids)].doubles + 32) for q in range(count))
    srv = S.StilesServer(shapes, data_bytes=2 * data, max_requests=count, precision=PREC[case["prec"]], device=DEV)
    for m, g in enumerate(grids):
        base = torch.zeros(g.doubles, dtype=torch.float64, device=DEV)
        rb, ra = W.sweep_base_packed(g.nt, g.b, g.w, g.a, 64 * seed + m, base)
        torch.cuda.synchronize()  # the server copies on a stream of its own
        srv.set_base(m, base, rb, ra)
    r = random.Random(seed)
    points = [(q % len(grids), 10.0 ** r.uniform(-1, 1), r.uniform(0.5, 0.99)) for q in range(count)]
    out = [torch.zeros(grids[m].doubles, dtype=torch.float64).pin_memory() for m, _, _ in points]
    return {"case": case, "server": srv, "points": points, "out": out, "grids": grids}


def _run_server(state):
    srv, points, out = state["server"], state["points"], state["out"]
    logdet = [0.0] * len(points)
    srv.start(30.0)
    waiting, left = list(range(len(points))), len(points)
    while left:
        while waiting:
            m, tau, rho = points[waiting[0]]
            if srv.submit(m, tau, rho, tag=waiting[0]) is None:
                break
            waiting.pop(0)
        for request, tag in srv.poll():
            code, info, logdet[tag] = srv.result(request)
            if code != S.STILES_OK:
                raise S.StilesError(code, "request")
            srv.sigma(request, out[tag])
            srv.release(request)
            left -= 1
    srv.stop()
    return {"logdet": np.array(logdet),
            "Sigma": [state["grids"][p[0]].parts(o) for p, o in zip(points, out)]}


def run(state):
    if "server" in state:
        return _run_server(state)
    if "batch" in state:
        bt = state["batch"]
        bt.factor_selinv()
        return {"L": bt.L, "Sigma": bt.S}
    st, op = state["st"], state["case"]["op"]
    if op == "factor":
        st.factor()
        return {"L": st.L, "logdet": st.logdet()}
    if op == "selinv":
        st.selinv()
        return {"Sigma": st.S}
    if op == "host":
        logdet = st.factor_selinv_host(state["A_host"], state["S_host"])
        return {"Sigma": state["S_host"], "logdet": logdet}
    st.factor_selinv()
    return {"L": st.L, "Sigma": st.S}


# ----------------------------------------------------------------- work ----
def _work(g, op, first=0):
    """Flops of the tile operations (POTRF, TRTRI, LAUUM m^3/3; TRSM, TRMM
    m k^2; SYRK and the symmetric Sigma_ii update m^2 k; GEMM 2 m n k), and
    each input tile read and each output tile written once."""
    flops = nbytes = 0.0
    for k in range(g.cols):
        m = float(g.rows(k))
        st = [float(g.rows(i)) for i in g.below(k)]
        column = 8.0 * (m * m + m * sum(st))
        if op == "selinv":
            nbytes += column
        else:
            nbytes += 2 * column
            flops += m ** 3 / 3 + sum(x * m * m + x * x * m for x in st)
            flops += sum(2.0 * st[i] * st[j] * m for i in range(len(st)) for j in range(i))
        if op != "factor" and k >= first:
            nbytes += column
            flops += 2 * m ** 3 / 3 + sum(2 * x * m * m for x in st) + 2.0 * m * sum(st) ** 2
    return {"bytes": nbytes, "flops": flops}


def work(case):
    if case["kind"] == "solo":
        return _work(Grid(case["nt"], case["b"], case["w"], case["a"]), case["op"], case["first"])
    grids = [Grid(*sh) for sh in _shapes(case)]
    if case["kind"] == "serve":
        grids = [grids[q % len(grids)] for q in range(case["requests"])]
    each = [_work(g, "fused") for g in grids]
    return {key: sum(e[key] for e in each) for key in ("bytes", "flops")}


# ---------------------------------------------------------------- exact ----
def _factor(g, A):
    """Packed Cholesky factor of the packed matrix A."""
    L = torch.zeros_like(A)
    part = A.clone()
    for k in range(g.cols):
        Lk = torch.linalg.cholesky(torch.tril(g.tile(part, k, k)))
        g.tile(L, k, k).copy_(Lk)
        st = g.below(k)
        X = {i: torch.linalg.solve_triangular(Lk, g.tile(part, i, k).t(), upper=False).t() for i in st}
        for i in st:
            g.tile(L, i, k).copy_(X[i])
            for j in st:
                if j <= i:
                    g.tile(part, i, j).sub_(X[i] @ X[j].t())
    return L


def _invert(g, L, first=0):
    """Packed selected inverse from the packed factor, tile columns >= first."""
    Sg = torch.zeros_like(L)
    for i in range(g.cols - 1, first - 1, -1):
        Li = g.tile(L, i, i)
        eye = torch.eye(g.rows(i), dtype=torch.float64, device=L.device)
        inv = torch.linalg.solve_triangular(Li, eye, upper=False)
        st = g.below(i)
        U = {k: g.tile(L, k, i) @ inv for k in st}
        D = inv.t() @ inv
        for j in st:
            X = -sum((g.tile(Sg, j, k) if j >= k else g.tile(Sg, k, j).t()) @ U[k] for k in st)
            g.tile(Sg, j, i).copy_(X)
            D = D - X.t() @ U[j]
        g.tile(Sg, i, i).copy_(0.5 * (D + D.t()))
    return Sg


def _logdet(g, L):
    return float(2.0 * sum(torch.log(g.tile(L, k, k).diagonal()).sum() for k in range(g.cols)))


def _exact_server(case, seed):
    shapes = _shapes(case)
    grids = [Grid(*sh) for sh in shapes]
    r = random.Random(seed)
    bases = []
    for m, g in enumerate(grids):
        base = torch.zeros(g.doubles, dtype=torch.float64, device=DEV)
        bases.append((base,) + tuple(W.sweep_base_packed(g.nt, g.b, g.w, g.a, 64 * seed + m, base)))
    logdet, sigma = [], []
    for q in range(case["requests"]):
        m, tau, rho = q % len(grids), 10.0 ** r.uniform(-1, 1), r.uniform(0.5, 0.99)
        g, (base, rb, ra) = grids[m], bases[m]
        A = rho * base
        for k in range(g.cols):
            if g.a:
                g.tile(A, g.nt, k).copy_(g.tile(base, g.nt, k))
            r0 = k * g.b
            g.tile(A, k, k).diagonal().copy_((tau + rho * rb + ra)[r0:r0 + g.rows(k)])
        L = _factor(g, A)
        logdet.append(_logdet(g, L))
        sigma.append([p.cpu() for p in g.parts(_invert(g, L))])
    return {"logdet": np.array(logdet), "Sigma": sigma}


def exact(case, seed):
    if case["kind"] == "serve":
        return _exact_server(case, seed)
    if case["kind"] == "batch":
        grids, off = [Grid(*sh) for sh in _shapes(case)], [0]
        for g in grids:  # each matrix starts at a multiple of 32 doubles
            off.append(off[-1] + (g.doubles + 31) // 32 * 32)
        L = torch.zeros(off[-1], dtype=torch.float64, device=DEV)
        Sg = torch.zeros_like(L)
        for m, g in enumerate(grids):
            A = torch.zeros(g.doubles, dtype=torch.float64, device=DEV)
            W.random_arrowhead_packed(g.nt, g.b, g.w, g.a, 64 * seed + m, A)
            Lm = _factor(g, A)
            L[off[m]:off[m] + g.doubles] = Lm
            Sg[off[m]:off[m] + g.doubles] = _invert(g, Lm)
        return {"L": L, "Sigma": Sg}
    g, op = Grid(case["nt"], case["b"], case["w"], case["a"]), case["op"]
    L = _factor(g, _matrix(case, g, seed))
    if op == "factor":
        return {"L": L, "logdet": _logdet(g, L)}
    Sg = _invert(g, L, case["first"])
    if op == "selinv":
        return {"Sigma": Sg}
    if op == "host":
        return {"Sigma": Sg.cpu(), "logdet": _logdet(g, L)}
    return {"L": L, "Sigma": Sg}
