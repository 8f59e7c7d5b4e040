"""The work that users of the solver library have it do, through its public calls.

Kinds of case (every mesh, discretisation and hierarchy is one of `synth`'s
recipes, the inputs of this repository's tests and benchmark):

  product   one block-sparse product on caller memory (gasa_bsr_mv, _f32, _ds):
            a Krylov method of the caller's own on A_0, a residual, a transfer
            through P_0 or R_0, or a coarse operator
  sweep     one block-Jacobi smoothing step on caller memory
  vcycle    one V-cycle on a resident hierarchy: the preconditioner inside a
            caller's own Krylov method
  solve     a whole solve from a right-hand side in host memory
  setup     a hierarchy from an assembled operator, its first V-cycle and one
            solve: what a program with one system to solve runs
  serve     a batch of requests over several resident meshes, sent to the
            request server and collected

Meshes: `tri` (SIPG Poisson, triangles), `tet` (SIPG Poisson, Kuhn tetrahedra),
`quad` (LDG convection-diffusion, quadrilaterals); `n` cells per side, `p` the
polynomial order, `r` the candidate vectors of the hierarchy.
"""
import functools
import math

import numpy as np
import torch

from paper_2504_13373_gb300 import gasa
from synth import configs, serving

TOL = 1e-10
PRECISION = {"fp64": gasa.GASA_PREC_FP64, "mixed32": gasa.GASA_PREC_MIXED32,
             "mixed16": gasa.GASA_PREC_MIXED16}
MODE = {"assign": gasa.GASA_MV_ASSIGN, "residual": gasa.GASA_MV_RESIDUAL, "add": gasa.GASA_MV_ADD}
DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a residual in a caller's loop on the smallest resident mesh of the benchmark
        dict(name="residual_tri_p1_32", kind="product", mesh="tri", n=32, p=1, r=12, pe=0.0,
             matrix="A", level=0, dtype="fp64", mode="residual"),
        # a caller's product with a coarse operator of a 3-D hierarchy: wide blocks, long rows
        dict(name="product_tet_p2_16_level1", kind="product", mesh="tet", n=16, p=2, r=80, pe=0.0,
             matrix="A", level=1, dtype="fp32", mode="assign"),
        # the outer product of a mixed-precision Krylov method, 3-D, an odd grid
        dict(name="outer_tet_p2_23_ds", kind="product", mesh="tet", n=23, p=2, r=8, pe=0.0,
             matrix="A", level=0, dtype="ds", mode="assign"),
        # the smoothing step of the benchmark's mesh
        dict(name="sweep_tri_p3_256", kind="sweep", mesh="tri", n=256, p=3, r=4, pe=0.0,
             dtype="fp32"),
        # the benchmark's preconditioner
        dict(name="vcycle_tri_p3_256_mixed32", kind="vcycle", mesh="tri", n=256, p=3, r=4, pe=0.0,
             precision="mixed32"),
        # the 3-D preconditioner, whose coarse levels outweigh level 0
        dict(name="vcycle_tet_p2_16_mixed32", kind="vcycle", mesh="tet", n=16, p=2, r=80, pe=0.0,
             precision="mixed32"),
        # FP16 blocks, a grid that is no power of two (padded coarse levels)
        dict(name="vcycle_tri_p3_90_mixed16", kind="vcycle", mesh="tri", n=90, p=3, r=4, pe=0.0,
             precision="mixed16"),
        # the FP64 preconditioner, nonsymmetric
        dict(name="vcycle_quad_p2_128_fp64", kind="vcycle", mesh="quad", n=128, p=2, r=36,
             pe=100.0, precision="fp64"),
        # the smallest whole solve (CG): latency
        dict(name="solve_tri_p1_32_mixed32", kind="solve", mesh="tri", n=32, p=1, r=12, pe=0.0,
             precision="mixed32"),
        # a whole GMRES solve
        dict(name="solve_quad_p2_96_mixed32", kind="solve", mesh="quad", n=96, p=2, r=36,
             pe=100.0, precision="mixed32"),
        # one system from its assembled operator to its solution
        dict(name="setup_tet_p2_8", kind="setup", mesh="tet", n=8, p=2, r=80, pe=0.0,
             precision="mixed32"),
        # a burst of requests over three resident meshes
        dict(name="serve_24", kind="serve", precision="mixed32", requests=24,
             mesh_a="tri", n_a=16, p_a=3, mesh_b="quad", n_b=32, p_b=2, mesh_c="tet", n_c=4, p_c=3),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]; odd ones among them."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_mesh(rng, scale=1.0):
    """A mesh family, order, size, candidate count and Peclet number."""
    mesh, p, hi = rng.choice([("tri", 1, 160), ("tri", 2, 128), ("tri", 3, 96), ("tet", 1, 14),
                              ("tet", 2, 10), ("quad", 1, 128), ("quad", 2, 96)])
    lo = 3 if mesh == "tet" else 8
    n = _log_int(rng, lo, max(lo + 1, int(hi * scale)))
    nb = _block(mesh, p)
    r = min((8 if mesh == "tet" else 4) * nb, 80)
    if mesh == "tri" and p == 3 and rng.random() < 0.5:
        r = 4
    pe = rng.choice([1.0, 100.0, 1e4]) if mesh == "quad" else 0.0
    return dict(mesh=mesh, n=n, p=p, r=r, pe=pe)


def draw(rng):
    kind = rng.choice(["product", "product", "sweep", "vcycle", "vcycle", "solve", "setup",
                       "serve"])
    if kind == "serve":
        return dict(kind="serve", precision=rng.choice(["mixed32", "fp64", "mixed16"]),
                    requests=rng.randint(3, 24),
                    mesh_a="tri", n_a=_log_int(rng, 8, 20), p_a=rng.randint(1, 2),
                    mesh_b="quad", n_b=_log_int(rng, 8, 32), p_b=rng.randint(1, 2),
                    mesh_c="tet", n_c=_log_int(rng, 3, 6), p_c=rng.randint(1, 2))
    if kind in ("product", "sweep"):
        c = dict(kind=kind, **_draw_mesh(rng))
        if kind == "sweep":
            c.update(dtype=rng.choice(["fp32", "fp64"]))
        else:
            dtype = rng.choice(["fp64", "fp32", "ds"])
            c.update(dtype=dtype, mode="assign", matrix="A", level=0)
            if dtype != "ds":
                c.update(mode=rng.choice(["assign", "residual", "add"]),
                         matrix=rng.choice(["A", "P", "R"]), level=rng.choice([0, 0, 1]))
        return c
    if kind == "vcycle":
        return dict(kind=kind, precision=rng.choice(["mixed32", "mixed32", "fp64", "mixed16"]),
                    **_draw_mesh(rng))
    c = dict(kind=kind, precision=rng.choice(["mixed32", "fp64"]),
             **_draw_mesh(rng, 0.5 if kind == "setup" else 0.4))
    return c


# ---------------------------------------------------------------------------
# operators and hierarchies
# ---------------------------------------------------------------------------
def _block(mesh, p):
    if mesh == "quad":
        return (p + 1) ** 2
    return (p + 1) * (p + 2) // 2 if mesh == "tri" else (p + 1) * (p + 2) * (p + 3) // 6


@functools.lru_cache(maxsize=8)
def _problem(mesh, n, p, r, pe, seed):
    """The assembled system of a mesh (host arrays) and its element aggregates."""
    if mesh == "tri":
        return configs.poisson2d(n, p, r=r, seed=seed)
    if mesh == "tet":
        return configs.poisson3d(n, p, r=r, seed=seed)
    return configs.convdiff2d(n, p, pe, r=r, seed=seed)


def _case_problem(case, seed=configs.SEED):
    return _problem(case["mesh"], case["n"], case["p"], case["r"], case["pe"], seed)


class Hierarchy:
    """A set-up context on its own stream, released with its last reference."""

    def __init__(self, pr, device_operator=None):
        self.stream = torch.cuda.Stream()
        self.ctx = gasa.gasa_create(0, self.stream)
        self.n = pr.n_dofs
        self.levels = pr.n_levels
        self.info = self.setup(pr, device_operator)

    def setup(self, pr, device_operator=None):
        opt = gasa.gasa_default_options(
            dim=pr.dim, n_cand=pr.r, seed=configs.SEED,
            solver=gasa.GASA_SOLVER_CG if pr.solver == "cg" else gasa.GASA_SOLVER_GMRES)
        rp, col, val = device_operator or (pr.A.row_ptr, pr.A.col, pr.A.val.ravel())
        return gasa.gasa_setup(self.ctx, rp, col, val, pr.A.b, pr.agg_of, opt,
                               adj_ptr=pr.adj_ptr, adj_idx=pr.adj_idx, centroids=pr.centroids,
                               on_device=device_operator is not None)

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            gasa.gasa_destroy(self.ctx)
            self.ctx = None


def _read_bsr(h, level, which):
    """(row_ptr, col, val, block columns) of A_k, P_k or R_k from the device."""
    sh = gasa.gasa_level_shape(h.ctx, level)
    rows, br, bc, cols = sh["units"], sh["s"], sh["s"], sh["units"]
    nnzb, base = sh["nnzb"], gasa.GASA_LV_A_ROWPTR
    if which != "A":
        units_next = gasa.gasa_level_shape(h.ctx, level + 1)["units"]
        nnzb = sh["P_nnzb"]
        if which == "P":
            bc, cols, base = sh["s_next"], units_next, gasa.GASA_LV_P_ROWPTR
        else:
            rows, br, base = units_next, sh["s_next"], gasa.GASA_LV_R_ROWPTR
    rp = gasa.gasa_get_level(h.ctx, level, base, np.empty(rows + 1, np.int32))
    col = gasa.gasa_get_level(h.ctx, level, base + 1, np.empty(nnzb, np.int32))
    val = gasa.gasa_get_level(h.ctx, level, base + 2, np.empty(nnzb * br * bc, np.float64))
    return rp, col, val.reshape(nnzb, br, bc), cols


@functools.lru_cache(maxsize=4)
def _operator(mesh, n, p, r, pe, matrix, level):
    pr = _problem(mesh, n, p, r, pe, configs.SEED)
    if matrix == "A" and level == 0:
        return pr.A.row_ptr, pr.A.col, pr.A.val, pr.A.n
    level = min(level, pr.n_levels - (1 if matrix == "A" else 2))
    return _read_bsr(Hierarchy(pr), level, matrix)


def _case_operator(case):
    return _operator(case["mesh"], case["n"], case["p"], case["r"], case["pe"],
                     case.get("matrix", "A"), case.get("level", 0))


@functools.lru_cache(maxsize=32)
def _level_work(mesh, n, p, r, pe, solve=False):
    """(matrix values, dofs of level 0, values of A_0, CG or GMRES iterations) of a hierarchy:
    the values of A_k, W_k, P_k and R_k on every smoothed level and of the coarsest inverse."""
    pr = _problem(mesh, n, p, r, pe, configs.SEED)
    h = Hierarchy(pr)
    values = 0
    for k in range(h.levels):
        sh = gasa.gasa_level_shape(h.ctx, k)
        if k + 1 == h.levels:
            values += (sh["units"] * sh["s"]) ** 2
        else:
            values += sh["nnzb"] * sh["s"] ** 2 + sh["units"] * sh["s"] ** 2
            values += 2 * sh["P_nnzb"] * sh["s"] * sh["s_next"]
    it = 0
    if solve:
        b, x = configs.rhs(1, pr.n_dofs), np.empty(pr.n_dofs)
        it = gasa.gasa_solve(h.ctx, b, x, TOL, gasa.GASA_PREC_FP64).iterations
    return values, pr.n_dofs, pr.A.nnzb * pr.A.b ** 2, it


def _serve_specs(case):
    out = []
    for j in "abc":
        mesh, n, p = case["mesh_" + j], case["n_" + j], case["p_" + j]
        r = min((8 if mesh == "tet" else 4) * _block(mesh, p), serving.R_CAP)
        out.append((mesh, n, p, r, 100.0 if mesh == "quad" else 0.0))
    return out


# ---------------------------------------------------------------------------
# what a program holds before the call
# ---------------------------------------------------------------------------
def _normal(seed, n, stream=0):
    g = torch.Generator(device=DEV).manual_seed(1000003 * (int(seed) + 1) + stream)
    return torch.randn(n, dtype=torch.float64, device=DEV, generator=g)


def _up(a):
    return torch.as_tensor(a).to(DEV)


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _split(v):
    hi = v.float()
    return hi, (v - hi.double()).float()


def _product_inputs(case, seed):
    rp, col, val, cols = _case_operator(case)
    rows, (br, bc) = len(rp) - 1, val.shape[1:]
    x = _normal(seed, cols * bc, 1)
    b = _normal(seed, rows * br, 2)
    if case["dtype"] == "fp32":
        x, b = x.float().double(), b.float().double()
    return rp, col, val, x, b, rows, br, bc


def _prepare_product(case, seed):
    rp, col, val, x, b, rows, br, bc = _product_inputs(case, seed)
    st = dict(kind="product", dtype=case["dtype"], mode=MODE[case["mode"]], rows=rows, br=br,
              bc=bc, rp=_up(rp), col=_up(col), adds=case["mode"] == "add")
    val = _up(val).reshape(-1)
    if case["dtype"] == "ds":
        st["ahi"], st["alo"] = _split(val)
        st["xhi"], st["xlo"] = _split(x)
        st["y"] = torch.zeros(rows * br, dtype=torch.float64, device=DEV)
        return st
    t = torch.float32 if case["dtype"] == "fp32" else torch.float64
    st.update(val=val.to(t), x=x.to(t), b=b.to(t))
    st["y"] = torch.zeros(rows * br, dtype=t, device=DEV)
    return st


def _sweep_weights(case):
    """w D^-1 of the level-0 operator (w = 1/2) in FP64, from the library's own block inverse."""
    rp, col, val, _ = _case_operator(case)
    n, bs = len(rp) - 1, val.shape[1]
    W = torch.empty(n * bs * bs, dtype=torch.float64, device=DEV)
    gasa.gasa_block_inverse(n, bs, _up(rp), _up(col), _up(val).reshape(-1), 0.5, W)
    return W


def _prepare_sweep(case, seed):
    rp, col, val, x, b, rows, bs, _ = _product_inputs(case, seed)
    t = torch.float32 if case["dtype"] == "fp32" else torch.float64
    return dict(kind="sweep", dtype=case["dtype"], rows=rows, bs=bs, rp=_up(rp), col=_up(col),
                val=_up(val).reshape(-1).to(t), W=_sweep_weights(case).to(t), x=x.to(t),
                b=b.to(t), out=torch.empty(rows * bs, dtype=t, device=DEV))


def _prepare_vcycle(case, seed):
    h = Hierarchy(_case_problem(case))
    st = dict(kind="vcycle", h=h, precision=PRECISION[case["precision"]],
              single=case["precision"] != "fp64", r=_normal(seed, h.n),
              z=torch.empty(h.n, dtype=torch.float64, device=DEV))
    torch.cuda.synchronize()
    return st


def _prepare_solve(case, seed):
    h = Hierarchy(_case_problem(case))
    return dict(kind="solve", h=h, precision=PRECISION[case["precision"]],
                b=_normal(seed, h.n).cpu().numpy(), x=np.empty(h.n))


def _setup_problem(case, seed):
    # another seed is another mesh: the operator is this call's input
    return _case_problem(case, configs.SEED + int(seed) % 1000)


def _prepare_setup(case, seed):
    pr = _setup_problem(case, seed)
    h = Hierarchy.__new__(Hierarchy)
    h.stream = torch.cuda.Stream()
    h.ctx = gasa.gasa_create(0, h.stream)
    st = dict(kind="setup", pr=pr, h=h, precision=PRECISION[case["precision"]],
              A=(_up(pr.A.row_ptr), _up(pr.A.col), _up(pr.A.val).reshape(-1)),
              b=_normal(seed, pr.n_dofs), z=torch.empty(pr.n_dofs, dtype=torch.float64, device=DEV),
              x=torch.empty(pr.n_dofs, dtype=torch.float64, device=DEV))
    torch.cuda.synchronize()
    return st


class Server:
    """A request server with three resident meshes."""

    def __init__(self, problems):
        self.hierarchies = [Hierarchy(pr) for pr in problems]
        self.srv = gasa.gasa_server_create(0, 40 << 30, 8)
        self.ids = [gasa.gasa_server_add_mesh(self.srv, h.ctx) for h in self.hierarchies]

    def __del__(self):
        if getattr(self, "srv", None) is not None:
            gasa.gasa_server_destroy(self.srv)
            self.srv = None


def _serve_rhs(case, seed):
    """Right-hand sides per mesh: request i goes to mesh i mod 3."""
    out = []
    for j, spec in enumerate(_serve_specs(case)):
        n = _problem(*spec, configs.SEED).n_dofs
        count = len(range(j, case["requests"], 3))
        out.append(_normal(seed, max(count, 1) * n, 10 + j).reshape(-1, n)[:count].cpu().numpy())
    return out


def _prepare_serve(case, seed):
    srv = Server([_problem(*spec, configs.SEED) for spec in _serve_specs(case)])
    rhs = _serve_rhs(case, seed)
    return dict(kind="serve", srv=srv, precision=PRECISION[case["precision"]], rhs=rhs,
                requests=case["requests"], x=[np.empty_like(b) for b in rhs])


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    return globals()["_run_" + st["kind"]](st)


def _run_product(st):
    if st["dtype"] == "ds":
        gasa.gasa_bsr_mv_ds(st["rows"], st["br"], st["bc"], st["rp"], st["col"], st["ahi"],
                            st["alo"], st["xhi"], st["xlo"], st["y"])
        return st["y"]
    y = st["y"]
    if st["adds"]:
        y.copy_(st["b"])          # the correction u += P e starts from the smoothed u
    f = gasa.gasa_bsr_mv_f32 if st["dtype"] == "fp32" else gasa.gasa_bsr_mv
    f(st["mode"], st["rows"], st["br"], st["bc"], st["rp"], st["col"], st["val"], st["x"],
      st["b"], y)
    return y


def _run_sweep(st):
    f = gasa.gasa_jacobi_sweep_f32 if st["dtype"] == "fp32" else gasa.gasa_jacobi_sweep
    f(st["rows"], st["bs"], st["rp"], st["col"], st["val"], st["W"], st["x"], st["b"], st["out"])
    return st["out"]


def _run_vcycle(st):
    with torch.cuda.stream(st["h"].stream):
        gasa.gasa_vcycle(st["h"].ctx, st["r"], st["z"], st["precision"])
        # the FP32 V-cycle's result is an FP32 vector widened to FP64; a flexible Krylov
        # method keeps it in FP32, as the library's own does (exact)
        return st["z"].float() if st["single"] else st["z"]


def _run_solve(st):
    gasa.gasa_solve(st["h"].ctx, st["b"], st["x"], TOL, st["precision"])
    return st["x"]


def _run_setup(st):
    h, pr = st["h"], st["pr"]
    with torch.cuda.stream(h.stream):
        info = h.setup(pr, st["A"])
        gasa.gasa_vcycle(h.ctx, st["b"], st["z"], gasa.GASA_PREC_FP64)
        gasa.gasa_solve(h.ctx, st["b"], st["x"], TOL, st["precision"], on_device=True)
        return {"x": st["x"], "z": st["z"], "omega": np.array(info.omega[:info.n_levels - 1])}


def _run_serve(st):
    srv, seen = st["srv"], [0, 0, 0]
    tickets = []
    for i in range(st["requests"]):
        j = i % 3
        tickets.append((gasa.gasa_server_submit(srv.srv, srv.ids[j], st["rhs"][j][seen[j]], TOL,
                                                st["precision"]), j, seen[j]))
        seen[j] += 1
    gasa.gasa_server_drain(srv.srv, 60.0)
    for t, j, k in tickets:
        status, _ = gasa.gasa_server_poll(srv.srv, t, st["x"][j][k])
        if status != gasa.GASA_OK:
            raise RuntimeError(f"request ended with status {status}")
    return st["x"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("product", "sweep"):
        rp, col, val, cols = _case_operator(case)
        rows, (br, bc) = len(rp) - 1, val.shape[1:]
        w = 4 if case["dtype"] == "fp32" else 8      # ds: two 4-byte words per value
        extra = {"assign": 0, "residual": 1, "add": 1}.get(case.get("mode"), 0)
        nbytes = col.size * (br * bc * w + 4) + 4 * len(rp) + cols * bc * w
        nbytes += rows * br * w * (1 + extra)
        flops = 2.0 * val.size
        if kind == "sweep":
            nbytes += rows * br * br * w + rows * br * w
            flops += 2.0 * rows * br * br
        return {"bytes": float(nbytes), "flops": flops}
    if kind == "serve":
        nbytes = flops = 0.0
        for j, spec in enumerate(_serve_specs(case)):
            values, n, _, it = _level_work(*spec, solve=True)
            q = len(range(j, case["requests"], 3))
            nbytes += it * math.ceil(q / 8) * values * (8 if case["precision"] == "fp64" else 4)
            nbytes += q * n * 16
            flops += 2.0 * it * q * values
        return {"bytes": nbytes, "flops": flops}
    values, n, a0, it = _level_work(case["mesh"], case["n"], case["p"], case["r"], case["pe"],
                                    solve=kind != "vcycle")
    w = {"fp64": 8, "mixed32": 4, "mixed16": 4}[case["precision"]]
    nbytes = values * w - (2 * a0 if case["precision"] == "mixed16" else 0)
    if kind == "vcycle":                             # every matrix of the cycle once, r and z
        return {"bytes": float(nbytes + 16 * n), "flops": 2.0 * values}
    solve = it * (nbytes + 8 * a0)                   # and A_0 in FP64 or its two words
    if kind == "solve":
        return {"bytes": float(solve + 16 * n), "flops": 2.0 * it * (values + a0)}
    return {"bytes": float(solve + 8 * (values + a0 + n * case["r"])),
            "flops": 2.0 * (it * (values + a0) + 10.0 * a0 * case["r"])}


# ---------------------------------------------------------------------------
# the same outputs in plain 64-bit torch
# ---------------------------------------------------------------------------
def _mv(op, x):
    """BSR product in FP64, in pieces of block entries that fit beside the rest."""
    rp, col, val = op[:3]
    rows, br, bc = rp.numel() - 1, val.shape[1], val.shape[2]
    y = torch.zeros(rows, br, dtype=torch.float64, device=DEV)
    row = torch.repeat_interleave(torch.arange(rows, device=DEV), (rp[1:] - rp[:-1]).long())
    xb = x.reshape(-1, bc)
    step = max(1, (1 << 26) // (br * bc))
    for k in range(0, col.numel(), step):
        part = torch.bmm(val[k:k + step], xb[col[k:k + step].long()].unsqueeze(2)).squeeze(2)
        y.index_add_(0, row[k:k + step], part)
    return y.reshape(-1)


def _banded_solve(pr, b):
    """A x = b by block elimination over runs of elements as long as the bandwidth, with one
    step of refinement; None where the blocks are too large to do quickly. b: dofs x k."""
    A = pr.A
    rows = np.repeat(np.arange(A.n), np.diff(A.row_ptr))
    run_ = int(np.abs(rows - A.col).max())
    if run_ * A.b > 5000:
        return None
    starts = list(range(0, A.n, run_))
    part = rows // run_
    blocks = {}
    val = _up(A.val)
    for i in range(len(starts)):
        ki = np.flatnonzero(part == i)
        for j in (i - 1, i, i + 1):
            k = ki[A.col[ki] // run_ == j]
            if k.size:
                h, w = min(run_, A.n - i * run_), min(run_, A.n - j * run_)
                D = torch.zeros(h, A.b, w, A.b, dtype=torch.float64, device=DEV)
                D[_up(rows[k] - i * run_), :, _up(A.col[k].astype(np.int64) - j * run_), :] = val[_up(k)]
                blocks[i, j] = D.reshape(h * A.b, w * A.b)
    op = (_up(A.row_ptr), _up(A.col), val)
    lu, low = [], []
    for i in range(len(starts)):
        D = blocks[i, i]
        if i:
            low.append(torch.linalg.lu_solve(*lu[-1], blocks[i, i - 1], left=False))
            D = D - low[-1] @ blocks[i - 1, i]
        lu.append(torch.linalg.lu_factor(D))

    def solve(v):
        ys = []
        for i, s in enumerate(starts):
            y = v[s * A.b:(s + run_) * A.b].clone()
            if i:
                y -= low[i - 1] @ ys[-1]
            ys.append(y)
        for i in reversed(range(len(starts))):
            if i + 1 < len(starts):
                ys[i] = ys[i] - blocks[i, i + 1] @ ys[i + 1]
            ys[i] = torch.linalg.lu_solve(*lu[i], ys[i])
        return torch.cat(ys)

    x = solve(b)
    res = b - torch.stack([_mv(op, x[:, c]) for c in range(b.shape[1])], 1)
    return x + solve(res)


def _exact_vcycle(case, seed):
    """One V-cycle with three steps before and after on the levels that the set-up made."""
    h = Hierarchy(_case_problem(case))
    last = h.levels - 1
    A, P, R, W = [], [], [], []
    for k in range(h.levels):
        def bsr(which):
            rp, col, val, _ = _read_bsr(h, k, which)
            return _up(rp), _up(col), _up(val)
        A.append(bsr("A"))
        if k < last:
            P.append(bsr("P"))
            R.append(bsr("R"))
            sh = gasa.gasa_level_shape(h.ctx, k)
            w = np.empty(sh["units"] * sh["s"] ** 2)
            W.append(_up(gasa.gasa_get_level(h.ctx, k, gasa.GASA_LV_W, w)).reshape(-1, sh["s"], sh["s"]))
    rp, col, val = A[last]
    m, s = rp.numel() - 1, val.shape[1]
    dense = torch.zeros(m, s, m, s, dtype=torch.float64, device=DEV)
    row = torch.repeat_interleave(torch.arange(m, device=DEV), (rp[1:] - rp[:-1]).long())
    dense[row, :, col.long(), :] = val

    def smooth(k, x, b):
        res = b - _mv(A[k], x)
        return x + torch.bmm(W[k], res.reshape(-1, W[k].shape[1], 1)).reshape(-1)

    def cycle(k, b):
        if k == last:
            return torch.linalg.solve(dense.reshape(m * s, m * s), b)
        x = torch.zeros_like(b)
        for _ in range(3):
            x = smooth(k, x, b)
        x = x + _mv(P[k], cycle(k + 1, _mv(R[k], b - _mv(A[k], x))))
        for _ in range(3):
            x = smooth(k, x, b)
        return x

    return cycle(0, _normal(seed, h.n))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("product", "sweep"):
        rp, col, val, x, b, rows, br, _ = _product_inputs(case, seed)
        v = _up(val)
        if case["dtype"] == "fp32":
            v = v.float().double()
        ax = _mv((_up(rp), _up(col), v), x)
        if kind == "sweep":
            W = _sweep_weights(case)
            if case["dtype"] == "fp32":
                W = W.float().double()
            return x + torch.bmm(W.reshape(rows, br, br), (b - ax).reshape(rows, br, 1)).reshape(-1)
        return {"assign": ax, "residual": b - ax, "add": b + ax}[case["mode"]]
    if kind == "vcycle":
        return _exact_vcycle(case, seed)
    if kind == "solve":
        pr = _case_problem(case)
        x = _banded_solve(pr, _normal(seed, pr.n_dofs).reshape(-1, 1))
        return None if x is None else x.reshape(-1)
    if kind == "setup":
        pr = _setup_problem(case, seed)
        x = _banded_solve(pr, _normal(seed, pr.n_dofs).reshape(-1, 1))
        return {"x": None if x is None else x.reshape(-1), "z": None, "omega": None}
    out = []
    for spec, b in zip(_serve_specs(case), _serve_rhs(case, seed)):
        x = _banded_solve(_problem(*spec, configs.SEED), _up(b.T.copy())) if b.size else None
        out.append(None if x is None else x.T.contiguous())
    return out
