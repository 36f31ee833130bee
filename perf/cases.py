"""Performance cases of the library: the calls its users make, over the range of sizes they make them at.

A case is a dict of plain values; ``prepare`` builds seeded inputs and the plan or network on the GPU, ``run``
makes one pass through the public entry points, ``work`` counts the bytes and operations the pass cannot do
without and ``exact`` gives the same outputs from FP64 torch.  The paths:

  single      one problem: Schur blocks, preconditioner, solve (FP32, or the FP64 path)
  pipeline    a ragged batch from QP data to lambda, launched directly or replayed as a captured graph
  host        the same from pinned host buffers
  resolve     the re-solve of a control loop: held blocks, a perturbed right-hand side, the previous solution
  noalloc     the allocation-free batched solve of a real-time loop
  full        full SPD cost blocks: Schur build, preconditioner, block-form solve
  build       Schur and preconditioner blocks of a batch
  step        right-hand side, primal step and true residual around a solve
  infer       warm-start network inference
  train       one training step of the warm-start network

Problems follow the repository's generators: A = I + h N(0, 1/nx), B = h N(0, 1), diag Q ~ U[0.1, 10],
diag R ~ U[0.1, 1], gamma ~ N(0, 1), nu = ceil(nx / 2).  The shapes of a batch come from the case alone
(``shapes``), the values from the seed.  A solve returns lambda, the iteration counts and the status codes;
its relres, the recurrence residual's norm at exit, restates the tolerance and is not returned.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2309_06427_gb300 import sspcg

DEV = "cuda"
KINDS = (sspcg.ARRAY_A, sspcg.ARRAY_B, sspcg.ARRAY_QD, sspcg.ARRAY_RD, sspcg.ARRAY_DIAG, sspcg.ARRAY_OFF,
         sspcg.ARRAY_VEC, sspcg.ARRAY_RFULL)
MLP_SHAPES = ((256, 1344), (256,), (256, 256), (256,), (32, 256), (32,))


def listed():
    return [
        {"name": "single nx2 N20 fp64", "path": "single", "N": 20, "nx": 2, "h": 0.05, "tol": 1e-8, "f64": True},
        {"name": "single nx14 N64", "path": "single", "N": 64, "nx": 14, "h": 0.01, "tol": 1e-6, "f64": False},
        {"name": "ragged batch 4096", "path": "pipeline", "nprob": 4096, "N_lo": 16, "N_hi": 128, "nx": "4,12,14,21",
         "h": 0.05, "tol": 1e-6, "shapes": 3, "graph": False, "kind": "sym"},
        {"name": "small batch 16384 graph", "path": "pipeline", "nprob": 16384, "N_lo": 8, "N_hi": 32, "nx": "2,4,6",
         "h": 0.05, "tol": 1e-6, "shapes": 6, "graph": True, "kind": "sym"},
        {"name": "host batch 512", "path": "host", "nprob": 512, "N_lo": 16, "N_hi": 128, "nx": "4,12,14,21",
         "h": 0.05, "tol": 1e-6, "shapes": 3, "kind": "sym"},
        {"name": "mpc resolve 1024", "path": "resolve", "nprob": 1024, "N_lo": 64, "N_hi": 512, "nx": "4-28",
         "h": 0.05, "tol": 1e-6, "shapes": 5},
        {"name": "noalloc 64 nx12 N32", "path": "noalloc", "nprob": 64, "N_lo": 32, "N_hi": 32, "nx": "12", "h": 0.05,
         "tol": 1e-6, "shapes": 7},
        {"name": "full cost 1024", "path": "full", "nprob": 1024, "N_lo": 16, "N_hi": 128, "nx": "4,12,14,21",
         "h": 0.05, "tol": 1e-6, "shapes": 3},
        {"name": "build 4096", "path": "build", "nprob": 4096, "N_lo": 16, "N_hi": 128, "nx": "4,12,14,21", "h": 0.05,
         "shapes": 3, "kind": "sym"},
        {"name": "kkt step 4096", "path": "step", "nprob": 4096, "N_lo": 16, "N_hi": 128, "nx": "4,12,14,21",
         "h": 0.05, "shapes": 3},
        {"name": "infer 4096 nx14 N64", "path": "infer", "nprob": 4096, "N_lo": 64, "N_hi": 64, "nx": "14", "h": 0.01,
         "shapes": 4},
        {"name": "train step 32", "path": "train", "nprob": 32, "N_lo": 64, "N_hi": 64, "nx": "14", "h": 0.01,
         "shapes": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["single", "single", "pipeline", "pipeline", "host", "resolve", "noalloc", "full", "build",
                       "step", "infer", "train"])
    if path == "single":
        if rng.random() < 0.4:
            return {"path": path, "N": _log_int(rng, 5, 60), "nx": rng.randint(1, 8), "h": 0.05, "tol": 1e-8,
                    "f64": True}
        nx = rng.randint(2, 28)
        return {"path": path, "N": _log_int(rng, max(8, 200 // nx), min(256, 4000 // nx)), "nx": nx,
                "h": rng.choice([0.01, 0.05]), "tol": 1e-6, "f64": False}
    lo = _log_int(rng, 4, 64)
    hi = lo + rng.randint(0, 64)
    nx = rng.choice(["4,12,14,21", "4-28", "%d" % rng.randint(2, 28), "%d,%d" % (rng.randint(2, 9), rng.randint(10, 28)),
                     "2,4,6"])
    c = {"path": path, "nprob": _log_int(rng, 16, 2048), "N_lo": lo, "N_hi": hi, "nx": nx, "h": 0.05,
         "shapes": rng.randint(100, 10 ** 6)}
    if path in ("pipeline", "host", "build"):
        c["kind"] = rng.choice(["sym", "sym", "sym", "add", "bj"])
    if path == "pipeline":
        c["graph"] = rng.random() < 0.5
    if path == "host":
        c["nprob"] = _log_int(rng, 8, 512)
    if path == "resolve":
        c["nprob"] = _log_int(rng, 16, 512)
        c["N_lo"], c["N_hi"] = 2 * lo, 2 * hi + rng.randint(0, 200)
    if path == "noalloc":
        c["nprob"] = _log_int(rng, 1, 256)
    if path == "full":
        c["nprob"] = _log_int(rng, 16, 512)
    if path == "train":
        c["nprob"] = rng.randint(4, 64)
    # no more work than the ragged batch of 4096
    N, m, _ = _shapes(c)
    most = 4096 * 73.0 * 200.0
    c["nprob"] = max(1, int(c["nprob"] * min(1.0, most / float(((N + 1.0) * m * m).sum()))))
    if path not in ("build", "step", "infer", "train"):
        c["tol"] = 1e-6
    return c


# ---------------------------------------------------------------------------
# Shapes, packed arrays
# ---------------------------------------------------------------------------
def _nu(nx):
    return (nx + 1) // 2


def _shapes(case):
    """(N, nx, nu) arrays of the case's problems: a function of the case alone."""
    if case["path"] == "single":
        return np.array([case["N"]]), np.array([case["nx"]]), np.array([_nu(case["nx"])])
    r = np.random.RandomState(case["shapes"])
    n = case["nprob"]
    if "-" in case["nx"]:
        lo, hi = (int(v) for v in case["nx"].split("-"))
        nx = r.randint(lo, hi + 1, n)
    else:
        nx = np.array([int(v) for v in case["nx"].split(",")])[r.randint(0, len(case["nx"].split(",")), n)]
    N = r.randint(case["N_lo"], case["N_hi"] + 1, n)
    return N, nx, (nx + 1) // 2


def _blocks(kind, N, nx, nu):
    """(blocks of a problem, shape of a block) of a packed array kind."""
    return {sspcg.ARRAY_A: (N, (nx, nx)), sspcg.ARRAY_B: (N, (nx, nu)), sspcg.ARRAY_QD: (N + 1, (nx,)),
            sspcg.ARRAY_RD: (N, (nu,)), sspcg.ARRAY_DIAG: (N + 1, (nx, nx)), sspcg.ARRAY_OFF: (N, (nx, nx)),
            sspcg.ARRAY_VEC: (N + 1, (nx,)), sspcg.ARRAY_RFULL: (N, (nu, nu))}[kind]


class Layout:
    """The packed arrays of a batch: every problem starts at a multiple of four values, in problem order.  One
    group of problems per nx; a group's blocks, problem by problem, are one tensor."""

    def __init__(self, N, nx, nu):
        self.N, self.nx, self.nu = N, nx, nu
        self.size, self.offs = {}, {}
        for kind in KINDS:
            blocks, shape = _blocks(kind, N.astype(np.int64), nx, nu)
            r4 = (blocks * math.prod(shape) + 3) // 4 * 4
            self.offs[kind] = np.concatenate([[0], np.cumsum(r4)[:-1]])
            self.size[kind] = max(int(r4.sum()), 4)
        self.groups = [(int(m), np.flatnonzero(nx == m)) for m in np.unique(nx)]
        self._idx = {}

    def index(self, kind, m, ids):
        """Positions of the group's values in the packed array, as [blocks, block shape]."""
        if (kind, m) not in self._idx:
            u = _nu(m)
            blocks, shape = _blocks(kind, self.N[ids].astype(np.int64), m, u)
            cnt = blocks * math.prod(shape)
            start = np.cumsum(cnt) - cnt
            at = torch.arange(int(cnt.sum()), device=DEV)
            shift = torch.repeat_interleave(torch.from_numpy(self.offs[kind][ids] - start).to(DEV),
                                            torch.from_numpy(cnt).to(DEV))
            self._idx[kind, m] = (at + shift).reshape(-1, *shape)
        return self._idx[kind, m]

    def pack(self, kind, parts, fill=0.0):
        """parts: one tensor per group, in the order of ``groups``."""
        flat = torch.full((self.size[kind],), fill, device=DEV, dtype=parts[0].dtype)
        for (m, ids), t in zip(self.groups, parts):
            flat[self.index(kind, m, ids).reshape(-1)] = t.reshape(-1)
        return flat

    def unpack(self, kind, flat):
        return [flat[self.index(kind, m, ids)] for m, ids in self.groups]

    def empty(self, kind, dtype=torch.float32):
        return torch.zeros(self.size[kind], dtype=dtype, device=DEV)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _inputs(case, seed):
    """The layout and the packed QP data of a case."""
    L = Layout(*_shapes(case))
    g, h = _gen(seed), case["h"]
    rows = {k: [] for k in ("A", "B", "qd", "rd", "gamma")}
    for m, ids in L.groups:
        u, n = _nu(m), int((L.N[ids]).sum())
        k = n + len(ids)
        rows["A"].append(torch.eye(m, device=DEV) + h / math.sqrt(m) * torch.randn(n, m, m, generator=g, device=DEV))
        rows["B"].append(h * torch.randn(n, m, u, generator=g, device=DEV))
        rows["qd"].append(0.1 + 9.9 * torch.rand(k, m, generator=g, device=DEV))
        rows["rd"].append(0.1 + 0.9 * torch.rand(n, u, generator=g, device=DEV))
        rows["gamma"].append(torch.randn(k, m, generator=g, device=DEV))
    kinds = {"A": sspcg.ARRAY_A, "B": sspcg.ARRAY_B, "qd": sspcg.ARRAY_QD, "rd": sspcg.ARRAY_RD,
             "gamma": sspcg.ARRAY_VEC}
    data = {n: L.pack(kinds[n], rows[n], 1.0 if n in ("qd", "rd") else 0.0) for n in rows}
    return L, data, g


def _full_cost(L, data, g):
    """Full SPD cost blocks Q = diag(qd) + M M^T / nx, R = diag(rd) + W W^T / nu."""
    Q, R = [], []
    qd, rd = L.unpack(sspcg.ARRAY_QD, data["qd"]), L.unpack(sspcg.ARRAY_RD, data["rd"])
    for a, b in zip(qd, rd):
        for out, d in ((Q, a), (R, b)):
            m = torch.randn(d.shape[0], d.shape[1], d.shape[1], generator=g, device=DEV)
            s = torch.diag_embed(d) + m @ m.transpose(1, 2) / d.shape[1]
            out.append((s + s.transpose(1, 2)) / 2)
    return L.pack(sspcg.ARRAY_DIAG, Q), L.pack(sspcg.ARRAY_RFULL, R)


def _plan(L, **kw):
    return sspcg.sspcg_plan_create(L.N, L.nx, L.nu, sspcg.options(**kw))


def _results(n, device=DEV, pin=False):
    mk = lambda dt: torch.zeros(n, dtype=dt, device=device, pin_memory=pin)
    return {"iters": mk(torch.int32), "relres": mk(torch.float64), "status": mk(torch.int32)}


def _work_blocks(L):
    return {"D": L.empty(sspcg.ARRAY_DIAG), "E": L.empty(sspcg.ARRAY_OFF), "PD": L.empty(sspcg.ARRAY_DIAG),
            "PE": L.empty(sspcg.ARRAY_OFF)}


def _network_params(g):
    """Flat FP32 parameters with weights ~ U(-1, 1) / sqrt(fan in) and small biases."""
    parts = []
    for s in MLP_SHAPES:
        scale = 1.0 / math.sqrt(s[1]) if len(s) == 2 else 0.05
        parts.append(((2 * torch.rand(s, generator=g, device=DEV) - 1) * scale).reshape(-1))
    return torch.cat(parts)


def _qp(d):
    return d["A"], d["B"], d["qd"], d["rd"]


def _out(d):
    return d["iters"], d["relres"], d["status"]


# ---------------------------------------------------------------------------
# prepare
# ---------------------------------------------------------------------------
def prepare(case, seed):
    path = case["path"]
    L, d, g = _inputs(case, seed)
    s = {"case": case, "path": path, **d}
    n = len(L.N)
    if path == "single":
        dt = torch.float64 if case["f64"] else torch.float32
        for k, kind in (("D", sspcg.ARRAY_DIAG), ("E", sspcg.ARRAY_OFF), ("PD", sspcg.ARRAY_DIAG),
                        ("PE", sspcg.ARRAY_OFF), ("lam", sspcg.ARRAY_VEC)):
            s[k] = L.empty(kind, dt)
        s["opts"] = sspcg.options(tol=case["tol"])
        s["shape"] = (int(L.N[0]), int(L.nx[0]), int(L.nu[0]))
        s["values"] = (s["shape"][0] + 1) * s["shape"][1]
        return {**s, **_results(1)}
    if path == "noalloc":
        plan = _plan(L, tol=case["tol"])
        s |= {"N": L.N, "nx": L.nx, "nu": L.nu, **_work_blocks(L), **_results(n), "lam": L.empty(sspcg.ARRAY_VEC)}
        sspcg.sspcg_build_schur_batched(plan, *_qp(s), s["D"], s["E"])
        sspcg.sspcg_build_precond_batched(plan, "sym", s["D"], s["E"], s["PD"], s["PE"], s["status"])
        s["opts"] = sspcg.options(tol=case["tol"])
        torch.cuda.synchronize()
        return s
    s["plan"] = plan = _plan(L, tol=case.get("tol", 1e-6), warm_start=2 if path == "resolve" else 0)
    if path == "host":
        for k in ("A", "B", "qd", "rd", "gamma"):
            s[k] = s[k].cpu().pin_memory()
        s["lam"] = torch.zeros(L.size[sspcg.ARRAY_VEC]).pin_memory()
        return {**s, **_results(n, "cpu", True)}
    if path == "step":
        s["c"], s["q"], s["mu"] = (torch.randn(L.size[sspcg.ARRAY_VEC], generator=g, device=DEV) for _ in range(3))
        s["r"] = torch.randn(L.size[sspcg.ARRAY_RD], generator=g, device=DEV)
        s["rhs"], s["dx"], s["du"] = L.empty(sspcg.ARRAY_VEC), L.empty(sspcg.ARRAY_VEC), L.empty(sspcg.ARRAY_RD)
        s["relres"] = torch.zeros(n, dtype=torch.float64, device=DEV)
        return s
    s |= {**_work_blocks(L), **_results(n), "lam": L.empty(sspcg.ARRAY_VEC)}
    if path == "full":
        s["Q"], s["R"] = _full_cost(L, d, g)
        s["status_build"] = torch.zeros_like(s["status"])
        return s
    if path == "build":
        return s
    if path == "pipeline":
        if case["graph"]:
            stream = torch.cuda.Stream()
            stream.wait_stream(torch.cuda.current_stream())
            sspcg.sspcg_plan_capture_pipeline(plan, case["kind"], *_qp(s), s["gamma"], s["D"], s["E"], s["PD"],
                                              s["PE"], s["lam"], *_out(s), stream)
            torch.cuda.synchronize()
        return s
    # the remaining paths hold the blocks of an earlier call
    sspcg.sspcg_build_schur_batched(plan, *_qp(s), s["D"], s["E"])
    sspcg.sspcg_build_precond_batched(plan, "sym", s["D"], s["E"], s["PD"], s["PE"], s["status"])
    if path in ("resolve", "train"):
        sspcg.sspcg_solve_qp_batched(plan, *_qp(s), s["PD"], s["PE"], s["gamma"], s["lam"], *_out(s))
    if path == "resolve":
        s["previous"] = s["lam"].clone()
        s["gamma"] = s["gamma"] * (1 + 0.01 * torch.randn(s["gamma"].shape, generator=g, device=DEV))
    if path in ("infer", "train"):
        s["net"] = sspcg.sspcg_mlp_create(int((L.N + 1).sum()))
        sspcg.sspcg_mlp_fit_normalisation(s["net"], plan, *_qp(s), s["gamma"], s["PD"])
        s["params"] = _network_params(g)
        sspcg.sspcg_mlp_set_params(s["net"], s["params"])
    if path == "train":
        s["hyper"] = sspcg.adam()
        s["loss"] = torch.zeros(1, dtype=torch.float64, device=DEV)
        s["grads"] = torch.zeros_like(s["params"])
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# run
# ---------------------------------------------------------------------------
def run(s):
    path = s["path"]
    if path == "single":
        (N, nx, nu), st = s["shape"], s["status"]
        if s["case"]["f64"]:
            sspcg.sspcg_build_schur_f64(N, nx, nu, *_qp(s), s["D"], s["E"])
            sspcg.sspcg_build_precond_f64(N, nx, "sym", s["D"], s["E"], s["PD"], s["PE"], st)
            sspcg.sspcg_solve_qp_f64(N, nx, nu, *_qp(s), s["PD"], s["PE"], s["gamma"], s["lam"], s["opts"], *_out(s))
        else:
            sspcg.sspcg_build_schur(N, nx, nu, *_qp(s), s["D"], s["E"])
            sspcg.sspcg_build_precond(N, nx, "sym", s["D"], s["E"], s["PD"], s["PE"], st)
            sspcg.sspcg_solve_qp(N, nx, nu, *_qp(s), s["PD"], s["PE"], s["gamma"], s["lam"], s["opts"], *_out(s))
        return {"lam": s["lam"][:s["values"]], "iters": s["iters"], "status": st}
    if path == "pipeline":
        if s["case"]["graph"]:
            sspcg.sspcg_plan_launch(s["plan"])
        else:
            sspcg.sspcg_pipeline_batched(s["plan"], s["case"]["kind"], *_qp(s), s["gamma"], s["D"], s["E"], s["PD"],
                                         s["PE"], s["lam"], *_out(s))
    elif path == "host":
        sspcg.sspcg_pipeline_host(s["plan"], s["case"]["kind"], *_qp(s), s["gamma"], s["lam"], *_out(s))
    elif path == "resolve":
        s["lam"].copy_(s["previous"])
        sspcg.sspcg_solve_qp_batched(s["plan"], *_qp(s), s["PD"], s["PE"], s["gamma"], s["lam"], *_out(s))
    elif path == "noalloc":
        sspcg.sspcg_solve_qp_batched_noalloc(s["N"], s["nx"], s["nu"], *_qp(s), s["PD"], s["PE"], s["gamma"], s["lam"],
                                             s["opts"], *_out(s))
    elif path == "full":
        sspcg.sspcg_build_schur_full_batched(s["plan"], s["A"], s["B"], s["Q"], s["R"], s["D"], s["E"],
                                             s["status_build"])
        sspcg.sspcg_build_precond_batched(s["plan"], "sym", s["D"], s["E"], s["PD"], s["PE"], s["status"])
        sspcg.sspcg_solve_batched(s["plan"], s["D"], s["E"], s["PD"], s["PE"], s["gamma"], s["lam"], *_out(s))
        return {"D": s["D"], "E": s["E"], "lam": s["lam"], "iters": s["iters"], "status": s["status"],
                "status_build": s["status_build"]}
    elif path == "build":
        sspcg.sspcg_build_schur_batched(s["plan"], *_qp(s), s["D"], s["E"])
        sspcg.sspcg_build_precond_batched(s["plan"], s["case"]["kind"], s["D"], s["E"], s["PD"], s["PE"], s["status"])
        return {k: s[k] for k in ("D", "E", "PD", "PE", "status")}
    elif path == "step":
        sspcg.sspcg_form_gamma_batched(s["plan"], *_qp(s), s["c"], s["q"], s["r"], s["rhs"])
        sspcg.sspcg_recover_step_batched(s["plan"], *_qp(s), s["q"], s["r"], s["mu"], s["dx"], s["du"])
        sspcg.sspcg_residual_qp_batched(s["plan"], *_qp(s), s["rhs"], s["mu"], s["relres"])
        return {k: s[k] for k in ("rhs", "dx", "du", "relres")}
    elif path == "infer":
        sspcg.sspcg_mlp_infer(s["net"], s["plan"], *_qp(s), s["gamma"], s["PD"], s["lam"])
        return {"lam": s["lam"]}
    elif path == "train":
        sspcg.sspcg_mlp_train_step(s["net"], s["plan"], 0, s["plan"].nprob, *_qp(s), s["gamma"], s["D"], s["E"],
                                   s["PD"], s["lam"], s["hyper"], s["loss"])
        sspcg.sspcg_mlp_get_grads(s["net"], s["grads"])
        sspcg.sspcg_mlp_get_params(s["net"], s["params"])
        return {"loss": s["loss"], "grads": s["grads"], "params": s["params"]}
    return {"lam": s["lam"], "iters": s["iters"], "status": s["status"]}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _iterations(N, case):
    """Typical PCG iterations of the generators' problems (symmetric stair, tol 1e-6; measured means)."""
    it = 7.4 * np.sqrt(N + 1.0) * (2.8 if case["h"] < 0.03 else 1.0)
    return it * {"add": 1.2, "bj": 1.9}.get(case.get("kind"), 1.0) * (0.7 if case["path"] == "resolve" else 1.0)


def work(case):
    N, nx, nu = (v.astype(np.float64) for v in _shapes(case))
    path = case["path"]
    qp = (N * nx * nx + N * nx * nu + (N + 1) * nx + N * nu)  # A, B, diag Q, diag R
    vec, diag, off = (N + 1) * nx, (N + 1) * nx * nx, N * nx * nx
    schur = N * (nx * nx * (nx + nu))  # multiply-adds, the upper triangle counted twice over
    schur = 0.5 * schur + off + N * nx * nu
    inverse = (N + 1) * nx ** 3 / 2
    stair = 2 * N * nx ** 3 if case.get("kind", "sym") != "bj" else 0 * N
    solve = _iterations(N, case) * (2 * (off + N * nx * nu) + diag + 2 * off + 10 * vec)
    if path in ("single", "pipeline", "host"):
        b, f = qp + 2 * vec, schur + inverse + stair + solve
    elif path in ("resolve", "noalloc"):
        b, f = qp + diag + off + (3 if path == "resolve" else 2) * vec, solve
    elif path == "full":
        r = N * nu * nu
        full = (N + 1) * nx ** 3 / 2 + N * nu ** 3 / 2 + N * (nx ** 3 + nx * nu * nu + nx * nx * (nx + nu) / 2)
        b = N * nx * nx + N * nx * nu + diag + r + diag + off + 2 * vec
        f = full + inverse + stair + _iterations(N, case) * (2 * diag + 4 * off + 10 * vec)
    elif path == "build":
        b, f = qp + 2 * (diag + off), schur + inverse + stair
    elif path == "step":
        b, f = qp + 7 * vec + 2 * N * nu, 4 * (off + N * nx * nu)
    else:
        rows = (N + 1)
        net = rows * (1344 * 256 + 256 * 256 + 256 * 32)
        if path == "infer":
            b, f = qp + 2 * vec + diag + 418336 / len(N), net
        else:
            b, f = qp + 2 * vec + 2 * diag + off + 10 * 418336 / len(N), 3 * net + 4 * (diag + 2 * off)
    return {"bytes": 4.0 * float(b.sum()), "flops": 2.0 * float(f.sum())}


# ---------------------------------------------------------------------------
# exact: the same outputs in FP64 torch
# ---------------------------------------------------------------------------
def _starts(N):
    """Index of each block row k >= 1 of the problems among the group's block rows, problem by problem."""
    kn, first = [], 0
    for n in N:
        kn.append(first + np.arange(1, n + 1))
        first += n + 1
    return torch.from_numpy(np.concatenate(kn)).to(DEV)


def _schur64(A, B, Qi, Ri, later):
    """FP64 Schur blocks (D, E) of a group: A, B per off-diagonal block, Qi, Ri inverse cost blocks (matrices);
    later: knot index of each off-diagonal block's row."""
    D, AQ = Qi.clone(), A @ Qi[later - 1]
    D[later] += AQ @ A.transpose(1, 2) + (B @ Ri) @ B.transpose(1, 2)
    return D, -AQ


def _solve64(D, E, gamma, N):
    """Block-tridiagonal solve of every problem of a group (block Thomas, problems side by side)."""
    P, m, top = len(N), D.shape[1], int(max(N)) + 1
    first = np.concatenate([[0], np.cumsum(N + 1)[:-1]])
    eye = torch.eye(m, dtype=torch.float64, device=DEV)
    n = torch.from_numpy(N).to(DEV)
    at, ae = torch.from_numpy(first).to(DEV), torch.from_numpy(first - np.arange(P)).to(DEV)
    kept, y, prev = [], [], None
    for k in range(top):
        has, hase = (k <= n), ((k <= n) & (k > 0))
        d = torch.where(has[:, None, None], D[torch.where(has, at + k, 0)], eye)
        g = torch.where(has[:, None], gamma[torch.where(has, at + k, 0)], 0.0)
        if k:
            e = torch.where(hase[:, None, None], E[torch.where(hase, ae + k - 1, 0)], 0.0)
            w = torch.cholesky_solve(e.transpose(1, 2), prev).transpose(1, 2)  # E D'^-1
            d, g = d - w @ e.transpose(1, 2), g - (w @ y[-1][:, :, None])[:, :, 0]
            kept[-1] = (kept[-1], e)
        prev = torch.linalg.cholesky(d)
        kept.append(prev)
        y.append(g)
    x = [None] * top
    for k in range(top - 1, -1, -1):
        c, rhs = (kept[k][0], y[k]) if k < top - 1 else (kept[k], y[k])
        if k < top - 1:
            rhs = rhs - (kept[k][1].transpose(1, 2) @ x[k + 1][:, :, None])[:, :, 0]
        x[k] = torch.cholesky_solve(rhs[:, :, None], c)[:, :, 0]
    return torch.stack(x, 1)[torch.arange(top, device=DEV)[None, :] <= n[:, None]]


def _features64(A, B, qd, rd, gamma, dj, later, m, u, k):
    """The network's raw feature rows of a group (column layout of sspcg_mlp_features)."""
    X = torch.zeros(k, 1344, dtype=torch.float64, device=DEV)
    a = torch.zeros(len(later), 28, 28, dtype=torch.float64, device=DEV)
    a[:, :m, :m] = A
    b = torch.zeros(len(later), 28, 14, dtype=torch.float64, device=DEV)
    b[:, :m, :u] = B
    X[later, :784], X[later, 784:1176] = a.reshape(-1, 784), b.reshape(-1, 392)
    X[later, 1176:1176 + m], X[later, 1204:1204 + u] = qd[later - 1], rd
    X[:, 1218:1218 + m], X[:, 1246:1246 + m], X[:, 1274:1274 + m] = qd, gamma, dj
    X[:, 1302] = m / 28
    return X


def exact(case, seed):
    path = case["path"]
    L, d, g = _inputs(case, seed)
    if path == "resolve" and case["nprob"] * case["N_hi"] > 600000:
        return None
    un = lambda kind, t: [v.double() for v in L.unpack(kind, t)]
    A, B = un(sspcg.ARRAY_A, d["A"]), un(sspcg.ARRAY_B, d["B"])
    qd, rd, gamma = un(sspcg.ARRAY_QD, d["qd"]), un(sspcg.ARRAY_RD, d["rd"]), un(sspcg.ARRAY_VEC, d["gamma"])
    Ns = [L.N[ids] for _, ids in L.groups]
    later = [_starts(N) for N in Ns]
    if path == "step":
        c, q, mu = (un(sspcg.ARRAY_VEC, torch.randn(L.size[sspcg.ARRAY_VEC], generator=g, device=DEV)) for _ in range(3))
        r = un(sspcg.ARRAY_RD, torch.randn(L.size[sspcg.ARRAY_RD], generator=g, device=DEV))
        rhs, dx, du = [], [], []
        mv = lambda M, x: (M @ x[:, :, None])[:, :, 0]
        for i, at in enumerate(later):
            s = c[i] + q[i] / qd[i]
            s[at] -= mv(A[i], q[i][at - 1] / qd[i][at - 1]) + mv(B[i], r[i] / rd[i])
            t = q[i] - mu[i]
            t[at - 1] += mv(A[i].transpose(1, 2), mu[i][at])
            rhs.append(s)
            dx.append(t / qd[i])
            du.append((r[i] + mv(B[i].transpose(1, 2), mu[i][at])) / rd[i])
        # the residual norm is taken of the FP32 right-hand side the call was given: no value here
        return {"rhs": L.pack(sspcg.ARRAY_VEC, rhs), "dx": L.pack(sspcg.ARRAY_VEC, dx),
                "du": L.pack(sspcg.ARRAY_RD, du), "relres": None}
    if path == "full":
        Qf, Rf = _full_cost(L, d, g)
        Qi = [torch.linalg.inv(v) for v in un(sspcg.ARRAY_DIAG, Qf)]
        Ri = [torch.linalg.inv(v) for v in un(sspcg.ARRAY_RFULL, Rf)]
    else:
        Qi, Ri = [torch.diag_embed(1 / v) for v in qd], [torch.diag_embed(1 / v) for v in rd]
    DE = [_schur64(*v) for v in zip(A, B, Qi, Ri, later)]
    if path in ("build", "infer", "train"):
        PD = [torch.linalg.inv(D) for D, _ in DE]
    if path == "build":
        c = {"sym": 1.0, "add": 0.5, "bj": 0.0}[case["kind"]]
        PE = [-c * P[at] @ E @ P[at - 1] for P, (_, E), at in zip(PD, DE, later)]
        return {"D": L.pack(sspcg.ARRAY_DIAG, [D for D, _ in DE]), "E": L.pack(sspcg.ARRAY_OFF, [E for _, E in DE]),
                "PD": L.pack(sspcg.ARRAY_DIAG, PD), "PE": L.pack(sspcg.ARRAY_OFF, PE), "status": None}
    if path in ("infer", "train"):
        X = []
        for i, (m, ids) in enumerate(L.groups):
            dj = (PD[i] @ gamma[i][:, :, None])[:, :, 0]
            X.append(_features64(A[i], B[i], qd[i], rd[i], gamma[i], dj, later[i], m, _nu(m), len(dj)))
        rows = sum(len(x) for x in X)
        mean = sum(x.sum(0) for x in X) / rows
        ms = sum(x.square().sum(0) for x in X) / rows
        var = sum((x - mean).square().sum(0) for x in X) / rows
        inv = torch.where(var.sqrt() <= 1e-6 * ms.sqrt(), 0.0, 1 / var.sqrt().clamp_min(1e-300))
        flat = _network_params(g).double()
        if path == "train":
            flat.requires_grad_(True)
        W, at = [], 0
        for sh in MLP_SHAPES:
            n = int(np.prod(sh))
            W.append(flat[at:at + n].reshape(sh))
            at += n
        Y = []
        for x in X:
            x = (x - mean) * inv
            x = torch.relu(x @ W[0].T + W[1])
            x = torch.relu(x @ W[2].T + W[3])
            Y.append(x @ W[4].T + W[5])
        Y = [y[:, :m] for y, (m, _) in zip(Y, L.groups)]
        if path == "infer":
            return {"lam": L.pack(sspcg.ARRAY_VEC, Y)}
        loss = 0.0
        for y, (D, E), gm, at, N in zip(Y, DE, gamma, later, Ns):
            mv = lambda M, x: (M @ x[:, :, None])[:, :, 0]
            low = torch.zeros_like(y).index_add(0, at, mv(E, y[at - 1]))
            up = torch.zeros_like(y).index_add(0, at - 1, mv(E.transpose(1, 2), y[at]))
            u = mv(D, y) + low + up - gm
            owner = torch.repeat_interleave(torch.arange(len(N), device=DEV), torch.from_numpy(N + 1).to(DEV))
            tot = lambda v: torch.zeros(len(N), dtype=torch.float64, device=DEV).index_add(0, owner, v.square().sum(1))
            loss = loss + (tot(u) / tot(gm)).sum()
        loss = loss / len(L.N)
        grads, = torch.autograd.grad(loss, flat)
        return {"loss": loss.detach().reshape(1), "grads": grads, "params": None}
    if path == "resolve":
        gp = d["gamma"] * (1 + 0.01 * torch.randn(d["gamma"].shape, generator=g, device=DEV))
        gamma = un(sspcg.ARRAY_VEC, gp)
    lam = L.pack(sspcg.ARRAY_VEC, [_solve64(D, E, gm, N) for (D, E), gm, N in zip(DE, gamma, Ns)])
    if path == "single":
        lam = lam[:(int(L.N[0]) + 1) * int(L.nx[0])]
    if path == "full":
        return {"D": L.pack(sspcg.ARRAY_DIAG, [D for D, _ in DE]), "E": L.pack(sspcg.ARRAY_OFF, [E for _, E in DE]),
                "lam": lam, "iters": None, "status": None, "status_build": None}
    return {"lam": lam, "iters": None, "status": None}
