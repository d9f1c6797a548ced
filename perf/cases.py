"""The calls a user of the library makes, as measurable cases.

Each case is one pass through the public entry points of
``paper_2006_16147_gb300.amg``: a solve on a hierarchy that is kept, a time
step that builds the hierarchy anew and solves once, a block solve of several
right-hand sides, a batch of independent systems, and the solve server. The
matrices are the model problems of the repository (7-point Poisson, jump
coefficients, 2D anisotropy), assembled on the GPU.

Right-hand sides are either b = A x* with x* ~ U[-1, 1] ("uniform") or N(0, 1)
entries ("normal"); the solution of the first kind is x* itself, of the second
(constant coefficients only) it comes from sine transforms in 64 bits.
"""
import math
import random

import torch

from paper_2006_16147_gb300 import amg, workloads

DEV = "cuda"
VA3 = dict(smooth_p=1, pre=4, post=4, omega_rule=1)


def listed():
    return [
        # the smallest call: one solve on a cached hierarchy, all launch latency
        dict(name="solve_poisson_32", kind="solve", op="poisson", nx=32, ny=32, nz=32, fp32=False),
        # an implicit time step on a small odd box: setup and solve, latency and host reads
        dict(name="step_poisson_61x47x33", kind="step", op="poisson", nx=61, ny=47, nz=33, fp32=False),
        # the paper's cycle for this aggregation: the K-cycle on every intermediate level
        dict(name="solve_kcycle_101x96x83", kind="solve", op="poisson", nx=101, ny=96, nz=83, fp32=False, cycle=32),
        # a served 2D anisotropic operator
        dict(name="solve_aniso2d_2048", kind="solve", op="aniso2d", nx=2048, ny=2048, nz=1, fp32=False),
        # a served 3D operator with the FP32 V-cycle
        dict(name="solve_fp32_poisson_192", kind="solve", op="poisson", nx=192, ny=192, nz=192, fp32=True),
        # the headline: hierarchy and solution of a 16.8M-unknown system
        dict(name="step_poisson_256", kind="step", op="poisson", nx=256, ny=256, nz=256, fp32=False),
        # jump coefficients (stalled coarsening, iterative coarsest level), flexible CG
        dict(name="step_fp32_varcoef_256", kind="step", op="varcoef", nx=256, ny=256, nz=256, fp32=True),
        # the paper's GPU setting: smoothed prolongator, l1-Jacobi 4+4
        dict(name="step_va3_poisson_128", kind="step", op="poisson", nx=128, ny=128, nz=128, fp32=False, va3=True),
        # many load cases of one operator
        dict(name="block_fp32_poisson_128x64", kind="block", op="poisson", nx=128, ny=128, nz=128, k=64, fp32=True),
        # a few load cases on an odd box, FP64
        dict(name="block_poisson_75x64x49x7", kind="block", op="poisson", nx=75, ny=64, nz=49, k=7, fp32=False),
        # 256 independent systems of uneven size
        dict(name="many_256_systems", kind="many", m=256, lo=16, hi=64, fp32=False),
        # the solve server: requests of 1 to 16 columns over three resident operators, host to host
        dict(name="serve_3_operators", kind="serve", requests=12, kmax=16, edge=64, fp32=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """Three edges around one log-uniform size, odd ones as likely as even ones."""
    e = _log(rng, lo, hi)
    near = lambda: max(lo, min(hi, int(round(e * rng.uniform(0.75, 1.25)))))  # noqa: E731
    return dict(nx=near(), ny=near(), nz=near())


def draw(rng):
    kind = rng.choice(["solve", "solve", "step", "step", "step", "block", "many", "serve"])
    fp32 = rng.random() < 0.4
    if kind == "solve":
        op = rng.choice(["poisson", "poisson", "varcoef", "aniso2d"])
        if op == "aniso2d":
            return dict(kind=kind, op=op, nx=_log(rng, 128, 2048), ny=_log(rng, 128, 2048), nz=1, fp32=fp32)
        if op == "poisson" and rng.random() < 0.3:
            return dict(kind=kind, op=op, **_box(rng, 32, 160), fp32=fp32, cycle=rng.choice([1, 2, 32]))
        return dict(kind=kind, op=op, **_box(rng, 32, 224), fp32=fp32)
    if kind == "step":
        op = rng.choice(["poisson", "poisson", "varcoef", "va3"])
        if op == "va3":
            return dict(kind=kind, op="poisson", **_box(rng, 32, 128), fp32=False, va3=True)
        return dict(kind=kind, op=op, **_box(rng, 32, 224), fp32=fp32)
    if kind == "block":
        c = _box(rng, 32, 112)
        return dict(kind=kind, op=rng.choice(["poisson", "poisson", "varcoef"]), **c, k=_log(rng, 2, 64), fp32=fp32)
    if kind == "many":
        return dict(kind=kind, m=_log(rng, 16, 256), lo=rng.randint(8, 24), hi=rng.randint(28, 60), fp32=fp32)
    return dict(kind=kind, requests=rng.randint(3, 12), kmax=rng.randint(1, 16), edge=rng.randint(32, 72), fp32=fp32)


# ------------------------------------------------------------ operators ----
class _Op:
    """7-point operator on an nx*ny*nz box from face coefficients (0 at no face);
    unknown (i, j, k) is row i + nx (j + ny k)."""

    def __init__(self, cx, cy, cz, nx, ny, nz):
        self.shape = (nz, ny, nx)
        self.n = nx * ny * nz
        self.cx, self.cy, self.cz = cx, cy, cz
        self.diag = (cx[:, :, :-1] + cx[:, :, 1:]) + (cy[:, :-1] + cy[:, 1:]) + (cz[:-1] + cz[1:])

    def csr(self):
        nz, ny, nx = self.shape
        idx = torch.arange(self.n, dtype=torch.int32, device=DEV).view(self.shape)
        col = torch.stack([idx + o for o in (-nx * ny, -nx, -1, 0, 1, nx, nx * ny)], -1)
        val = torch.stack([-self.cz[:-1], -self.cy[:, :-1], -self.cx[:, :, :-1], self.diag, -self.cx[:, :, 1:],
                           -self.cy[:, 1:], -self.cz[1:]], -1)
        keep = torch.ones(self.shape + (7,), dtype=torch.bool, device=DEV)
        keep[0, :, :, 0] = False
        keep[:, 0, :, 1] = False
        keep[:, :, 0, 2] = False
        keep[:, :, -1, 4] = False
        keep[:, -1, :, 5] = False
        keep[-1, :, :, 6] = False
        ptr = torch.zeros(self.n + 1, dtype=torch.int32, device=DEV)
        ptr[1:] = torch.cumsum(keep.view(self.n, 7).sum(1, dtype=torch.int32), 0)
        return ptr, col[keep].contiguous(), val[keep].contiguous()

    def apply(self, x):
        """A x for x of shape (n,) or (n, k)."""
        v = x.reshape(self.shape + (-1,))
        u = lambda c: c.unsqueeze(-1)  # noqa: E731
        y = u(self.diag) * v
        y[1:] -= u(self.cz[1:-1]) * v[:-1]
        y[:-1] -= u(self.cz[1:-1]) * v[1:]
        y[:, 1:] -= u(self.cy[:, 1:-1]) * v[:, :-1]
        y[:, :-1] -= u(self.cy[:, 1:-1]) * v[:, 1:]
        y[:, :, 1:] -= u(self.cx[:, :, 1:-1]) * v[:, :, :-1]
        y[:, :, :-1] -= u(self.cx[:, :, 1:-1]) * v[:, :, 1:]
        return y.reshape(x.shape)


def _gen(seed, part):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 7919 * part + 17)


def _operator(op, nx, ny, nz, seed):
    f64 = dict(dtype=torch.float64, device=DEV)
    if op == "varcoef":
        # log-coefficient N(0, 2^2) per node, harmonic mean on every face
        g = torch.randn((nz + 2, ny + 2, nx + 2), generator=_gen(seed, 1), **f64)
        kap = torch.exp(2.0 * g)
        hm = lambda a, b: 2.0 * a * b / (a + b)  # noqa: E731
        return _Op(hm(kap[1:-1, 1:-1, :-1], kap[1:-1, 1:-1, 1:]), hm(kap[1:-1, :-1, 1:-1], kap[1:-1, 1:, 1:-1]),
                   hm(kap[:-1, 1:-1, 1:-1], kap[1:, 1:-1, 1:-1]), nx, ny, nz)
    kx, ky, kz = (1.0, 1e-2, 0.0) if op == "aniso2d" else (1.0, 1.0, 1.0)
    one = torch.ones((), **f64)
    return _Op((kx * one).expand(nz, ny, nx + 1), (ky * one).expand(nz, ny + 1, nx), (kz * one).expand(nz + 1, ny, nx),
               nx, ny, nz)


def _csr(A):
    ptr, col, val = A.csr()
    return ptr, col, val, torch.ones(A.n, dtype=torch.float64, device=DEV)


def _uniform(n, k, seed, part=2):
    shape = (n,) if k is None else (n, k)
    return torch.rand(shape, generator=_gen(seed, part), dtype=torch.float64, device=DEV).mul_(2.0).sub_(1.0)


def _normal(n, k, seed, part=3):
    shape = (n,) if k is None else (n, k)
    return torch.randn(shape, generator=_gen(seed, part), dtype=torch.float64, device=DEV)


def _sine(n):
    i = torch.arange(1, n + 1, dtype=torch.float64, device=DEV)
    S = math.sqrt(2.0 / (n + 1)) * torch.sin(torch.outer(i, i) * (math.pi / (n + 1)))
    return S, 2.0 - 2.0 * torch.cos(i * (math.pi / (n + 1)))


def _sine_solve(op, nx, ny, nz, b):
    """A^-1 b of a constant-coefficient operator: diagonal in the sine basis of the three axes."""
    k = (1.0, 1e-2, 0.0) if op == "aniso2d" else (1.0, 1.0, 1.0)
    (Sx, lx), (Sy, ly), (Sz, lz) = _sine(nx), _sine(ny), _sine(nz)
    lam = (k[2] * lz)[:, None, None] + (k[1] * ly)[None, :, None] + (k[0] * lx)[None, None, :]

    def turn(v):
        v = torch.einsum("ai,kjic->kjac", Sx, v)
        v = torch.einsum("bj,kjac->kbac", Sy, v)
        return torch.einsum("dk,kbac->dbac", Sz, v)

    v = b.reshape(nz, ny, nx, -1)
    return turn(turn(v) / lam.unsqueeze(-1)).reshape(b.shape)


# ---------------------------------------------------------------- cases ----
def _options(case):
    o = dict(precision=amg.AMG_FP32_VCYCLE if case["fp32"] else amg.AMG_FP64)
    if case.get("op") == "varcoef":
        o["krylov"] = 1                      # flexible CG, as the coarsest solve may be iterative
    if case.get("cycle"):
        o["cycle"] = case["cycle"]
    if case.get("va3"):
        o.update(VA3)
    return o


def _box_of(case):
    return case["op"], case["nx"], case["ny"], case["nz"]


def _edges(case):
    """Edges of a batch's systems, uniform in lo..hi, fixed by the case."""
    return workloads.batch_edges(case["m"], 5, case["lo"], case["hi"])


def _serve_boxes(case):
    e = case["edge"]
    return [("poisson", e, e, e), ("aniso2d", 8 * e, 8 * e, 1), ("varcoef", e, e, e)]


def _serve_requests(case):
    """(operator, columns) of each request in order of arrival, fixed by the case: every operator and a request of
    the largest size are among them."""
    g = random.Random(1000 * case["requests"] + case["kmax"])
    reqs = [(g.randrange(3), g.randint(1, case["kmax"])) for _ in range(case["requests"])]
    return [(i if i < 3 else hid, case["kmax"] if i == 0 else k) for i, (hid, k) in enumerate(reqs)]


def _serve_rhs(case, seed, ops, r, hid, k):
    box = _serve_boxes(case)[hid]
    if box[0] == "varcoef":
        return ops[hid].apply(_uniform(ops[hid].n, k, seed, 100 + r))
    return _normal(ops[hid].n, k, seed, 100 + r)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "many":
        systems = [_csr(_operator("poisson", e, e, e, seed)) for e in _edges(case)]
        b = _normal(sum(e ** 3 for e in _edges(case)), None, seed)
        return dict(kind=kind, systems=systems, b=b, m=case["m"], opts=_options(case))
    if kind == "serve":
        hs, ops = [], []
        for box in _serve_boxes(case):
            A = _operator(*box, seed)
            o = _options(case)
            if box[0] == "varcoef":
                o["krylov"] = 1
            hs.append(amg.amg_setup(*_csr(A), **o))
            ops.append(A)
        reqs = [(hid, _serve_rhs(case, seed, ops, r, hid, k).cpu().numpy())
                for r, (hid, k) in enumerate(_serve_requests(case))]
        return dict(kind=kind, server=amg.Server(hs, slots=16), reqs=reqs)
    A = _operator(*_box_of(case), seed)
    s = dict(kind=kind, opts=_options(case))
    if kind == "step":
        s["A"] = _csr(A)
    else:
        s["h"] = amg.amg_setup(*_csr(A), **s["opts"])
    if kind == "block" and case["op"] != "varcoef":
        s["b"] = _normal(A.n, case["k"], seed)
    else:
        s["b"] = A.apply(_uniform(A.n, case.get("k"), seed)).contiguous()
    return s


def run(state):
    kind = state["kind"]
    if kind == "solve":
        x = torch.zeros_like(state["b"])
        info = amg.amg_solve(state["h"], state["b"], x)
        return dict(x=x, iterations=info["iterations"])
    if kind == "step":
        h = amg.amg_setup(*state["A"], **state["opts"])
        x = torch.zeros_like(state["b"])
        info = amg.amg_solve(h, state["b"], x)
        rep = amg.amg_hierarchy_info(h)
        h.close()
        return dict(x=x, iterations=info["iterations"], rows=sum(rep["n"]), entries=sum(rep["nnz"]))
    if kind == "block":
        X = torch.zeros_like(state["b"])
        infos = amg.amg_solve_batch(state["h"], state["b"], X)
        return dict(x=X, iterations=sum(i["iterations"] for i in infos))
    if kind == "many":
        h = amg.amg_setup_many(state["systems"], **state["opts"])
        x = torch.zeros_like(state["b"])
        infos = amg.amg_solve_many(h, state["b"], x, state["m"])
        h.close()
        return dict(x=x, iterations=sum(i["iterations"] for i in infos))
    srv = state["server"]
    sent = [srv.submit(hid, B) for hid, B in state["reqs"]]
    while srv.step():
        pass
    srv.poll()
    return dict(x=[X for _, X in sent])


def exact(case, seed):
    kind = case["kind"]
    if kind == "many":
        b = _normal(sum(e ** 3 for e in _edges(case)), None, seed)
        out, at = [], 0
        for e in _edges(case):
            out.append(_sine_solve("poisson", e, e, e, b[at:at + e ** 3]))
            at += e ** 3
        return dict(x=torch.cat(out), iterations=None)
    if kind == "serve":
        boxes = _serve_boxes(case)
        out = []
        for r, (hid, k) in enumerate(_serve_requests(case)):
            op, nx, ny, nz = boxes[hid]
            n = nx * ny * nz
            if op == "varcoef":
                out.append(_uniform(n, k, seed, 100 + r))
            else:
                out.append(_sine_solve(op, nx, ny, nz, _normal(n, k, seed, 100 + r)))
        return dict(x=[x.cpu() for x in out])
    op, nx, ny, nz = _box_of(case)
    n, k = nx * ny * nz, case.get("k")
    if kind == "block" and op != "varcoef":
        x = _sine_solve(op, nx, ny, nz, _normal(n, k, seed))
    else:
        x = _uniform(n, k, seed)
    return dict(x=x, iterations=None) if kind != "step" else dict(x=x, iterations=None, rows=None, entries=None)


def _sizes(op, nx, ny, nz):
    n = nx * ny * nz
    nnz = 7 * n - 2 * (nx * ny + ny * nz + nx * nz)
    return n, nnz


def work(case):
    """Matrix, right-hand sides and solutions once each; the products of one pass of CG's least work, 2 per entry and
    column."""
    kind = case["kind"]
    parts = []
    if kind == "many":
        parts = [(_sizes("poisson", e, e, e), 1) for e in _edges(case)]
    elif kind == "serve":
        reqs = _serve_requests(case)
        parts = [(_sizes(*box), sum(k for hid, k in reqs if hid == i)) for i, box in enumerate(_serve_boxes(case))]
    else:
        parts = [(_sizes(*_box_of(case)), case.get("k") or 1)]
    b = sum(12.0 * nnz + 4.0 * n + 16.0 * n * k for (n, nnz), k in parts)
    return {"bytes": b, "flops": sum(2.0 * nnz * k for (_, nnz), k in parts)}
