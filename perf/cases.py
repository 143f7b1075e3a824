"""The work that is timed when the library's speed is followed: calls that a
user's program makes, through the public entry points of
``paper_2212_01110_gb300.spock``, over the sizes, tree shapes, forms and
precisions that the library is used with.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs and handles a program has before the call
    run(state)           one pass
    work(case)           bytes and flops a pass cannot do without
    exact(case, seed)    what run() returns, in plain FP64 torch

A case is a dict of plain values:
    call      "solve" (spock_solve_dev, a fixed number of SPOCK iterations, as
              a control loop with an iteration budget runs it), "cp"
              (spock_cp_step_dev), "operators" (L, L*, prox f, prox g* and T one
              by one), "batch" (spock_batch_solve_dev), "sensitivity"
              (spock_grad_dev and spock_adjoint_dev)
    branch, branching, N   children per node of the first `branching` stages,
              then one child per node up to the horizon N; with "ragged" each
              node of those stages has 1..branch children, drawn from it
    nx, nu    state and input dimension
    system    "orthogonal": A = 0.95 x orthogonal, dense B, diagonal Q ~ U(0.5, 2),
              R = 0.1 I, Dirichlet child probabilities, AV@R a ~ U(0.1, 0.9);
              "thermal": the data-center system (tridiagonal A(w), B = I, two
              disturbance values with probabilities 0.3 and 0.7, R = 10 I, a = 0.95)
    form      "box", or "general": full cost matrices and polyhedral rows
    precision 64 or 32
    steps     SPOCK iterations, CP iterations or applications of J^T
    warm      the solve starts from a stored pair (closed-loop control)
    count     instances of a batch
Outputs of the FP32 mode are handed on as 32-bit numbers, which they are.
"""
import math

import numpy as np
import torch

from paper_2212_01110_gb300 import spock


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(call, branch, branching, N, nx, nu, system="orthogonal", form="box", precision=64, steps=1, memory=3,
          warm=False, ragged=0, count=1):
    return {"call": call, "branch": branch, "branching": branching, "N": N, "nx": nx, "nu": nu, "system": system,
            "form": form, "precision": precision, "steps": steps, "memory": memory, "warm": warm, "ragged": ragged,
            "count": count}


def listed():
    return [
        # the smallest problem (15 nodes), a short solve: one launch, latency only
        dict(_case("solve", 2, 3, 3, 3, 2, steps=25), name="solve_15_nodes_f64"),
        # the smallest call: one evaluation of T on that problem
        dict(_case("cp", 2, 3, 3, 3, 2), name="cp_15_nodes_f64"),
        # a closed-loop control step: the thermal system, N = 10, nx = nu = 20
        # (2,047 nodes, full binary tree), warm start, an iteration budget
        dict(_case("solve", 2, 10, 10, 20, 20, "thermal", steps=8, warm=True), name="closed_loop_2047_nodes_f64"),
        # the paper's time-to-tolerance system (nx = nu = 50), FP32 iterations
        dict(_case("solve", 2, 11, 11, 50, 50, "thermal", precision=32, steps=6), name="thermal_4095_nodes_f32"),
        # the benchmark's workload: 62,805 nodes, nx = 50, nu = 20, in FP64 ...
        dict(_case("solve", 4, 6, 20, 50, 20, steps=4), name="large_62805_nodes_f64"),
        # ... and its FP32 mode, on the shorter horizon with the same 4,096 chains
        dict(_case("solve", 4, 6, 10, 50, 20, precision=32, steps=6), name="chains_21845_nodes_f32"),
        # vanilla CP on a mid-size tree in FP32
        dict(_case("cp", 3, 5, 9, 24, 9, precision=32, steps=10), name="cp_1336_nodes_f32"),
        # the operators one by one on a ragged tree with odd sizes
        dict(_case("operators", 5, 4, 7, 33, 15, ragged=3), name="operators_ragged_f64"),
        # a heterogeneous batch (horizons, branchings and sizes of its own per instance)
        dict(_case("batch", 4, 3, 12, 30, 10, precision=32, steps=6, count=48), name="batch_48_f32"),
        # the same call in FP64, smaller instances
        dict(_case("batch", 3, 2, 8, 16, 6, steps=6, count=24), name="batch_24_f64"),
        # general form: full Q, R, Q_N and coupled constraint rows
        dict(_case("cp", 4, 4, 6, 50, 20, form="general", steps=5), name="general_853_nodes_f64"),
        # gradients of the optimal cost and of the control law (607 nodes)
        dict(_case("sensitivity", 3, 4, 10, 20, 8, steps=20), name="sensitivity_607_nodes_f64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve", "solve", "cp", "operators", "batch", "sensitivity"])
    if call == "batch":
        return _case("batch", rng.randint(2, 4), rng.randint(1, 3), rng.randint(4, 12), rng.randint(8, 30),
                     rng.randint(3, 10), precision=rng.choice([32, 64]), steps=rng.randint(3, 6),
                     memory=rng.choice([3, 5]), count=_log_int(rng, 4, 48))
    if call == "sensitivity":
        branch = rng.randint(2, 4)
        return _case(call, branch, rng.randint(1, {2: 6, 3: 4, 4: 3}[branch]), rng.randint(7, 12), rng.randint(3, 30),
                     rng.randint(2, 12), steps=rng.randint(5, 25))
    system = "orthogonal" if call == "operators" else rng.choice(["orthogonal", "orthogonal", "thermal"])
    form = "general" if call == "cp" and system == "orthogonal" and rng.random() < 0.4 else "box"
    branch = 2 if system == "thermal" else rng.randint(2, 5)
    most = _log_int(rng, 2, 200 if form == "general" else 2048)          # scenarios
    branching = max(1, int(math.log(most) / math.log(branch) + 1e-9))
    N = branching if system == "thermal" else branching + rng.choice([0, 0, 1, 2, 3, 5, 8])
    nx = _log_int(rng, 2, 64)
    nu = nx if system == "thermal" else max(1, min(40, int(nx * rng.uniform(0.2, 1.2))))
    ragged = rng.randint(1, 1000) if call == "operators" or rng.random() < 0.3 else 0
    return _case(call, branch, branching, N, nx, nu, system, form, rng.choice([64, 32]) if call != "operators" else 64,
                 rng.randint(2, 6), rng.choice([0, 3, 3, 5]) if call == "solve" else 3,
                 call == "solve" and rng.random() < 0.5, 0 if system == "thermal" else ragged)


# ---------------------------------------------------------------------------
# trees and data
# ---------------------------------------------------------------------------
class _Tree:
    """Breadth-first tree: ancestors, children counts, stages and the offsets
    of every block of z and eta (include/spock.h)."""

    def __init__(self, c):
        rng = np.random.RandomState(c["ragged"]) if c["ragged"] else None
        counts, width = [], 1
        anc, begin = [np.array([-1])], [0, 1]
        for t in range(c["N"]):
            if t >= c["branching"]:
                m = np.ones(width, np.int64)
            elif rng is None:
                m = np.full(width, c["branch"])
            else:
                m = rng.randint(1, c["branch"] + 1, width)
            counts.append(m)
            anc.append(np.repeat(np.arange(begin[-2], begin[-1]), m))
            width = int(m.sum())
            begin.append(begin[-1] + width)
        self.anc, self.begin = np.concatenate(anc).astype(np.int32), begin
        self.n, self.nl, self.N = begin[-1], begin[-2], c["N"]
        self.m = np.concatenate(counts).astype(np.int64)              # children of nonleaf nodes
        self.c0 = 1 + np.concatenate([[0], np.cumsum(self.m)[:-1]])   # first child
        self.sib = np.arange(1, self.n) - self.c0[self.anc[1:]]       # place among the siblings, nonroot nodes


def _gen(seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _data(c, t, seed):
    """Problem data of the case as FP64 tensors (on the GPU), x0 included."""
    dev = _device()
    g = _gen(seed, dev)
    f = dict(dtype=torch.float64, device=dev)
    rand = lambda *s: torch.rand(*s, generator=g, **f)     # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=g, **f)   # noqa: E731
    n, nx, nu = t.n, c["nx"], c["nu"]
    d = {"nx": nx, "nu": nu}
    par = torch.as_tensor(t.anc[1:].astype(np.int64), device=dev)
    if c["system"] == "thermal":
        w = torch.as_tensor(np.concatenate([[0], t.sib]), device=dev).double()
        j = torch.arange(nx, **f)
        A = torch.diag_embed(1 + w[:, None] / 2 * (1 + j / nx))
        A += 0.01 * (torch.diag(torch.ones(nx - 1, **f), 1) + torch.diag(torch.ones(nx - 1, **f), -1))
        B = torch.eye(nx, nu, **f).repeat(n, 1, 1)
        prob = torch.where(w == 0, 0.3, 0.7)
        Q, R, a, xlim, ulim = torch.ones(n, nx, **f), torch.full((n, nu), 10.0, **f), torch.full((n,), 0.95, **f), 1.0, 1.5
        x0 = 0.3 * (2 * rand(nx) - 1)
    else:
        A = torch.eye(nx, **f).repeat(n, 1, 1)
        for _ in range(4):   # product of reflections: dense orthogonal matrices
            v = randn(n, nx, 1)
            v /= v.norm(dim=1, keepdim=True)
            A -= 2 * v @ (v.transpose(1, 2) @ A)
        A *= 0.95
        B = randn(n, nx, nu) / math.sqrt(nx)
        e = -torch.log(rand(n - 1).clamp_min(1e-12))           # Dirichlet(1) per node, floored
        s = torch.zeros(t.nl, **f).index_add_(0, par, e)
        e = (e / s[par]).clamp_min(1e-3)
        s = torch.zeros(t.nl, **f).index_add_(0, par, e)
        prob = torch.cat([torch.ones(1, **f), e / s[par]])
        Q, R, a, xlim, ulim = 0.5 + 1.5 * rand(n, nx), torch.full((n, nu), 0.1, **f), 0.1 + 0.8 * rand(n), 5.0, 1.0
        x0 = randn(nx).clamp(-4.0, 4.0)
    A[0], B[0], prob[0] = 0, 0, 1
    d.update(A=A, B=B, prob=prob, Q=Q, R=R, QN=torch.ones(n, nx, **f), a=a, x0=x0)
    box = {"xmin": torch.full((n, nx), -xlim, **f), "umin": torch.full((n, nu), -ulim, **f)}
    if c["form"] == "box":
        d.update(box, xmax=-box["xmin"], umax=-box["umin"])
        return d
    def full(diag, k):   # D (I / 2 + M M' / k) D
        M = randn(n, k, k)
        M = 0.5 * torch.eye(k, **f) + M @ M.transpose(1, 2) / k
        M = diag.sqrt()[:, :, None] * M * diag.sqrt()[:, None, :]
        return 0.5 * (M + M.transpose(1, 2))
    rows, rowsN = 10, 6   # coupled rows next to the box rows
    G = torch.cat([torch.eye(nx + nu, **f).repeat(n, 1, 1), randn(n, rows, nx + nu) / math.sqrt(nx + nu)], 1)
    GN = torch.cat([torch.eye(nx, **f).repeat(n, 1, 1), randn(n, rowsN, nx) / math.sqrt(nx)], 1)
    lo = torch.cat([box["xmin"], box["umin"], torch.full((n, rows), -3.0, **f)], 1)
    loN = torch.cat([box["xmin"], torch.full((n, rowsN), -3.0, **f)], 1)
    d.update(Q=full(Q, nx), R=full(R, nu), QN=full(d["QN"], nx), Gx=G[:, :, :nx].contiguous(),
             Gu=G[:, :, nx:].contiguous(), GN=GN, cmin=lo, cmax=-lo, cNmin=loN, cNmax=-loN)
    return d


def _norm_bound(c, t, d):
    """An upper bound of ||L|| from the column groups of L (a program that
    gives its own step size has one)."""
    nx = c["nx"]
    par = torch.as_tensor(t.anc[1:].astype(np.int64), device=d["A"].device)
    if c["form"] == "box":
        w = torch.cat([d["Q"], d["R"]], 1)[1:]
        s = torch.zeros(t.nl, w.shape[1], dtype=w.dtype, device=w.device).index_add_(0, par, w)
        best = max(float(s.max()), float(d["QN"].max())) + 1.0
    else:
        M = torch.zeros(t.nl, nx + c["nu"], nx + c["nu"], dtype=torch.float64, device=d["A"].device)
        M[:, :nx, :nx].index_add_(0, par, d["Q"][1:])
        M[:, nx:, nx:].index_add_(0, par, d["R"][1:])
        G = torch.cat([d["Gx"], d["Gu"]], 2)[:t.nl]
        M += G.transpose(1, 2) @ G
        GN = d["GN"][t.nl:]
        best = max(float(torch.linalg.matrix_norm(M).max()),
                   float(torch.linalg.matrix_norm(GN.transpose(1, 2) @ GN + d["QN"][t.nl:]).max()))
    return math.sqrt(max(best, 5.0))


def _problem(t, d):
    h = {k: (v.cpu().numpy() if isinstance(v, torch.Tensor) else v) for k, v in d.items()}
    h["anc"] = t.anc
    return spock.Problem(h)


def _instances(c, seed):
    """Cases of a batch's instances: sizes of their own within the batch's."""
    rng = np.random.RandomState(1234 + c["count"])
    out = []
    for i in range(c["count"]):
        b = int(rng.randint(2, c["branch"] + 1))
        k = int(rng.randint(1, c["branching"] + 1))
        out.append(dict(c, call="solve", branch=b, branching=k, N=int(rng.randint(k, c["N"] + 1)),
                        nx=int(rng.randint(max(2, c["nx"] // 3), c["nx"] + 1)),
                        nu=int(rng.randint(max(1, c["nu"] // 3), c["nu"] + 1)), count=1))
    return out


def _start(c, n_z, n_eta, seed):
    """A stored primal-dual pair."""
    g = _gen(seed + 7919, _device())
    v = 0.5 * torch.randn(n_z + n_eta, generator=g, dtype=torch.float64, device=_device())
    return v[:n_z].clone(), v[n_z:].clone()


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c, dev = case, _device()
    f = dict(dtype=torch.float64, device=dev)
    prec = spock.SPOCK_FP64 if c["precision"] == 64 else spock.SPOCK_FP32
    s = {"case": c, "prec": prec}
    if c["call"] in ("solve", "batch"):
        s["settings"] = spock.spock_default_settings(memory=c["memory"], precision=prec, max_iter=c["steps"],
                                                     eps_abs=1e-12, eps_rel=1e-12, fp64_tail=0)
    if c["call"] == "batch":
        s["problems"], s["x0"] = [], []
        for i, q in enumerate(_instances(c, seed)):
            t = _Tree(q)
            d = _data(q, t, seed * 1000 + i)
            s["problems"].append(_problem(t, d))
            s["x0"].append(d["x0"].contiguous())
        s["z"] = torch.zeros(sum(p.n_z for p in s["problems"]), **f)
        s["eta"] = torch.zeros(sum(p.n_eta for p in s["problems"]), **f)
        s["zs"] = list(s["z"].split([p.n_z for p in s["problems"]]))
        s["etas"] = list(s["eta"].split([p.n_eta for p in s["problems"]]))
        s["batch"] = _Batch([p.handle for p in s["problems"]])
        return s
    t = _Tree(c)
    d = _data(c, t, seed)
    p = s["problem"] = _problem(t, d)
    s["x0"] = d["x0"].contiguous()
    s["z"], s["eta"] = torch.zeros(p.n_z, **f), torch.zeros(p.n_eta, **f)
    s["alpha"] = 0.95 / _norm_bound(c, t, d)
    if c["call"] == "solve" and c["warm"]:
        # the pair that an earlier call for a neighbouring state left
        s["z0"], s["eta0"] = torch.zeros_like(s["z"]), torch.zeros_like(s["eta"])
        spock.spock_cp_step_dev(p.handle, 0.9 * s["x0"], 40, 0.0, spock.SPOCK_FP64, s["z0"], s["eta0"])
    elif c["call"] == "cp":
        s["z0"], s["eta0"] = _start(c, p.n_z, p.n_eta, seed)
    elif c["call"] == "operators":
        s["z"], s["eta"] = _start(c, p.n_z, p.n_eta, seed)
        s["out"] = {k: torch.empty(p.n_z if k in ("Lt", "proxf", "Tz") else p.n_eta, **f)
                    for k in ("L", "Lt", "proxf", "proxg", "Tz", "Teta")}
    elif c["call"] == "sensitivity":
        spock.spock_cp_step_dev(p.handle, s["x0"], 200, 0.0, spock.SPOCK_FP64, s["z"], s["eta"])
        n, nx, nu = t.n, c["nx"], c["nu"]
        shapes = {"g_x0": (nx,), "g_A": (n, nx, nx), "g_B": (n, nx, nu), "g_Q": (n, nx), "g_R": (n, nu), "g_QN": (n, nx)}
        s["value"] = {k: torch.zeros(*v, **f) for k, v in shapes.items()}
        s["policy"] = {k: torch.zeros(*v, **f) for k, v in shapes.items()}
        s["g_z"] = torch.zeros(p.n_z, **f)
        s["g_z"][1 + n * nx] = 1.0   # the first entry of u^0
    return s


class _Batch:
    """Owner of a batch handle."""

    def __init__(self, handles):
        self.handle = spock.spock_batch_create(handles)

    def __del__(self):
        spock.spock_free(self.handle)


def _handed_on(s, z, eta):
    return {"z": z.clone(), "eta": eta.clone()} if s["case"]["precision"] == 64 else {"z": z.float(), "eta": eta.float()}


def run(state):
    s, c = state, state["case"]
    if c["call"] == "batch":
        infos = spock.spock_batch_solve_dev(s["batch"].handle, s["x0"], s["settings"], s["zs"], s["etas"], 0)
        out = _handed_on(s, s["z"], s["eta"])
        out["iterations"] = np.array([i.iterations for i in infos])
        return out
    p = s["problem"].handle
    if c["call"] == "solve":
        if c["warm"]:
            s["z"].copy_(s["z0"])
            s["eta"].copy_(s["eta0"])
        info = spock.spock_solve_dev(p, s["x0"], s["settings"], s["z"], s["eta"], int(c["warm"]))
        return dict(_handed_on(s, s["z"], s["eta"]), iterations=info.iterations)
    if c["call"] == "cp":
        s["z"].copy_(s["z0"])
        s["eta"].copy_(s["eta0"])
        xi = spock.spock_cp_step_dev(p, s["x0"], c["steps"], s["alpha"], s["prec"], s["z"], s["eta"])
        return dict(_handed_on(s, s["z"], s["eta"]), xi=xi)
    if c["call"] == "operators":
        o, z, eta = s["out"], s["z"], s["eta"]
        spock.spock_apply_L_dev(p, z, o["L"])
        spock.spock_apply_Lt_dev(p, eta, o["Lt"])
        spock.spock_prox_f_dev(p, s["x0"], s["alpha"], z, o["proxf"])
        spock.spock_prox_gconj_dev(p, s["alpha"], eta, o["proxg"])
        spock.spock_T_dev(p, s["x0"], s["alpha"], z, eta, o["Tz"], o["Teta"])
        return o
    spock.spock_grad_dev(p, s["z"], s["eta"], s["prec"], **s["value"])
    spock.spock_adjoint_dev(p, s["z"], s["eta"], s["g_z"], c["steps"], 1e-14, **s["policy"])
    return {"value": s["value"], "policy": s["policy"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _work_T(c):
    """(bytes, flops) of one evaluation of T: the factors of both passes ([A | B]
    and K in each direction, the node block of the backward pass; the passes run
    in opposite orders over the tree), the rows of L, z and eta in and out."""
    t = _Tree(c)
    nx, nu, n, nl = c["nx"], c["nu"], t.n, t.nl
    fac = 2 * (n - 1) * nx * (nx + nu) + nl * (3 * nu * nx + nu * nu)
    nc, ncN = (nx + nu, nx) if c["form"] == "box" else (nx + nu + 10, nx + 6)
    nz = 1 + n * nx + nl * nu + int((4 * t.m + 1).sum())
    ne = int((2 * t.m + 2).sum()) + nl * nc + (n - 1) * (nx + nu + 2) + (n - nl) * (ncN + nx + 2)
    par = 2 * n * (nx + nu) + n * (nx + nu) + (n - nl) * nx       # bounds, roots of the cost weights
    if c["form"] == "general":
        par += nl * nc * (nx + nu) + (n - 1) * (nx * nx + nu * nu) // 2 + (n - nl) * (ncN * nx + nx * nx // 2)
    return (fac + par + 2 * (nz + ne)) * (c["precision"] // 8), 2 * fac + 4 * par + 12 * (nz + ne)


def work(case):
    c = case
    if c["call"] == "batch":
        parts = [_work_T(q) for q in _instances(c, 0)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    else:
        b, f = _work_T(c)
    # a solve evaluates T once at the start and at least once per iteration
    k = {"solve": c["steps"] + 1, "batch": c["steps"] + 1, "cp": c["steps"], "operators": 2, "sensitivity": c["steps"] + 1}
    return {"bytes": int(b * k[c["call"]]), "flops": int(f * k[c["call"]])}


# ---------------------------------------------------------------------------
# the operators in plain torch, FP64
# ---------------------------------------------------------------------------
class _Plain:
    """z and eta as blocks: per node x; per nonleaf node u; y in rows (three
    arrays: one entry per child, one entry per child, one per nonleaf node);
    tau and s per nonroot node; s0."""

    def __init__(self, c, t, d):
        self.c, self.t, self.d = c, t, d
        dev = d["A"].device
        T = lambda a: torch.as_tensor(np.asarray(a, np.int64), device=dev)   # noqa: E731
        nx, nu, n, nl, m = c["nx"], c["nu"], t.n, t.nl, t.m
        box = c["form"] == "box"
        nc, ncN = (nx + nu, nx) if box else (d["Gx"].shape[1], d["GN"].shape[1])
        self.par, p = T(t.anc[1:]), t.anc[1:]
        z2 = 1 + n * nx + nl * nu + np.concatenate([[0], np.cumsum(4 * m + 1)])
        el = np.concatenate([[0], np.cumsum(2 * m + 2 + nc)])
        sib, mp = t.sib, m[p]
        rows = lambda start, k: T(np.asarray(start)[:, None] + np.arange(k))   # noqa: E731
        self.z = {"s0": T([0]), "x": rows(1 + nx * np.arange(n), nx), "u": rows(1 + n * nx + nu * np.arange(nl), nu),
                  "y1": T(z2[p] + sib), "y2": T(z2[p] + mp + sib), "y3": T(z2[:-1] + 2 * m),
                  "tau": T(z2[p] + 2 * mp + 1 + sib), "s": T(z2[p] + 3 * mp + 1 + sib)}
        er = el[-1] + (nx + nu + 2) * np.arange(n - 1)
        ef = er[-1] + nx + nu + 2 + (ncN + nx + 2) * np.arange(n - nl)
        self.e = {"y1": T(el[p] + sib), "y2": T(el[p] + mp + sib), "y3": T(el[:-1] + 2 * m), "sb": T(el[:-1] + 2 * m + 1),
                  "c": rows(el[:-1] + 2 * m + 2, nc), "nr": rows(er, nx + nu + 2), "cN": rows(ef, ncN),
                  "lf": rows(ef + ncN, nx + 2)}
        self.n_z, self.n_e = int(z2[-1]), int(ef[-1] + ncN + nx + 2)
        if box:
            self.q, self.r, self.qn = d["Q"].sqrt(), d["R"].sqrt(), d["QN"].sqrt()
            self.lo, self.hi = torch.cat([d["xmin"], d["umin"]], 1)[:nl], torch.cat([d["xmax"], d["umax"]], 1)[:nl]
            self.loN, self.hiN = d["xmin"][nl:], d["xmax"][nl:]
        else:
            up = lambda M: torch.linalg.cholesky(M).transpose(1, 2)   # noqa: E731
            self.q, self.r, self.qn = up(d["Q"]), up(d["R"]), up(d["QN"])
            self.G, self.GN = torch.cat([d["Gx"], d["Gu"]], 2)[:nl], d["GN"][nl:]
            self.lo, self.hi, self.loN, self.hiN = d["cmin"][:nl], d["cmax"][:nl], d["cNmin"][nl:], d["cNmax"][nl:]
        self.box = box
        self._factor()

    def _mul(self, F, x):
        return F * x if self.box else (F @ x[:, :, None])[:, :, 0]

    def _tmul(self, F, w):
        return F * w if self.box else (F.transpose(1, 2) @ w[:, :, None])[:, :, 0]

    def _sum(self, v):
        """Sum over the children of each nonleaf node of a value per nonroot node."""
        return torch.zeros((self.t.nl,) + v.shape[1:], dtype=v.dtype, device=v.device).index_add_(0, self.par, v)

    def L(self, z):
        nl, c, p, d = self.t.nl, self.c, self.par, self.d
        v = {k: z[i] for k, i in self.z.items()}
        out = torch.empty(self.n_e, dtype=z.dtype, device=z.device)
        e = self.e
        s = torch.cat([v["s0"], v["s"]])
        for k in ("y1", "y2", "y3"):
            out[e[k]] = v[k]
        out[e["sb"]] = s[:nl] - self._sum(d["prob"][1:] * v["y1"]) - v["y3"]
        xu = torch.cat([v["x"][:nl], v["u"]], 1)
        out[e["c"]] = xu if self.box else (self.G @ xu[:, :, None])[:, :, 0]
        half = lambda w: 0.5 * torch.stack([w, w], 1)   # noqa: E731
        out[e["nr"]] = torch.cat([self._mul(self.q[1:], v["x"][p]), self._mul(self.r[1:], v["u"][p]), half(v["tau"])], 1)
        xl = v["x"][nl:]
        out[e["cN"]] = xl if self.box else (self.GN @ xl[:, :, None])[:, :, 0]
        out[e["lf"]] = torch.cat([self._mul(self.qn[nl:], xl), half(s[nl:])], 1)
        return out

    def Lt(self, eta):
        nl, nx, nu, d = self.t.nl, self.c["nx"], self.c["nu"], self.d
        w = {k: eta[i] for k, i in self.e.items()}
        out = torch.empty(self.n_z, dtype=eta.dtype, device=eta.device)
        nr = w["nr"]
        xu = w["c"] if self.box else (self.G.transpose(1, 2) @ w["c"][:, :, None])[:, :, 0]
        xu = xu + self._sum(torch.cat([self._tmul(self.q[1:], nr[:, :nx]), self._tmul(self.r[1:], nr[:, nx:nx + nu])], 1))
        xl = w["cN"] if self.box else (self.GN.transpose(1, 2) @ w["cN"][:, :, None])[:, :, 0]
        out[self.z["x"]] = torch.cat([xu[:, :nx], xl + self._tmul(self.qn[nl:], w["lf"][:, :nx])])
        out[self.z["u"]] = xu[:, nx:]
        out[self.z["y1"]] = w["y1"] - d["prob"][1:] * w["sb"][self.par]
        out[self.z["y2"]] = w["y2"]
        out[self.z["y3"]] = w["y3"] - w["sb"]
        out[self.z["tau"]] = 0.5 * (nr[:, -2] + nr[:, -1])
        s = torch.cat([w["sb"], 0.5 * (w["lf"][:, -2] + w["lf"][:, -1])])
        out[self.z["s0"]], out[self.z["s"]] = s[:1], s[1:]
        return out

    def _factor(self):
        """The Riccati recursion of the projection on the dynamics, per stage."""
        t, A, B, nx, nu = self.t, self.d["A"], self.d["B"], self.c["nx"], self.c["nu"]
        eye = lambda k, j: torch.eye(j, dtype=A.dtype, device=A.device).repeat(k, 1, 1)   # noqa: E731
        P = eye(t.begin[-1] - t.begin[-2], nx)
        self.K, self.H, self.Ab, self.PB = [None] * t.N, [None] * t.N, [None] * (t.N + 1), [None] * (t.N + 1)
        for s in range(t.N - 1, -1, -1):
            b0, b1, b2 = t.begin[s:s + 3]
            q = self.par[b1 - 1:b2 - 1] - b0
            Ac, Bc = A[b1:b2], B[b1:b2]
            PB = P @ Bc
            H = eye(b1 - b0, nu).index_add_(0, q, Bc.transpose(1, 2) @ PB)
            F = torch.zeros(b1 - b0, nu, nx, dtype=A.dtype, device=A.device).index_add_(0, q, PB.transpose(1, 2) @ Ac)
            H = torch.linalg.cholesky(H)
            K = -torch.cholesky_solve(F, H)
            Ab = Ac + Bc @ K[q]
            P = (eye(b1 - b0, nx) + K.transpose(1, 2) @ K).index_add_(0, q, Ab.transpose(1, 2) @ (P @ Ab))
            P = 0.5 * (P + P.transpose(1, 2))
            self.K[s], self.H[s], self.Ab[s + 1], self.PB[s + 1] = K, H, Ab, PB

    def prox_f(self, z, x0, alpha):
        t, B, d = self.t, self.d["B"], self.d
        mv = lambda M, v: (M @ v[:, :, None])[:, :, 0]   # noqa: E731
        mtv = lambda M, v: (M.transpose(1, 2) @ v[:, :, None])[:, :, 0]   # noqa: E731
        xb, ub = z[self.z["x"]], z[self.z["u"]]
        out = z.clone()
        out[0] -= alpha
        q, ds = -xb[t.nl:], [None] * t.N
        for s in range(t.N - 1, -1, -1):
            b0, b1, b2 = t.begin[s:s + 3]
            k = self.par[b1 - 1:b2 - 1] - b0
            g = ub[b0:b1].clone().index_add_(0, k, -mtv(B[b1:b2], q))
            dd = torch.cholesky_solve(g[:, :, None], self.H[s])[:, :, 0]
            add = mtv(self.Ab[s + 1], q + mv(self.PB[s + 1], dd[k]))
            q = (mtv(self.K[s], dd - ub[b0:b1]) - xb[b0:b1]).index_add_(0, k, add)
            ds[s] = dd
        x, xs, us = x0[None, :], [x0[None, :]], []
        for s in range(t.N):
            b0, b1, b2 = t.begin[s:s + 3]
            k = self.par[b1 - 1:b2 - 1] - b0
            us.append(mv(self.K[s], x) + ds[s])
            x = mv(self.Ab[s + 1], x[k]) + mv(B[b1:b2], ds[s][k])
            xs.append(x)
        out[self.z["x"]], out[self.z["u"]] = torch.cat(xs), torch.cat(us)
        # kernel of a y1 - y2 + y3 - tau - s per child
        v, p = {k: z[i] for k, i in self.z.items()}, self.par
        a = d["a"][:t.nl]
        r = a[p] * v["y1"] - v["y2"] + v["y3"][p] - v["tau"] - v["s"]
        cc = a * a + 3
        lam = (r - (self._sum(r) / (cc + self._sum(torch.ones_like(r))))[p]) / cc[p]
        for k, step in (("y1", -a[p] * lam), ("y2", lam), ("tau", lam), ("s", lam), ("y3", -self._sum(lam))):
            out[self.z[k]] = v[k] + step
        return out

    def prox_g(self, eta, alpha):
        w = eta / alpha
        out = w.clone()
        for k in ("y1", "y2", "sb"):
            out[self.e[k]] = w[self.e[k]].clamp_min(0)
        out[self.e["c"]] = w[self.e["c"]].clamp(self.lo, self.hi)
        out[self.e["cN"]] = w[self.e["cN"]].clamp(self.loN, self.hiN)
        for k in ("nr", "lf"):
            y = w[self.e[k]]
            sh = torch.zeros_like(y[0])
            sh[-2], sh[-1] = 0.5, -0.5
            y = y - sh
            t, nv = y[:, -1:], y[:, :-1].norm(dim=1, keepdim=True)
            sc = 0.5 * (nv + t)
            proj = torch.cat([sc / nv * y[:, :-1], sc], 1)
            proj = torch.where(nv <= t, y, torch.where(nv <= -t, torch.zeros_like(y), proj))
            out[self.e[k]] = proj + sh
        return eta - alpha * out

    def T(self, z, eta, x0, alpha):
        zp = self.prox_f(z - alpha * self.Lt(eta), x0, alpha)
        return zp, self.prox_g(eta + alpha * self.L(2 * zp - z), alpha)

    def norm(self):
        """||L|| of the box form: the largest norm of its column groups."""
        b2 = 1 + self._sum(self.d["prob"][1:] ** 2)
        xu = 1 + self._sum(torch.cat([self.q[1:], self.r[1:]], 1) ** 2)
        ys = (2 + b2 + b2.sqrt() * (b2 + 4).sqrt()) / 2
        return math.sqrt(max(float(xu.max()), float(ys.max()), 1 + float((self.qn[self.t.nl:] ** 2).max())))

    def gradient(self, z, eta):
        """The Lagrangian's derivatives at (z, eta) (box form)."""
        t, nl, nx, nu, p = self.t, self.t.nl, self.c["nx"], self.c["nu"], self.par
        w = self.Lt(eta)[self.z["x"]]
        lam = -w
        for s in range(t.N - 1, -1, -1):
            b1, b2 = t.begin[s + 1:s + 3]
            lam.index_add_(0, p[b1 - 1:b2 - 1], (self.d["A"][b1:b2].transpose(1, 2) @ lam[b1:b2, :, None])[:, :, 0])
        x, u, nr = z[self.z["x"]], z[self.z["u"]], eta[self.e["nr"]]
        zero = lambda *s: torch.zeros(*s, dtype=z.dtype, device=z.device)   # noqa: E731
        g = {"g_x0": -lam[0], "g_A": zero(t.n, nx, nx), "g_B": zero(t.n, nx, nu), "g_Q": zero(t.n, nx),
             "g_R": zero(t.n, nu), "g_QN": zero(t.n, nx)}
        g["g_A"][1:] = -lam[1:, :, None] * x[p][:, None, :]
        g["g_B"][1:] = -lam[1:, :, None] * u[p][:, None, :]
        g["g_Q"][1:] = nr[:, :nx] * x[p] / (2 * self.q[1:])
        g["g_R"][1:] = nr[:, nx:nx + nu] * u[p] / (2 * self.r[1:])
        g["g_QN"][nl:] = eta[self.e["lf"]][:, :nx] * x[nl:] / (2 * self.qn[nl:])
        return g


def exact(case, seed):
    """Calls whose result is a fixed composition of the operators.  A solve's
    iterate follows decisions taken from rounded norms, and the adjoint's an
    unfinished Krylov iteration, so these have none."""
    c = case
    if c["call"] in ("solve", "batch"):
        return None
    t = _Tree(c)
    d = _data(c, t, seed)
    P, alpha, x0 = _Plain(c, t, d), 0.95 / _norm_bound(c, t, d), d["x0"]
    if c["call"] == "sensitivity":
        z, eta = torch.zeros(P.n_z, dtype=x0.dtype, device=x0.device), torch.zeros(P.n_e, dtype=x0.dtype, device=x0.device)
        for _ in range(200):
            z, eta = P.T(z, eta, x0, 0.99 / P.norm())
        return {"value": P.gradient(z, eta), "policy": dict.fromkeys(("g_x0", "g_A", "g_B", "g_Q", "g_R", "g_QN"))}
    z, eta = _start(c, P.n_z, P.n_e, seed)
    if c["call"] == "operators":
        Tz, Te = P.T(z, eta, x0, alpha)
        return {"L": P.L(z), "Lt": P.Lt(eta), "proxf": P.prox_f(z, x0, alpha), "proxg": P.prox_g(eta, alpha),
                "Tz": Tz, "Teta": Te}
    for _ in range(c["steps"]):
        z, eta, zp, ep = *P.T(z, eta, x0, alpha), z, eta
    xi = None
    if c["precision"] == 64:
        rz, re = zp - z, ep - eta
        xi = max(float((rz / alpha - P.Lt(re)).abs().max()), float((re / alpha - P.L(rz)).abs().max()))
    return {"z": z, "eta": eta, "xi": xi}
