"""Timed cases of the field-solve library: what a user's program calls, over the range of
meshes, tearings, precisions, solvers and calls that the workloads, the tests and the benchmark use.

A case is one call pattern ("call") on one mesh and tearing:

* march     one Newmark step of a field march in progress (dd_step_scaled), the per-step hot path;
* default   one step exactly as a first-time user writes it: FieldSolver with default parameters;
* pic       one PIC cycle (push, deposit, field step, Faraday) with the beam in flight;
* gradient  one evaluation of the probe objective and its gradients: new materials, factorisation,
            forward march, adjoint march (probe_objective(...).backward());
* refactor  new materials, factorisation, one step (an optimisation or finite-difference loop);
* coupled / schur   one application of an interface operator in FP64.

Fields start from a few cavity modes (edge integrals, amplitudes from the seed) that are already
ringing, plus the workloads' Gaussian line pulse, so that the solves see fields of ordinary shape.
Meshes are Kuhn boxes of cubic cells (side 1/n of the longest unit edge), optionally jittered.
"""
import functools
import math

import numpy as np
import torch

from paper_2204_13254_gb300 import adjoint as A
from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

WARM_STEPS = 3      # steps marched before the timed one: the march is under way, its graphs are captured
PIC_STEPS = 24      # PIC cycles before the timed one: the beam is in the domain
GRAD_STEPS = 6      # forward steps of one objective evaluation


# ---- cases ------------------------------------------------------------------------------------

def _case(name, call, nx, ny, nz, cell, dt, kx=0, ky=0, kz=0, rcb=0, jitter=False, eps=False, precision="fp64",
          solver="gmres", scheme="dp1", graph=True, tuned=False, members=1, particles=0):
    """nx, ny, nz cells of side `cell`; blocks kx, ky, kz or `rcb` bisected parts; dt = 2 x the explicit limit."""
    return dict(name=name, call=call, nx=nx, ny=ny, nz=nz, cell=cell, dt=dt, kx=kx, ky=ky, kz=kz, rcb=rcb,
                jitter=jitter, eps=eps, precision=precision, solver=solver, scheme=scheme, graph=graph, tuned=tuned,
                members=members, particles=particles)


def listed():
    return [
        # the smallest problem with the library's own defaults (FP64, Schur CG, eager launches, stats read): a
        # first-time user's step, all latency
        _case("cavity8_default", "default", 8, 8, 8, 1 / 8, 0.05808, 2, 2, 2, solver="cg", graph=False),
        # the same problem as a long march runs it: mixed precision, coupled GMRES, CUDA-graph steps
        _case("cavity8_mixed", "march", 8, 8, 8, 1 / 8, 0.05808, 2, 2, 2, precision="mixed"),
        # the beam problem: 10^5 macro-particles in flight, mixed-precision field solve
        _case("beam16x16x32_pic", "pic", 16, 16, 32, 1 / 16, 0.02879, 4, 4, 8, precision="mixed", particles=100000),
        # Robin transmission (MFETI-DP2) on the same box, mixed precision
        _case("box16x16x32_dp2", "march", 16, 16, 32, 1 / 16, 0.02879, 4, 4, 8, precision="mixed", scheme="dp2"),
        # the Schur-complement interface system by CG in mixed precision, subdomains of 6^3 cubes
        _case("cavity24_schur_mixed", "march", 24, 24, 24, 1 / 24, 0.01916, 4, 4, 4, precision="mixed", solver="cg"),
        # 16 field problems on one set of operators (a parameter study in the sources)
        _case("cavity24_ensemble16", "march", 24, 24, 24, 1 / 24, 0.01916, 4, 4, 4, precision="mixed", members=16,
              tuned=True),
        # jittered mesh, 300 bisected subdomains of uneven size (ragged tiles), mixed precision
        _case("jitter64_rcb300_mixed", "march", 64, 32, 32, 1 / 32, 0.011826, rcb=300, jitter=True, precision="mixed",
              tuned=True),
        # the largest: the 48^3 cavity, the benchmark's own problem, in mixed precision and in FP64
        _case("cavity48_mixed", "march", 48, 48, 48, 1 / 48, 0.009579, 8, 8, 8, precision="mixed", tuned=True),
        _case("cavity48_fp64", "march", 48, 48, 48, 1 / 48, 0.009579, 8, 8, 8, tuned=True),
        # inverse design: objective and gradients on the 32^3 cavity with new random materials
        _case("cavity32_eps_gradient", "gradient", 32, 32, 32, 1 / 32, 0.02027, 8, 8, 4, eps=True),
        # new materials, factorisation and one step on a ragged tearing of a jittered mesh
        _case("jitter32_refactor", "refactor", 32, 16, 16, 1 / 16, 0.02365, rcb=40, jitter=True, eps=True),
        # the FP64 interface operator alone, as an outside Krylov solver or an analysis calls it
        _case("cavity32_coupled_apply", "coupled", 32, 32, 32, 1 / 32, 0.01437, 8, 8, 4),
    ]


def draw(rng):
    """A case of the same ranges: calls, sizes (log-uniform, odd ones included), tearings and options."""
    call = rng.choice(["march", "march", "march", "march", "default", "pic", "gradient", "refactor", "coupled", "schur"])
    n = [int(round(math.exp(rng.uniform(math.log(5), math.log(40))))) for _ in range(3)]
    while n[0] * n[1] * n[2] > 30000:
        n[rng.randrange(3)] -= 1
    if call in ("gradient", "pic"):
        n = [max(v, 8) for v in n]
    cells = n[0] * n[1] * n[2]
    per = math.exp(rng.uniform(math.log(30), math.log(300)))    # cells per subdomain
    parts = max(2, min(int(round(cells / per)), 600))
    jitter = call != "pic" and rng.random() < 0.5
    eps = call in ("gradient", "refactor")
    cell = 1.0 / max(n)
    dt = cell * (0.378 if jitter else 0.46) * (1.4 if eps else 1.0)
    members = rng.choice([1, 1, 2, 5, 16]) if call == "march" and cells < 6000 else 1
    solver = "cg" if call == "default" or (members == 1 and call in ("march", "pic") and rng.random() < 0.25) else "gmres"
    scheme = "dp2" if call == "march" and solver == "gmres" and rng.random() < 0.25 else "dp1"
    if scheme == "dp2" and members > 1:
        scheme = "dp1"
    precision = rng.choice(["fp64", "mixed"]) if call in ("march", "pic") else "fp64"
    if members > 1:
        precision = "mixed"
    case = _case("", call, n[0], n[1], n[2], cell, dt, rcb=parts, jitter=jitter, eps=eps, precision=precision,
                 solver=solver, scheme=scheme, graph=call != "default" and rng.random() < 0.8,
                 tuned=rng.random() < 0.5 and call == "march", members=members,
                 particles=int(round(math.exp(rng.uniform(math.log(1000), math.log(100000))))) if call == "pic" else 0)
    del case["name"]
    return case


# ---- inputs -----------------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _mesh(nx, ny, nz, cell, kx, ky, kz, rcb, jitter):
    """xyz, tets, part, number of subdomains, box side lengths."""
    L = (nx * cell, ny * cell, nz * cell)
    xyz, tets = W.kuhn_box(nx, ny, nz, *L)
    rng = np.random.default_rng(7)
    if jitter:
        xyz, rng = W.jitter_nodes(xyz, cell, L, 0.2, seed=7)
    if rcb:
        part = W.rcb_partition(W.tet_centroids(xyz, tets), rcb, rng.uniform(0.6, 1.4, size=rcb))
        return xyz, tets, part, rcb, L
    return xyz, tets, W.block_partition(nx, ny, nz, kx, ky, kz), kx * ky * kz, L


def _geometry(case):
    return _mesh(case["nx"], case["ny"], case["nz"], case["cell"], case["kx"], case["ky"], case["kz"], case["rcb"],
                 case["jitter"])


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Edges:
    """Interior edges of the mesh: sorted node pairs, oriented from the lower to the higher id."""

    def __init__(self, case, dev):
        xyz, tets, part, n_sub, L = _geometry(case)
        self.xyz = torch.as_tensor(xyz, device=dev)
        t = torch.as_tensor(tets, device=dev).long()
        self.tets, self.part, self.n_sub, self.n_nodes, self.L = t, torch.as_tensor(part, device=dev).long(), n_sub, len(xyz), L
        N = self.n_nodes
        ea, eb = t[:, [0, 0, 0, 1, 1, 2]], t[:, [1, 2, 3, 2, 3, 3]]
        key = torch.minimum(ea, eb) * N + torch.maximum(ea, eb)
        self.sign = torch.where(ea < eb, 1.0, -1.0).to(torch.float64)
        ukey, inv = torch.unique(key, return_inverse=True)
        f = torch.cat([t[:, [1, 2, 3]], t[:, [0, 2, 3]], t[:, [0, 1, 3]], t[:, [0, 1, 2]]]).sort(dim=1).values
        self.faces, cnt = torch.unique((f[:, 0] * N + f[:, 1]) * N + f[:, 2], return_counts=True)
        wall = self.faces[cnt == 1]
        a, b, c = wall // (N * N), wall // N % N, wall % N
        pec = torch.isin(ukey, torch.cat([a * N + b, a * N + c, b * N + c]))
        self.key = ukey[~pec]
        self.n = self.key.numel()
        dof = torch.full_like(ukey, -1)
        dof[~pec] = torch.arange(self.n, device=dev)
        self.tet_dof = dof[inv]
        self.lo, self.hi = self.key // N, self.key % N

    def dofs(self, lo, hi):
        """dof of each node pair, -1 on the wall."""
        k = lo * self.n_nodes + hi
        p = torch.searchsorted(self.key, k).clamp(max=self.n - 1)
        return torch.where(self.key[p] == k, p, -1)

    def source(self, case):
        """1 on the z-directed line of edges through the middle of the box."""
        pairs = torch.as_tensor(W.z_line_node_pairs(case["nx"], case["ny"], case["nz"], case["nx"] // 2, case["ny"] // 2),
                                device=self.key.device)
        v = torch.zeros(self.n, dtype=torch.float64, device=self.key.device)
        d = self.dofs(pairs[:, 0], pairs[:, 1])
        v[d[d >= 0]] = 1.0
        return v

    def modes(self, rng, times):
        """Edge values at each time of five ringing cavity modes with amplitudes from rng."""
        mid, vec = 0.5 * (self.xyz[self.lo] + self.xyz[self.hi]), self.xyz[self.hi] - self.xyz[self.lo]
        out = [torch.zeros(self.n, dtype=torch.float64, device=mid.device) for _ in times]
        for _ in range(5):
            m, amp, phase = rng.integers(1, 4, 3), rng.normal(size=3), rng.uniform(0, 2 * math.pi)
            kv = [math.pi * int(m[a]) / self.L[a] for a in range(3)]
            s = [torch.sin(kv[a] * mid[:, a]) for a in range(3)]
            c = [torch.cos(kv[a] * mid[:, a]) for a in range(3)]
            v = (amp[0] * c[0] * s[1] * s[2] * vec[:, 0] + amp[1] * s[0] * c[1] * s[2] * vec[:, 1] +
                 amp[2] * s[0] * s[1] * c[2] * vec[:, 2])
            w = math.sqrt(kv[0] ** 2 + kv[1] ** 2 + kv[2] ** 2)
            for o, t in zip(out, times):
                o += math.cos(w * t + phase) * v
        return out


def _start_fields(case, E, seed):
    """(e^0, e^-1) of every member, members one after the other."""
    e = [E.modes(np.random.default_rng([seed, 17, r]), (0.0, -case["dt"])) for r in range(case["members"])]
    return torch.cat([a for a, _ in e]), torch.cat([b for _, b in e])


def _pulse(case, n, t0=20.0):
    """Second differences of the integrated pulse, one per step, then nothing."""
    t = case["dt"] * np.arange(-1, n + 1, dtype=np.float64)
    g = W.gaussian_pulse_G(t, t0 * case["dt"], 6.0 * case["dt"])
    return [float(v) for v in g[2:] - 2.0 * g[1:-1] + g[:-2]]


def _eps(case, seed, n_tets, dev):
    """Random materials U[1, 4] per tet."""
    return torch.as_tensor(np.random.default_rng([seed, 3]).uniform(1.0, 4.0, n_tets), device=dev)


def _beam(case, seed):
    """Injected during the first 16 cycles, slow enough to stay in flight for a long march."""
    xyz, _, _, _, L = _geometry(case)
    rng = np.random.default_rng([seed, 5])
    n = case["particles"]
    off = np.clip(rng.normal(0.0, 0.05 * min(L[:2]), size=(n, 2)), -0.45 * min(L[:2]), 0.45 * min(L[:2]))
    x = np.column_stack([L[0] / 2 + off[:, 0], L[1] / 2 + off[:, 1], np.zeros(n)])
    return x, np.tile([0.0, 0.0, 0.05], (n, 1)), rng.uniform(0.0, 16 * case["dt"], n), -1e-6, -1.0


def _probes(L, cell):
    """Four points a few cells off the source line."""
    c = [v / 2 for v in L]
    return np.array([[c[0] + 1.7 * cell, c[1] + 0.3 * cell, c[2] - 1.4 * cell], [c[0] - 2.3 * cell, c[1] + 1.2 * cell, c[2]],
                     [c[0] + 0.6 * cell, c[1] - 2.1 * cell, c[2] + 2.2 * cell], [c[0] - 1.1 * cell, c[1] - 1.6 * cell, c[2]]])


def _params(case):
    if case["call"] == "default":
        return None
    mixed = case["precision"] == "mixed"
    kw = dict(precision=D.DD_MIXED if mixed else D.DD_FP64, tol=1e-5 if mixed else 1e-10, max_refine=6,
              refine_tol=1e-10 if mixed else 1e-12, chunk=2 if case["graph"] else 8, use_graph=int(case["graph"]),
              solver=D.DD_SOLVER_SCHUR_CG if case["solver"] == "cg" else D.DD_SOLVER_COUPLED_GMRES,
              scheme=D.DD_SCHEME_DP2 if case["scheme"] == "dp2" else D.DD_SCHEME_DP1, members=case["members"])
    if case["call"] in ("gradient", "refactor", "coupled", "schur"):
        kw["tol"] = 1e-12
    return D.make_params(**kw)


def prepare(case, seed):
    dev, dt, call = _device(), case["dt"], case["call"]
    xyz, tets, part, n_sub, L = _geometry(case)
    E = _Edges(case, dev)
    s = dict(call=call, dt=dt)
    if call == "gradient":
        s["march"] = A.ProbeMarch(dict(xyz=xyz, tets=tets, part=part, n_sub=n_sub, probes=_probes(L, case["cell"]),
                                       source_pairs=W.z_line_node_pairs(case["nx"], case["ny"], case["nz"],
                                                                        case["nx"] // 2, case["ny"] // 2),
                                       d2g=_pulse(case, GRAD_STEPS, t0=4.0), dt=dt), params=_params(case))
        s["eps"] = _eps(case, seed, len(tets), dev)
        s["amp"] = torch.tensor(1.0 + 0.001 * (seed % 97), dtype=torch.float64, device=dev)
        return s
    fs = D.FieldSolver(xyz, tets, part, n_sub, params=_params(case))
    if call == "pic":
        fs.set_beam(*_beam(case, seed))
    fs.bind()
    fs.factor(dt)
    s["fs"] = fs
    if case["tuned"]:
        D.dd_autotune(fs.h)
    if call in ("coupled", "schur"):
        n = fs.n_lambda + (fs.sizes.n_corner if call == "coupled" else 0)
        s["u"] = torch.as_tensor(np.random.default_rng([seed, 1]).normal(size=n), device=dev)
        return s
    s["out"] = torch.empty(fs.n_dof, dtype=torch.float64, device=dev)
    if call == "pic":
        s["x"] = torch.empty(3 * case["particles"], dtype=torch.float64, device=dev)
        s["status"] = torch.empty(case["particles"], dtype=torch.int32, device=dev)
        s["G"], s["prev"] = torch.empty_like(s["out"]), torch.empty_like(s["out"])
        s["b"] = torch.empty(D.dd_pic_state(fs.h), dtype=torch.float64, device=dev)
        for _ in range(PIC_STEPS):
            D.dd_pic_step(fs.h, stats=False)
        return s
    s["source"] = torch.cat([(1.0 + 0.25 * r) * E.source(case) for r in range(case["members"])])
    if call == "refactor":
        s["eps"], s["scale"] = _eps(case, seed, len(tets), dev), 1.0 + 0.001 * (seed % 97)
        return s
    s["pulse"], s["step"] = _pulse(case, 60), 0
    fs.set_state(*_start_fields(case, E, seed), 0)
    for _ in range(WARM_STEPS):
        _step(s)
    return s


def _step(s):
    k = s["step"]
    s["step"] = k + 1
    if s["call"] == "default":
        s["fs"].step(s["source"] * s["pulse"][k] if k < len(s["pulse"]) else None, s["out"])
    elif k < len(s["pulse"]):
        D.dd_step_scaled(s["fs"].h, s["source"], s["pulse"][k], s["out"], stats=False)
    else:
        D.dd_step(s["fs"].h, None, s["out"], stats=False)
    return s["out"]


def run(state):
    s = state
    call = s["call"]
    if call == "gradient":
        eps, amp = s["eps"].detach().requires_grad_(), s["amp"].detach().requires_grad_()
        J = A.probe_objective(eps, amp, s["march"], GRAD_STEPS)
        J.backward()
        return {"J": J.detach(), "eps": eps.grad, "amp": amp.grad}
    fs = s["fs"]
    if call == "coupled":
        return fs.coupled_apply(s["u"])
    if call == "schur":
        return fs.schur_apply(s["u"])
    if call == "refactor":
        D.dd_set_eps(fs.h, s["eps"])
        fs.factor(s["dt"])
        D.dd_step_scaled(fs.h, s["source"], s["scale"], s["out"], stats=False)
        return s["out"]
    if call == "pic":
        D.dd_pic_step(fs.h, stats=False)
        D.dd_get_state(fs.h, s["out"], s["prev"])
        D.dd_pic_state(fs.h, s["x"], s["status"], s["G"], s["b"])
        return {"e": s["out"], "x": s["x"], "status": s["status"], "G": s["G"], "b": s["b"]}
    return _step(s)


# ---- what a pass cannot do without ------------------------------------------------------------

@functools.lru_cache(maxsize=16)
def _local_sizes(*geometry):
    """Per subdomain: interior, interface and corner unknowns; and the number of unknowns."""
    case = dict(zip(("nx", "ny", "nz", "cell", "kx", "ky", "kz", "rcb", "jitter"), geometry))
    E = _Edges(case, torch.device("cpu"))
    sub, dof, mult = _tear(E)
    m = mult[dof]
    return [torch.bincount(sub[sel], minlength=E.n_sub).double() for sel in (m == 1, m == 2, m > 2)], E.n, E.n_sub


def _tear(E):
    """Local copies (subdomain, dof), sorted, and the number of copies of each dof."""
    d = E.tet_dof.reshape(-1)
    s = E.part[:, None].expand(-1, 6).reshape(-1)
    key = torch.unique((s * E.n + d)[d >= 0])
    sub, dof = key // E.n, key % E.n
    return sub, dof, torch.bincount(dof, minlength=E.n)


def work(case):
    """The factored local operators (symmetric, each distinct element once, at the precision they are applied in),
    read once, with one multiplication and one addition per element and right-hand side; the fields and sources read
    and written once.  The interface operator alone: its [interface | corner] block.  A factorisation: the symmetric
    inverse of every local matrix (n^3 flops) and its storage written once.  A gradient: that, and two operator
    reads' arithmetic per forward and per backward step."""
    (nI, nG, nC), n, n_sub = _local_sizes(*(case[k] for k in ("nx", "ny", "nz", "cell", "kx", "ky", "kz", "rcb",
                                                              "jitter")))
    ns, g, R = nI + nG + nC, nG + nC, case["members"]
    elem = 4 if case["precision"] == "mixed" else 8
    full = float((ns * (ns + 1) / 2).sum())
    block = float((g * (g + 1) / 2).sum())
    if case["call"] in ("coupled", "schur"):
        u = float(nG.sum()) / 2 + (float(nC.sum()) / 4 if case["call"] == "coupled" else 0.0)
        return {"bytes": 8 * block + 16 * u, "flops": 4 * block}
    step = {"bytes": elem * full + R * 8.0 * 4 * n, "flops": 4.0 * R * full}
    if case["call"] == "pic":
        step["bytes"] += case["particles"] * (2 * 56 + 28) + 8.0 * 3 * n
    if case["call"] in ("refactor", "gradient"):
        steps = 1 if case["call"] == "refactor" else 3 * GRAD_STEPS
        return {"bytes": 8 * full + 8 * 6.0 * case["nx"] * case["ny"] * case["nz"] + steps * 8.0 * 4 * n,
                "flops": float((ns ** 3).sum()) + steps * step["flops"]}
    return step


# ---- what it should give, in 64 bits ----------------------------------------------------------

class _Fem:
    """Whitney edge elements: element matrices and assembled sparse matrices, in 64 bits."""

    def __init__(self, case, dev, eps=None):
        E = self.E = _Edges(case, dev)
        X = E.xyz[E.tets]
        Dm = X[:, 1:] - X[:, :1]
        self.vol = torch.linalg.det(Dm).abs() / 6.0
        inv = torch.linalg.inv(Dm).transpose(1, 2)                     # gradients of lambda_1..3
        self.grad = torch.cat([-inv.sum(1, keepdim=True), inv], 1)
        a, b = [0, 0, 0, 1, 1, 2], [1, 2, 3, 2, 3, 3]
        G = self.grad @ self.grad.transpose(1, 2)
        M = (torch.ones(4, 4, dtype=torch.float64, device=dev) + torch.eye(4, dtype=torch.float64, device=dev)) / 20.0
        ab = lambda Q, p, q: Q[..., p, :][..., :, q]  # noqa: E731
        self.T = self.vol[:, None, None] * (ab(M, a, a) * ab(G, b, b) - ab(M, a, b) * ab(G, b, a) -
                                            ab(M, b, a) * ab(G, a, b) + ab(M, b, b) * ab(G, a, a))
        curl = 2.0 * torch.linalg.cross(self.grad[:, a], self.grad[:, b])
        self.S = self.vol[:, None, None] * (curl @ curl.transpose(1, 2))
        ss = E.sign[:, :, None] * E.sign[:, None, :]
        self.T, self.S = self.T * ss, self.S * ss
        eps = torch.ones_like(self.vol) if eps is None else eps
        self.A = self.matrix(eps[:, None, None] * self.T + case["dt"] ** 2 / 4 * self.S)
        self.K = self.matrix(self.S)

    def matrix(self, elem, rows=None, n=None):
        """Sparse matrix of element matrices; `rows` maps (tet, local edge) to an unknown, -1 for none."""
        r = self.E.tet_dof if rows is None else rows
        n = self.E.n if n is None else n
        i, j = r[:, :, None].expand(-1, 6, 6), r[:, None, :].expand(-1, 6, 6)
        keep = (i >= 0) & (j >= 0)
        key = i[keep] * n + j[keep]
        ukey, inv = torch.unique(key, return_inverse=True)
        val = torch.zeros(ukey.numel(), dtype=torch.float64, device=key.device).index_add_(0, inv, elem[keep])
        ptr = torch.searchsorted(ukey // n, torch.arange(n + 1, device=key.device))
        return torch.sparse_csr_tensor(ptr, ukey % n, val, (n, n))


def _diagonal(A):
    n = A.shape[0]
    row = torch.repeat_interleave(torch.arange(n, device=A.device), A.crow_indices().diff())
    on = row == A.col_indices()
    d = torch.ones(n, dtype=torch.float64, device=A.device)
    d[row[on]] = A.values()[on]
    return d


def _cg(A, B, dinv):
    """A X = B by Jacobi CG on every column, to the last digits."""
    X = torch.zeros_like(B)
    R = B.clone()
    Z = dinv[:, None] * R
    P, rz = Z.clone(), (R * Z).sum(0)
    stop = rz.clone() * 1e-31
    for k in range(1000):
        Q = A @ P
        pq = (P * Q).sum(0)
        alpha = torch.where(pq > 0, rz / pq, torch.zeros_like(pq))
        X += alpha * P
        R -= alpha * Q
        if k % 50 == 49:
            R = B - A @ X
        Z = dinv[:, None] * R
        rz_new = (R * Z).sum(0)
        if k % 5 == 4 and bool((rz_new <= stop).all()):
            break
        P = Z + torch.where(rz > 0, rz_new / rz, torch.zeros_like(rz)) * P
        rz = rz_new
    return X


def _interface_exact(case, seed):
    """The interface operators from the torn system: B_r A_rr^-1 B_r^T with the corners free (coupled) or tied (schur)."""
    dev = _device()
    F = _Fem(case, dev)
    E = F.E
    sub, dof, mult = _tear(E)
    lam = torch.nonzero(mult == 2)[:, 0]
    cor = torch.nonzero(mult > 2)[:, 0]
    r = mult[dof] <= 2
    # unknowns: every local copy of an r dof, then the corners
    local = torch.full((sub.numel(),), -1, device=dev)
    nr = int(r.sum())
    local[r] = torch.arange(nr, device=dev)
    cid = torch.full((E.n,), -1, device=dev)
    cid[cor] = torch.arange(cor.numel(), device=dev)
    local[~r] = nr + cid[dof[~r]]
    pos = torch.searchsorted(sub * E.n + dof, (E.part[:, None] * E.n + E.tet_dof).clamp(min=0))
    rows = torch.where(E.tet_dof >= 0, local[pos.clamp(max=sub.numel() - 1)], -1)
    n = nr + cor.numel()
    M = F.matrix(F.T + case["dt"] ** 2 / 4 * F.S, rows, n)
    first = torch.searchsorted(dof.sort().values, lam)          # copies of a dof in subdomain order
    order = torch.argsort(dof * E.n_sub + sub)
    s1, s2 = local[order[first]], local[order[first + 1]]
    u = torch.as_tensor(np.random.default_rng([seed, 1]).normal(
        size=lam.numel() + (cor.numel() if case["call"] == "coupled" else 0)), device=dev)
    b = torch.zeros(n, 1, dtype=torch.float64, device=dev)
    b[s1, 0], b[s2, 0] = u[:lam.numel()], -u[:lam.numel()]
    dinv = 1.0 / _diagonal(M)
    if case["call"] == "schur":
        x = _cg(M, b, dinv)[:, 0]
        return x[s1] - x[s2]
    c = torch.zeros(n, 1, dtype=torch.float64, device=dev)
    c[nr:, 0] = u[lam.numel():]
    Mc = (M @ c)
    rhs = b + Mc
    rhs[nr:] = 0.0

    class Interior:     # the r block of M, with the corner rows and columns left out
        def __matmul__(self, P):
            Q = M @ P
            Q[nr:] = 0.0
            return Q

    z = _cg(Interior(), rhs, dinv)
    zc = (M @ z)[nr:, 0]
    return torch.cat([z[s1, 0] - z[s2, 0], Mc[nr:, 0] - zc])


def _kuhn_locate(E, case, x):
    """The tet of each point of an unjittered box, by barycentric coordinates among its cube's six tets."""
    n = torch.tensor([case["nx"], case["ny"], case["nz"]], device=x.device)
    q = torch.minimum((x / case["cell"]).floor().long().clamp(min=0), n - 1)
    return (q[:, 0] + n[0] * (q[:, 1] + n[1] * q[:, 2]))[:, None] * 6 + torch.arange(6, device=x.device)


def _pic_exact(case, seed):
    """The PIC cycle with every path cut at the grid planes x_a = i h and x_a - x_b = i h that bound the tets."""
    dev, dt, h = _device(), case["dt"], case["cell"]
    F = _Fem(case, dev)
    E = F.E
    x, v, t_inj, q, qm = _beam(case, seed)
    x, v, t_inj = (torch.as_tensor(w, device=dev) for w in (x, v, t_inj))
    status = torch.zeros(len(t_inj), dtype=torch.int32, device=dev)
    N = E.n_nodes
    fa, fb, fc = E.faces // (N * N), E.faces // N % N, E.faces % N
    fe = torch.stack([E.dofs(fa, fb), E.dofs(fb, fc), E.dofs(fa, fc)], 1)
    fs = torch.tensor([1.0, 1.0, -1.0], dtype=torch.float64, device=dev)

    def curl(e):
        return (torch.where(fe >= 0, e[fe.clamp(min=0)], torch.zeros((), dtype=torch.float64, device=dev)) * fs).sum(1)

    def lam(t, p):
        l3 = (F.grad[t][:, 1:] @ (p - E.xyz[E.tets[t, 0]])[:, :, None])[:, :, 0]
        return torch.cat([1.0 - l3.sum(1, keepdim=True), l3], 1)

    def locate(p):
        c = _kuhn_locate(E, case, p)
        low = torch.stack([lam(c[:, k], p).min(1).values for k in range(6)], 1)
        return c[torch.arange(len(p), device=dev), low.argmax(1)]

    la, lb = [0, 0, 0, 1, 1, 2], [1, 2, 3, 2, 3, 3]
    planes = torch.tensor([[1, 0, 0], [0, 1, 0], [0, 0, 1], [1, -1, 0], [0, 1, -1], [1, 0, -1]], dtype=torch.float64,
                          device=dev) / h

    def fields(p, e, b):
        t = locate(p)
        l, g = lam(t, p), F.grad[t]
        d = E.tet_dof[t]
        ev = torch.where(d >= 0, e[d.clamp(min=0)], torch.zeros((), dtype=torch.float64, device=dev)) * E.sign[t]
        Ex = (ev[:, :, None] * (l[:, la, None] * g[:, lb] - l[:, lb, None] * g[:, la])).sum(1)
        Bx = torch.zeros_like(Ex)
        for f in ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2)):
            nodes, order = E.tets[t][:, list(f)].sort(dim=1)
            loc = torch.tensor(f, device=dev)[order]
            fid = torch.searchsorted(E.faces, (nodes[:, 0] * N + nodes[:, 1]) * N + nodes[:, 2])
            at = torch.arange(len(p), device=dev)
            ga, gb, gc = (g[at, loc[:, k]] for k in range(3))
            wa, wb, wc = (l[at, loc[:, k], None] for k in range(3))
            Bx += 2.0 * b[fid][:, None] * (wa * torch.linalg.cross(gb, gc) + wb * torch.linalg.cross(gc, ga) +
                                           wc * torch.linalg.cross(ga, gb))
        return Ex, Bx

    e0 = e1 = torch.zeros(E.n, dtype=torch.float64, device=dev)
    G, dep0, b = torch.zeros_like(e0), torch.zeros_like(e0), torch.zeros(len(E.faces), dtype=torch.float64, device=dev)
    dinv = 1.0 / _diagonal(F.A)
    for k in range(PIC_STEPS + 1):
        t0, t1 = k * dt, (k + 1) * dt
        fly = status == 1
        new = (status == 0) & (t_inj <= t1)
        if bool(fly.any()):
            Ex, Bx = fields(x[fly], e1, b)
            vm = v[fly] + 0.5 * qm * dt * Ex
            tv = 0.5 * qm * dt * Bx
            vp = vm + torch.linalg.cross(vm, tv)
            v[fly] = vm + torch.linalg.cross(vp, 2.0 * tv / (1.0 + (tv * tv).sum(1, keepdim=True))) + 0.5 * qm * dt * Ex
        tau = torch.where(fly, dt, t1 - t_inj.clamp(min=t0))
        status[new] = 1
        act = status == 1
        p0, p1 = x[act], x[act] + tau[act, None] * v[act]
        u0, u1 = p0 @ planes.T, p1 @ planes.T
        up = u1 > u0
        plane = torch.where(up, u0.floor() + 1.0, u0.ceil() - 1.0)       # the first plane ahead of each family
        cut = torch.where(u1 != u0, (plane - u0) / (u1 - u0), torch.ones_like(u0)).clamp(0.0, 1.0)
        cuts = torch.cat([torch.zeros_like(cut[:, :1]), cut.sort(dim=1).values, torch.ones_like(cut[:, :1])], 1)
        dep = torch.zeros_like(e0)
        for c in range(cuts.shape[1] - 1):
            a, z = p0 + cuts[:, c, None] * (p1 - p0), p0 + cuts[:, c + 1, None] * (p1 - p0)
            on = cuts[:, c + 1] > cuts[:, c]
            if not bool(on.any()):
                continue
            a, z = a[on], z[on]
            t = locate(0.5 * (a + z))
            l0, l1 = lam(t, a), lam(t, z)
            w = q * E.sign[t] * (l0[:, la] * l1[:, lb] - l0[:, lb] * l1[:, la])
            d = E.tet_dof[t]
            dep.index_add_(0, d[d >= 0], w[d >= 0])
        x[act] = p1
        G = G + dep
        rhs = -dt * dt * (F.K @ e1[:, None]) - (dep - dep0)[:, None]
        e2 = 2.0 * e1 - e0 + _cg(F.A, rhs, dinv)[:, 0]
        b = b - 0.5 * dt * (curl(e2) + curl(e1))
        e0, e1, dep0 = e1, e2, dep
    inside = bool(((x > 0.0) & (x < torch.tensor(E.L, dtype=torch.float64, device=dev))).all())
    if not inside:      # a particle that reached a wall stops there: not followed here
        return None
    return {"e": e1, "x": x.reshape(-1), "status": status, "G": G, "b": b}


def exact(case, seed):
    call, dt, dev = case["call"], case["dt"], _device()
    if call in ("coupled", "schur"):
        return _interface_exact(case, seed)
    if call == "pic":
        return _pic_exact(case, seed)
    eps = _eps(case, seed, len(_geometry(case)[1]), dev) if case["eps"] else None
    F = _Fem(case, dev, eps)
    dinv = 1.0 / _diagonal(F.A)
    src = F.E.source(case)[:, None]
    if call == "refactor":
        return _cg(F.A, -(1.0 + 0.001 * (seed % 97)) * src, dinv)[:, 0]
    if call == "gradient":
        return _gradient_exact(case, seed, F, dinv, src[:, 0])
    R = case["members"]
    e1, e0 = (v.reshape(R, -1).T.contiguous() for v in _start_fields(case, F.E, seed))
    src = torch.cat([(1.0 + 0.25 * r) * src for r in range(R)], 1)
    pulse = _pulse(case, 60)
    for k in range(WARM_STEPS + 1):
        e0, e1 = e1, 2.0 * e1 - e0 + _cg(F.A, -dt * dt * (F.K @ e1) - pulse[k] * src, dinv)
    return e1.T.reshape(-1)


def _gradient_exact(case, seed, F, dinv, src):
    dev, dt, E = _device(), case["dt"], F.E
    amp, pulse = 1.0 + 0.001 * (seed % 97), _pulse(case, GRAD_STEPS, t0=4.0)
    pts = torch.as_tensor(_probes(E.L, case["cell"]), device=dev)
    rows = []       # E at each probe: a [3, 6] map of its tet's edge values
    for p in pts:
        l3 = (F.grad[:, 1:] @ (p - E.xyz[E.tets[:, 0]])[:, :, None])[:, :, 0]
        l = torch.cat([1.0 - l3.sum(1, keepdim=True), l3], 1)
        t = int(torch.nonzero((l >= -1e-12).all(1))[0, 0])
        a, b = [0, 0, 0, 1, 1, 2], [1, 2, 3, 2, 3, 3]
        Wt = (l[t, a, None] * F.grad[t, b] - l[t, b, None] * F.grad[t, a]) * E.sign[t, :, None]
        d = E.tet_dof[t]
        rows.append((d[d >= 0], Wt[d >= 0]))
    solve = lambda v: _cg(F.A, v[:, None], dinv)[:, 0]  # noqa: E731
    K = lambda v: (F.K @ v[:, None])[:, 0]  # noqa: E731
    zero = torch.zeros(E.n, dtype=torch.float64, device=dev)
    e = {-1: zero, 0: zero}
    J = torch.zeros((), dtype=torch.float64, device=dev)
    for k in range(GRAD_STEPS):
        e[k + 1] = 2.0 * e[k] - e[k - 1] + solve(-dt * dt * K(e[k]) - amp * pulse[k] * src)
        for d, Wt in rows:
            J += ((e[k + 1][d] @ Wt) ** 2).sum()
    e[-1] = zero
    mu1 = mu2 = zero
    geps = torch.zeros(len(E.tets), dtype=torch.float64, device=dev)
    gamp = torch.zeros((), dtype=torch.float64, device=dev)
    local = lambda v: torch.where(E.tet_dof >= 0, v[E.tet_dof.clamp(min=0)], torch.zeros((), dtype=torch.float64,  # noqa: E731
                                                                                      device=dev))
    for k in range(GRAD_STEPS, 0, -1):
        seed_v = zero.clone()
        for d, Wt in rows:
            seed_v.index_add_(0, d, 2.0 * (Wt @ (e[k][d] @ Wt)))
        mu0 = 2.0 * mu1 - mu2 + solve(-dt * dt * K(mu1) + seed_v)
        acc = e[k] - 2.0 * e[k - 1] + e.get(k - 2, zero)
        geps -= (local(mu0)[:, :, None] * F.T * local(acc)[:, None, :]).sum((1, 2))
        gamp -= pulse[k - 1] * (mu0 @ src)
        mu1, mu2 = mu0, mu1
    return {"J": J, "eps": geps, "amp": gamp}
