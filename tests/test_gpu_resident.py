"""The mixed-precision coupled GMRES and the Schur CG as one kernel (operators resident in
shared memory) against the kernel-per-stage solve (which sym_fp32 = 0 selects): the
same Arnoldi counts up to FP32 rounding of the stopping test (cold solves), fields equal
to the refinement tolerance; one, two and four CTAs per SM, short and long restarts, both
schemes, eager and graph steps; a spent budget and a non-finite source are reported."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def march(w, dt, n, **kw):
    prm = D.make_params(**{**dict(precision=D.DD_MIXED, tol=1e-5, refine_tol=1e-11, max_refine=8,
                                  solver=D.DD_SOLVER_COUPLED_GMRES), **kw})
    fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, w.eps, w.mu, params=prm).bind()
    fs.factor(dt)
    src = torch.tensor(np.random.default_rng(2).standard_normal(fs.n_dof), device="cuda")
    out = torch.empty_like(src)
    fields, iters = [], []
    D.dd_profile(fs.h, 1, read=False)
    for k in range(n):
        iters.append(D.dd_step_scaled(fs.h, src, 1.0 / (1 + k), out)["iters"])
        fields.append(out.clone())
    D.dd_profile(fs.h, 0, read=False)
    launches = D.dd_profile(fs.h)["total_launches"]
    fs.close()
    return fields, iters, launches


# 8 subdomains (one CTA per SM), 216 (two), 512 of 2^3 cubes (four); a ragged bisection
def problem(kind):
    if kind == "ragged":
        n, L = (9, 7, 8), (9 / 7, 1.0, 8 / 7)
        xyz, tets = W.kuhn_box(*n, *L)
        xyz, rng = W.jitter_nodes(xyz, 1 / 7, L, 0.2, seed=3)
        part = W.rcb_partition(W.tet_centroids(xyz, tets), 11, rng.uniform(0.6, 1.4, size=11))
        return W.Workload("ragged", xyz, tets, part, 11, None, 1.0, 6, W.z_line_node_pairs(*n, 4, 3)), 0.05
    n, k = {"sub8": (8, 2), "sub216": (12, 6), "sub512": (16, 8)}[kind]
    return W.box(n, n, n, k, k, k), 0.46 / n


@pytest.mark.parametrize("kind", ["sub8", "sub216", "sub512", "ragged"])
@pytest.mark.parametrize("kw", [dict(), dict(restart=7, use_graph=1, chunk=2), dict(restart=32, precond=0),
                                dict(scheme=D.DD_SCHEME_DP2, use_graph=1)])
def test_resident_solve_matches_staged(kind, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w, dt = problem(kind)
    f1, i1, l1 = march(w, dt, 4, **kw)
    f0, i0, l0 = march(w, dt, 4, sym_fp32=0, **kw)
    assert l1 < l0 / 2                      # the resident form is the one in use
    for a, b in zip(f1, f0):
        assert torch.linalg.norm(a - b) <= 1e-9 * torch.linalg.norm(b)
    # one cold solve to a fixed tolerance: the residuals differ by FP32 rounding, so the stopping
    # test falls on the same Arnoldi step or on its neighbour (a later refinement pass takes its
    # tolerance from the residual before it, so counts of whole steps are not comparable)
    one = dict(max_refine=1, refine_tol=1.0, warm_start=0)
    for a, b in zip(march(w, dt, 3, **kw, **one)[1], march(w, dt, 3, sym_fp32=0, **kw, **one)[1]):
        assert abs(a - b) <= 1
    f2, i2, _ = march(w, dt, 4, **kw)       # fixed summation order: bitwise reproducible
    assert i2 == i1 and all(torch.equal(a, b) for a, b in zip(f1, f2))


@pytest.mark.parametrize("kind", ["sub8", "sub216", "ragged"])
@pytest.mark.parametrize("graph", [0, 1])
def test_resident_cg(kind, graph):
    """Mixed against the kernel-per-stage CG (sym_fp32 = 0); FP64 against the coupled GMRES
    (another kernel family) to the solves' tolerance."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w, dt = problem(kind)
    cg = dict(solver=D.DD_SOLVER_SCHUR_CG, use_graph=graph)
    f1, _, l1 = march(w, dt, 4, **cg)
    f0, _, l0 = march(w, dt, 4, sym_fp32=0, **cg)
    assert l1 < l0 / 2
    for a, b in zip(f1, f0):
        assert torch.linalg.norm(a - b) <= 1e-9 * torch.linalg.norm(b)
    one = dict(max_refine=1, refine_tol=1.0, warm_start=0)
    for a, b in zip(march(w, dt, 3, **cg, **one)[1], march(w, dt, 3, sym_fp32=0, **cg, **one)[1]):
        assert abs(a - b) <= 1
    d = dict(precision=D.DD_FP64, tol=1e-13, max_it=2000)
    f2, _, l2 = march(w, dt, 4, **cg, **d)
    f3, _, _ = march(w, dt, 4, **d)
    h = D.dd_setup(w.xyz, w.tets, w.part, w.n_sub)
    m = D.dd_get_maps(h)
    D.dd_destroy(h)
    if (m["n_gam"] + m["n_cor"]).max() <= 150:   # the FP64 rows of a larger block do not fit a CTA
        assert l2 < 4 * 25
    for a, b in zip(f2, f3):
        assert torch.linalg.norm(a - b) <= 1e-10 * torch.linalg.norm(b)
    f4, _, _ = march(w, dt, 4, **cg, **d)
    assert all(torch.equal(a, b) for a, b in zip(f2, f4))


def test_resident_budget_and_nonfinite():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w, dt = problem("sub8")
    for graph in (0, 1):
        prm = D.make_params(precision=D.DD_MIXED, tol=1e-6, max_it=3, max_refine=1, use_graph=graph,
                            solver=D.DD_SOLVER_COUPLED_GMRES)
        fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, params=prm).bind()
        fs.factor(dt)
        src = torch.tensor(np.random.default_rng(2).standard_normal(fs.n_dof), device="cuda")
        st = D.dd_step(fs.h, src, None, raise_on_error=False)
        assert st["rc"] == D.DD_ERR_NO_CONVERGENCE and st["iters"] == 3
        src[5] = float("nan")
        assert D.dd_step(fs.h, src, None, raise_on_error=False)["rc"] == D.DD_ERR_NONFINITE
        fs.set_params(D.make_params(precision=D.DD_MIXED, tol=1e-6, max_refine=6, use_graph=graph,
                                    solver=D.DD_SOLVER_COUPLED_GMRES))
        z = torch.zeros(fs.n_dof, dtype=torch.float64, device="cuda")
        fs.set_state(z, z, 0)
        st = D.dd_step(fs.h, None, None)    # zero right-hand side: nothing to do
        assert st["iters"] == 0 and not fs.get_state()[0].any()
        fs.close()
