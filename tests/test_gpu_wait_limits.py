"""Every bounded device wait of a step, made to run out by dd_set_wait_limit: the step is
reported as DD_ERR_TIMEOUT and not taken, the context stays usable, and the march goes on
as if nothing had happened.  One problem per kernel that waits: the fixed-point FP64 GEMV
(64 subdomains), the one-kernel Arnoldi and CG steps (8 large subdomains, dense FP64
GEMVs, which wait for nothing), the one-kernel interface solves of small tearings (216
subdomains) in FP64 and mixed precision.  No GPU fault is involved.

Tolerances: the solves after the interrupted step start cold, so the fields agree with
those of an undisturbed march to the tolerance of the solves (FP64 1e-13, mixed 1e-11)
times a margin for the steps between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GMRES, CG = D.DD_SOLVER_COUPLED_GMRES, D.DD_SOLVER_SCHUR_CG
PROBLEMS = {
    "fixed_gmres": (16, 4, D.DD_FP64, GMRES), "fixed_cg": (16, 4, D.DD_FP64, CG),
    "step_gmres": (12, 2, D.DD_FP64, GMRES), "step_cg": (12, 2, D.DD_FP64, CG),
    "resident_cg64": (12, 6, D.DD_FP64, CG), "resident_cg32": (12, 6, D.DD_MIXED, CG),
    "resident_gmres32": (12, 6, D.DD_MIXED, GMRES),
}


def solver(kind, graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, k, prec, solver_ = PROBLEMS[kind]
    w = W.box(n, n, n, k, k, k)
    mixed = prec == D.DD_MIXED
    prm = D.make_params(precision=prec, tol=1e-5 if mixed else 1e-13, refine_tol=1e-11, max_refine=8, max_it=2000,
                        solver=solver_, use_graph=graph)
    fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, w.eps, w.mu, params=prm).bind()
    fs.factor(0.46 / n)
    return fs


def march(fs, interrupt):
    src = torch.tensor(np.random.default_rng(2).standard_normal(fs.n_dof), device="cuda")
    out = torch.empty_like(src)
    fields = []
    for k in range(4):
        if interrupt and k == 2:
            e0, e1, step = fs.get_state()
            D.dd_set_wait_limit(fs.h, 4)
            st = D.dd_step_scaled(fs.h, src, 1.0 / (1 + k), out, stats=True, raise_on_error=False)
            D.dd_set_wait_limit(fs.h, 0)
            assert st["rc"] == D.DD_ERR_TIMEOUT, st
            assert "wait" in D.lib().dd_last_error(fs.h).decode()
            f0, f1, step2 = fs.get_state()
            assert step2 == step and torch.equal(f0, e0) and torch.equal(f1, e1)
        D.dd_step_scaled(fs.h, src, 1.0 / (1 + k), out)
        fields.append(out.clone())
    return fields


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("kind", list(PROBLEMS))
def test_wait_that_runs_out_is_reported(kind, graph):
    runs = []
    for interrupt in (False, True):
        fs = solver(kind, graph)
        try:
            runs.append(march(fs, interrupt))
        finally:
            fs.close()
    for a, b in zip(*runs):
        assert torch.linalg.norm(a - b) <= 1e-9 * torch.linalg.norm(b)


@pytest.mark.parametrize("kind", ["fixed_gmres", "fixed_cg"])
def test_wait_behind_the_interface_solve(kind):
    """Only the last GEMVs of an eager FP64 step give up: the solve has converged by then, and
    the error word alone tells.  The word is set by hand before the step (it is sticky): 24
    bytes in front of the limit that dd_set_wait_limit writes."""
    fs = solver(kind, 0)
    try:
        src = torch.tensor(np.random.default_rng(2).standard_normal(fs.n_dof), device="cuda")
        out = torch.empty_like(src)
        D.dd_step(fs.h, src, out)
        words = fs.ws_view.view(torch.int32)
        D.dd_set_wait_limit(fs.h, 1987654321)
        at = torch.nonzero(words == 1987654321).flatten()
        D.dd_set_wait_limit(fs.h, 0)
        assert at.numel() == 1 and words[at].item() == 0
        words[at - 6] = 1
        st = D.dd_step(fs.h, src, out, stats=True, raise_on_error=False)
        assert st["rc"] == D.DD_ERR_TIMEOUT and fs.get_state()[2] == 1
        assert words[at - 6].item() == 0
        assert D.dd_step(fs.h, src, out, stats=True)["rc"] == D.DD_OK
    finally:
        fs.close()


@pytest.mark.parametrize("scheme", [D.DD_SCHEME_DP1, D.DD_SCHEME_DP2])
def test_operator_calls(scheme):
    """The operator calls only launch, and nobody reads the error word after them: they wait for
    nothing, and leave nothing behind that a later step would report."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.box(16, 16, 16, 4, 4, 4)
    fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, params=D.make_params(solver=GMRES, scheme=scheme, tol=1e-12)).bind()
    try:
        fs.factor(0.03)
        nc, gen = fs.sizes.n_corner, torch.Generator().manual_seed(1)
        calls = [lambda u, v: D.dd_dp2_apply(fs.h, u, v)]
        sizes = [2 * fs.n_lambda + nc]
        if scheme == D.DD_SCHEME_DP1:
            calls = [lambda u, v: D.dd_coupled_apply(fs.h, u, v), lambda u, v: D.dd_schur_apply(fs.h, u, v),
                     lambda u, v: D.dd_schur_apply_static(fs.h, u, v)]
            sizes = [fs.n_lambda + nc, fs.n_lambda, fs.n_lambda]
        src = torch.randn(fs.n_dof, dtype=torch.float64, generator=gen).cuda()
        for call, n in zip(calls, sizes):
            u = torch.randn(n, dtype=torch.float64, generator=gen).cuda()
            a, b, c = (torch.zeros_like(u) for _ in range(3))
            call(u, a)
            D.dd_set_wait_limit(fs.h, 4)
            call(u, b)
            D.dd_set_wait_limit(fs.h, 0)
            assert torch.isfinite(a).all() and torch.equal(a, b)
            assert D.dd_step(fs.h, src, None, stats=True)["rc"] == D.DD_OK
            call(u, c)
            assert torch.equal(a, c)
    finally:
        fs.close()


def test_factorisation():
    """The tensor-core elimination: reported as what it is (its pivots say nothing then), nothing
    factored, nothing left behind, and the next factorisation is as good as the first."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.cavity(8, 2)
    fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub,
                       params=D.make_params(solver=GMRES, factor_mode=D.DD_FACTOR_TENSOR)).bind()
    try:
        u = torch.randn(fs.n_lambda + fs.sizes.n_corner, dtype=torch.float64,
                        generator=torch.Generator().manual_seed(1)).cuda()
        fs.factor(0.05)
        a = fs.coupled_apply(u)
        for _ in range(2):
            D.dd_set_wait_limit(fs.h, 4)
            with pytest.raises(D.DDError) as e:
                fs.factor(0.05)
            assert e.value.code == D.DD_ERR_TIMEOUT
            D.dd_set_wait_limit(fs.h, 0)
            with pytest.raises(D.DDError) as e:
                fs.coupled_apply(u)
            assert e.value.code == D.DD_ERR_STATE
        fs.factor(0.05)
        assert torch.equal(fs.coupled_apply(u), a)
    finally:
        fs.close()
