"""One handle stepped in FP64, in mixed precision and in FP64 again, on a tearing whose FP64
operators are packed in fixed point (they share their storage with the FP32 ones): every
result equals, bit for bit, that of a handle that has only ever had that precision;
autotuning in between leaves the packed operators as they are; and the operator calls, in FP64
whatever the handle's precision, are the same."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def close(a, b):   # to the tolerance of the solve
    return bool(torch.linalg.norm(a - b) <= 1e-11 * torch.linalg.norm(b))


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("solver", [D.DD_SOLVER_COUPLED_GMRES, D.DD_SOLVER_SCHUR_CG])
def test_switch(solver, graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.box(16, 16, 16, 4, 4, 4)
    prms = {p: D.make_params(precision=p, tol=1e-12 if p == D.DD_FP64 else 1e-5, refine_tol=1e-11, max_refine=8,
                             solver=solver, use_graph=graph) for p in (D.DD_FP64, D.DD_MIXED)}
    rng = np.random.default_rng(3)

    def handle(prec):
        fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, params=prms[prec]).bind()
        fs.factor(0.03)
        return fs

    one = {p: handle(p) for p in prms}
    both = handle(D.DD_FP64)
    n = both.n_dof
    e0, e1, src = (torch.tensor(rng.standard_normal(n), device="cuda") for _ in range(3))
    u = torch.tensor(rng.standard_normal(both.n_lambda + both.sizes.n_corner), device="cuda")

    def step(fs):
        out = torch.empty_like(src)
        fs.set_state(e0, e1, 0)
        D.dd_step(fs.h, src, out)
        return out

    want = {p: step(one[p]) for p in prms}
    assert torch.linalg.norm(want[D.DD_MIXED] - want[D.DD_FP64]) <= 1e-8 * torch.linalg.norm(want[D.DD_FP64])
    applied = one[D.DD_FP64].coupled_apply(u)
    assert torch.equal(applied, one[D.DD_MIXED].coupled_apply(u))
    try:
        for prec in (D.DD_FP64, D.DD_MIXED, D.DD_FP64, D.DD_MIXED):
            both.set_params(prms[prec])
            assert torch.equal(step(both), want[prec])
            assert torch.equal(both.coupled_apply(u), applied)
        both.set_params(prms[D.DD_FP64])
        D.dd_autotune(both.h)
        assert close(both.coupled_apply(u), applied)   # (its dense form is tuned)
        same = torch.equal if solver == D.DD_SOLVER_COUPLED_GMRES else close   # (the CG's dense kinds are tuned)
        assert same(step(both), want[D.DD_FP64])
        both.factor(0.02)                         # and a new factorisation packs for the precision in force
        both.factor(0.03)
        assert same(step(both), want[D.DD_FP64])
    finally:
        both.close()
        for fs in one.values():
            fs.close()
