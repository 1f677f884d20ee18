"""The one-kernel vector part of a CG iteration over the number of multipliers: one, two
and four elements a thread (28,224, 108,000 and 190,080 multipliers on 152
multiprocessors), in FP64 and mixed precision, eager and captured.  Reference: the same
step by the coupled GMRES on the same tearing (other operators, other vector kernels),
to the parity bounds of the solvers (1e-10; mixed precision 1e-8)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, k", [(24, 8), (40, 10), (48, 12)])
def test_step_over_sizes(n, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.cavity(n, k)
    gen = torch.Generator().manual_seed(3)

    def step(prec, solver, graph):
        mixed = prec == D.DD_MIXED
        prm = D.make_params(precision=prec, tol=1e-4 if mixed else 1e-13, refine_tol=1e-11, max_refine=10, max_it=500,
                            solver=solver, use_graph=graph)
        fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, w.eps, w.mu, prm).bind()
        fs.factor(0.46 / n)
        src = torch.randn(fs.n_dof, dtype=torch.float64, generator=gen.manual_seed(3)).cuda()
        out = torch.empty_like(src)
        fs.step(src, out)
        fs.close()
        return out

    ref = step(D.DD_FP64, D.DD_SOLVER_COUPLED_GMRES, 0)
    for prec, graph in ((D.DD_FP64, 0), (D.DD_FP64, 1), (D.DD_MIXED, 0), (D.DD_MIXED, 1)):
        got = step(prec, D.DD_SOLVER_SCHUR_CG, graph)
        assert (got - ref).norm() <= (1e-8 if prec == D.DD_MIXED else 1e-10) * ref.norm()
