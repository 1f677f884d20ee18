"""The one-kernel Arnoldi step over the number of unknowns: one, two and four elements
a thread (the last block partly filled, or nearly every multiprocessor's), and the
three-kernel form beyond; in FP32 and FP64, eager and captured, with the longest restart
(33 sums a pass).  The sizes are reached with copies of one small problem, each with a
source of its own; every member's first step equals the sparse direct solve
A e^1 = -d2g, to the parity bounds of the solver (1e-10; mixed precision 1e-8)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import scipy.sparse.linalg as spla

from oracle import fem, newmark
from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("prec", [D.DD_FP64, D.DD_MIXED])
@pytest.mark.parametrize("fill", [0.3, 0.99, 1.01, 2.2, 4.2])   # of one element a thread, 512 threads per multiprocessor
def test_step_over_sizes(fill, prec, graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.cavity(12, 6)
    dt = 0.04
    h = D.dd_setup(w.xyz, w.tets, w.part, w.n_sub, w.eps, w.mu)
    sz = D.dd_get_sizes(h)
    D.dd_destroy(h)
    cap = 512 * torch.cuda.get_device_properties(0).multi_processor_count
    R = max(1, int(fill * cap) // int(sz.n_lambda + sz.n_corner))
    mixed = prec == D.DD_MIXED
    prm = D.make_params(precision=prec, tol=1e-4 if mixed else 1e-12, refine_tol=1e-10, max_refine=8, max_it=500, restart=32,
                        solver=D.DD_SOLVER_COUPLED_GMRES, use_graph=graph, members=R)
    fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, w.eps, w.mu, prm).bind()
    fs.factor(dt)
    nd = fs.n_dof_member
    src = np.random.default_rng(7).standard_normal((R, nd))
    out = torch.empty(fs.n_dof, dtype=torch.float64, device="cuda")
    fs.step(torch.tensor(src.reshape(-1), device="cuda"), out)
    fs.close()
    space = fem.EdgeSpace(w.xyz, w.tets, w.eps, w.mu)
    A, _ = newmark.newmark_matrices(*space.assemble(), dt)
    want = spla.splu(A.tocsc()).solve(-src.T).T
    err = np.linalg.norm(out.cpu().numpy().reshape(R, nd) - want, axis=1) / np.linalg.norm(want, axis=1)
    assert err.max() <= (1e-8 if mixed else 1e-10)
