"""FP64 DP2 steps on the packed fixed-point tiles (the two-sided multipliers as their input):
the first step from rest equals the sparse direct solve, on block and on ragged
subdomains, eager and captured.

Tolerance: the solve's 1e-13 of the interface right-hand side, three decades for the
recovery from it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import scipy.sparse.linalg as spla

from oracle import fem, newmark
from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("kind", ["blocks", "ragged"])
def test_step_from_rest(kind, graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if kind == "blocks":
        w = W.box(16, 16, 16, 4, 4, 4)
        xyz, tets, part, n_sub, dt = w.xyz, w.tets, w.part, w.n_sub, 0.03
    else:
        n, L = (16, 14, 13), (16 / 14, 1.0, 13 / 14)
        xyz, tets = W.kuhn_box(*n, *L)
        xyz, rng = W.jitter_nodes(xyz, 1 / 14, L, 0.2, seed=5)
        part, n_sub, dt = W.rcb_partition(W.tet_centroids(xyz, tets), 50, rng.uniform(0.6, 1.4, size=50)), 50, 0.027
    space = fem.EdgeSpace(xyz, tets)
    A, _ = newmark.newmark_matrices(*space.assemble(), dt)
    src = np.random.default_rng(6).standard_normal(space.n)
    ref = spla.splu(A.tocsc()).solve(-src)
    fs = D.FieldSolver(xyz, tets, part, n_sub, params=D.make_params(
        tol=1e-13, max_it=2000, solver=D.DD_SOLVER_COUPLED_GMRES, scheme=D.DD_SCHEME_DP2, use_graph=graph)).bind()
    fs.factor(dt)
    m = fs.maps()
    assert D.dd_get_gemv_bytes(fs.h, "coupled", D.DD_FP64)[1] < 0.8 * 8 * float(((m["n_gam"] + m["n_cor"]).astype(float) ** 2).sum())
    out = torch.empty(space.n, dtype=torch.float64, device="cuda")
    fs.step(torch.tensor(src, device="cuda"), out)
    fs.close()
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)
