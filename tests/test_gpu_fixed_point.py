"""FP64 GEMVs on the packed fixed-point tiles: the coupled operator equals the CPU
oracle's, a step the sparse direct solve, on block subdomains (tile rows of 64 and a
remainder) and on a ragged bisection (remainders of every size: short, narrow and
diagonal tiles); inputs of ordinary and of widely spread magnitude, zero, NaN.

Tolerances: the fixed-point sums round at 2^-57 of their scale, n <= 700 terms, so the
operator is off by less than 1e-14 of its norm; the oracle's Cholesky solves (condition
number of A_rr below 1e3) bound the comparison at 1e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import scipy.sparse.linalg as spla

from oracle import dd as odd
from oracle import fem, newmark
from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def problem(kind):
    if kind == "blocks":
        w = W.box(16, 16, 16, 4, 4, 4)
        return w.xyz, w.tets, w.part, w.n_sub, 0.03
    n, L = (16, 14, 13), (16 / 14, 1.0, 13 / 14)
    xyz, tets = W.kuhn_box(*n, *L)
    xyz, rng = W.jitter_nodes(xyz, 1 / 14, L, 0.2, seed=5)
    part = W.rcb_partition(W.tet_centroids(xyz, tets), 50, rng.uniform(0.6, 1.4, size=50))
    return xyz, tets, part, 50, 0.027


@pytest.mark.parametrize("kind", ["blocks", "ragged"])
def test_coupled_operator_and_step(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets, part, n_sub, dt = problem(kind)
    space = fem.EdgeSpace(xyz, tets)
    maps = odd.DDMaps(space, part, n_sub)
    solver = odd.DDSolver(space, maps, dt)
    fs = D.FieldSolver(xyz, tets, part, n_sub,
                       params=D.make_params(tol=1e-13, max_it=2000, solver=D.DD_SOLVER_COUPLED_GMRES)).bind()
    fs.factor(dt)
    g = maps.n_lambda + maps.n_corner
    m = fs.maps()   # the packed form is the one in use: about half of the dense bytes
    dense = 8 * float(((m["n_gam"] + m["n_cor"]).astype(np.float64) ** 2).sum())
    assert D.dd_get_gemv_bytes(fs.h, "coupled", D.DD_FP64)[1] < 0.8 * dense
    rng = np.random.default_rng(1)
    inputs = [rng.standard_normal(g), rng.standard_normal(g) * 10.0 ** rng.uniform(-12, 12, g), np.zeros(g),
              1e-250 * rng.standard_normal(g)]
    for u in inputs:
        got = fs.coupled_apply(torch.tensor(u, device="cuda")).cpu().numpy()
        ref = solver.coupled_apply(u)
        assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    bad = inputs[0].copy()
    bad[3] = np.nan
    assert np.isnan(fs.coupled_apply(torch.tensor(bad, device="cuda")).cpu().numpy()).any()
    # one step from rest: A e^1 = -d2g
    T, S = space.assemble()
    A, _ = newmark.newmark_matrices(T, S, dt)
    src = rng.standard_normal(space.n)
    out = torch.empty(space.n, dtype=torch.float64, device="cuda")
    fs.step(torch.tensor(src, device="cuda"), out)
    ref = spla.splu(A).solve(-src)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
    src[5] = np.nan   # a non-finite source is reported and the step is not taken
    st = D.dd_step(fs.h, torch.tensor(src, device="cuda"), None, raise_on_error=False)
    assert st["rc"] == D.DD_ERR_NONFINITE
    e_n, _, step = fs.get_state()
    assert step == 1 and torch.equal(e_n, out)
    fs.close()
