"""Operator calls of a handle whose FP64 steps run on packed fixed-point tiles: row by row
what the dense FP64 form gives (a DD_MIXED handle of the same factors, which has no
fixed-point tiles), bit for bit.  Inputs of ordinary size, and inputs whose entries spread
over many orders of magnitude inside a subdomain, whose far rows a common scale would
drown: one entry, decaying pulses, a few entries in a hundred; tiny, zero and non-finite
inputs.  Block and ragged tearings, both schemes, every call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CALLS = {"coupled": D.DD_SCHEME_DP1, "schur": D.DD_SCHEME_DP1, "schur_static": D.DD_SCHEME_DP1, "dp2": D.DD_SCHEME_DP2}


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
@pytest.mark.parametrize("call", list(CALLS))
def test_rows_are_the_dense_forms(call, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    xyz, tets, part, n_sub, dt = problem(kind)
    fixed, dense = (D.FieldSolver(xyz, tets, part, n_sub, params=D.make_params(
        solver=D.DD_SOLVER_COUPLED_GMRES, scheme=CALLS[call], precision=p)).bind() for p in (D.DD_FP64, D.DD_MIXED))
    for fs in (fixed, dense):
        fs.factor(dt)
    m = fixed.maps()   # the steps' form is the packed one: about half of the dense bytes
    bytes_dense = 8 * float(((m["n_gam"] + m["n_cor"]).astype(np.float64) ** 2).sum())
    assert D.dd_get_gemv_bytes(fixed.h, "coupled", D.DD_FP64)[1] < 0.8 * bytes_dense
    nl, nc = fixed.n_lambda, fixed.sizes.n_corner
    n = {"coupled": nl + nc, "schur": nl, "schur_static": nl, "dp2": 2 * nl + nc}[call]
    fn = {"coupled": D.dd_coupled_apply, "schur": D.dd_schur_apply, "schur_static": D.dd_schur_apply_static,
          "dp2": D.dd_dp2_apply}[call]

    def run(fs, u):
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        fn(fs.h, torch.as_tensor(u, device="cuda"), out)
        return out.cpu().numpy()

    rng = np.random.default_rng(4)
    sub = m["mult_sub"][:, 0]
    rank = rng.permutation(n)
    inputs = [rng.standard_normal(n), rng.standard_normal(n) * 10.0 ** rng.uniform(-10, 0, n), np.exp(-60.0 * rank / n),
              np.exp(-12.0 * rank / n), rng.standard_normal(n) * (rng.random(n) < 0.03),
              np.where(np.resize(sub, n) == 21, 1.0, 1e-9) * rng.standard_normal(n), 1e-250 * rng.standard_normal(n),
              np.zeros(n)] + [np.eye(1, n, at)[0] for at in (3, nl // 2 + 7, n - 2)]
    for bad in (np.nan, np.inf):
        inputs.append(inputs[0].copy())
        inputs[-1][nl // 3] = bad
    for k, u in enumerate(inputs):
        assert np.array_equal(run(fixed, u), run(dense, u), equal_nan=True), k
    fixed.close()
    dense.close()
