"""The tensor-core elimination against the FP64 one over materials whose permittivity varies by
up to eight decades from tet to tet (rows of very different scale inside a pivot block):
the operators of both agree in the norm and row by row, as two FP64 eliminations of the
same matrices would.

Tolerance: an FP64 elimination of n rows is off by about sqrt(n) 2^-53 of the scale of a
row (the roundings of n updates, independent of each other), two of them by twice that;
n = 604 here.  It has to hold for nine rows out of ten (the tenth may be small by
cancellation), and in the norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("decades", [0, 2, 4])
def test_rows_over_material_contrast(decades):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.box(16, 16, 16, 4, 4, 4)
    eps = 10.0 ** np.random.default_rng(1).uniform(-decades, decades, len(w.tets))
    rows = []
    for mode in (D.DD_FACTOR_FP64, D.DD_FACTOR_TENSOR):
        fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub, eps, 1.0,
                           D.make_params(solver=D.DD_SOLVER_COUPLED_GMRES, factor_mode=mode)).bind()
        fs.factor(0.03)
        assert fs.sizes.max_ns == 604
        u = np.random.default_rng(2).standard_normal(fs.n_lambda + fs.sizes.n_corner)
        rows.append(fs.coupled_apply(torch.tensor(u, device="cuda")).cpu().numpy())
        fs.close()
    want, got = rows
    tol = 2 * np.sqrt(604) * 2.0**-53
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
    assert np.quantile(np.abs(got - want) / np.abs(want), 0.9) <= tol
