"""Pivot blocks of the tensor-core elimination over their conditioning: inverted in FP32
and corrected (time steps of ordinary size), or swept in FP64 where FP32 loses the
block (a curl-curl matrix with a vanishing mass term: condition numbers 7, 3e3, 3e5,
9e8; from the second on some FP32 sweeps leave residuals above their bounds, in the
last they meet pivots that are not positive).

Tolerance: an elimination of n rows is off by n 2^-53 of the condition number; both sides
of the comparison are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dd as odd
from oracle import fem
from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [0.05, 2.0, 20.0, 1000.0])
def test_coupled_operator_over_conditioning(dt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = W.cavity(6, 2)
    space = fem.EdgeSpace(w.xyz, w.tets)
    maps = odd.DDMaps(space, w.part, w.n_sub)
    ref = odd.DDSolver(space, maps, dt)
    n = max(maps.nr)
    cond = max(np.linalg.cond(a[:k, :k]) for a, k in zip(ref.A, maps.nr))
    fs = D.FieldSolver(w.xyz, w.tets, w.part, w.n_sub,
                       params=D.make_params(solver=D.DD_SOLVER_COUPLED_GMRES, factor_mode=D.DD_FACTOR_TENSOR)).bind()
    fs.factor(dt)
    u = np.random.default_rng(0).standard_normal(maps.n_lambda + maps.n_corner)
    got = fs.coupled_apply(torch.tensor(u, device="cuda")).cpu().numpy()
    fs.close()
    want = ref.coupled_apply(u)
    assert np.linalg.norm(got - want) <= 2 * n * 2.0**-53 * cond * np.linalg.norm(want)
