"""Device memory of a handle (no GPU needed): the packed FP64 operators and the scratch of the
tensor-core elimination take no room of their own.  The bounds are what the dense
operators, their FP32 copies, the packed FP32 tiles and the vectors of these problems took
in all before there were packed FP64 operators."""
import pytest

from paper_2204_13254_gb300 import dd as D
from paper_2204_13254_gb300 import workloads as W


@pytest.mark.parametrize("n, k, members, limit", [(16, 4, 1, 324861440), (24, 4, 1, 2777904128), (8, 2, 1, 30364160),
                                                  (16, 4, 4, 610137344)])
@pytest.mark.parametrize("precision", [D.DD_FP64, D.DD_MIXED])
def test_workspace_bytes(n, k, members, limit, precision):
    w = W.box(n, n, n, k, k, k)
    h = D.dd_setup(w.xyz, w.tets, w.part, w.n_sub, w.eps, w.mu,
                   D.make_params(precision=precision, members=members, solver=D.DD_SOLVER_COUPLED_GMRES))
    try:
        assert D.dd_get_sizes(h).workspace_bytes <= limit
    finally:
        D.dd_destroy(h)
