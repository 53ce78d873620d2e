"""Solvers after the multigrid hierarchy of a handle was built anew: a graph captured with the old
hierarchy holds its freed level buffers and must not be replayed."""
import numpy as np
import pytest

from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host  # noqa: F401

pytestmark = pytest.mark.gpu


# 32,768 rows: above the sizes of the one-launch solvers, so both take cycle graphs in mode 1
@pytest.mark.parametrize("solver", ["cg", "gmres"])
@pytest.mark.parametrize("kind", ["amg", "amg_jr"])
def test_solve_after_rebuild(g, solver, kind):  # noqa: F811
    A = P.poisson3d_matrix(32)
    n = len(A[0]) - 1
    b = dev(P.uniform_pm1(101, n))
    pc = g.params(kind, direction="symmetric", omega=0.7 if kind == "amg_jr" else 1.0)

    def solve(h):
        h.set_graph_mode(1)
        x = dev(np.zeros(n))
        info = (g.cg_solve(h, b, x, 1e-8, 200, pc) if solver == "cg"
                else g.gmres_solve(h, b, x, 30, 1e-8, 200, pc))
        return info.iters, host(x).tobytes()

    first, second = dict(coarse_size=64), dict(coarse_size=2000, theta=0.1)
    fresh = {}
    for name, cfg in (("first", first), ("second", second)):
        h = g.gs2_setup(A)
        h.amg_setup(**cfg)
        fresh[name] = solve(h)
    assert fresh["first"] != fresh["second"]
    h = g.gs2_setup(A)
    for name, cfg in (("first", first), ("second", second), ("first", first), ("second", second)):
        h.amg_setup(**cfg)
        assert solve(h) == fresh[name]
        assert solve(h) == fresh[name]
