"""Exact Gauss-Seidel on triangles of few levels, which are solved by a launch per level (up to two
levels at these sizes): one level, two levels of rows that take 1, 4 and 16 lanes with remainders, and
three levels, the first count that goes back to one launch.  Against the FP64 oracle, 1e-12 relative
as for every FP64 sweep (rows are reduced in another order, a few ulps an entry)."""
import numpy as np
import pytest

import oracle
from paper_2104_01196_gb300 import problems as P
import paper_2104_01196_gb300 as lib
from test_gpu_parity import dev, g, host, rel, rhs_and_x0  # noqa: F401

pytestmark = pytest.mark.gpu


def layered(n, levels, mean, seed):
    """Rows in `levels` groups; a row couples to `mean` rows of the group before on average, both
    ways (so that the upper triangle has as many levels), 0 to 2 mean of them."""
    rng = np.random.RandomState(seed)
    M = np.zeros((n, n))
    size = n // levels
    for i in range(size, size * levels):
        first = (i // size - 1) * size
        k = rng.randint(1, 2 * mean + 1)
        c = first + rng.choice(size, min(k, size), replace=False)
        M[i, c] = rng.uniform(-1, 1, len(c))
        M[c, i] = rng.uniform(-1, 1, len(c))
    M[np.arange(n), np.arange(n)] = 1.0 + 1.5 * np.abs(M).sum(1)
    return P.dense_to_csr(M)


@pytest.mark.parametrize("levels", [1, 2, 3])
@pytest.mark.parametrize("n,mean", [(33, 2), (700, 3), (700, 20), (601, 90)])
@pytest.mark.parametrize("direction", [0, 1, 2])
def test_few_levels(g, levels, n, mean, direction):  # noqa: F811
    A = layered(n, levels, mean, 10 * levels + mean)
    b, x0 = rhs_and_x0(A, 121)
    h = g.gs2_setup(A)
    for sweeps, omega in ((1, 1.0), (2, 1.2)):
        x = dev(x0)
        g.gs_apply(h, dev(b), x, sweeps, omega, direction)
        assert rel(host(x), oracle.gs(A, b, x0, sweeps, omega, direction)) <= 1e-12
    assert h.stats()["levels_lower"] == levels
    # as a preconditioner (from x = 0) and in the hybrid form
    info = g.gmres_solve(h, dev(b), dev(np.zeros(n)), 30, 1e-10, 200,
                         g.params("gs", direction="symmetric"))
    assert info.ok
    pc = g.params("gs", direction=direction, parts=2)
    x = dev(x0)
    g.relax_apply(h, dev(b), x, pc)
    h.check()


# a half sweep is the residual and one launch a level
@pytest.mark.parametrize("levels,launches", [(1, 2), (2, 3), (3, 3)])
def test_launches(g, levels, launches):  # noqa: F811
    A = layered(300, levels, 3, levels)
    b, x0 = rhs_and_x0(A, 122)
    h = g.gs2_setup(A)
    x = dev(x0)
    g.gs_apply(h, dev(b), x, 1, 1.0, g.FORWARD)
    before = lib.launch_count()
    g.gs_apply(h, dev(b), x, 1, 1.0, g.FORWARD)
    assert lib.launch_count() - before == launches
