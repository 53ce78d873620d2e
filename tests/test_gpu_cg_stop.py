"""CG's stop flag: set once every block of the launch that sets it is done.

A flag that a launch sets while some of its blocks have yet to start lets the threads of such a
block disagree about leaving before a block barrier; on a breakdown (p.q = 0) the block then updates
x with whatever alpha it finds.
"""
import numpy as np
import pytest

from test_gpu_parity import dev, g, host  # noqa: F401

pytestmark = pytest.mark.gpu


def signs(n):
    """diag(1, -1, 1, ...): with b = 1 and n even, p.q = sum of +-1 = 0 in the first iteration."""
    d = np.where(np.arange(n) % 2 == 0, 1.0, -1.0)
    return np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), d


# one block of the vector kernels, a few, and more blocks than run at once; graphs (1) and separate
# launches (2); a breakdown leaves x as it was, in every repetition
@pytest.mark.parametrize("n", [64, 20002, 600002])
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("pc", [None, "jr"])
def test_breakdown_leaves_x(g, n, mode, pc):  # noqa: F811
    A = signs(n)
    h = g.gs2_setup(A)
    h.set_graph_mode(mode)
    b = dev(np.ones(n))
    for _ in range(20):
        x = dev(np.zeros(n))
        info = g.cg_solve(h, b, x, 1e-8, 50, None if pc is None else g.params(pc))
        assert g.STATUS[info.status] == "BREAKDOWN" and info.iters == 0
        assert not host(x).any()
    # the handle solves as before afterwards: b in the span of one eigenvalue, one iteration
    e = np.where(np.arange(n) % 2 == 0, 3.0, 0.0)
    x = dev(np.zeros(n))
    info = g.cg_solve(h, dev(e), x, 1e-8, 50, None if pc is None else g.params(pc))
    assert info.ok and info.iters == 1 and np.array_equal(host(x), e)


# converged after k iterations or stopped by the limit: the same bits from graphs and from separate
# launches, in every repetition, and the limit counts as before
@pytest.mark.parametrize("limit", [1, 15, 16, 17, 5000])
def test_stop_is_the_same_in_every_mode(g, limit):  # noqa: F811
    from paper_2104_01196_gb300 import problems as P
    A = P.poisson3d_matrix(33)
    n = len(A[0]) - 1
    b = dev(P.uniform_pm1(91, n))
    h = g.gs2_setup(A)
    pc = g.params("gs2", direction="symmetric")
    seen = set()
    for mode in (1, 2, 1, 2):
        h.set_graph_mode(mode)
        x = dev(np.zeros(n))
        info = g.cg_solve(h, b, x, 1e-10, limit, pc)
        assert info.ok == (limit == 5000) and (info.ok or info.iters == limit)
        seen.add((info.iters, host(x).tobytes()))
    assert len(seen) == 1
