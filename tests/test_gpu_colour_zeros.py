"""Multicolour sweeps of a matrix with stored zeros: a stored zero times an infinity or a NaN is a NaN,
as in the other layouts, while a slot that the row does not have contributes nothing."""
import numpy as np
import pytest

import oracle
from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1000, 1), (40, 40)])
@pytest.mark.parametrize("zero", [0.0, -0.0])
def test_stored_zero(g, dims, zero):  # noqa: F811
    A = P.poisson2d_matrix(dims[0]) if dims[1] > 1 else P.dense_to_csr(
        4.0 * np.eye(dims[0]) - np.eye(dims[0], k=1) - np.eye(dims[0], k=-1))
    n = len(A[0]) - 1
    rows = np.repeat(np.arange(n), np.diff(A[0]))
    # the last row of the last colour: its neighbours read its x before it is overwritten
    color = oracle.coloring(A)
    color = np.asarray(color[0] if isinstance(color, tuple) else color)
    src = int(np.flatnonzero(color == color.max())[-1])
    hit = np.flatnonzero((A[1] == src) & (rows != src))
    va = A[2].copy()
    va[hit] = zero
    h = g.gs2_setup((A[0], A[1], va))
    b, x0 = P.uniform_pm1(111, n), P.uniform_pm1(112, n)
    for bad in (np.inf, np.nan):
        x1 = x0.copy()
        x1[src] = bad
        x = dev(x1)
        g.mtgs_apply(h, dev(b), x, 1, 1.0, g.FORWARD)
        got = host(x)
        assert np.isnan(got[rows[hit]]).all()
    # finite everywhere otherwise
    x = dev(x0)
    g.mtgs_apply(h, dev(b), x, 2, 0.9, g.SYMMETRIC)
    assert np.isfinite(host(x)).all()
