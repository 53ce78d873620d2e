"""Sweeps without an inner sweep in the one-launch form: a half sweep's residual reads other rows'
x right before the update writes it, with no inner sweep's barrier between them.

The row kernels (which a profiled handle takes) separate the two by a launch, and reduce a row in
the same order: the results are equal bit for bit, in every repetition.
"""
import numpy as np
import pytest

import oracle
from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host, rel, rhs_and_x0  # noqa: F401

pytestmark = pytest.mark.gpu


# one CTA, a cluster of full warps, one whose last CTA is short, and the largest (16 x 512 rows)
@pytest.mark.parametrize("name", ["poisson2d_8", "poisson2d_64", "poisson2d_61", "poisson3d_20"])
@pytest.mark.parametrize("direction", [0, 1, 2])
@pytest.mark.parametrize("omega", [1.0, 0.8])
def test_no_inner_sweep(g, name, direction, omega):  # noqa: F811
    kind, size = name.split("_")
    A = getattr(P, kind + "_matrix")(int(size))
    b, x0 = rhs_and_x0(A, 81)
    h = g.gs2_setup(A)
    pc = g.params("gs2", outer=6, inner=0, omega=omega, direction=direction)
    h.profile(True)
    x = dev(x0)
    g.gs2_apply_ex(h, dev(b), x, pc)
    rows = host(x)
    h.profile(False)
    assert rel(rows, oracle.gs2(A, b, x0, 6, 0, omega, 1.0, direction)) <= 1e-12
    for _ in range(50):
        x = dev(x0)
        g.gs2_apply_ex(h, dev(b), x, pc)
        assert np.array_equal(host(x), rows)


# inner sweeps, relaxed and damped: the same bits as the row kernels too
@pytest.mark.parametrize("name", ["poisson2d_64", "poisson3d_17"])
@pytest.mark.parametrize("outer,inner,omega,gamma", [
    (2, 1, 0.9, 1.0), (1, 2, 1.0, 0.7), (2, 3, 0.9, 0.7), (1, 3, 1.1, 1.0)])
def test_inner_sweeps(g, name, outer, inner, omega, gamma):  # noqa: F811
    kind, size = name.split("_")
    A = getattr(P, kind + "_matrix")(int(size))
    b, x0 = rhs_and_x0(A, 82)
    h = g.gs2_setup(A)
    pc = g.params("gs2", outer=outer, inner=inner, omega=omega, gamma=gamma, direction="symmetric")
    out = []
    for profiled in (True, False):
        h.profile(profiled)
        x = dev(x0)
        g.gs2_apply_ex(h, dev(b), x, pc)
        out.append(host(x))
    assert np.array_equal(out[0], out[1])
