"""Row kernels at the edges of their layouts, against the FP64 oracle.

Tolerance as for every FP64 sweep: rows are reduced in another order and
scaled by a precomputed D^{-1}, a few ulps per entry, so 1e-12 relative.
"""
import numpy as np
import pytest

import oracle
from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host, rel, rhs_and_x0  # noqa: F401

pytestmark = pytest.mark.gpu
TOL = 1e-12


def band_matrix(n, width, seed):
    """n rows on `width` diagonals, the main one and others near and far on either side; entries
    outside [0, n) dropped, so the chunks at both ends are narrower."""
    far = [-(n // 3) - 1, -7, -1, 1, 2, n // 4 + 3, -3, 5, -(n // 2)]
    offs = sorted({0, *far[:width - 1]})
    val = P.uniform_pm1(seed, n * len(offs)).reshape(n, len(offs))
    rp, ci, va = [0], [], []
    for i in range(n):
        for q, o in enumerate(offs):
            if 0 <= i + o < n:
                ci.append(i + o)
                va.append(len(offs) + 1.0 + val[i, q] if o == 0 else val[i, q])
        rp.append(len(ci))
    return np.array(rp, np.int64), np.array(ci, np.int32), np.array(va)


# every unrolled stencil width (1 to 8 slots) and the first one beyond, on rows that fill a warp,
# miss it by one, exceed it by one, and take several chunks per warp's neighbourhood
@pytest.mark.parametrize("width", range(1, 10))
@pytest.mark.parametrize("n", [31, 32, 33, 1000])
def test_stencil_widths(g, width, n):  # noqa: F811
    A = band_matrix(n, width, 7 * width + n)
    b, x0 = rhs_and_x0(A, 5)
    h = g.gs2_setup(A)
    # (31 to 33 rows pad by more than 20% in some widths and stay row tiles)
    assert n < 1000 or h.stats()["offset_frac_a"] == 1.0
    y = dev(np.zeros(n))
    g.gs2_spmv(h, dev(b), y)
    assert rel(host(y), oracle.spmv(A, b)) <= TOL
    for omega in (1.0, 0.9):
        x = dev(x0)
        g.gs2_apply(h, dev(b), x, 1, 2, omega, g.SYMMETRIC)
        assert rel(host(x), oracle.gs2(A, b, x0, 1, 2, omega, 1.0, oracle.SYMMETRIC)) <= TOL
    x = dev(x0)
    g.jr_apply(h, dev(b), x, 2, 0.8)
    assert rel(host(x), oracle.jr(A, b, x0, 2, 0.8)) <= TOL
    x = dev(x0)
    g.mtgs_apply(h, dev(b), x, 1, 1.1, g.SYMMETRIC)
    assert rel(host(x), oracle.mtgs(A, b, x0, 1, 1.1, oracle.SYMMETRIC)) <= TOL


def chain_matrix(n):
    """Every row needs the one before it (and, backwards, the one after it): n levels of one row."""
    i = np.arange(n)
    M = np.zeros((n, n))
    M[i, i] = 4.0
    M[i[1:], i[:-1]] = -1.0 + 0.001 * i[1:]
    M[i[:-1], i[1:]] = 0.5
    return P.dense_to_csr(M)


# the triangular solve: one row, chains of single rows, levels that fill a chunk and exceed it, and
# rows that take 1, 4 and 16 lanes with a remainder of every size, one of them longer than a group
TRI = {
    "n1": (np.array([0, 1]), np.array([0], np.int32), np.array([3.0])),
    "chain_2": chain_matrix(2),
    "chain_300": chain_matrix(300),
    "one_level_65": P.dense_to_csr(np.diag(np.arange(1.0, 66.0))),
    "stencil_33": P.poisson2d_matrix(33),
    "stencil_3d_9": P.poisson3d_matrix(9),
    "lanes_1_long_row": P.random_csr(700, 3, mean_offdiag=4.0, long_rows=[(650, 300)]),
    "lanes_4": P.random_csr(500, 4, mean_offdiag=20.0),
    "lanes_16": P.random_csr(400, 5, mean_offdiag=90.0, long_rows=[(390, 380)]),
}


@pytest.mark.parametrize("name", list(TRI))
@pytest.mark.parametrize("direction", [0, 1, 2])
def test_triangular_solve(g, name, direction):  # noqa: F811
    A = TRI[name]
    b, x0 = rhs_and_x0(A, 21)
    h = g.gs2_setup(A)
    for sweeps, omega in ((1, 1.0), (2, 1.2)):
        x = dev(x0)
        g.gs_apply(h, dev(b), x, sweeps, omega, direction)
        assert rel(host(x), oracle.gs(A, b, x0, sweeps, omega, direction)) <= TOL
    h.check()


# NaN right-hand sides -- the pattern that marks an unsolved row among them -- reach the rows that
# depend on them and no others, and nothing waits for them
@pytest.mark.parametrize("bits", [0x7ff8000000000000, 0xffffffffffffffff, 0xfff8000000000001])
def test_triangular_solve_nan(g, bits):  # noqa: F811
    A = chain_matrix(100)
    b, x0 = rhs_and_x0(A, 22)
    b[40] = np.array([bits], np.uint64).view(np.float64)[0]
    h = g.gs2_setup(A)
    x = dev(x0)
    g.gs_apply(h, dev(b), x, 1, 1.0, 0)
    h.check()
    got = host(x)
    assert np.isnan(got[40:]).all() and not np.isnan(got[:40]).any()


def uneven_matrix(n, mean, longest, seed):
    """Row lengths spread evenly over 1 .. longest around `mean`, unsorted columns."""
    M = P.random_csr(n, seed, mean_offdiag=mean, empty_frac=0.1,
                     long_rows=[(n // 2, longest)] if longest else [])
    return M


# lane slices: every lane count, rows in order and sorted by length, empty rows, n not a multiple of
# a chunk or of the sort's window, and a row too long for them (row tiles)
LANES = {
    "uneven_1500": uneven_matrix(1500, 9.0, 0, 31),
    "uneven_1024": uneven_matrix(1024, 9.0, 60, 32),
    "uneven_5003": uneven_matrix(5003, 14.0, 100, 33),
    "uneven_40001": uneven_matrix(40001, 3.0, 0, 34),
    "long_777": uneven_matrix(777, 40.0, 130, 35),
    "long_90": uneven_matrix(90, 60.0, 80, 36),
    "too_long_4000": uneven_matrix(4000, 6.0, 3000, 37),
}


@pytest.mark.parametrize("name", list(LANES))
def test_lane_slices(g, name):  # noqa: F811
    A = LANES[name]
    n = len(A[0]) - 1
    b, x0 = rhs_and_x0(A, 41)
    h = g.gs2_setup(A)
    y = dev(np.zeros(n))
    g.gs2_spmv(h, dev(b), y)
    assert rel(host(y), oracle.spmv(A, b)) <= TOL
    for inner, omega in ((1, 1.0), (2, 0.9)):
        x = dev(x0)
        g.gs2_apply(h, dev(b), x, 1, inner, omega, g.SYMMETRIC)
        assert rel(host(x), oracle.gs2(A, b, x0, 1, inner, omega, 1.0, oracle.SYMMETRIC)) <= TOL
    x = dev(x0)
    g.jr_apply(h, dev(b), x, 2, 0.8)
    assert rel(host(x), oracle.jr(A, b, x0, 2, 0.8)) <= TOL
    x = dev(x0)
    g.mtgs_apply(h, dev(b), x, 1, 1.1, g.SYMMETRIC)
    assert rel(host(x), oracle.mtgs(A, b, x0, 1, 1.1, oracle.SYMMETRIC)) <= TOL


# an infinity in x reaches the rows that hold its column, as an infinity, and no padding slot
def test_lane_slices_infinity(g):  # noqa: F811
    A = LANES["uneven_5003"]
    n = len(A[0]) - 1
    x = P.uniform_pm1(43, n)
    x[[0, 777]] = np.inf
    h = g.gs2_setup(A)
    y = dev(np.zeros(n))
    g.gs2_spmv(h, dev(x), y)
    rows = np.repeat(np.arange(n), np.diff(A[0]))
    hit = np.zeros(n, bool)
    hit[rows[np.isin(A[1], [0, 777])]] = True
    got = host(y)
    assert np.isfinite(got[~hit]).all() and not np.isfinite(got[hit]).any()
    one = np.zeros(n, int)
    np.add.at(one, rows[np.isin(A[1], [0, 777])], 1)
    assert np.isinf(got[one == 1]).all()


# colours of stencils of every width (offsets count from a colour row's row in A), odd sizes and a
# chunk at each end, and an infinity that may reach only the rows that hold its column
@pytest.mark.parametrize("width", [3, 5, 7, 9])
def test_colour_rows_infinity(g, width):  # noqa: F811
    n = 1003
    A = band_matrix(n, width, width)
    h = g.gs2_setup(A)
    b, x0 = rhs_and_x0(A, 51)
    x = dev(x0)
    g.mtgs_apply(h, dev(b), x, 2, 0.9, g.FORWARD)
    assert rel(host(x), oracle.mtgs(A, b, x0, 2, 0.9, oracle.FORWARD)) <= TOL
    # b = inf at the last row of the last colour: x there, and nowhere else, in one forward sweep
    color = oracle.coloring(A)
    color = np.asarray(color[0] if isinstance(color, tuple) else color)
    last = int(np.flatnonzero(color == color.max())[-1])
    b2 = b.copy()
    b2[last] = np.inf
    x = dev(x0)
    g.mtgs_apply(h, dev(b2), x, 1, 1.0, g.FORWARD)
    got = host(x)
    assert np.isinf(got[last]) and np.isfinite(np.delete(got, last)).all()
    # x = inf at row 0: every row of a colour that holds column 0 and is updated before row 0's
    # own colour takes it; row 0 is in the first colour, so it is overwritten first
    x1 = x0.copy()
    x1[0] = np.inf
    x = dev(x1)
    g.mtgs_apply(h, dev(b), x, 1, 1.0, g.FORWARD)
    assert np.isfinite(host(x)).all()


# small stencil systems in one launch: one row, one and several CTAs with a last one short, both
# size lines and one row beyond, more neighbours than it takes (row kernels), unsorted rows (row
# kernels), every direction, damping, no inner sweep, several sweeps
SMALL = {
    "n1": (np.array([0, 1]), np.array([0], np.int32), np.array([3.0])),
    "band_64": band_matrix(64, 3, 61),
    "band_65": band_matrix(65, 7, 62),
    "grid_4096": P.poisson2d_matrix(64),
    "grid_4225": P.poisson2d_matrix(65),
    "grid3d_8000": P.poisson3d_matrix(20),
    "grid_8281": P.poisson2d_matrix(91),
    "band_9_wide": band_matrix(300, 9, 63),
    "unsorted": P.random_csr(300, 64, mean_offdiag=2.0),
}


@pytest.mark.parametrize("name", list(SMALL))
@pytest.mark.parametrize("direction", [0, 1, 2])
def test_small_sweeps(g, name, direction):  # noqa: F811
    A = SMALL[name]
    b, x0 = rhs_and_x0(A, 71)
    h = g.gs2_setup(A)
    for outer, inner, omega, gamma in ((1, 1, 1.0, 1.0), (2, 2, 0.9, 1.0), (1, 0, 0.8, 1.0),
                                       (1, 3, 1.0, 1.0), (2, 3, 0.9, 0.7)):
        x = dev(x0)
        g.gs2_apply_ex(h, dev(b), x, g.params("gs2", outer=outer, inner=inner, omega=omega,
                                              gamma=gamma, direction=direction))
        ref = oracle.gs2(A, b, x0, outer, inner, omega, gamma, direction)
        assert rel(host(x), ref) <= TOL, (outer, inner, omega, gamma)


# the same call through the row kernels (which a profiled handle takes): the same bits, also where
# b and x hold infinities and NaN
@pytest.mark.parametrize("name", ["grid_4096", "band_65", "grid3d_8000"])
def test_small_sweeps_equal_row_kernels(g, name):  # noqa: F811
    A = SMALL[name]
    b, x0 = rhs_and_x0(A, 72)
    h = g.gs2_setup(A)
    for special in (False, True):
        if special:
            b[3], x0[40], x0[50] = np.inf, np.nan, -np.inf
        out = []
        for profiled in (False, True):
            h.profile(profiled)
            x = dev(x0)
            g.gs2_apply_ex(h, dev(b), x, g.params("gs2", inner=3, direction="symmetric"))
            out.append(host(x))
        h.profile(False)
        fine = np.isfinite(out[1])
        if special:  # (the row kernels' zero slots may turn more rows into NaN)
            assert np.isfinite(out[0][fine]).all() and (~np.isfinite(out[0])).any()
        assert np.array_equal(out[0][fine], out[1][fine])
