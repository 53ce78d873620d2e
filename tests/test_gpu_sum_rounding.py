"""A row's products are summed from zero and meet the row's operand (b, rhat) in one subtraction.

The operand is 2^54 here and the products are small integers (quarters of them in the prescaled
matrices), so every sum of products is exact in any order and one subtraction rounds once; a sum that
starts at the operand would round after every product.  The expected values are the same formulas in
numpy, equal bit for bit: the diagonal is 4, omega is 1, and a triangle's row has at most two entries.
"""
import numpy as np
import pytest

import oracle
from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host  # noqa: F401

pytestmark = pytest.mark.gpu


def uneven(n, seed):
    """Rows of 1 to about 60 entries of +-1 around a diagonal of 4, unsorted."""
    rng = np.random.RandomState(seed)
    rp, ci, va = [0], [], []
    for i in range(n):
        k = min(int(np.exp(2.0 + 0.8 * rng.randn())), 60)
        cols = rng.choice(n, k, replace=False)
        cols = np.append(cols[cols != i], i)
        rng.shuffle(cols)
        ci.extend(cols)
        va.extend(np.where(cols == i, 4.0, rng.choice([-1.0, 1.0], len(cols))))
        rp.append(len(ci))
    return np.array(rp, np.int64), np.array(ci, np.int32), np.array(va)


# the one-launch sweeps (n <= 4,096), stencil rows, and rows on several lanes
MATS = {"grid_60": P.poisson2d_matrix(60), "grid_130": P.poisson2d_matrix(130),
        "uneven_3000": uneven(3000, 1), "uneven_20000": uneven(20000, 2)}


class Ref:
    def __init__(self, A):
        self.A, self.n = A, len(A[0]) - 1
        self.row = np.repeat(np.arange(self.n), np.diff(A[0]))
        self.low, self.up = A[1] < self.row, A[1] > self.row

    def times(self, x, keep=None, scale=1.0):
        k = slice(None) if keep is None else keep
        return np.bincount(self.row[k], (self.A[2][k] * scale) * x[self.A[1][k]], self.n)

    def rhat(self, b, x):
        return 0.25 * (b - self.times(x))


def vectors(n):
    rng = np.random.RandomState(7)
    return 2.0 ** 54 * rng.choice([-1.0, 1.0], n), rng.choice([-3.0, -1.0, 1.0, 3.0], n)


@pytest.mark.parametrize("name", list(MATS))
def test_residual(g, name):  # noqa: F811
    m = Ref(MATS[name])
    b, x0 = vectors(m.n)
    h = g.gs2_setup(m.A)
    x = dev(x0)
    g.jr_apply(h, dev(b), x, 1, 1.0)
    assert np.array_equal(host(x), x0 + m.rhat(b, x0))


@pytest.mark.parametrize("name", ["grid_60", "grid_130"])
@pytest.mark.parametrize("inner", [1, 3])
def test_inner_sweeps(g, name, inner):  # noqa: F811
    m = Ref(MATS[name])
    b, x0 = vectors(m.n)
    h = g.gs2_setup(m.A)
    for form in ("noncompact", "compact"):
        want = x0
        for keep, other in ((m.low, m.up), (m.up, m.low)):
            rh = m.rhat(b, want) if form == "noncompact" else 0.25 * b - m.times(want, other, 0.25)
            gg = rh
            for _ in range(inner):
                gg = rh - m.times(gg, keep, 0.25)
            want = want + gg if form == "noncompact" else gg
        x = dev(x0)
        g.gs2_apply_ex(h, dev(b), x, g.params("gs2", inner=inner, direction="symmetric", form=form))
        assert np.array_equal(host(x), want), form


@pytest.mark.parametrize("name", ["grid_60", "grid_130"])
def test_exact_and_multicolour_sweeps(g, name):  # noqa: F811
    m = Ref(MATS[name])
    b, x0 = vectors(m.n)
    h = g.gs2_setup(m.A)
    rp, ci, va = m.A
    rh, gg = m.rhat(b, x0), np.zeros(m.n)
    for i in range(m.n):
        k = slice(rp[i], rp[i + 1])
        low = ci[k] < i
        gg[i] = rh[i] - (va[k][low] * 0.25 * gg[ci[k][low]]).sum()
    x = dev(x0)
    g.gs_apply(h, dev(b), x, 1, 1.0, g.FORWARD)
    assert np.array_equal(host(x), x0 + gg)
    color = oracle.coloring(m.A)
    color = np.asarray(color[0] if isinstance(color, tuple) else color)
    want = x0.copy()
    for c in range(color.max() + 1):
        s = m.times(want, m.low | m.up, 0.25)
        want = np.where(color == c, 0.25 * b - s, want)
    x = dev(x0)
    g.mtgs_apply(h, dev(b), x, 1, 1.0, g.FORWARD)
    assert np.array_equal(host(x), want)


# a row's total meets its last entry in one rounding also where the row is summed on several lanes:
# an even number of ones, then a last entry of 2^53, is exact that way; a one added to 2^53 on its own
# is lost
@pytest.mark.parametrize("n,mean", [(3000, 11), (20000, 11), (120000, 14), (900, 60)])
def test_last_entry(g, n, mean):  # noqa: F811
    rng = np.random.RandomState(n)
    count = 2 * np.clip((mean / 2.0 * np.exp(0.6 * rng.randn(n))).astype(int), 0, 60)
    rp = np.concatenate([[0], np.cumsum(count + 1)]).astype(np.int64)
    row = np.repeat(np.arange(n), count + 1)
    k = np.arange(len(row)) - rp[row]
    ci = np.where(k == count[row], row, (row + 1 + k) % n).astype(np.int32)
    va = np.where(k == count[row], 2.0 ** 53, 1.0)
    h = g.gs2_setup((rp, ci, va))
    y = dev(np.zeros(n))
    g.gs2_spmv(h, dev(np.ones(n)), y)
    assert np.array_equal(host(y), 2.0 ** 53 + count)


# ... and in the local blocks of the hybrid form
@pytest.mark.parametrize("n,mean", [(3000, 11), (20000, 11)])
def test_last_entry_hybrid(g, n, mean):  # noqa: F811
    rng = np.random.RandomState(n + 1)
    count = 2 * np.clip((mean / 2.0 * np.exp(0.6 * rng.randn(n))).astype(int), 0, 60)
    rp = np.concatenate([[0], np.cumsum(count + 1)]).astype(np.int64)
    row = np.repeat(np.arange(n), count + 1)
    k = np.arange(len(row)) - rp[row]
    half = n // 2  # two blocks, each row's columns inside its own
    lo, size = np.where(row < half, 0, half), np.where(row < half, half, n - half)
    ci = np.where(k == count[row], row, lo + (row - lo + 1 + k) % size).astype(np.int32)
    va = np.where(k == count[row], 2.0 ** 53, 1.0)
    h = g.gs2_setup((rp, ci, va))
    # one sweep without an inner one from x = 1, b = 0: x - (2^53 + count) / 2^53
    x = dev(np.ones(n))
    g.relax_apply(h, dev(np.zeros(n)), x, g.params("gs2", inner=0, parts=2))
    want = 1.0 - (2.0 ** 53 + count) * 2.0 ** -53
    assert np.array_equal(host(x), want)
