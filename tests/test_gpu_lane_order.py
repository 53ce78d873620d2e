"""Which lanes sum a row, told from the result: with x = 1 every product is exact, so the rounding of
a row's sum is that of its order of additions, and the product A x in lane slices is predicted bit for
bit -- K parts of consecutive entries, each from the first on, a butterfly over the parts, and with
more lanes than the row tiles' (A holds its diagonal) the last entry after that.
"""
import numpy as np
import pytest

import oracle
from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host, rel  # noqa: F401

pytestmark = pytest.mark.gpu


def matrix(n, count, seed):
    """count[i] entries around row i, the diagonal at a place of its own, positive values of one size
    and a diagonal of their sum's (so that additions round)."""
    rng = np.random.RandomState(seed)
    rp = np.concatenate([[0], np.cumsum(count)]).astype(np.int64)
    row = np.repeat(np.arange(n), count)
    k = np.arange(rp[-1]) - rp[row]
    ci = ((row + k - (rng.randint(0, 1 << 30, n) % count)[row]) % n).astype(np.int32)
    va = rng.uniform(0.5, 1.5, rp[-1])
    diag = ci == row
    assert diag.sum() == n
    va[diag] = 1.5 * count
    return rp, ci, va


def lane_sum(v, K, held):
    seg, s = -(-len(v) // K), []
    for l in range(K):
        lo, hi = l * seg, min((l + 1) * seg, len(v))
        if held:
            lo, hi = max(lo - 1, 0), min((l + 1) * seg - 1, len(v) - 1)
        t = 0.0
        for a in v[lo:max(hi, lo)]:
            t += a
        s.append(t)
    while len(s) > 1:
        h = len(s) // 2
        s = [s[i] + s[i + h] for i in range(h)]
    return s[0] + v[-1] if held else s[0]


def predicted(A, K, held):
    rp, _, va = A
    return np.array([lane_sum(va[rp[i]:rp[i + 1]].tolist(), K, held) for i in range(len(rp) - 1)])


def lengths(n, low, high, seed):
    return np.random.RandomState(seed).randint(low, high + 1, n)


# every number of lanes, in order (lengths within a slot of one another) and sorted in windows (spread),
# n not a multiple of a chunk or of the window, and as many rows of four lanes as need no more of
# them; (n, shortest, longest row, lanes, whether the last entry is held back)
@pytest.mark.parametrize("n,low,high,K,held", [
    (90001, 2, 12, 1, False), (3000, 5, 6, 2, True), (20001, 1, 12, 2, True),
    (2999, 13, 16, 4, True), (5003, 1, 24, 4, True), (20001, 50, 70, 4, False),
    (3001, 23, 24, 8, True), (2050, 30, 32, 8, True), (1999, 60, 64, 16, True),
    (1500, 30, 130, 16, True)])
def test_lanes(g, n, low, high, K, held):  # noqa: F811
    A = matrix(n, lengths(n, low, high, n), 3)
    h = g.gs2_setup(A, precisions=("fp32", "fp16"))
    y = dev(np.zeros(n))
    g.gs2_spmv(h, dev(np.ones(n)), y)
    one = predicted(A, 1, False)
    want = predicted(A, K, held)
    assert K == 1 or not np.array_equal(want, one)
    assert np.array_equal(host(y), want)
    # the triangles, in every precision, against the oracle (its tolerance: FP32 triangles round
    # their values to 6e-8 and FP16 ones to 5e-4, and a sweep's result adds up rows of them)
    b, x0 = P.uniform_pm1(131, n), P.uniform_pm1(132, n)
    for precision, tol in (("fp64", 1e-12), ("fp32", 1e-5), ("fp16", 1e-2)):
        x = dev(x0)
        g.gs2_apply_ex(h, dev(b), x, g.params("gs2", inner=2, direction="symmetric",
                                              precision=precision))
        ref = oracle.gs2(A, b, x0, 1, 2, 1.0, 1.0, oracle.SYMMETRIC)
        assert rel(host(x), ref) <= tol, precision


# a long-row matrix of 128 MB and more on few rows (12 bytes an entry): one lane a row
def test_few_streaming_rows(g):  # noqa: F811
    n = 100003
    A = matrix(n, lengths(n, 108, 120, 5), 7)
    assert 12 * A[0][-1] >= 128 << 20
    h = g.gs2_setup(A)
    y = dev(np.zeros(n))
    g.gs2_spmv(h, dev(np.ones(n)), y)
    rp, _, va = A
    s = np.zeros(n)
    for k in range(120):
        has = rp[:-1] + k < rp[1:]
        s[has] += va[rp[:-1][has] + k]
    assert np.array_equal(host(y), s)


# a pack of uneven systems (rows sorted in windows that reach over several systems, and systems that
# finish before others): each as in a pack of one, bit for bit
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_pack_of_uneven_systems(g, precision):  # noqa: F811
    sizes = [1700, 333, 5000, 64, 2900, 777]
    As, bs = [], []
    for s, n in enumerate(sizes):
        rp, ci, va = matrix(n, lengths(n, 1, 14, 40 + s), 50 + s)
        row = np.repeat(np.arange(n), np.diff(rp))
        va[ci == row] *= 0.6 + 0.2 * s  # from barely to strongly dominant
        As.append((rp, ci, va))
        bs.append(P.uniform_pm1(60 + s, n))
    pc = g.params("gs2", direction="symmetric", precision=precision)

    def solve(which):
        h = g.pack_setup([As[s] for s in which])
        h.set_graph_mode(1)
        x = dev(np.zeros(sum(sizes[s] for s in which)))
        infos = g.pack_gmres(h, dev(np.concatenate([bs[s] for s in which])), x, 20, 1e-10, 500, pc)
        assert all(i.ok for i in infos)
        return [i.iters for i in infos], np.split(host(x), np.cumsum([sizes[s] for s in which])[:-1])

    iters, xs = solve(range(len(sizes)))
    assert len(set(iters)) > 1
    for s in range(len(sizes)):
        it, x = solve([s])
        assert it == [iters[s]] and np.array_equal(x[0], xs[s]), s
