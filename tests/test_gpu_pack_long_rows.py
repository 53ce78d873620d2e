"""Packs of long rows: how a row is summed depends on neither the number of systems nor on whether
the pack's matrix fits L2 (5 systems of 24^3 nodes: 186 MB of entries on 207,360 rows; 9: 335 MB on
373,248), so a system's result is that of a pack of one, bit for bit."""
import numpy as np
import pytest

from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [5, 9])
@pytest.mark.parametrize("precision", ["none", "fp64", "fp32"])
def test_long_rows_as_in_a_pack_of_one(g, count, precision):  # noqa: F811
    pr = P.elasticity3d(24)
    n = pr.n
    pc = None if precision == "none" else g.params("gs2", inner=2, omega=0.8,
                                                   direction="symmetric", precision=precision)
    rhs = [P.uniform_pm1(200 + s, n) for s in range(count)]

    def solve(systems):
        h = g.pack_setup([pr.A] * len(systems))
        h.set_graph_mode(1)
        x = dev(np.zeros(n * len(systems)))
        infos = g.pack_gmres(h, dev(np.concatenate([rhs[s] for s in systems])), x, 20, 1e-8, 30, pc)
        assert all(i.iters == 30 for i in infos)
        return host(x).reshape(len(systems), n)

    packed = solve(range(count))
    for s in (0, count - 1):
        assert np.array_equal(packed[s], solve([s])[0]), s
