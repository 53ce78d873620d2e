"""Bytes of the per-kernel profile: what a row kernel reads of its matrix.  Columns count where the
layout stores them; a stencil's offset chunks store none."""
import numpy as np
import pytest

from paper_2104_01196_gb300 import problems as P
from test_gpu_parity import dev, g, host  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["stencil", "scattered"])
def test_spmv_bytes(g, name):  # noqa: F811
    A = P.poisson2d_matrix(80) if name == "stencil" else P.random_csr(6400, 5, mean_offdiag=6.0)
    n, nnz = len(A[0]) - 1, len(A[1])
    h = g.gs2_setup(A)
    assert (h.stats()["offset_frac_a"] == 1.0) == (name == "stencil")
    h.profile(True)
    y = dev(np.zeros(n))
    g.gs2_spmv(h, dev(np.ones(n)), y)
    got = h.profile_read()["spmv"]["bytes"]
    h.profile(False)
    # values and columns; x and y; at most four bytes a row each of pointers and row order
    least = (8 if name == "stencil" else 12) * nnz + 16 * n
    assert least <= got <= least + 8 * n + 64
