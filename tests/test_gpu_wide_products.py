"""Rows of a sparse product with more distinct columns than a shared-memory
table takes (768): what is emitted from a table in global memory, in one chunk
of 2048 columns, at its edges and in several chunks, bit for bit the oracle's.
Every row of these coarse operators is full or nearly so; `widest` is the
widest row's length, n_c where it is full."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_17517_gb300 as G  # noqa: E402
from tests.test_gpu_parity import _check_setup  # noqa: E402
from tests.test_gpu_shape_edges import General  # noqa: E402
from tests.test_gpu_sparse_products import random_matrix  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.build()
    G.lib()


@pytest.mark.parametrize("n,seed,widest", [(1166, 0, 768), (1178, 0, 769), (1592, 0, 1024), (3142, 0, 2048),
                                           (3138, 1, 2049), (6354, 5, 4124)])
def test_widest_row(n, seed, widest):
    c = General(random_matrix(n, 60, seed), max_levels=2, trunc_rtol=0.0, coarse_poly_order=4, poly_order=2,
                r_drop=0.0, a_drop=0.0)
    assert np.diff(c.Ho.A_coarse.rowptr).max() == widest
    _check_setup(c)


def test_wide_rows_cost_their_entries():
    """About a thousand full rows of some hundred thousand products each: this
    setup takes 16 ms on a GB300.  Ranking every entry against its whole
    table, sized by the products, took 2.7 s; 200 ms lies far from both."""
    A = random_matrix(1592, 200, 0)
    arrays = [torch.tensor(a, device="cuda") for a in (A.rowptr, A.col.astype(np.int32), A.val)]
    opts = G.airg_options_default(max_levels=2, trunc_rtol=0.0, coarse_poly_order=4, poly_order=2, r_drop=0.0,
                                  a_drop=0.0)
    ms = []
    for _ in range(3):
        h = G.airg_setup(*arrays, opts)
        ms.append(G.airg_setup_info(h)["setup_ms"])
        G.airg_free(h)
    assert min(ms) < 200.0, ms
