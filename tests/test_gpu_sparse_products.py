"""Sparse products of the setup on general matrices: rows whose numbers of
products and distinct columns fall on every path of the product (lane groups
of 8 and 32, shared-memory tables with bitmap or counted ranks, tables in
global memory).  Every level must match the CPU oracle bit for bit: the
products are sums in a fixed order, so the tolerance is zero."""
import os
import subprocess
import sys
from types import SimpleNamespace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_17517_gb300 as G  # noqa: E402
from oracle import airg as O  # noqa: E402
from tests.test_gpu_parity import _check_setup  # noqa: E402

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OPTS = dict(max_levels=3, trunc_rtol=0.0, coarse_poly_order=4, poly_order=2, coarse_min_rows=4)


def random_matrix(n, per_row, seed):
    """Diagonally dominant, `per_row` off-diagonal entries a row anywhere."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(n, dtype=np.int64), per_row)
    cols = rng.integers(0, n, n * per_row)
    keep = rows != cols
    key = np.unique(rows[keep] * n + cols[keep])
    rows = np.concatenate([key // n, np.arange(n)])
    cols = np.concatenate([key % n, np.arange(n)])
    vals = np.concatenate([-rng.uniform(0.1, 1.0, key.size), np.full(n, 1.5 * per_row)])
    o = np.lexsort((cols, rows))
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, rows + 1, 1)
    return O.CSR(n, n, np.cumsum(rp), cols[o].astype(np.int64), vals[o])


def check(n, per_row):
    A = random_matrix(n, per_row, 31 * n + per_row)
    h = G.airg_setup(torch.tensor(A.rowptr, device="cuda"), torch.tensor(A.col.astype(np.int32), device="cuda"),
                     torch.tensor(A.val, device="cuda"), G.airg_options_default(**OPTS))
    _check_setup(SimpleNamespace(Ho=O.setup(A, O.Options(**OPTS)), h=h))


# products per row of the restrictor and RAP products: a few; around 32; a few
# hundred; thousands with more than 768 distinct columns; columns up to 70,000
# apart
@pytest.mark.parametrize("n,per_row", [(500, 1), (900, 3), (700, 14), (2600, 60), (70000, 6)])
def test_products_of_general_matrices(n, per_row):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.build()
    check(n, per_row)


def test_products_in_small_pieces():
    """The same with scratch pieces and global tables of 4096 entries."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    code = "import sys; sys.path.insert(0, %r); import tests.test_gpu_sparse_products as T; T.check(2600, 60)" % ROOT
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                       env=dict(os.environ, AIRG_SPGEMM_SLOTS="4096"))
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
