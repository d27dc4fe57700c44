"""The Gram-Schmidt columns of the setup meet at a bounded grid barrier.  A
launch that gives up waiting costs time and nothing else: the column is taken
again with one launch per dot, and every bit of the hierarchy is the
oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_17517_gb300 as G  # noqa: E402
from synthetic import workload  # noqa: E402
from tests.test_gpu_parity import Case, _check_setup, _check_solve  # noqa: E402
from tests.test_gpu_shape_edges import General, random_matrix  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.build()
    G.lib()


def _dots(h):
    return G.airg_setup_info(h)["exact_dots"]


# the dots of a column that gave up are counted as run and run again, so a
# larger count shows that a launch did give up (no polls at all: the first
# block to arrive at any barrier does)
def test_levels_without_polls(monkeypatch):
    w = workload("grid", (160, 120))
    plain = Case(w)
    monkeypatch.setenv("AIRG_COLUMN_SPINS", "0")
    c = Case(w)
    assert _dots(c.h) > _dots(plain.h)
    _check_setup(c)
    _check_solve(c)


@pytest.mark.parametrize("n,gives_up", [(2048, False), (2049, True), (77825, True), (311297, True), (622593, False)])
def test_columns_without_polls(n, gives_up, monkeypatch):
    A = random_matrix(n, 2, n)
    plain = General(A, max_levels=1, coarse_poly_order=6)
    monkeypatch.setenv("AIRG_COLUMN_SPINS", "0")
    c = General(A, max_levels=1, coarse_poly_order=6)
    assert (_dots(c.h) > _dots(plain.h)) == gives_up
    assert np.array_equal(G.airg_export_vector(c.h, 0, 3), G.airg_export_vector(plain.h, 0, 3))
    _check_setup(c)
