"""Row kernels of operators whose slices are at most two entries wide: the
layout reports the variant that runs.  One slice a warp is only run where it
is asked for, and gives the bits of two and four."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_17517_gb300 as G  # noqa: E402
from tests.test_gpu_shape_edges import banded  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.build()
    G.lib()


def _one_level(A, prec):
    return G.airg_setup(torch.tensor(A.rowptr, device="cuda"), torch.tensor(A.col.astype(np.int32), device="cuda"),
                        torch.tensor(A.val, device="cuda"),
                        G.airg_options_default(max_levels=1, coarse_poly_order=4, precision=prec))


@pytest.mark.parametrize("prec", [G.AIRG_FP64, G.AIRG_MIXED_FP32])
@pytest.mark.parametrize("n,width", [(33, 1), (1000, 1), (999, 2), (300001, 1), (300001, 2)])
def test_variant_of_narrow_slices(n, width, prec, monkeypatch):
    A = banded(n, width)
    b = torch.tensor(np.random.default_rng(n).standard_normal(n), device="cuda")
    # timed: never the variant with one slice a warp, however often
    for _ in range(6):
        h = _one_level(A, prec)
        assert G.airg_operator_layout_info(h, 0, "coarse")["r"] in (2, 4)
        G.airg_free(h)
    xs = []
    for r in (1, 2, 4):
        monkeypatch.setenv("AIRG_ROWS_PER_WARP", str(r))
        h = _one_level(A, prec)
        assert G.airg_operator_layout_info(h, 0, "coarse")["r"] == r
        x, info = G.airg_solve(h, b, rtol=1e-10)
        assert info.converged
        xs.append(x)
        G.airg_free(h)
    assert torch.equal(xs[0], xs[1]) and torch.equal(xs[0], xs[2])
